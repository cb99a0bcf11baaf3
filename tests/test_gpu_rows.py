"""The row kernels of the V-cycle at the shapes where they can go wrong: rows split over 1 to 32 lanes,
slices with few rows, levels of a handful of rows, and rows longer than a lane's first chunk. One FP64
cycle of a chain against the same cycle written with scipy on the operators that the library exports.
Both sides round the same products and sums in different orders: 1e-11 relative, the bound of the parity
tests for one cycle."""
import numpy as np
import pytest
import torch

from paper_0912_1976_gb300 import inputs as I
from paper_0912_1976_gb300 import vemg as V

pytestmark = pytest.mark.gpu

CASES = {
    # thousands of rows per colour on the finest level, tens below: 1 to 4 lanes a row
    "layers": (lambda: I.make_mesh(90, 83, 14, I.depth_sines(1e-2), z_jitter=0.3, seed=61), {}),
    # coarse rows of 30 and more entries: up to 16 lanes a row
    "unstructured": (lambda: I.make_mesh(34, 31, 13, I.depth_sines(1e-1), z_jitter=0.3, xy_jitter=0.2, seed=62), {}),
    # coarsened down to a few rows
    "deep": (lambda: I.make_mesh(9, 7, 5, I.depth_sines(1e-2), z_jitter=0.3, seed=63), dict(coarse_max=3, max_levels=16)),
    # one column of hexes: slices that are never full
    "column": (lambda: I.make_mesh(1, 1, 37, I.depth_sines(1e-1), z_jitter=0.3, seed=64), dict(coarse_max=5)),
}


def _cycle(h, chain, l, b):
    nlev = V.vemg_get_size(h, "nlev", chain)
    A = V.vemg_get_csr(h, "lev.A", chain, l).tocsr()
    if l == nlev - 1 and V.vemg_get_size(h, "direct", chain):
        return np.linalg.solve(A.toarray(), b)
    colour = V.vemg_get_int(h, "lev.colour", chain, l)
    d = A.diagonal()
    rows = [np.nonzero(colour == c)[0] for c in range(colour.max() + 1)]

    def sweep(x, order):
        for c in order:
            i = rows[c]
            x[i] += (b[i] - A[i] @ x) / d[i]

    x = np.zeros_like(b)
    sweep(x, range(len(rows)))
    if l < nlev - 1:
        P = V.vemg_get_csr(h, "lev.P", chain, l)
        x += P @ _cycle(h, chain, l + 1, P.T @ (b - A @ x))
    sweep(x, reversed(range(len(rows))))
    return x


@pytest.mark.parametrize("name", list(CASES))
def test_cycle_matches_the_exported_operators(name):
    make, opts = CASES[name]
    m = make()
    vm = V.Mesh.from_inputs(m)
    h = V.vemg_setup(V.vemg_assemble(vm), vm, V.vemg_default_options(bc=V.VEMG_DIRICHLET_TOP, **opts))
    b = np.random.default_rng(5).standard_normal(V.vemg_get_size(h, "lev.n", 1, 0))
    x = V.vemg_vcycle(h, 1, torch.from_numpy(b).cuda()).cpu().numpy()
    ref = _cycle(h, 1, 0, b)
    assert np.linalg.norm(x - ref) <= 1e-11 * np.linalg.norm(ref)


@pytest.mark.parametrize("precision", [V.VEMG_PREC_FP32, V.VEMG_PREC_BF16])
@pytest.mark.parametrize("power", [-70, 70])
def test_solution_scales_exactly_with_the_right_hand_side(precision, power):
    """FP32 cycles convert between FP64 and FP32 vectors. A right-hand side scaled by a power of two keeps
    every operation inside the normal range, so x scales by it bit for bit."""
    m = I.make_mesh(24, 20, 12, I.depth_sines(1e-2), z_jitter=0.3, seed=65)
    vm = V.Mesh.from_inputs(m)
    h = V.vemg_setup(V.vemg_assemble(vm), vm, V.vemg_default_options(precision=precision))
    b = torch.from_numpy(I.normal_loads(m.n, 66)).cuda()
    x, i1 = V.vemg_solve(h, b, rtol=1e-8)
    y, i2 = V.vemg_solve(h, b * 2.0 ** power, rtol=1e-8)
    assert i1["status"] == i2["status"] == "OK" and i1["iters"] == i2["iters"]
    assert torch.equal(y, x * 2.0 ** power)
    Y, infos = V.vemg_solve_batch(h, torch.stack([b, b * 2.0 ** power]), rtol=1e-8)
    assert infos[0]["status"] == infos[1]["status"] == "OK" and torch.equal(Y[1], Y[0] * 2.0 ** power)


@pytest.mark.parametrize("bc", [V.VEMG_NEUMANN, V.VEMG_DIRICHLET_TOP])
@pytest.mark.parametrize("precision", [V.VEMG_PREC_FP64, V.VEMG_PREC_BF16])
def test_single_steps_repeat_and_share_the_solve_vectors(bc, precision):
    """vemg_precond runs from a graph from its second call on, and the single steps work in the solve's
    vectors: the same bits call after call, in place, between solves and beside other steps."""
    m = I.make_mesh(23, 19, 11, I.depth_sines(1e-2), z_jitter=0.3, seed=67)
    vm = V.Mesh.from_inputs(m)
    h = V.vemg_setup(V.vemg_assemble(vm), vm, V.vemg_default_options(bc=bc, precision=precision))
    n = V.vemg_get_size(h, "n") - (V.vemg_get_size(h, "mtop") if bc == V.VEMG_DIRICHLET_TOP else 0)
    r = torch.from_numpy(np.random.default_rng(8).standard_normal(n)).cuda()
    b = torch.from_numpy(I.normal_loads(m.n, 68)).cuda()
    z, y, v = V.vemg_precond(h, r), V.vemg_spmv(h, r), None
    x, _ = V.vemg_solve(h, b, rtol=1e-8)
    for _ in range(3):
        assert torch.equal(V.vemg_precond(h, r), z) and torch.equal(V.vemg_spmv(h, r), y)
        w = V.vemg_vcycle(h, 1, r[:V.vemg_get_size(h, "lev.n", 1, 0)].contiguous())
        assert v is None or torch.equal(v, w)
        v = w
        assert torch.equal(V.vemg_solve(h, b, rtol=1e-8)[0], x)
    for step, want in ((V.vemg_precond, z), (V.vemg_spmv, y)):
        t = r.clone()
        assert torch.equal(step(h, t, t), want)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    assert torch.equal(V.vemg_precond(h, r, stream=side), z)
