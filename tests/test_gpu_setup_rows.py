"""The setup's kernels with a warp per row at the row lengths where they change form: sorts of 256 and of
more entries, products of 512 and of more distinct columns. A dense symmetric matrix over a mesh of one
layer has rows of any wanted length: every row of A has 2 t entries and every row of A E~ has t, t nodes
on top. Only the setup runs; no cycle."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_0912_1976_gb300 import inputs as I
from paper_0912_1976_gb300 import vemg as V

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kx, ky", [(15, 7), (42, 2), (31, 15), (26, 18)])   # 128, 129, 512, 513 nodes on top
def test_dense_rows(kx, ky):
    m = I.make_mesh(kx, ky, 1, I.depth_sines(1e-1), z_jitter=0.3, seed=71)
    vm = V.Mesh.from_inputs(m)
    n = vm.n
    w = np.random.default_rng(6).uniform(0.5, 1.5, (n, n))
    w = np.triu(w, 1) + np.triu(w, 1).T
    dense = np.diag(w.sum(1)) - w
    # columns in descending order: the permuted rows have to be sorted
    rp = torch.arange(0, n * n + 1, n, dtype=torch.int32, device="cuda")
    ci = torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda").repeat(n)
    v = torch.from_numpy(np.ascontiguousarray(dense[:, ::-1]).ravel()).cuda()
    A = SimpleNamespace(n=n, c=V.vemg_csr(n, n * n, rp.data_ptr(), ci.data_ptr(), v.data_ptr()))
    torch.cuda.synchronize()
    h = V.vemg_setup(A, vm, V.vemg_default_options())
    order = np.asarray(V.vemg_get_int(h, "new2old"))
    want = dense[np.ix_(order, order)]
    got = V.vemg_get_csr(h, "A").tocsr()
    assert got.has_sorted_indices and np.array_equal(got.toarray(), want)
    # a dense level: every row has a colour of its own
    assert np.array_equal(np.sort(V.vemg_get_int(h, "lev.colour", 1, 0)), np.arange(V.vemg_get_size(h, "lev.n", 1, 0)))
    E = V.vemg_get_csr(h, "E").toarray()
    Ac = V.vemg_get_csr(h, "Ac").tocsr()
    assert np.array_equal(np.diff(Ac.indptr), np.full(E.shape[1], E.shape[1]))
    # each side: two products with at most n terms per sum
    bound = 4 * (n + 2) * 2.0 ** -53 * (abs(E).T @ abs(want) @ abs(E))
    assert (abs(Ac.toarray() - E.T @ want @ E) <= bound).all()


def _assemble(xyz, tets):
    return V.vemg_assemble(V.Mesh(xyz, tets, np.zeros(len(xyz), np.uint8), np.zeros((1, 3), np.int32))).to_host()


@pytest.mark.parametrize("n, ne", [(33, 60), (48, 600)])   # a block's rows fit shared memory; they do not
def test_assembly_adds_elements_in_order(n, ne):
    """The matrix of arbitrary tetrahedra, bit for bit the sum of one-element matrices in element order."""
    rng = np.random.default_rng(n)
    xyz = rng.uniform(size=(n, 3))
    tets = np.array([rng.permutation(n)[:4] for _ in range(ne)], np.int32)
    tets[: (n + 3) // 4] = np.resize(rng.permutation(n), (n + 3) // 4 * 4).reshape(-1, 4)   # no node left out
    d = xyz[tets]
    flip = np.linalg.det(d[:, 1:] - d[:, :1]) < 0
    tets[flip, 2:] = tets[flip, 3:1:-1]
    want, seen = np.zeros((n, n)), np.zeros((n, n), bool)
    for t in tets:
        want[np.ix_(t, t)] += _assemble(xyz[t], np.arange(4, dtype=np.int32)[None]).toarray()
        seen[np.ix_(t, t)] = True
    got = _assemble(xyz, tets)
    assert (got.nnz > 1024) == (ne > 100) and got.nnz == seen.sum()
    assert np.array_equal(got.toarray(), want)


def test_setups_side_by_side():
    """Colourings run beside the coarsening on streams of their own: two threads that set up different
    problems at once, and a setup that fails while its colourings run, leave every colour as it is."""
    from concurrent.futures import ThreadPoolExecutor

    meshes = [V.Mesh.from_inputs(I.make_mesh(k, k + 3, 11, I.depth_sines(1e-2), z_jitter=0.3, seed=k)) for k in (40, 57)]

    def colours(vm):
        with torch.cuda.stream(torch.cuda.Stream()):
            h = V.vemg_setup(V.vemg_assemble(vm), vm, V.vemg_default_options())
            return [V.vemg_get_int(h, "lev.colour", c, l) for c in (0, 1) for l in range(V.vemg_get_size(h, "nlev", c))]

    alone = [colours(vm) for vm in meshes]
    bad = V.Mesh.from_inputs(I.make_mesh(40, 43, 11, I.depth_sines(1e-2), z_jitter=0.3, seed=40))
    bad.top_tris[0] = bad.n   # out of range: found after the colouring of A_bar began
    with ThreadPoolExecutor(2) as pool:
        for _ in range(3):
            both = list(pool.map(colours, meshes))
            with pytest.raises(V.VemgError):
                V.vemg_setup(V.vemg_assemble(bad), bad, V.vemg_default_options())
            for got, want in zip(both, alone):
                assert len(got) == len(want) and all(np.array_equal(a, b) for a, b in zip(got, want))
