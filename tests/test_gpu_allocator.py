"""The device allocator that a caller installs (vemg_set_allocator): the library asks for no alignment
beyond that of its elements, and does with what its results and their inputs take."""
import contextlib
import ctypes as C

import numpy as np
import pytest
import torch

from paper_0912_1976_gb300 import inputs as I
from paper_0912_1976_gb300 import vemg as V

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _allocator(shift=0, budget=1 << 40, largest=1 << 40):
    """Blocks `shift` bytes past a 512-byte boundary, `budget` bytes of them at a time, none over `largest`."""
    held = {}

    @C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p)
    def alloc(nbytes, ctx):
        if sum(b for _, b in held.values()) + nbytes > budget or nbytes > largest:
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes) + shift)
        held[p + shift] = p, nbytes
        return p + shift

    @C.CFUNCTYPE(None, C.c_void_p, C.c_void_p)
    def free(ptr, ctx):
        torch.cuda.caching_allocator_delete(held.pop(ptr)[0])

    L = V.lib()
    assert L.vemg_set_allocator(C.cast(alloc, C.c_void_p), C.cast(free, C.c_void_p), None) == V.VEMG_OK
    try:
        yield held
    finally:
        L.vemg_set_allocator(None, None, None)
        assert not held   # everything allocated under it was released before it went


def _case(nx, ny, nz):
    m = I.make_mesh(nx, ny, nz, I.depth_sines(1e-2), z_jitter=0.3, seed=81)
    return m, V.Mesh.from_inputs(m)


@pytest.mark.parametrize("shift", [8, 16])
@pytest.mark.parametrize("shape", [(5, 4, 3), (21, 19, 9)])
def test_blocks_aligned_to_their_elements_only(shape, shift):
    """Assembly, load, solves and batches under such an allocator: the same bits as under cudaMalloc."""
    m, vm = _case(*shape)
    f = torch.from_numpy(I.normal_loads(m.n, 82)).cuda()

    def results():
        A = V.vemg_assemble(vm)
        out = [t.clone() for t in A.tensors()] + [V.vemg_load(vm, f)]
        for prec in (V.VEMG_PREC_FP64, V.VEMG_PREC_BF16):
            h = V.vemg_setup(A, vm, V.vemg_default_options(precision=prec))
            out.append(V.vemg_solve(h, f, rtol=1e-9)[0])
            V.vemg_batch_set_tuning(h, 4, (4, 4, 4), (2, 2, 2))   # no shapes chosen by time
            out.append(V.vemg_solve_batch(h, torch.stack([f, 2 * f, -f]), rtol=1e-9)[0])
            h.destroy()
        A.free()
        torch.cuda.synchronize()
        return [t.cpu().numpy() for t in out]

    want = results()
    with _allocator(shift):
        got = results()
    assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("spare", [1 << 17, 1 << 21])   # bytes for all temporary arrays
def test_assembly_within_its_result(spare):
    """What assembly needs beside the mesh, its incidence lists and the matrix fits in little memory; the
    matrix has the same bits then. Less than the matrix itself is refused, and leaves nothing behind."""
    m, vm = _case(40, 38, 11)
    A = V.vemg_assemble(vm)
    want = [t.cpu().numpy() for t in A.tensors()]
    A.free()
    ne, nnz = vm.tets.shape[0], len(want[1])
    result = 12 * nnz + 4 * (m.n + 1)
    # the mesh starts in a block of at most 1 MiB; rows' lengths, counts and their scans, 24 bytes a node
    need = 24 * m.n + 32 * ne + 4 * (m.n + 1) + (1 << 20) + 24 * m.n
    with _allocator(budget=need + result + spare):
        A = V.vemg_assemble(vm)
        got = [t.cpu().numpy() for t in A.tensors()]
        A.free()
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
    with _allocator(budget=result // 2), pytest.raises(V.VemgError) as e:
        V.vemg_assemble(vm)
    assert e.value.code == V.VEMG_ENOMEM


def test_no_block_larger_than_an_array():
    """The library allocates many arrays at once where it can; an allocator that gives no block larger than
    the largest array serves it too."""
    m, vm = _case(5, 4, 3)
    b = torch.from_numpy(I.normal_loads(m.n, 83)).cuda()

    def solutions():
        A = V.vemg_assemble(vm)
        h = V.vemg_setup(A, vm, V.vemg_default_options())
        V.vemg_batch_set_tuning(h, 4, (4, 4, 4), (2, 2, 2))
        out = [V.vemg_solve(h, b, rtol=1e-9)[0], V.vemg_solve_batch(h, torch.stack([b, -b, 2 * b]), rtol=1e-9)[0]]
        h.destroy()
        A.free()
        return out

    want = solutions()
    # 120 nodes: nothing that grows with the mesh is over 120 x 120 doubles, and partial sums of at most
    # 608 blocks, 8 reductions and 5 sums take 195 KB
    with _allocator(largest=1 << 18):
        got = solutions()
    assert all(torch.equal(x, y) for x, y in zip(got, want))


@pytest.mark.parametrize("engine", [False, True])
def test_refused_batch_leaves_nothing_behind(engine):
    """A batch or an engine for which the memory does not suffice: VEMG_ENOMEM, and what it had allocated
    until then is given back; the hierarchy goes on."""
    m, vm = _case(21, 19, 9)
    b = torch.from_numpy(I.normal_loads(m.n, 84)).cuda()
    A = V.vemg_assemble(vm)
    h = V.vemg_setup(A, vm, V.vemg_default_options())
    want = V.vemg_solve(h, b, rtol=1e-9)[0]
    # 16 columns: the first three of the six vectors fit
    with _allocator(budget=4 * 16 * 8 * m.n) as held, pytest.raises(V.VemgError) as e:
        if engine:
            V.Engine(h, 16)
        else:
            V.vemg_solve_batch(h, b.repeat(16, 1), rtol=1e-9)
    assert e.value.code == V.VEMG_ENOMEM and not held
    assert torch.equal(V.vemg_solve(h, b, rtol=1e-9)[0], want)
    assert torch.isfinite(V.vemg_solve_batch(h, b.repeat(16, 1), rtol=1e-9)[0]).all()
