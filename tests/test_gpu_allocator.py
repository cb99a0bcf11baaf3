"""The device allocator that a caller installs (vemg_set_allocator): the library asks for no alignment
beyond that of its elements."""
import contextlib
import ctypes as C

import numpy as np
import pytest
import torch

from paper_0912_1976_gb300 import inputs as I
from paper_0912_1976_gb300 import vemg as V

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _allocator(shift):
    """Blocks `shift` bytes past a 512-byte boundary."""
    held = {}

    @C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p)
    def alloc(nbytes, ctx):
        p = torch.cuda.caching_allocator_alloc(int(nbytes) + shift)
        held[p + shift] = p
        return p + shift

    @C.CFUNCTYPE(None, C.c_void_p, C.c_void_p)
    def free(ptr, ctx):
        torch.cuda.caching_allocator_delete(held.pop(ptr))

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
