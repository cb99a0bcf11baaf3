"""The dense coarsest solve at the edges of its 32 x 32 tiles: chains of a single level, whose V-cycle is
the explicit inverse G of D, against numpy: D = A, and on the singular surface chain D = A + sigma 1 1^T,
sigma = tr(A) / n^2, with G projected on the complement of the constants on both sides. An inverse from a Cholesky factor has a relative error of order n u cond(D), u = 2^-53."""
import numpy as np
import pytest
import torch

from paper_0912_1976_gb300 import inputs as I
from paper_0912_1976_gb300 import vemg as V

pytestmark = pytest.mark.gpu

# rows of A_bar = (nx + 1)(ny + 1) nz, of the surface operator (nx + 1)(ny + 1)
MESHES = [(1, 1, 1), (3, 7, 1), (2, 10, 1), (3, 3, 4), (4, 12, 1), (3, 7, 31), (10, 30, 3), (31, 31, 1)]


@pytest.mark.parametrize("nx,ny,nz", MESHES)
def test_one_level_chains_apply_the_inverse(nx, ny, nz):
    m = I.make_mesh(nx, ny, nz, I.depth_sines(1e-2), z_jitter=0.3, seed=51)
    vm = V.Mesh.from_inputs(m)
    h = V.vemg_setup(V.vemg_assemble(vm), vm, V.vemg_default_options())
    for chain in (0, 1):
        n = V.vemg_get_size(h, "lev.n", chain, 0)
        assert V.vemg_get_size(h, "nlev", chain) == 1 and V.vemg_get_size(h, "direct", chain) == 1
        assert n == (nx + 1) * (ny + 1) * (nz if chain else 1)
        A = V.vemg_get_csr(h, "lev.A", chain, 0).toarray()
        b = np.random.default_rng(n).standard_normal(n)
        D, c = (A + np.trace(A) / n ** 2, b - b.mean()) if chain == 0 else (A, b)
        w, Q = np.linalg.eigh(D)
        x = Q @ ((Q.T @ c) / w)
        if chain == 0:
            x -= x.mean()
        v = V.vemg_vcycle(h, chain, torch.from_numpy(b).cuda()).cpu().numpy()
        bound = 8.0 * n * 2.0 ** -53 * (w[-1] / w[0]) * np.linalg.norm(b) / w[0]
        assert np.linalg.norm(v - x) <= bound, (n, np.linalg.norm(v - x), bound)
