"""gd_solve of systems on either side of the size up to which every free dof is a coarse
unknown (1,024 dofs) and of the grid sizes that run as one cluster (8 and 16 CTAs).  Against
SuperLU on the same values: the solve stops at a relative residual of 1e-12, so the residual
evaluated here is held to 2e-12 and x to 1e-12 times a condition number of at most 1e5.
With the FP32 inverse as the preconditioner (error at most about 1e5 x 6e-8 = 6e-3 per
application, two applications per iteration) 1e-12 takes three iterations; ten are allowed."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

from gpu_common import smooth_state
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_03411_gb300 import build as build_mod
    build_mod.build()
    import paper_2604_03411_gb300.binding as B
    return torch, B


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("coarse", [1536, 800])
@pytest.mark.parametrize("shape", [(1, 1), (6, 5), (8, 8), (13, 11), (17, 17), (18, 17), (25, 20), (1, 1, 1), (3, 3, 2),
                                   (6, 5, 5), (6, 6, 5)])
def test_solve(env, shape, coarse, precision):
    torch, B = env
    mesh = I.uniaxial_bc_2d(I.structured_q4(*shape)) if len(shape) == 2 else I.biaxial_bc_3d(I.structured_hex8(*shape))
    rng = np.random.default_rng(6)
    prob = I.Problem("t", mesh, I.icnn_weights(rng, 3, 8), I.icnn_weights(rng, 1, 8), I.Material(), np.array([0.1]))
    h = B.gd_create(prob, B.gd_default_options(precision=B.GD_FP64 if precision == "fp64" else B.GD_MIXED,
                                               coarse=coarse))
    d, k = smooth_state(mesh, rng, u_amp=0.02, noise=0.0, phi_amp=0.1, kappa_amp=0.05)
    rowptr, colidx = B.gd_csr_pattern(h)
    vals = torch.zeros(colidx.size, dtype=torch.float64 if precision == "fp64" else torch.float32, device="cuda")
    dd = torch.tensor(d.ravel(), device="cuda")
    B.gd_assemble(h, dd, torch.tensor(k.ravel(), device="cuda"), torch.zeros_like(dd), vals, None, None,
                  B.GD_ASM_TANGENT)
    n = dd.numel()
    free = np.ones(n, bool)
    free[mesh.bc_node.astype(np.int64) * mesh.ndof + mesh.bc_comp] = False
    b = rng.standard_normal(n)
    b[~free] = 0.0
    x = torch.zeros_like(dd)
    it, rel = B.gd_solve(h, torch.tensor(b, device="cuda"), x, vals)
    assert rel <= 1e-12
    if n <= min(coarse, 1024):
        assert B.gd_coarse_info(h) == (mesh.n_nodes, int(free.sum()))
        assert it <= 10
    x = x.cpu().numpy()
    assert np.all(x[~free] == 0.0)
    K = sp.csr_matrix((vals.double().cpu().numpy(), colidx, rowptr), shape=(n, n))[free][:, free].tocsc()
    assert np.linalg.norm(K @ x[free] - b[free]) <= 2e-12 * np.linalg.norm(b)
    xr = spla.spsolve(K, b[free])
    assert np.linalg.norm(x[free] - xr) <= 1e-7 * np.linalg.norm(xr)
