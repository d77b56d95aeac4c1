"""The branch of a point close to the yield surface, from FP64 calls: networks whose second-layer
units are in the flat part of softplus and that have no skip weights, so that the normalisation by
N'(0) amplifies an absolute error of the FP32 evaluation that decides clear cases, and states
moved by up to 1e-3 from the root of every loading point.  A point's branch agrees with the
oracle's unless its trial value is within 1e-9 of the switch, and with it the results: max|gpu -
oracle| <= 1e-10 max|oracle|."""
import numpy as np
import pytest

from gpu_common import compare_assembly, gpu_assemble, oracle_assemble, smooth_state
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("dim,w", [(2, 8), (2, 24), (3, 17)])
@pytest.mark.parametrize("bias", [-6.0, -8.0, -10.0])
def test_near_the_yield_surface(bias, dim, w):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_03411_gb300 import build as build_mod
    build_mod.build()
    import oracle
    import paper_2604_03411_gb300.binding as B
    mesh = I.uniaxial_bc_2d(I.structured_q4(5, 3)) if dim == 2 else I.biaxial_bc_3d(I.structured_hex8(3, 2, 2))
    psi, yld = I.icnn_pair(5, w, w)
    W1, b1, W2, B2, b2, w3, b3 = np.split(yld.params, np.cumsum([w, w, w * w, w, w, w]))     # views
    B2[:], b3[:] = 0.0, 0.0
    b2 += bias
    prob = I.Problem("t", mesh, psi, yld, I.Material(), np.array([0.1]))
    rng = np.random.default_rng(3)
    dofs, kappa = smooth_state(mesh, rng, u_amp=0.06)
    _, _, k, qi = oracle_assemble(oracle, prob, dofs, kappa)
    kappa = np.where(qi[..., 5] > 0.5, k, kappa) * (1.0 + 1e-3 * rng.uniform(-1.0, 1.0, kappa.shape))
    h = B.gd_create(prob, B.gd_default_options())
    Rg, Kg, kg, lg = gpu_assemble(B, torch, h, dofs, kappa)
    Ro, Ko, ko, qi = oracle_assemble(oracle, prob, dofs, kappa)
    assert qi[..., 5].any() and not (qi[..., 5] > 0.5).all()
    eR, eK, ek, fl = compare_assembly(Rg, Kg, kg, lg, Ro, Ko, ko, qi, TOL)
    assert fl and eR < TOL and eK < TOL and ek < TOL, (eR, eK, ek, fl)
