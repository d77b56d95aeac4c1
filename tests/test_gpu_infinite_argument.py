"""The argument q = psi_e + qcoef (phi - kappa) / f_d(kappa) of the yield network is infinite where
f_d underflows (kappa far above its scale 1 / eta_d).  At q = +inf the trial value is +inf: the
point loads, no finite kappa solves it and nothing finite may come out of it (a Newton step then
reports GD_ERR_NAN).  At q = -inf the point is elastic, as for the oracle.  The points beside it
in the same warp are untouched: their kappa agrees with the oracle's to 1e-10."""
import numpy as np
import pytest

from gpu_common import gpu_assemble, oracle_assemble, smooth_state
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_03411_gb300 import build as build_mod
    build_mod.build()
    import oracle
    import paper_2604_03411_gb300.binding as B
    return torch, B, oracle


def setup(w, elem, kappa_n, phi):
    mesh = I.uniaxial_bc_2d(I.structured_q4(3, 2))
    psi, yld = I.icnn_pair(5, w, w)
    prob = I.Problem("far", mesh, psi, yld, I.Material(), np.array([0.1]))
    dofs, kappa = smooth_state(mesh, np.random.default_rng(3), u_amp=0.06)
    kappa[elem] = kappa_n
    dofs[mesh.conn[elem], 2] = phi
    return prob, dofs, kappa


@pytest.mark.parametrize("w", [3, 8, 16, 64])
def test_fp64_above(env, w):
    torch, B, _ = env
    prob, dofs, kappa = setup(w, list(range(6)), 800.0, 900.0)
    h = B.gd_create(prob, B.gd_default_options())
    R, K, k, l = gpu_assemble(B, torch, h, dofs, kappa)
    assert l.all() and not np.isfinite(k).any() and not np.isfinite(R).all()


@pytest.mark.parametrize("w", [3, 8, 16, 64])
@pytest.mark.parametrize("points", ["one element", "some points", "all"])
def test_fp64_below(env, w, points):
    torch, B, oracle = env
    elem = {"one element": [2], "some points": [0, 5], "all": list(range(6))}[points]
    prob, dofs, kappa = setup(w, elem, 800.0, 0.1)
    if points == "some points":
        kappa[elem, 1:3] = 0.2
    far = kappa > 700.0
    h = B.gd_create(prob, B.gd_default_options())
    R, K, k, l = gpu_assemble(B, torch, h, dofs, kappa)
    _, _, ko, qi = oracle_assemble(oracle, prob, dofs, kappa)
    assert not l[far].any() and np.array_equal(k[far], kappa[far])
    near = ~far
    assert np.array_equal(l[near] > 0, qi[..., 5][near] > 0.5)
    if near.any():
        assert np.abs(k[near] - ko[near]).max() <= 1e-10 * np.abs(ko[near]).max()
