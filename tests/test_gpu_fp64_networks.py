"""FP64 element kernel at the edges of its network and CTA mappings: widths that are no
multiple of the lanes per point or of the output chunk, rows of very different scale
(each has its own fixed-point exponent), pre-activations beyond the range of the softplus
polynomials, meshes that change the CTA width.  Bar as in test_gpu_assemble.py: the results
are FP64 sums, so max|gpu - oracle| <= 1e-10 max|oracle|."""
import numpy as np
import pytest

from gpu_common import compare_assembly, gpu_assemble, oracle_assemble, smooth_state
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-10


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


def make(dim, shape, w_psi, w_y, seed=7, scale=None):
    mesh = I.uniaxial_bc_2d(I.structured_q4(*shape)) if dim == 2 else I.biaxial_bc_3d(I.structured_hex8(*shape))
    rng = np.random.default_rng(seed)
    psi, yld = I.icnn_weights(rng, 3, w_psi), I.icnn_weights(rng, 1, w_y)
    if scale is not None:
        for net in (psi, yld):
            w, n = net.width, net.n_in
            W2 = net.params[w * n + w:w * n + w + w * w].reshape(w, w)
            W2 *= (scale ** rng.uniform(-1.0, 1.0, w))[:, None]
    return I.Problem("t", mesh, psi, yld, I.Material(), np.array([0.1]))


def check(env, prob, u_amp=0.06, phi_amp=0.3, smooth=False):
    torch, B, oracle = env
    rng = np.random.default_rng(3)
    if smooth:          # nodal noise scaled by the element size: fine meshes stay far from inversion
        dofs, kappa = smooth_state(prob.mesh, rng, u_amp=u_amp, phi_amp=phi_amp, kappa_amp=0.3)
    else:
        dofs, kappa = I.random_state(prob.mesh, rng, u_amp=u_amp, phi_amp=phi_amp, kappa_amp=0.3)
    h = B.gd_create(prob, B.gd_default_options())
    Rg, Kg, kg, lg = gpu_assemble(B, torch, h, dofs, kappa)
    Ro, Ko, ko, qi = oracle_assemble(oracle, prob, dofs, kappa)
    eR, eK, ek, fl = compare_assembly(Rg, Kg, kg, lg, Ro, Ko, ko, qi, TOL)
    assert eR < TOL and eK < TOL and ek < TOL and fl, (eR, eK, ek, fl)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("w_psi,w_y", [(1, 2), (5, 3), (17, 30), (33, 15), (63, 61)])
def test_widths(env, dim, w_psi, w_y):
    check(env, make(dim, (5, 3) if dim == 2 else (3, 2, 2), w_psi, w_y))


@pytest.mark.parametrize("dim", [2, 3])
def test_rows_of_different_scale(env, dim):
    check(env, make(dim, (5, 3) if dim == 2 else (3, 2, 2), 24, 20, scale=30.0))


def test_large_pre_activations(env):
    """Strains of order 1 and weights of order 10: layer-1 pre-activations past 64."""
    prob = make(2, (6, 4), 16, 8)
    prob.psi.params[:48] *= 120.0
    check(env, prob, u_amp=0.25)


@pytest.mark.parametrize("shape", [(1, 1), (2, 1), (13, 47), (31, 41), (37, 67), (70, 71)])
def test_cta_widths_q4(env, shape):
    """8, 16 and 32 points per CTA, full and ragged, one and several batches per CTA."""
    check(env, make(2, shape, 8, 8), smooth=True)


@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 6, 7), (7, 9, 8), (11, 10, 11)])
def test_cta_widths_hex8(env, shape):
    check(env, make(3, shape, 8, 8), smooth=True)
