"""FP64 element kernel on networks that a calibration may end with, whose fixed-point sums would lose
bits: second-layer units far in the flat part of softplus (without skip weights, so that the
normalisation by N'(0) amplifies what is left of them), first-layer units over many orders of
magnitude whose weights undo that, and states close to the yield surface.  The results are FP64 sums: max|gpu - oracle| <= 1e-10
max|oracle|, and a point's branch agrees unless its trial value is within 1e-9 of the switch."""
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


def parts(net):
    """Views of the packed parameters: W1, b1, W2, A2, b2, w3, a3."""
    w, n = net.width, net.n_in
    cut = np.cumsum([w * n, w, w * w, w * n, w, w])
    W1, b1, W2, A2, b2, w3, a3 = np.split(net.params, cut)
    return W1.reshape(w, n), b1, W2.reshape(w, w), A2.reshape(w, n), b2, w3, a3


def problem(dim, w, **mat):
    mesh = I.uniaxial_bc_2d(I.structured_q4(5, 3)) if dim == 2 else I.biaxial_bc_3d(I.structured_hex8(3, 2, 2))
    psi, yld = I.icnn_pair(5, w, w)
    return I.Problem("t", mesh, psi, yld, I.Material(**mat), np.array([0.1]))


def check(env, prob, near_yield=False):
    torch, B, oracle = env
    rng = np.random.default_rng(3)
    dofs, kappa = smooth_state(prob.mesh, rng, u_amp=0.06)
    if near_yield:      # the root of every loading point, moved by up to 1e-3
        _, _, k, qi = oracle_assemble(oracle, prob, dofs, kappa)
        kappa = np.where(qi[..., 5] > 0.5, k, kappa) * (1.0 + 1e-3 * rng.uniform(-1.0, 1.0, kappa.shape))
    h = B.gd_create(prob, B.gd_default_options())
    Rg, Kg, kg, lg = gpu_assemble(B, torch, h, dofs, kappa)
    Ro, Ko, ko, qi = oracle_assemble(oracle, prob, dofs, kappa)
    assert np.isfinite(Ro).all() and qi[..., 5].any() and not (qi[..., 5] > 0.5).all()
    eR, eK, ek, fl = compare_assembly(Rg, Kg, kg, lg, Ro, Ko, ko, qi, TOL)
    assert eR < TOL and eK < TOL and ek < TOL and fl, (eR, eK, ek, fl)


def without_skips(net, bias):
    _, _, _, A2, b2, _, a3 = parts(net)
    A2[:] = 0.0
    a3[:] = 0.0
    b2 += bias


@pytest.mark.parametrize("near_yield", [False, True])
@pytest.mark.parametrize("dim,w", [(2, 8), (2, 24), (3, 17)])
@pytest.mark.parametrize("bias", [-8.0, -10.0, -15.0, -20.0, -30.0, -60.0])
def test_flat_second_layer(env, bias, dim, w, near_yield):
    prob = problem(dim, w, mu_e=float(np.exp(-bias)))
    without_skips(prob.psi, bias)
    without_skips(prob.yld, bias)
    check(env, prob, near_yield)


@pytest.mark.parametrize("dim,w", [(2, 9), (2, 32), (3, 24)])
@pytest.mark.parametrize("spread", [8.0, 16.0])
def test_small_weights_on_large_activations(env, spread, dim, w):
    """b1 down to -spread, W2's columns scaled by exp(-b1 - spread) or less: every unit counts alike."""
    prob = problem(dim, w)
    for net in (prob.psi, prob.yld):
        W1, b1, W2, A2, b2, w3, a3 = parts(net)
        d = -np.linspace(0.0, spread, w)
        b1 += d
        W2 *= 10.0 * np.exp(-d)[None, :] / np.exp(spread / 2)
        A2[:] = 0.0
        a3[:] = 0.0
    check(env, prob)


def test_batch_of_ordinary_and_flat_networks(env):
    """Every specimen of a batch takes its own networks' form: a point's history and branch are those of
    the specimen alone, to the last bit."""
    torch, B, _ = env
    probs, states = [], []
    for i, (bias, w) in enumerate([(0.0, 8), (-20.0, 17), (-4.0, 24), (0.0, 32), (-60.0, 9)]):
        prob = problem(2, w)
        if bias:
            without_skips(prob.psi, bias)
            without_skips(prob.yld, bias)
        probs.append(prob)
        states.append(smooth_state(prob.mesh, np.random.default_rng(i), u_amp=0.06))
    alone = [gpu_assemble(B, torch, B.gd_create(p, B.gd_default_options()), d, k)[2:] for p, (d, k) in zip(probs, states)]
    h = B.gd_create_batch(probs, B.gd_default_options())
    _, _, kg, lg = gpu_assemble(B, torch, h, np.concatenate([d for d, _ in states]), np.concatenate([k for _, k in states]))
    assert np.array_equal(kg, np.concatenate([a[0] for a in alone]))
    assert np.array_equal(lg, np.concatenate([a[1] for a in alone]))
