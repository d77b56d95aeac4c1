"""The adjoint's element kernel gives a batch of 32 points to 32, 16, ... or one warp, by
the mesh size, ragged in the batches.  Few elements: gd_backward against the oracle's FP64
discrete adjoint on every weight, bar 1e-8 of the largest component (both are exact
derivatives of converged paths).  Up to 21,140 elements: a directional derivative against
fourth-order central differences of the path, bar 1e-5."""
import numpy as np
import pytest

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
    return B, oracle


def tight(B):
    return B.gd_default_options(newton_rtol=1e-12, newton_atol=1e-14, krylov_rtol=1e-13, krylov_max=50000)


@pytest.mark.parametrize("shape", [(1, 1), (5, 3), (2, 2, 1)])
def test_every_weight_of_small_meshes(env, shape):
    B, oracle = env
    mesh = I.uniaxial_bc_2d(I.structured_q4(*shape)) if len(shape) == 2 else I.uniaxial_bc_3d(I.structured_hex8(*shape))
    psi, yld = I.icnn_pair(11, 8, 8)
    load = np.array([0.25, 0.4])
    prob = I.Problem("shares", mesh, psi, yld, I.Material(beta_d=10.0, c_d=10.0 * 0.1 ** 2), load)
    w = np.array([1.0, -0.5])
    go, reac_o = oracle.adjoint_gradient(oracle.Model.from_problem(prob), mesh, load, w, rtol=1e-13, atol=1e-15)
    h = B.gd_create(prob, tight(B))
    reac, rep = B.gd_run_load_path(h)
    assert rep.step_cuts == 0
    g = B.gd_backward(h, w)
    assert np.abs(g - go).max() <= 1e-8 * np.abs(go).max()


@pytest.mark.parametrize("shape", [(34, 31), (53, 47), (71, 60), (105, 97), (151, 140)])
def test_direction_on_larger_meshes(env, shape):
    B, _ = env
    mesh = I.uniaxial_bc_2d(I.structured_q4(*shape, shape[0] / shape[1], 1.0))
    psi, yld = I.icnn_pair(4, 8, 8)
    prob = I.Problem("shares", mesh, psi, yld, I.Material(beta_d=10.0, c_d=10.0), np.array([0.05, 0.1]))
    theta = np.concatenate([psi.params, yld.params])
    w = np.array([1.0, -0.5])
    h = B.gd_create(prob, tight(B))

    def loss(th):
        B.gd_set_params(h, th[:psi.params.size], th[psi.params.size:])
        B.gd_set_state(h, np.zeros((mesh.n_nodes, 3)), np.zeros((mesh.n_elems, 4)), 0)
        reac, rep = B.gd_run_load_path(h)
        assert rep.step_cuts == 0
        return float(w @ reac)

    v = np.random.default_rng(3).standard_normal(theta.size) * np.maximum(np.abs(theta), 0.1)
    s = 1e-3
    fd = (8.0 * (loss(theta + s * v) - loss(theta - s * v)) - (loss(theta + 2 * s * v) - loss(theta - 2 * s * v))) / (12 * s)
    loss(theta)
    g = B.gd_backward(h, w)
    assert abs(g @ v - fd) <= 1e-5 * abs(fd)
