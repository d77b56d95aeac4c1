"""A held load: the second step finds every point on its yield surface, and the rounding of
Phi_d decides which of them load.  The gradient has to follow the branches of the tangent that it
transposes.  One element (its sums have one order, so a state and its flags repeat to the last
bit), forty networks; the reference is the discrete adjoint with the oracle's partial derivatives,
each point put on the branch that gd_assemble reports there by a relative 1e-9 of its history.
Bar: 1e-6 of the largest component."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from gpu_common import gpu_assemble
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TIGHT = dict(newton_rtol=1e-13, newton_atol=1e-15, krylov_rtol=1e-13)


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


def reference(oracle, prob, states, flags, w):
    """dL/dtheta of sum_s w_s F_s with the given states (d, kappa) and branches of every step."""
    m, mesh = oracle.Model.from_problem(prob), prob.mesh
    n, c = mesh.n_nodes * mesh.ndof, mesh.conn[0]
    edm = oracle.element_dof_map(mesh)[0]
    bidx, _ = oracle.dirichlet(mesh)
    free = np.setdiff1d(np.arange(n), bidx)
    er = np.zeros(n)
    er[mesh.react_node.astype(np.int64) * mesh.ndof + mesh.react_comp] = 1.0
    grad, mu = np.zeros(m.n_theta), np.zeros(4)
    for s in range(len(states) - 1, -1, -1):
        d = states[s][0].ravel()
        kp = states[s - 1][1].ravel() if s else np.zeros(4)
        kp = np.where(flags[s].ravel() > 0, kp * (1.0 - 1e-9), kp * (1.0 + 1e-9))
        R, Ke, _, qi, _ = m.assemble(mesh, d, kp.reshape(1, 4))
        assert np.array_equal(qi[0, :, 5] > 0.5, flags[s].ravel() > 0)
        K = oracle.global_matrix(mesh, Ke)
        dR, dk, dRk, dkk, dkd = m.element_sens(mesh.coords[c], d.reshape(-1, mesh.ndof)[c], kp)
        dR_th, dR_kp, rhs = np.zeros((n, m.n_theta)), np.zeros((n, 4)), w[s] * (K.T @ er)
        dR_th[edm], dR_kp[edm] = dR, dRk
        np.add.at(rhs, edm, mu @ dkd)
        lam = np.zeros(n)
        lam[free] = spla.spsolve(K[free][:, free].T.tocsc(), rhs[free])
        grad += w[s] * (er @ dR_th) + mu @ dk - lam @ dR_th
        mu = w[s] * (er @ dR_kp) + mu * dkk - lam @ dR_kp
    return grad


@pytest.mark.parametrize("first", [0, 20])
def test_gradient_of_a_held_load(env, first):
    torch, B, oracle = env
    w, held = np.array([0.25, 1.0]), []
    for seed in range(first, first + 20):
        mesh = I.uniaxial_bc_2d(I.structured_q4(1, 1))
        psi, yld = I.icnn_pair(seed, 8, 8)
        prob = I.Problem("held", mesh, psi, yld, I.Material(), np.array([0.3, 0.3]))
        h = B.gd_create(prob, B.gd_default_options(**TIGHT))
        states, flags, kp = [], [], np.zeros((1, 4))
        for _ in range(2):
            B.gd_newton_step(h)
            d, kappa = B.gd_get_fields(h)[:2]
            flags.append(gpu_assemble(B, torch, h, d, kp)[3])
            kp = np.array(kappa).reshape(1, 4)
            states.append((np.array(d), kp))
        held.append(flags[1])
        g = B.gd_backward(h, w)
        ref = reference(oracle, prob, states, flags, w)
        assert np.abs(g - ref).max() <= 1e-6 * np.abs(ref).max(), (seed, flags[1].tolist())
    assert np.any(held) and not np.all(held), "points of both branches"
