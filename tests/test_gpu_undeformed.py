"""A body without strain, damage or history is elastic: psi_e = 0, G(0) = 0 and so Phi_d(0) = 0,
whatever the networks (N(0), N_k(0) and their derivatives are the normalising constants).  Over
fifty networks per case: no loading flag, the history unchanged to the last bit, no residual,
and the tangent of the FP64 oracle (1e-10 of its largest entry; the penalty block is beta_d
there, and beta_d (1 - dkappa/dphi) on a loading point)."""
import numpy as np
import pytest

from gpu_common import gpu_assemble, oracle_assemble
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu
NETS = 50


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


def problem(dim, seed, w, energy):
    mesh = I.uniaxial_bc_2d(I.structured_q4(3, 2)) if dim == 2 else I.uniaxial_bc_3d(I.structured_hex8(1, 2, 1))
    psi, yld = I.icnn_pair(seed, *w)
    return I.Problem("zero", mesh, psi, yld, I.Material(energy=energy), np.array([0.1]))


@pytest.mark.parametrize("dim,w,energy", [(2, (8, 8), I.ENERGY_ICNN_RAW), (2, (17, 64), I.ENERGY_ICNN_ISO),
                                          (3, (64, 24), I.ENERGY_ICNN_RAW), (3, (16, 3), I.ENERGY_ICNN_ISO)])
def test_zero_state_is_elastic(env, dim, w, energy):
    torch, B, oracle = env
    probs = [problem(dim, s, w, energy) for s in range(NETS)]
    h = B.gd_create(probs[0], B.gd_default_options())
    n, nq = probs[0].mesh.n_nodes * (dim + 1), (probs[0].mesh.n_elems, 2 ** dim)
    for s, p in enumerate(probs):
        B.gd_set_params(h, p.psi.params, p.yld.params)
        R, K, k, l = gpu_assemble(B, torch, h, np.zeros(n), np.zeros(nq))
        assert not l.any() and not k.any(), (s, int(l.sum()), np.abs(k).max())
        _, Ko, _, _ = oracle_assemble(oracle, p, np.zeros(n), np.zeros(nq))
        d = np.abs((K - Ko).data).max() if (K - Ko).nnz else 0.0
        assert np.abs(R).max() < 1e-14 and d <= 1e-10 * np.abs(Ko.data).max(), s


def test_zero_state_of_a_batch(env):
    torch, B, _ = env
    probs = [problem(2, s, (8 + s % 9, 3 + s % 17), I.ENERGY_ICNN_RAW) for s in range(NETS)]
    h = B.gd_create_batch(probs, B.gd_default_options())
    n = sum(p.mesh.n_nodes for p in probs) * 3
    ne = sum(p.mesh.n_elems for p in probs)
    R, K, k, l = gpu_assemble(B, torch, h, np.zeros(n), np.zeros((ne, 4)))
    assert not l.any() and not k.any(), (int(l.sum()), np.abs(k).max())
