"""CUDA-core FP32 networks of the mixed element kernel, four points of an element at a time:
widths around the lane groups (16 and 32 units, and two units per lane beyond), the
identity yield function, ragged batches of elements, and a batch whose specimens change
networks inside a warp's 32 points.  Tolerance of the mixed kernel against the oracle:
2e-5 of the largest entry (FP32 roundoff 6e-8 through ~1e3 operations per entry)."""
import numpy as np
import pytest

from gpu_common import gpu_assemble, oracle_assemble, rel_err, smooth_state
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 2e-5


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


def specimen(rng, shape, wp, wy):
    mesh = I.uniaxial_bc_2d(I.structured_q4(*shape)) if len(shape) == 2 else I.biaxial_bc_3d(I.structured_hex8(*shape))
    yld = I.icnn_weights(rng, 1, wy) if wy else I.ICNN(1, 0, np.zeros(1))
    return I.Problem("u", mesh, I.icnn_weights(rng, 3, wp), yld, I.Material(), np.array([0.1]))


@pytest.mark.parametrize("shape", [(3, 1), (7, 5), (1, 1, 1), (3, 2, 1)])
@pytest.mark.parametrize("wp,wy", [(1, 1), (16, 17), (17, 16), (31, 33), (33, 32), (64, 64), (8, 0)])
def test_widths(env, shape, wp, wy):
    torch, B, oracle = env
    rng = np.random.default_rng(7)
    prob = specimen(rng, shape, wp, wy)
    h = B.gd_create(prob, B.gd_default_options(precision=B.GD_MIXED, icnn_mma=B.GD_ICNN_CUDA_CORES))
    d, k = smooth_state(prob.mesh, rng)
    Rg, Kg, kg, lg = gpu_assemble(B, torch, h, d, k, precision="mixed")
    Ro, Ko, ko, qi = oracle_assemble(oracle, prob, d, k)
    assert rel_err(Rg, Ro) < TOL
    assert np.abs((Kg - Ko).data).max() < TOL * np.abs(Ko.data).max()
    assert np.abs(kg - ko).max() < TOL
    assert np.all(kg >= k)


def test_specimens_of_other_networks_in_one_warp(env):
    torch, B, oracle = env
    rng = np.random.default_rng(8)
    probs = [specimen(rng, s, wp, wy) for s, wp, wy in
             [((3, 1), 16, 8), ((2, 1), 32, 17), ((1, 1), 5, 33), ((4, 3), 24, 24), ((5, 1), 40, 16)]]
    h = B.gd_create_batch(probs, B.gd_default_options(precision=B.GD_MIXED))
    states = [smooth_state(p.mesh, rng) for p in probs]
    d = np.concatenate([s[0] for s in states])
    k = np.concatenate([s[1] for s in states])
    Rg, Kg, kg, lg = gpu_assemble(B, torch, h, d, k, precision="mixed")
    no, eo, _ = B.gd_batch_layout(h)
    for i, p in enumerate(probs):
        Ro, Ko, ko, qi = oracle_assemble(oracle, p, *states[i])
        rows = slice(3 * no[i], 3 * no[i + 1])
        assert rel_err(Rg[rows], Ro) < TOL
        assert np.abs((Kg[rows, rows] - Ko).data).max() < TOL * np.abs(Ko.data).max()
        assert np.abs(kg[eo[i]:eo[i + 1]] - ko).max() < TOL
