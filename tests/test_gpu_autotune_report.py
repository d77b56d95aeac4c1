"""gd_autotune times a launch choice only where the launcher follows it: small systems launch the
CTAs that they fill (or one cluster) whatever the CTAs per SM, and the 4 x 4 block products have one
mapping.  What is not timed is -1."""
import numpy as np
import pytest

from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_03411_gb300 import build as build_mod
    build_mod.build()
    import paper_2604_03411_gb300.binding as binding
    return binding


def tuned(B, mesh, mixed):
    psi, yld = I.icnn_pair(5, 8, 8)
    prob = I.Problem("t", mesh, psi, yld, I.Material(), np.array([0.02, 0.04]))
    o = B.gd_default_options(precision=B.GD_MIXED) if mixed else B.gd_default_options()
    h = B.gd_create(prob, o)
    return B.gd_autotune(h)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("shape,one_grid", [((8, 8), True), ((30, 20), True), ((4, 4, 4), True), ((20, 20, 20), False)])
def test_what_is_timed(B, shape, one_grid, mixed):
    """81 to 651 nodes fill less than one CTA per SM, 9,261 nodes 290 or more CTAs."""
    mesh = I.uniaxial_bc_2d(I.structured_q4(*shape)) if len(shape) == 2 else I.uniaxial_bc_3d(I.structured_hex8(*shape))
    t = tuned(B, mesh, mixed)
    us = [t.krylov_us[i] for i in range(4)]
    timed = [v for v in us if v > 0]
    assert us[0] > 0 and us[t.krylov_ctas_per_sm - 1] == min(timed)
    assert len(timed) == 1 if one_grid else len(timed) >= 2
    up = [t.krylov_us_up[i] for i in range(3)]
    if len(shape) == 3:
        assert t.krylov_up == 1 and all(v == -1.0 for v in up)
    else:
        assert up[[1, 2, 4].index(t.krylov_up)] > 0
    assert all(t.krylov_us_lanes[i] == -1.0 for i in range(3))
