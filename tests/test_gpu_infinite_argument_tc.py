"""The tensor-core kernel pads its networks to a multiple of 16 units with zero weights.  An
infinite argument of the yield network (f_d underflows in FP32 where eta_d kappa is past 104) must
not meet them: at q = +inf the trial value is +inf and the point loads, whatever the width, and
at q = -inf it is elastic and keeps its history."""
import numpy as np
import pytest

from gpu_common import gpu_assemble, smooth_state
from paper_2604_03411_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [8, 16, 23, 32])
def test_bf16(w):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_03411_gb300 import build as build_mod
    build_mod.build()
    import paper_2604_03411_gb300.binding as B
    mesh = I.uniaxial_bc_2d(I.structured_q4(5, 4))
    psi, yld = I.icnn_pair(5, w, w)
    prob = I.Problem("far", mesh, psi, yld, I.Material(), np.array([0.1]))
    dofs, kappa = smooth_state(mesh, np.random.default_rng(3), u_amp=0.06)
    kappa[:] = 200.0
    h = B.gd_create(prob, B.gd_default_options(precision=B.GD_MIXED, icnn_mma=B.GD_ICNN_BF16))
    for phi, loads in ((250.0, True), (0.1, False)):
        dofs[:, 2] = phi
        try:
            R, K, k, l = gpu_assemble(B, torch, h, dofs, kappa, "mixed")
        except B.GDError as e:           # no finite root: reported, too
            assert loads and "LOCAL_SOLVE" in str(e)
            continue
        assert (l > 0).all() if loads else not l.any()
        assert np.array_equal(k, kappa) if not loads else not np.isfinite(k).any()
