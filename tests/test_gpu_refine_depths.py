"""Refinement residual at the depth counts where its register tiles (64 depths per load of a warp, up
to four) begin and end, with an odd number of rows per warp left over, in both forms, against the
FP64 oracle.

Tolerance 1e-5 relative L2, as for every mixed inversion: FP32 rows of the residual at alpha = 1e-2,
FP64-accurate rows at alpha = 1e-4 (the damping each form is chosen for).
"""
import numpy as np
import pytest

from oracle import edt2d
from tests.gpu_helpers import rel_l2, small_workload, dev
from tests.test_gpu_edges import data, mixed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("resid,alpha", [(1, 1e-2), (2, 1e-4)])
@pytest.mark.parametrize("nz", [63, 64, 65, 128, 129, 191, 192, 193, 256])
def test_depth_tiles_of_the_residual(nz, resid, alpha):
    wl = small_workload(nx=32, nz=nz, nf=5, alpha=alpha)
    D = data(wl, 9)
    _, vh_or = edt2d.invert(wl, D)
    s = mixed(wl, resid=resid)
    s.invert(dev(D))
    st = s.stats()
    assert st.n_notpd == 0 and st.n_nonfinite == 0
    assert rel_l2(s.vhat().cpu().numpy(), vh_or) < 1e-5
