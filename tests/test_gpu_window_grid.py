"""Kernel rows of the window geometry on a grid (transform over y first, then the window sum by cosine
and sine transforms) at the forms where their indexing can go wrong, against the FP64 oracle: every
window shape, x and y spacings that differ (no transposed planes), one depth and depth counts around
the tiles of 8; and the Gram of window rows at its depth tiles.

Tolerance 1e-5 relative L2 on Vhat, as for the other window shapes: FP32 rows and one refinement step
at alpha = 1e-3.
"""
import numpy as np
import pytest

from oracle import edt3d
from tests.gpu_helpers import rel_l2, dev
from tests.test_gpu_window import born_data, workload, solver

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WINDOWS = [(1, 1), (2, 1), (4, 1), (8, 1), (16, 1), (2, 2), (4, 4), (8, 8), (16, 16), (4, 2), (8, 4), (16, 8)]


def check(wl):
    D = born_data(wl, salt=23)
    _, vh_or = edt3d.invert(wl, D)
    s = solver(wl)
    s.invert(dev(D.astype(np.complex64)), out_dtype=torch.float32)
    st = s.stats()
    assert st.n_notpd == 0 and st.n_nonfinite == 0
    want = np.stack([vh_or[m[1], m[0]] for m in edt3d.pair_representatives(wl)])
    assert rel_l2(s.vhat().cpu().numpy(), want) < 1e-5, rel_l2(s.vhat().cpu().numpy(), want)


@pytest.mark.parametrize("wx,wy", WINDOWS)
def test_every_window(wx, wy):
    check(workload(32, 32, wx, wy, nf=2, nz=5, alpha=1e-3))


@pytest.mark.parametrize("n,nz", [(32, 1), (32, 8), (32, 16), (64, 17), (128, 33)])
def test_depth_tiles(n, nz):
    check(workload(n, n, 4, 4, nf=2, nz=nz, alpha=1e-3))


@pytest.mark.parametrize("n,w", [(32, 8), (64, 4)])
def test_spacings_differ(n, w):
    wl = workload(n, n, w, w, nf=2, nz=6, alpha=1e-3)
    wl.dy = 1.25 * wl.dx
    check(wl)


@pytest.mark.parametrize("nz", [31, 127, 128, 129, 225, 256])
def test_gram_depths(nz):
    """Depth counts at the edges of the Gram's 32-depth groups and 128-row halves (its rows arrive in
    bulk, an odd count with a padding depth)."""
    check(workload(64, 1, 4, 1, nf=4, nz=nz, alpha=1e-2))
