"""The FP64 depth march over stacks where its recursion splits the layers over lanes (more than 64
layers over few wavenumbers), rescales (every eighth layer) and evaluates in chunks of 4 or 16
depths, against the oracle: 1e-12 as for the other stacks, elementwise 1e-10."""
import numpy as np
import pytest

from oracle import edt2d
from tests.gpu_helpers import rel_l2, small_workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,nf,nlayer", [
    (16, 9, 1, 1), (16, 5, 3, 64), (16, 33, 3, 65), (32, 17, 5, 130), (64, 40, 3, 1025),
    (64, 16, 2, 2), (512, 20, 40, 70),
])
def test_green_stacks(nx, nz, nf, nlayer):
    from paper_0905_0238_gb300 import Config, Solver, EDT_FP64
    # alternating velocities: strong reflections at every interface
    rng = np.random.default_rng(nlayer)
    depth = 10.0 * nz
    tops = np.concatenate([[0.0], np.sort(rng.uniform(0.01, 1.0, nlayer - 1)) * depth])
    vel = 2500.0 + 800.0 * np.where(np.arange(nlayer) % 2, 1.0, -1.0) * rng.uniform(0.2, 1.0, nlayer)
    wl = small_workload(nx=nx, nz=nz, nf=nf, fmin=5.0, fmax=40.0, layers=(tops, vel))
    g = Solver(Config.from_workload(wl, precision=EDT_FP64)).green().cpu().numpy()
    want = edt2d.green_table(wl)[:, : nx // 2 + 1, :]
    assert rel_l2(g, want) < 1e-12
    assert np.max(np.abs(g - want) / np.abs(want)) < 1e-10
