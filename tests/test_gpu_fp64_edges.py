"""FP64 path at the edges of its tiles, against the FP64 oracle: the Gram's 2 x 2 tiles of the lower
triangle (odd and smallest depth counts, one and several groups of tiles) with its rows split over
CTAs (few subproblems) and not (many), and the Jacobi solver's smallest, odd and largest systems with
absolute, relative and no truncation.

Tolerances: 1e-10 on Vhat for the damped solve, 1e-8 for the truncated SVD, as for the other FP64 cases
(cond(G + lam I) 2^-53 below 1e-11; the truncation threshold at least 2 % from every singular value).
"""
import numpy as np
import pytest

from oracle import edt2d
from tests.gpu_helpers import rel_l2, small_workload
from tests.test_gpu_solvers import data, separated_tol, solve_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz", [(32, 1), (32, 2), (32, 63), (32, 126), (32, 127), (512, 3), (512, 200)])
def test_gram_tiles(nx, nz):
    wl = small_workload(nx=nx, nz=nz, nf=4, alpha=1e-3, dx=10.0 if nx == 32 else 4.0)
    D = data(wl, 21)
    _, vh_or = edt2d.invert(wl, D)
    _, vh = solve_gpu(wl, D)
    assert rel_l2(vh, vh_or) < 1e-10


@pytest.mark.parametrize("nz", [1, 2, 3, 64, 65, 95, 96])
def test_jacobi_sizes(nz):
    wl = small_workload(nx=32, nz=nz, nf=6, alpha=1e-3)
    D = data(wl, 22)
    tol = separated_tol(wl, D, [3e-3, 2e-3, 5e-3, 1.5e-3, 7e-3, 1.2e-2, 2.5e-2])
    _, vh_or = edt2d.invert(wl, D, solver="tsvd", tsvd_tol=-tol)
    _, vh = solve_gpu(wl, D, solver=1, tsvd_tol=-tol)
    assert rel_l2(vh, vh_or) < 1e-8


def test_jacobi_without_truncation():
    """A threshold far below every singular value keeps them all: two depths, well conditioned."""
    wl = small_workload(nx=32, nz=2, nf=6, alpha=1e-3)
    D = data(wl, 23)
    _, vh_or = edt2d.invert(wl, D, solver="tsvd", tsvd_tol=1e-30)
    _, vh = solve_gpu(wl, D, solver=1, tsvd_tol=1e-30)
    assert rel_l2(vh, vh_or) < 1e-8


@pytest.mark.parametrize("nz,dz", [(3, 60.0), (8, 60.0), (13, 60.0), (33, 40.0)])
def test_jacobi_with_a_threshold_of_zero(nz, dz):
    """tsvd_tol = 0 keeps every positive singular value, and every pair is rotated to its own diagonal:
    the least-squares solution.  Compared where the system's condition is below 1e3: its square, which
    the normal matrix has, times the FP64 rounding of nz sums gives 1e-8."""
    from paper_0905_0238_gb300 import Config, Solver, EDT_FP64
    wl = small_workload(nx=32, nz=nz, nf=12, dz=dz, alpha=1e-3)
    D = data(wl, 24)
    s = Solver(Config.from_workload(wl, precision=EDT_FP64, solver=1, tsvd_tol=0.0))
    s.invert(torch.from_numpy(D).cuda())
    vh, D2, seen = s.vhat().cpu().numpy(), edt2d.data_transform(D), 0
    for m in range(wl.nx // 2 + 1):
        want, system = edt2d.solve_wavenumber(wl, D2, m, return_system=True, solver="tsvd", tsvd_tol=0.0)
        if "Ahat" not in system:             # no row is kept
            assert not vh[m].any()
            continue
        sv = np.linalg.svd(system["Ahat"], compute_uv=False)
        if sv[-1] * 1e3 > sv[0]:
            assert rel_l2(vh[m], want) < 1e-8, m
            seen += 1
    assert seen >= 6
