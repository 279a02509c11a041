"""A pivot that is not positive, in the first, a middle and the last column of a 32-column diagonal block
and in the first and a later block of the double-float factorisation: the subproblem is reported not
positive definite with a zero solution, and other subproblems are not affected.

The pivot is placed without damping (alpha = 0) by a thin, very slow layer between two depth samples: the
wave through it decays by exp(-eps h / c), beyond the range of FP64, so every kernel row is exactly zero
at the samples below it, and so is the pivot of the first of them.  The tolerance of the unaffected
requests, 1e-5, is that of every mixed solve.
"""
import copy

import numpy as np
import pytest

import synth
from oracle import stream1d
from synth import stream
from tests.gpu_helpers import rel_l2, small_workload, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COLUMNS = [0, 1, 15, 30, 31, 32, 33, 50, 63, 64]


def absorbing(column, dz):
    """Layers whose samples (j + 1/2) dz, j >= column, lie below the slow layer."""
    top = column * dz - 0.1 * dz if column else 0.1 * dz
    return np.array([0.0, top, top + 0.2 * dz]), np.array([1500.0, 1e-3, 2000.0])


@pytest.mark.parametrize("column", COLUMNS)
def test_line(column):
    from paper_0905_0238_gb300 import Config, Solver, EDT_MIXED
    nz, dz = 70, 40.0
    wl = small_workload(nx=32, nz=nz, nf=24, dx=20.0, dz=dz, alpha=0.0, layers=absorbing(column, dz))
    s = Solver(Config.from_workload(wl, precision=EDT_MIXED))
    D = synth.rng_for(1, salt=3).standard_normal((24, 32, 32)).astype(np.complex64)
    G = s.gram(dev(D))[0].cpu().numpy()
    assert not G[:, column:, :].any() and np.all(np.diagonal(G, axis1=1, axis2=2)[:, :column] > 0)
    for _ in range(2):                  # and again on the same context
        V = s.invert(dev(D)).cpu().numpy()
        assert s.stats().n_notpd == wl.nx // 2 + 1
        assert not V.any()


def test_stream():
    from paper_0905_0238_gb300 import Stream, edt
    rng = synth.rng_for(4, salt=970)
    subs, bad = [], []
    for i, column in enumerate(COLUMNS):
        sub = stream.sub1d_random(rng, nz_range=(96, 96), rows_range=(400, 400), layers_range=(6, 6))
        a = stream1d.kernel_rows(sub)
        sub.data = (a @ rng.standard_normal((sub.nz, 2))).astype(np.complex64)
        subs.append(sub)
        off = copy.copy(sub)
        off.alpha = 0.0
        off.layer_top, off.layer_vel = absorbing(column, sub.dz)
        subs.append(off)
    v, status = Stream(max_batch=8).solve(subs)
    for i, (sub, got, code) in enumerate(zip(subs, v, status)):
        if i % 2:
            assert code == edt.EDT_ENOTPD and not got.any()
        else:
            assert code == 0 and rel_l2(got, stream1d.solve(sub)) < 1e-5
