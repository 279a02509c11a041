"""Contexts of different sizes used in turn in one process: a later context with fewer depths or points
must not take away the shared memory that an earlier one's kernels launch with.  The earlier context's
result is the same, bit for bit, before and after the later one is created and used."""
import numpy as np
import pytest

import synth
from tests.gpu_helpers import small_workload, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solver(kind, nx, nz):
    from paper_0905_0238_gb300 import Config, Solver, EDT_FP64, EDT_GEOM_WINDOW, EDT_MIXED
    kw = {"fp64": dict(precision=EDT_FP64), "mixed": dict(precision=EDT_MIXED),
          "mixed one pass": dict(precision=EDT_MIXED, passes=1), "native Cholesky": dict(precision=EDT_MIXED, chol_df=2),
          "tsvd": dict(precision=EDT_FP64, solver=1, tsvd_tol=-1e-2),
          "disk": dict(precision=EDT_FP64, kz_disk=2.2)}.get(kind)
    wl = small_workload(nx=nx, nz=nz, nf=4, alpha=1e-2)
    if kw is None:
        kw = dict(precision=EDT_MIXED, geometry=EDT_GEOM_WINDOW, fold=0, ny=1, dy=wl.dx, wx=4, wy=1)
    return Solver(Config.from_workload(wl, **kw)), wl


def _data(kind, wl, salt):
    shape = (4, 1, wl.nx, 1, 4) if kind == "window" else (4, wl.nx, wl.nx)
    rng = synth.rng_for(2, salt=salt)
    return dev((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64))


@pytest.mark.parametrize("kind", ["fp64", "mixed", "mixed one pass", "native Cholesky", "tsvd", "disk", "window"])
@pytest.mark.parametrize("small", [(32, 16), (64, 16), (32, 95)])
def test_a_smaller_context_leaves_a_larger_one_alone(kind, small):
    big, wl = _solver(kind, 64, 96)
    D = _data(kind, wl, 1)
    want = big.invert(D).cpu().numpy()
    other, wl2 = _solver(kind, *small)
    V2 = other.invert(_data(kind, wl2, 2))
    assert torch.isfinite(V2).all()
    assert np.array_equal(big.invert(D).cpu().numpy(), want)


def test_calls_that_share_scratch_do_not_disturb_one_another():
    """The Gram's partial tiles, the folded residual planes and the reversed march's states share memory, as
    do the FP64 spectra, the Gram's parts and the truncated SVD's log: every call on a context that has
    made the others gives what it gives on a new context, bit for bit."""
    layers = (np.array([0.0, 60.0, 150.0, 250.0]), np.array([1500.0, 1800.0, 2300.0, 2900.0]))
    wl = small_workload(nx=64, nz=40, nf=4, alpha=1e-2, cutoff=0.0, layers=layers)
    from paper_0905_0238_gb300 import Config, Solver, EDT_MIXED
    new = lambda: Solver(Config.from_workload(wl, precision=EDT_MIXED))
    rng = synth.rng_for(2, salt=7)
    D = dev((rng.standard_normal((4, 64, 64)) + 1j * rng.standard_normal((4, 64, 64))).astype(np.complex64))
    V = dev(1e-8 * rng.standard_normal((64, 40)))

    def calls(solver):
        return dict(invert=lambda: [solver().invert(D)],
                    vjp=lambda: (lambda s: [s.invert(D), *s.invert_vjp(V, out_dtype=torch.complex64)][2:])(solver()),
                    misfit=lambda: [solver().misfit_grad(V, D)[2]],        # dJ/dc: no atomic sums
                    forward=lambda: [solver().forward(V)], gram=lambda: list(solver().gram(D)))

    want = {k: [a.cpu().numpy() for a in f()] for k, f in calls(new).items()}
    one = new()
    order = ["invert", "misfit", "vjp", "forward", "gram", "misfit", "invert", "vjp"]
    for k in order:
        for a, b in zip(calls(lambda: one)[k](), want[k]):
            assert np.array_equal(a.cpu().numpy(), b), k
    tsvd, wl2 = _solver("tsvd", 64, 96)
    D2 = _data("tsvd", wl2, 1)
    first, G = tsvd.invert(D2).cpu().numpy(), tsvd.gram(D2)[0].cpu().numpy()
    assert np.array_equal(tsvd.invert(D2).cpu().numpy(), first) and np.array_equal(tsvd.gram(D2)[0].cpu().numpy(), G)
