"""The spectral Born operator on the folded table index (forward model, misfit and its
gradients) at the sizes where its tiles, edge pairs and depth chunks begin and end, against the
oracle.

Every entry of a frequency plane comes from a pair of the table index 0..N/2 (eight entries to a
pair, four with the edge N/2, fewer distinct ones at 0 and on the diagonal): N = 16 leaves part of
a 32-wide tile empty, N = 64 fills one, N = 128 takes off-diagonal tiles.  Depths come in chunks
of 8 in the forward model and 32 to 128 in the gradients.

Tolerances: the mixed forward model holds each plane's sums to 2^-27 of the plane (float pairs, or FP64
where the sums cancel too far for those), so its error is that of the two FP32 transforms, at most
about 3 u per radix-2 stage (u = 2^-24) in the 2-norm, 2 * 7 * 3 u = 2.5e-6 for N = 128; FP64 1e-11 as
elsewhere.  The misfit's sums are FP32
over the depths and one lateral axis: 1e-5 as in test_gpu_grad."""
import numpy as np
import pytest

import synth
from oracle import edt2d, grad2d
from tests.gpu_helpers import rel_l2, small_workload, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LAYERS = (np.array([0.0, 60.0, 150.0, 250.0]), np.array([1500.0, 1800.0, 2300.0, 2900.0]))


def _workload(nx, nz, nf):
    return small_workload(nx=nx, nz=nz, nf=nf, fmin=8.0, fmax=35.0, cutoff=0.0, layers=LAYERS, alpha=1e-3)


def _solver(wl, precision):
    from paper_0905_0238_gb300 import Config, Solver
    return Solver(Config.from_workload(wl, precision=precision))


def _model(wl, salt):
    # every wavenumber present, so that every entry of the planes counts
    return 1e-8 * synth.rng_for(7, salt=salt).standard_normal((wl.nx, wl.nz))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 2.5e-6)])
@pytest.mark.parametrize("nx,nz,nf", [(16, 1, 2), (16, 9, 3), (32, 8, 2), (64, 33, 2), (128, 17, 2), (128, 70, 1)])
def test_forward_edges(precision, tol, nx, nz, nf):
    from paper_0905_0238_gb300 import EDT_FP64, EDT_MIXED
    wl = _workload(nx, nz, nf)
    V = _model(wl, 1)
    s = _solver(wl, EDT_FP64 if precision == "fp64" else EDT_MIXED)
    D = s.forward(dev(V)).cpu().numpy()
    assert rel_l2(D, edt2d.forward(wl, V)) < tol


@pytest.mark.parametrize("nx,nz,eps,depth,sigma", [
    (64, 200, 0.15, 800.0, 60.0), (128, 200, 0.15, 800.0, 120.0), (128, 200, 0.15, 800.0, 160.0),
    (64, 255, 5.0, 1200.0, 30.0), (64, 256, 10.0, 1600.0, 10.0),
])
def test_forward_of_models_whose_sums_cancel(nx, nz, eps, depth, sigma):
    """Smooth perturbations of a homogeneous reference, and deep ones under strong decay: the depth sums come
    to 1e-4 to 1e-10 of their terms, and every frequency keeps the accuracy of the transforms."""
    from paper_0905_0238_gb300 import EDT_MIXED
    wl = small_workload(nx=nx, nz=nz, nf=4, fmin=20.0, fmax=60.0, dx=12.5, dz=8.0, cutoff=0.0, eps=eps,
                        layers=(np.array([0.0]), np.array([2000.0])))
    x, z = np.arange(nx) * 12.5, (np.arange(nz) + 0.5) * 8.0
    V = 1e-8 * np.exp(-((x[:, None] - nx * 6.25) ** 2 + (z[None, :] - depth) ** 2) / (2 * sigma ** 2))
    D, want = _solver(wl, EDT_MIXED).forward(dev(V)).cpu().numpy(), edt2d.forward(wl, V)
    for f in range(4):
        assert rel_l2(D[f], want[f]) < 2.5e-6


@pytest.mark.parametrize("nx,nz,nf", [(64, 1, 2), (64, 65, 1), (64, 129, 1), (128, 7, 2), (256, 34, 1)])
def test_gradient_edges(nx, nz, nf):
    from paper_0905_0238_gb300 import EDT_MIXED
    wl = _workload(nx, nz, nf)
    V, D = _model(wl, 2), edt2d.forward(wl, _model(wl, 3))
    J, gV, gc = _solver(wl, EDT_MIXED).misfit_grad(dev(V), dev(D))
    assert abs(float(J.cpu()) / grad2d.misfit(wl, V, D) - 1) < 1e-5
    assert rel_l2(gV.cpu().numpy(), grad2d.grad_V(wl, V, D)) < 1e-5
    assert rel_l2(gc.cpu().numpy(), grad2d.grad_c(wl, V, D)) < 1e-5
    Vt = _solver(wl, EDT_MIXED).adjoint(dev(D)).cpu().numpy()
    assert rel_l2(Vt, edt2d.adjoint(wl, D)) < 1e-5


@pytest.mark.parametrize("scale", [1e-18, 1e-12, 1e12, 1e18, 1e20])
def test_misfit_does_not_depend_on_the_unit_of_the_data(scale):
    """Model and data times a factor: J and dJ/dc change by its square and dJ/dV by the factor, to
    the same 1e-5, although the squares of the residual, and its products with the model, leave the FP32
    range."""
    from paper_0905_0238_gb300 import EDT_MIXED
    wl = _workload(64, 40, 3)
    V, D = _model(wl, 2), edt2d.forward(wl, _model(wl, 3))
    J, gV, gc = _solver(wl, EDT_MIXED).misfit_grad(dev(scale * V), dev(scale * D))
    assert abs(float(J.cpu()) / scale / scale / grad2d.misfit(wl, V, D) - 1) < 1e-5
    assert rel_l2(gV.cpu().numpy() / scale, grad2d.grad_V(wl, V, D)) < 1e-5
    assert rel_l2(gc.cpu().numpy() / scale / scale, grad2d.grad_c(wl, V, D)) < 1e-5
