"""Launch counts that edt_get_stats reports: the same before and after the context has a workspace."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["line", "deep stack", "fp64", "window line", "window grid"])
def test_launch_counts_do_not_depend_on_the_workspace(kind):
    from paper_0905_0238_gb300 import Config, EDT_FP64, EDT_GEOM_WINDOW, EDT_MIXED, edt
    n = 40 if kind == "deep stack" else 3
    kw = dict(precision=EDT_FP64 if kind == "fp64" else EDT_MIXED)
    if kind.startswith("window"):
        grid = kind == "window grid"
        kw.update(geometry=EDT_GEOM_WINDOW, fold=0, ny=32 if grid else 1, dy=10.0, wx=4, wy=4 if grid else 1)
    cfg = Config(nx=32, dx=10.0, nz=20, dz=10.0, z0=0.0, freq_hz=np.array([8.0, 15.0]), eps=0.15,
                 layer_top=np.arange(n) * (200.0 / n), layer_vel=np.linspace(1500.0, 3000.0, n), alpha=1e-2,
                 cutoff=1.0, **kw)
    c, _arrays = cfg.c_config()
    ctx, nbytes = edt.edt_create(c)
    try:
        before = edt.edt_get_stats(ctx)
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        edt.edt_set_workspace(ctx, ws.data_ptr(), nbytes)
        after = edt.edt_get_stats(ctx)
        for name in ("launches_per_invert", "launches_per_grad", "freq_chunk", "gram_rows_padded"):
            assert getattr(before, name) == getattr(after, name), name
    finally:
        edt.edt_destroy(ctx)
