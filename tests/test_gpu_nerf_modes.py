"""The NeRF engine where test_gpu_nerf_shapes.py does not take it: E4M3 shading of every shape against the oracle,
and the plain method's colour rows at the same shapes, precisions and weight stages, with sample counts whose
runs of rows cross the halves of a tile.

E4M3 against the oracle's E4M3 mode: a sum that rounds to the other neighbour moves a colour by up to a quarter of an
E4M3 step of the last hidden activation (0.5 below 8) times the largest output weight (Xavier: sqrt(6 / (N + 3))); such
flips are few, so up to eight layers the root mean square stays within half the E4M3 mode's own distance from the
unrounded network (through fifteen E4M3 layers one flip becomes many: there the largest difference alone is checked)."""
import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

from .gpu_helpers import MARGIN, NOID, compare_volume, gpu_frame
from .test_gpu_nerf_shapes import STAGES, _scene

pytestmark = pytest.mark.gpu

SHAPES = [(64, 1, 1), (64, 3, 32), (128, 2, 7), (128, 8, 8), (256, 1, 8), (256, 2, 16), (256, 16, 5)]


def _check_e4m3(got, fp8, fp64, width, hidden):
    err, own = got - fp8, fp8 - fp64
    rms, own_rms, worst = np.sqrt((err ** 2).mean()), np.sqrt((own ** 2).mean()), np.abs(err).max()
    limit = 0.25 * 0.5 * np.sqrt(6 / (width + 3))
    print(f"E4M3: rms {rms:.2e} (the mode's own {own_rms:.2e}), max {worst:.2e} of {limit:.2e}")
    assert worst <= limit and (rms <= 0.5 * own_rms or hidden > 8)


@pytest.mark.parametrize("width,hidden,samples", SHAPES)
def test_e4m3_shading(orc, width, hidden, samples):
    from paper_2308_04669_gb300 import native
    sc = _scene(hidden, width, samples)
    px = sg.pixel_subset(sc.W, sc.H, 600, 8)
    g = gpu_frame(sc, precision=native.PREC_FP8, depth_source=1)
    hit = g["id"][px] != NOID
    px = px[hit]
    assert len(px) > 100
    kw = dict(depth_mode=orc.DEPTH_MARCH, march_n=128, march_b=4, n_threads=8)
    osc = orc.OracleScene(sc)
    q, n = (orc.steps23(osc, px, g["id"][px], g["depth"][px], quant=m, **kw)["rgba"] for m in (orc.QUANT_FP8, orc.QUANT_NONE))
    _check_e4m3(g["rgba"][px], q, n, width, hidden)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("width,hidden,samples", [(w, h, s) for (w, h, _), s in zip(SHAPES, (37, 100, 64, 37, 100, 64, 37))])
def test_plain_method_rows(orc, prec, width, hidden, samples):
    """Dense against the oracle; early termination within its bound of dense; every stage size within the order of a
    pair's partial sums (1e-5)."""
    import torch
    from paper_2308_04669_gb300 import native
    sc = _scene(hidden, width, 8)
    r = native.renderer_for(sc, precision=native.PREC_BF16 if prec == "bf16" else native.PREC_FP8)
    cam = r.camera(sc.eye, sc.target, sc.fov_deg)

    def frame(early):
        rgba = torch.empty(sc.W * sc.H, 4, device="cuda")
        r.render_march(cam, samples, early, rgba)
        torch.cuda.synchronize()
        r.sync()
        return rgba.cpu().numpy().astype(np.float64)

    dense, early = frame(0), frame(1)
    for b in STAGES:
        r.set_schedule([b] * len(native.SCHEDULE_KERNELS))
        assert np.abs(frame(0) - dense).max() <= 1e-5 and np.abs(frame(1) - early).max() <= 1e-5, b
    r.close()
    assert np.abs(early - dense).max() < 2e-3
    px = sg.pixel_subset(sc.W, sc.H, 300, 3)
    osc = orc.OracleScene(sc)
    q, vm = orc.volume_render(osc, samples, px=px, n_threads=8, quant=orc.QUANT_BF16 if prec == "bf16" else orc.QUANT_FP8,
                              margins=True)
    assert (q[:, 3] > 0.5).sum() > 20
    if prec == "bf16":
        compare_volume(dense[px], q, vm)
    else:
        keep = vm > MARGIN
        assert keep.mean() >= 0.95
        seen = keep & (q[:, 3] > 1e-3)
        _check_e4m3(dense[px][seen], q[seen], orc.volume_render(osc, samples, px=px, n_threads=8)[seen], width, hidden)
