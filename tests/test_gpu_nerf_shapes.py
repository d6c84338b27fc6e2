"""The NeRF engine at its widths, several depths and numbers of samples: in BF16 against the oracle at the
tolerance of the engine's other tests, and in both precisions at every way its weights are staged (a layer per
stage, two chunks, one chunk, odd numbers of chunks): the stage size never changes a result."""
import dataclasses

import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

from .gpu_helpers import frame_vs_oracle, gpu_frame

pytestmark = pytest.mark.gpu

STAGES = (1024, 8192, 12288, 16384, 24576, 36864, 49152, 65536)


def _scene(hidden, width, samples):
    base = sg.three_types_scene(96, 80)
    types = [sg.make_type(k, 3, t, 2, 64, hidden, width) for t, k in enumerate((sg.SDF_SPHERE, sg.SDF_TORUS, sg.SDF_BOX))]
    return dataclasses.replace(base, types=types, n_shade=samples)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("width,hidden,samples", [(64, 1, 1), (64, 3, 32), (128, 2, 7), (128, 8, 8), (256, 1, 8), (256, 2, 16),
                                                  (256, 16, 5)])
def test_nerf_shapes(orc, prec, width, hidden, samples):
    import torch
    from paper_2308_04669_gb300 import native
    p = native.PREC_BF16 if prec == "bf16" else native.PREC_FP8
    sc = _scene(hidden, width, samples)
    px = sg.pixel_subset(96, 80, 300, 8)
    g = gpu_frame(sc, precision=p, depth_source=1)
    assert g["stats"].status == 0
    if prec == "bf16":
        rep, _ = frame_vs_oracle(g, orc.OracleScene(sc), px=px, depth_mode=orc.DEPTH_MARCH, march_n=128, march_b=4,
                                 quant=orc.QUANT_BF16, n_threads=8)
        assert rep["hit"] > 50

    r = native.renderer_for(sc, precision=p)
    o = r.get_options()
    o.depth_source = 1
    r.set_options(o)
    n = sc.W * sc.H
    for b in STAGES:
        r.set_schedule([b] * len(native.SCHEDULE_KERNELS))
        rgba = torch.empty(n, 4, device="cuda")
        st = r.render(r.camera(sc.eye, sc.target, sc.fov_deg), r.lights(sc.lights), rgba=rgba, stats=True)
        torch.cuda.synchronize()
        assert st.status == 0, b
        assert np.array_equal(rgba.cpu().numpy().astype(np.float64), g["rgba"]), b
    r.close()
