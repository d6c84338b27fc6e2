"""The plain method's answers to deferred pairs: with a confidence bound of 1 every NeDF pair of an
untrained network is deferred, so the frame's depths, ids and shadows are the plain method's, bit for
bit, whether the pairs are few (a warp per pair) or many (a thread per pair)."""
import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

WARP_PAIRS = 32768      # kFallbackWarpPairs


@pytest.mark.parametrize("steps,bisect", [(1, 0), (37, 3), (256, 8)])
@pytest.mark.parametrize("size,many", [(40, False), (448, True)])
def test_deferred_pairs_equal_the_plain_method(size, many, steps, bisect):
    import torch
    from paper_2308_04669_gb300 import build, native
    build.build()
    sc = sg.stress_scene(size, size - 8, nerf=False, n_inst=64)
    r = native.renderer_for(sc, precision=native.PREC_BF16)
    cam, lights = r.camera(sc.eye, sc.target, sc.fov_deg), r.lights(sc.lights[:2])
    got = []
    for source in (native.DEPTH_NEDF, native.DEPTH_MARCH):
        o = r.get_options()
        o.depth_source, o.fallback_conf, o.march_steps, o.march_bisect = source, 1.0, steps, bisect
        r.set_options(o)
        n = sc.W * sc.H
        b = [torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"), None,
             torch.empty(n, device="cuda"), None]
        st = r.render(cam, lights, *b, stats=True)
        torch.cuda.synchronize()
        got.append([x.cpu().numpy() for x in b if x is not None] + [st])
    r.close()
    st = got[0][-1]
    assert st.fallback_pairs == st.primary_pairs + st.shadow_pairs and st.status == 0
    assert (st.primary_pairs > WARP_PAIRS) == many
    for a, b in zip(got[0][:3], got[1][:3]):
        assert np.array_equal(a, b)
