"""Plain-method labels on the GPU against the oracle's uniform march, for every SDF kind and at a bound
radius on either side of the limit up to which the label march skips samples."""
import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

from .gpu_helpers import DMARGIN, close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _scaled(kind, scale):
    p = [v * scale for v in sg.DEFAULT_PARAMS[kind]]
    if kind == sg.SDF_TWISTTORUS:
        p[2] = sg.DEFAULT_PARAMS[kind][2] / scale          # the twist is an angle per length
    return sg.make_type(kind, 7, 0, 4, 64, rb=scale, params=p)


@pytest.mark.parametrize("scale", [1.0, 100.0])
@pytest.mark.parametrize("kind", sorted(sg.DEFAULT_PARAMS))
def test_labels_of_every_kind_match_the_uniform_march(orc, kind, scale):
    """Hit bit-exact and m* within 1e-4 except at knife edges (a march test within DMARGIN of the
    surface, relative to the coordinates), as in test_training_rays_and_labels."""
    import torch
    from paper_2308_04669_gb300 import native
    n, steps, bisect = 1200, 97, 6
    ty = _scaled(kind, scale)
    one = sg.Scene("one", 8, 8, sg.f32([0, 0, 3 * scale]), sg.f32([0, 0, 0]), 40.0, sg.f32([[2, 3, 2]]), [ty],
                   np.zeros(1, np.uint32), sg.f32(np.eye(3).reshape(1, 9)), sg.f32([[0, 0, 0]]), sg.f32([1.0]))
    r = native.renderer_for(one)
    o, d = torch.empty(n, 3, device="cuda"), torch.empty(n, 3, device="cuda")
    m, h = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    r.make_labels(0, n, 11, steps, bisect, o, d, m, h)
    torch.cuda.synchronize()
    r.close()
    go, gd = o.cpu().numpy().astype(np.float64), d.cpu().numpy().astype(np.float64)
    osc = orc.OracleScene(one)
    om, oh = orc.train_labels(osc, 0, go, gd, steps, bisect)
    knife = np.zeros(n, bool)
    for i in range(n):
        _, q, dg = orc.query_diag(osc, 0, go[i], gd[i], need=np.inf, depth_mode=orc.DEPTH_MARCH, march_n=steps, march_b=bisect)
        dm = orc.query_diag(osc, 0, go[i], gd[i], need=1e-4 * scale, depth_mode=orc.DEPTH_MARCH, march_n=steps, march_b=bisect)[2]
        knife[i] = dg[1] <= DMARGIN or dm[1] <= DMARGIN or abs(q[3] - q[4]) < 1e-6 * scale
    gh = h.cpu().numpy() > 0.5
    assert np.array_equal(gh[~knife], oh[~knife] == 1)
    both = gh & (oh == 1) & ~knife
    assert close(m.cpu().numpy()[both], om[both], 1e-4, 1e-4).all()
    assert 0.05 < gh.mean() < 0.95 and knife.mean() < 0.05
