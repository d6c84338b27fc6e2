"""Gradients of batches that keep the training chains and the weight-gradient kernels on several tiles per block.

The gradient of 613 rays (five 128-row tiles, the last ragged) is compared with the oracle; then the same rays repeated 2^j
times, so that tiles hold other rows on every repetition and every block walks several of them.  A repetition
count that is a power of two scales the losses' averages, and with them every error signal and its BF16
rounding, exactly: loss and gradient are the 613 rays' up to the order of the FP32 sums.  A tile left out,
counted twice or paired with another's operand changes them by a tile's share."""
import dataclasses

import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

from .test_gpu_cls import _fine_centres

pytestmark = pytest.mark.gpu

N = 613
SMS = 152


def _rays(r, t, n, seed):
    import torch
    o, d = torch.empty(n, 3, device="cuda"), torch.empty(n, 3, device="cuda")
    m, h = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    r.make_labels(t, n, seed, 256, 8, o, d, m, h)
    return o, d, m, h


def _layers(g, shapes):
    at = 0
    for fi, fo in shapes:
        yield g[at:at + fi * fo + fo]
        at += fi * fo + fo
    assert at == len(g)


def _sum_error(tiles, splits):
    """Relative error of an FP32 sum over a split's tiles (eight 16-row products each) and then over the splits: an
    ulp per addition, and ten times that for cancellation between the terms."""
    return 10 * (8 * -(-tiles // splits) + splits) * 2.0 ** -23


def _check_repeats(r, t, rays, repeats, shapes, jobs):
    import torch
    n_par = sum(a * b + b for a, b in shapes)
    one = torch.zeros(n_par, device="cuda")
    loss = r.loss_grad(t, *rays, one)
    g1 = one.cpu().numpy().astype(np.float64)
    for k in repeats:
        tiles = -(-N * k // 128)
        big = torch.zeros(n_par, device="cuda")
        lk = r.loss_grad(t, *[torch.cat([x] * k).contiguous() for x in rays], big)
        assert abs(lk - loss) <= 1e-5 * abs(loss), (k, lk, loss)
        tol = _sum_error(tiles, max(1, min(SMS // jobs, tiles)))
        gk = big.cpu().numpy().astype(np.float64)
        err = [np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(_layers(gk, shapes), _layers(g1, shapes))]
        print(f"{k} repeats ({tiles} tiles): worst layer {max(err):.2e} of {tol:.2e} allowed; a tile's share {1 / tiles:.2e}")
        assert max(err) <= tol, (k, err)
    return g1


@pytest.mark.parametrize("hidden,width", [(1, 64), (1, 128), (6, 128), (16, 64), (16, 128)])
def test_regression_gradient(orc, hidden, width):
    """The 613 rays' gradient against the oracle's BF16 one with the bounds of the smaller batches' test (half the layer's own
    BF16 effect and 5e-4 of the largest element); then 307 and 613 tiles for at most 304 blocks."""
    from paper_2308_04669_gb300 import native
    base = sg.three_types_scene(8, 8, nerf=False)
    sc = dataclasses.replace(base, types=[sg.make_type(t.kind, 3, i, hidden, width) for i, t in enumerate(base.types)])
    r = native.renderer_for(sc, precision=native.PREC_BF16)
    rays = _rays(r, 1, N, 9)
    d = sc.types[1].nedf_dims
    shapes = list(zip(d[:-1], d[1:]))
    g = _check_repeats(r, 1, rays, (64, 128), shapes, hidden)
    r.close()
    args = [x.cpu().numpy().astype(np.float64) for x in rays[:3]] + [(rays[3].cpu().numpy() > 0.5).astype(np.int32)]
    osc = orc.OracleScene(sc)
    _, og = orc.nedf_loss_grad(osc, 1, *args, quant=orc.QUANT_BF16)
    _, og64 = orc.nedf_loss_grad(osc, 1, *args)
    scale = np.abs(og).max()
    for l, (a, b, c) in enumerate(zip(_layers(g, shapes), _layers(og, shapes), _layers(og64, shapes))):
        assert np.linalg.norm(a - b) <= 0.5 * np.linalg.norm(b - c) + 5e-4 * scale, l


def test_classifier_gradient(orc):
    """The 613 rays' gradient against the oracle's FP64 one with the bounds of the smaller batch's test; then 154 and 307 tiles
    for at most 152 blocks."""
    import torch
    from paper_2308_04669_gb300 import native
    sc = sg.classifier_scene(16, 16)
    r = native.renderer_for(sc, precision=native.PREC_BF16)
    o, d, m, h = _rays(r, 0, N, 4)
    m = torch.tensor(_fine_centres(m.cpu().numpy()), device="cuda")
    g = _check_repeats(r, 0, (o, d, m, h), (32, 64), sg.cls_layers(), 74)
    r.close()
    go, gd = o.cpu().numpy().astype(np.float64), d.cpu().numpy().astype(np.float64)
    X = np.array([orc.cls_features(a, b / np.linalg.norm(b), 1.0)[0] for a, b in zip(go, gd)])
    _, og = orc.cls_loss_grad(sc.types[0].nedf_w.astype(np.float64), X, m.cpu().numpy().astype(np.float64),
                               (h.cpu().numpy() > 0.5).astype(np.int32))
    assert np.linalg.norm(g - og) <= 5e-2 * np.linalg.norm(og)
    for l, (a, b) in enumerate(zip(_layers(g, sg.cls_layers()), _layers(og, sg.cls_layers()))):
        assert np.linalg.norm(a - b) <= 0.15 * np.linalg.norm(b), l
