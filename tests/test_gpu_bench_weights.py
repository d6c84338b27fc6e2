"""The committed weights of the bench's reference arm are what the bench's training gives, bit for bit (the
training is deterministic on one GPU model: 152 SMs)."""
import os

import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t", [0, 1, 2])
def test_training_reproduces_the_committed_weights(t):
    import torch
    from paper_2308_04669_gb300 import native
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the order of the weight gradients' sums follows the number of SMs")
    z = np.load(os.path.join(os.path.dirname(native.__file__), "data", "nedf_thousand_bench.npz"))
    sc = sg.thousand_scene(64, 64)
    r = native.renderer_for(sc, precision=native.PREC_BF16)
    r.make_labels(t, int(z["rays"]), 2 + t, 256, 8)
    for _ in range(int(z["steps"])):
        r.train_step(t, int(z["batch"]), 1e-3)
    w = r.get_nedf_weights(t, sc.types[t].nedf_w.shape[0])
    r.sync()
    r.close()
    assert np.array_equal(w.astype(np.float32), z[f"type{t}"])
