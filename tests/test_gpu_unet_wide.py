"""The network on images at least 128 pixels wide, where the blocks' second
convolutions pool their output and, in the backward pass, take their gradient
through the ReLU before them, inside the row kernel: against the BF16-emulating
oracle, with the bounds of test_gpu_unet.py.  Needs a GB300."""
import numpy as np
import pytest

from oracle import unet as ounet
from test_gpu_conv import bf16_round
from test_gpu_unet import _compare

pytestmark = pytest.mark.gpu


# levels 0 and 1 wide with ragged column blocks; level 2 too, as 64-column halves (few
# tiles) and whole; one row of pooled pixels a level at the bottom; a batch
@pytest.mark.parametrize("B, H, W", [(1, 16, 128), (2, 24, 264), (1, 32, 520), (1, 304, 520)])
def test_wide_network_matches_oracle(B, H, W):
    import torch
    import paper_1610_03918_gb300 as pg
    rng = np.random.default_rng(B + H + W)
    p = ounet.init_params(9)
    for n in p:
        p[n] = bf16_round(p[n]) if not n.endswith(".b") else rng.standard_normal(p[n].shape) * 0.05
    x = bf16_round(rng.standard_normal((B, H, W, 2)))
    t = rng.standard_normal((B, H, W))
    net = pg.Unet(B, H, W)
    net.set_params(ounet.flat(p).astype(np.float32))
    xd = torch.tensor(x, dtype=torch.float32, device="cuda")
    y = net.forward(xd).cpu().numpy()
    loss, g = net.gradients(xd, torch.tensor(t, dtype=torch.float32, device="cuda"))
    assert net.status() == pg.PIC_OK
    net.close()
    yo, _ = ounet.forward(p, x, q=bf16_round)
    assert np.linalg.norm(y - yo) / np.linalg.norm(yo) < 1e-2
    lo, go = ounet.loss_and_grads(p, x, t, q=bf16_round)
    assert loss == pytest.approx(lo, rel=1e-3)
    for name, (rel, cos) in _compare(g, go).items():
        assert rel < 0.15 and cos > 0.995, (name, rel, cos)
    # nothing but the last layers' own arithmetic and one data gradient before these
    for name in ("head.W", "head.b", "dec0b.W", "dec0b.b", "dec0a.b"):
        assert _compare(g, go)[name][0] < 1e-2, name
