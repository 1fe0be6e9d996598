"""pic_unet_forward into output arrays that the network's last kernel cannot store
into: the same values as into one it can.  Needs a GB300."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 4, 1, 2, 3])
def test_output_at_any_address(offset):
    import torch
    import paper_1610_03918_gb300 as pg
    B, H, W = 1, 16, 24
    rng = np.random.default_rng(3)
    net = pg.Unet(B, H, W)
    net.set_params((0.1 * rng.standard_normal(net.nparam)).astype(np.float32))
    x = torch.tensor(rng.standard_normal((B, H, W, 2)), dtype=torch.float32, device="cuda")
    want = net.forward(x)
    room = torch.full((4 * B * H * W + 8,), 7, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert pg.load_library().pic_unet_forward(net.h, x.data_ptr(), room.data_ptr() + offset) == pg.PIC_OK
    net.stream.synchronize()
    got = room.cpu().numpy()
    net.close()
    assert got[offset:offset + 4 * B * H * W].tobytes() == want.cpu().numpy().tobytes()
    assert (got[:offset] == 7).all() and (got[offset + 4 * B * H * W:] == 7).all()
