"""An Adam step re-packs the blob: whatever it held before (never packed, every
BF16 and FP32 place of it some finite value), it is then the one enzo_mlp_pack
makes of the updated weights, padding columns included."""
import pytest

import paper_1307_2265_gb300 as ez

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 300])
def test_step_leaves_the_packed_blob(n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    net = ez.MLP(seed=4)
    x, t = torch.randn(n, 6, device="cuda", generator=g), torch.randn(n, device="cuda", generator=g)
    net.blob.view(torch.bfloat16).fill_(0.0625)
    net.train_step(x, t, 1e-3)
    used = (64 * 16 + 2 * 64 * 64) * 2 // 4 + 193          # the tiles, then b1, b2, w3, b3
    got = net.blob.clone()
    net.pack()
    assert torch.equal(got[:used].view(torch.int32), net.blob[:used].view(torch.int32))
    assert int(net.status[12].item()) == 0
