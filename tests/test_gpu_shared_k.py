"""Shared k-blocks at sizes that take clusters of two, three, four and more shares: column counts that leave the last
share short, row counts that leave the last tile short, fp32 storage; against the library's plain kernel."""
import pytest
import torch

import paper_2309_06626_b200 as asx
from gpu_util import shares_k_blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f32", [False, True], ids=["bf16", "f32"])
@pytest.mark.parametrize("case", [
    # C_in, C_out, H, W, Nb, kept per image
    (512, 512, 7, 7, 64, 24), (256, 176, 14, 14, 9, 97), (512, 136, 7, 7, 40, 25), (1024, 512, 7, 7, 11, 35), (256, 80, 9, 11, 30, 99),
], ids=lambda c: "x".join(str(v) for v in c))
def test_shares_of_every_size(case, f32):
    cin, cout, H, W, Nb, kept = case
    gen = torch.Generator(device="cuda").manual_seed(cin + cout)
    dt = torch.float32 if f32 else torch.bfloat16

    def tf32(t):                                                  # values whose lower 13 mantissa bits are zero
        return (t.view(torch.int32) & ~0x1fff).view(torch.float32) if f32 else t.to(dt)
    x = tf32(torch.randn((Nb, H, W, cin), generator=gen, device="cuda"))
    w = tf32(torch.randn((cout, 3, 3, cin), generator=gen, device="cuda") * (9 * cin) ** -0.5)
    b = torch.randn((cout,), generator=gen, device="cuda")
    mask = torch.zeros(H * W, dtype=torch.uint8)
    mask[torch.randperm(H * W, generator=torch.Generator().manual_seed(1))[:kept]] = 1
    layer = asx.MaskedConvLayer(cin, cout, 3, 3, 1, 1)
    layer.set_mask(mask.numpy())
    base = asx.F32 if f32 else 0
    want = layer.run(x, w, b, flags=base | asx.ACT_RELU | asx.IMPL_NAIVE).float().clone()
    for flags in (asx.IMPL_ROW_GATHER, asx.IMPL_ROW_GATHER | asx.RECOMPACT):
        got = layer.run(x, w, b, flags=base | asx.ACT_RELU | flags).float()
        torch.cuda.synchronize()
        assert layer.device_status() == 0 and shares_k_blocks(layer)
        assert (got - want).norm() <= (2e-5 if f32 else 5e-3) * want.norm()
        assert not got.reshape(Nb, H * W, cout)[:, (mask == 0).cuda()].any()
    layer.close()
