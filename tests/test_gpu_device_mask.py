"""Kept-row lists at the limits between the one-pass and the two-pass forms, from a caller's buffer and through
set_mask with a mask that a kernel has just written."""
import numpy as np
import pytest
import torch

import oracle
import paper_2309_06626_b200 as asx
import workloads as wl
from gpu_util import to_dev_bf16

pytestmark = pytest.mark.gpu

ONE_PASS = 192 * 1024                    # largest mask of the one-pass form
ONE_SUB_TILE = 4096 * 8 * 148            # largest mask whose blocks take one 4096-row sub-tile each (148 SMs)


@pytest.mark.parametrize("rows", [1, 4095, 4096, 4097, 16384, 16385, ONE_PASS - 1, ONE_PASS, ONE_PASS + 1, ONE_SUB_TILE, ONE_SUB_TILE + 1])
@pytest.mark.parametrize("offset", [0, 3], ids=["aligned", "unaligned"])
def test_lists_at_the_limits(rows, offset):
    gen = torch.Generator(device="cuda").manual_seed(rows)
    mask = torch.randint(0, 3, (rows + offset,), generator=gen, device="cuda", dtype=torch.uint8)[offset:]
    want = np.flatnonzero(mask.cpu().numpy()).astype(np.int32)
    kept, count, _ = asx.compact_mask(mask)
    assert int(count.item()) == want.size
    assert np.array_equal(kept[:want.size].cpu().numpy(), want)
    layer = asx.MaskedConvLayer(8, 8, 1, 1, 1, 0)
    for m in (mask, torch.flip(mask, (0,)).contiguous()):       # the second one replaces the layer's copy of the first
        layer.set_mask(m)
        assert np.array_equal(layer.kept(), np.flatnonzero(m.cpu().numpy()).astype(np.int32))
    layer.close()


@pytest.mark.parametrize("cin,cout,k", [(64, 128, 3), (32, 48, 3), (128, 64, 1)])
def test_masks_change_from_pass_to_pass(cin, cout, k):
    """mask_from_activation, set_mask and three runs with no synchronisation in between, on rounds of other activations:
    the first run waits for the mask on the device, the second starts in stream order, the third overlaps."""
    spec = wl.LayerSpec("dyn", cin, cout, k, k, 1, k // 2, 24, 31, 5, 0, 1, "relu", wl.BASE_SEED + 900 + cin)
    w, b = wl.make_w(spec), wl.make_b(spec)
    wd, bd = to_dev_bf16(w), torch.from_numpy(b).cuda()
    layer = asx.MaskedConvLayer(cin, cout, k, k, 1, k // 2)
    gen = torch.Generator(device="cuda").manual_seed(7)
    xs = []
    for r in range(6):
        x = torch.relu(torch.randn((spec.Nb, spec.H, spec.W, cin), generator=gen, device="cuda")).to(torch.bfloat16)
        dead = torch.rand((spec.Nb, spec.H, spec.W, 1), generator=gen, device="cuda") < 0.15 * r
        xs.append(x.masked_fill(dead, 0))
    torch.cuda.synchronize()
    got = []
    for x in xs:
        mask = asx.mask_from_activation(x)
        layer.set_mask(mask)
        got.append((mask, [layer.run(x, wd, bd).clone() for _ in range(2)] + [layer.run(x, wd, bd, flags=asx.ACT_RELU | asx.RECOMPACT).clone()]))
    torch.cuda.synchronize()
    assert layer.device_status() == 0
    layer.close()
    for x, (mask, ys) in zip(xs, got):
        xf = x.float().cpu().numpy()
        m = oracle.mask_from_activation(xf.reshape(spec.M, cin))
        assert np.array_equal(mask.reshape(-1).cpu().numpy(), m)
        ref = oracle.masked_conv(xf, w, b, m, 1, k // 2, True).reshape(spec.M, cout)
        for y in ys:
            g = y.float().cpu().numpy().astype(np.float64).reshape(spec.M, cout)
            assert np.linalg.norm(g - ref) / np.linalg.norm(ref) < 5e-3
            assert not g[m == 0].any()


def test_host_mask_is_refused_under_capture():
    """The call fails, the layer keeps its mask and the capture goes on."""
    spec = wl.LayerSpec("capture", 64, 64, 3, 3, 1, 1, 20, 21, 2, 50, 1, "relu", wl.BASE_SEED + 950)
    x, w, b, mask = wl.make_x(spec), wl.make_w(spec), wl.make_b(spec), wl.make_layer_mask(spec)
    xd, wd, bd = to_dev_bf16(x), to_dev_bf16(w), torch.from_numpy(b).cuda()
    layer = asx.MaskedConvLayer(64, 64, 3, 3, 1, 1)
    layer.set_mask(mask)
    want = layer.run(xd, wd, bd).clone()
    pinned = torch.from_numpy(1 - mask).pin_memory()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for refused in (lambda: layer.set_mask(1 - mask), lambda: layer.set_mask(pinned),
                        lambda: layer.set_mask_random(spec.P, 0.5, 1, 3)):
            with pytest.raises(asx.AsxError) as e:
                refused()
            assert e.value.code == 7                         # ASX_ERR_CUDA
        y = layer.run(xd, wd, bd)
    y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    assert np.array_equal(layer.kept(), oracle.kept_list(mask))
    layer.set_mask(1 - mask)                                 # outside it is taken
    assert np.array_equal(layer.kept(), oracle.kept_list(1 - mask))
    del graph
    layer.close()


@pytest.mark.parametrize("per_row", [False, True], ids=["shared", "per_row"])
def test_a_graph_replayed_under_another_mask(per_row):
    """The direct form whose warps share the k range is launched for a number of kept rows: under a mask with as many it
    computes that one, under another it stores nothing but zeros, says so, and stays inside its tensors."""
    spec = wl.LayerSpec("replay", 64, 64, 3, 3, 1, 1, 13, 11, 3, 50, 1, "relu", wl.BASE_SEED + 951)
    x, w, b, mask = wl.make_x(spec), wl.make_w(spec), wl.make_b(spec), wl.make_layer_mask(spec, per_row)
    xd, wd, bd = to_dev_bf16(x), to_dev_bf16(w), torch.from_numpy(b).cuda()
    room = torch.full((spec.M + 256, 64), 7.0, dtype=torch.bfloat16, device="cuda")
    y = room[128:128 + spec.M].view(spec.Nb, spec.Ho, spec.Wo, 64)
    layer = asx.MaskedConvLayer(64, 64, 3, 3, 1, 1)
    layer.set_mask(mask)
    layer.run(xd, wd, bd, y, flags=asx.ACT_RELU | asx.IMPL_DIRECT_K)
    torch.cuda.synchronize()
    assert layer.last_run_form() == asx.FORM_DIRECT_K
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        layer.run(xd, wd, bd, y, flags=asx.ACT_RELU | asx.IMPL_DIRECT_K)
    more, fewer = mask.copy(), mask.copy()
    more[np.flatnonzero(mask == 0)[:5]] = 1
    fewer[np.flatnonzero(mask)[:7]] = 0
    for m in (mask, np.roll(mask, 3), more, fewer, np.zeros_like(mask), np.ones_like(mask), mask):
        layer.set_mask(m)
        y.fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        same = int(m.sum()) == int(mask.sum())
        assert layer.device_status() == (0 if same else 8)
        got, full = y.float().cpu().numpy().reshape(spec.M, 64), m if per_row else np.tile(m, spec.Nb)
        assert not got[full == 0].any()
        if same:
            ref = oracle.masked_conv(x, w, b, m, 1, 1, True).reshape(spec.M, 64)
            assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 5e-3
        else:
            assert (got[full != 0] == 7.0).all()
        assert bool((room[:128] == 7.0).all()) and bool((room[128 + spec.M:] == 7.0).all())
    del graph
    layer.close()
