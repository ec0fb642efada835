"""The two direct forms of the fused layer (operands gathered into registers; small filter matrices, few rows) against the CPU
oracle at the sizes where it can go wrong: channel counts that are whole 16-byte chunks and words of four bytes,
windows that reach over every edge, column ranges that end inside a 32- or 64-channel block, row counts around the
16-row tiles, lists rebuilt by several blocks."""
import numpy as np
import pytest
import torch

import oracle
import paper_2309_06626_b200 as asx
import workloads as wl
from gpu_util import check_against_oracle, make_problem, to_dev_bf16

pytestmark = pytest.mark.gpu

CASES = [
    # C_in, C_out, k, stride, pad, H, W, Nb, pct, block
    (8, 8, 1, 1, 0, 9, 7, 2, 30, 1),            # one chunk of a group of four
    (64, 32, 1, 1, 0, 16, 16, 2, 40, 2),        # two groups, all loaded first
    (96, 40, 1, 2, 0, 15, 17, 3, 50, 4),        # three groups, columns end inside the block
    (128, 136, 1, 1, 0, 12, 11, 2, 25, 1),      # four groups, three blocks of columns
    (32, 32, 3, 1, 1, 14, 15, 2, 30, 1),        # nine groups, odd count
    (24, 56, 3, 2, 1, 13, 12, 2, 50, 2),        # taps change inside a group
    (3, 64, 7, 2, 3, 32, 30, 2, 50, 4),         # words, leading half word
    (3, 32, 3, 2, 1, 18, 20, 1, 40, 2),
    (4, 24, 5, 2, 2, 14, 16, 2, 30, 1),         # words without a leading half
    (6, 16, 3, 1, 1, 10, 9, 2, 20, 1),
    (2, 48, 4, 2, 1, 18, 22, 2, 25, 4),
    (1, 8, 2, 2, 0, 16, 16, 3, 50, 1),
]


def _spec(c, seed=0):
    cin, cout, k, s, p, H, W, Nb, pct, blk = c
    return wl.LayerSpec("direct", cin, cout, k, k, s, p, H, W, Nb, pct, blk, "relu", wl.BASE_SEED + 8800 + seed)


@pytest.mark.parametrize("per_row", [False, True])
@pytest.mark.parametrize("case", CASES, ids=["-".join(map(str, c)) for c in CASES])
def test_against_the_oracle(case, per_row):
    spec = _spec(case)
    x, w, b, mask = make_problem(spec, per_row=per_row)
    for flags in (asx.ACT_RELU, asx.ACT_SILU | asx.RECOMPACT):
        check_against_oracle(spec, x, w, b, mask, flags | asx.IMPL_DIRECT, form=asx.FORM_DIRECT)
    check_against_oracle(spec, x, w, None, mask, asx.IMPL_DIRECT, form=asx.FORM_DIRECT)


K_CASES = [
    # few rows, the k range shared by eight warps: fewer groups than warps, one more, several turns
    (8, 8, 1, 1, 0, 9, 7, 2, 30, 1),
    (24, 56, 3, 2, 1, 13, 12, 2, 50, 2),
    (32, 40, 3, 1, 1, 7, 5, 1, 20, 1),
    (64, 72, 3, 1, 1, 9, 10, 1, 90, 4),
    (136, 64, 3, 2, 1, 8, 9, 3, 30, 1),
    (256, 48, 1, 1, 0, 11, 11, 2, 0, 1),
    (512, 32, 3, 1, 1, 6, 6, 1, 50, 4),
]


@pytest.mark.parametrize("per_row", [False, True])
@pytest.mark.parametrize("case", K_CASES, ids=["-".join(map(str, c)) for c in K_CASES])
def test_shared_k_range(case, per_row):
    spec = _spec(case, 4)
    x, w, b, mask = make_problem(spec, per_row=per_row)
    for flags in (asx.ACT_RELU | asx.RECOMPACT, asx.ACT_SILU):
        check_against_oracle(spec, x, w, b, mask, flags | asx.IMPL_DIRECT_K, form=asx.FORM_DIRECT_K)
    check_against_oracle(spec, x, w, None, mask, asx.IMPL_DIRECT_K, form=asx.FORM_DIRECT_K)


@pytest.mark.parametrize("impl", [asx.IMPL_DIRECT, asx.IMPL_DIRECT_K], ids=["direct", "direct_k"])
@pytest.mark.parametrize("kept", [0, 1, 15, 16, 17, 33, "all"])
def test_row_counts_around_a_tile(kept, impl):
    spec = _spec((32, 32, 3, 1, 1, 19, 21, 1, 0, 1))
    x, w, b, _ = make_problem(spec)
    mask = np.zeros(spec.P, np.uint8)
    if kept == "all":
        mask[:] = 1
    else:
        mask[np.random.default_rng(kept).permutation(spec.P)[:kept]] = 1
    check_against_oracle(spec, x, w, b, mask, asx.ACT_RELU | asx.RECOMPACT | impl)


@pytest.mark.parametrize("cin,cout,k,s,p,impl,form", [
    (3, 64, 7, 2, 3, asx.IMPL_DIRECT, asx.FORM_DIRECT), (5, 12, 3, 1, 1, asx.IMPL_DIRECT, asx.FORM_DIRECT),
    (32, 36, 1, 1, 0, asx.IMPL_DIRECT, asx.FORM_DIRECT), (8, 32, 3, 1, 1, asx.IMPL_DIRECT, asx.FORM_DIRECT),
    (36, 20, 3, 2, 1, asx.IMPL_DIRECT_K, asx.FORM_DIRECT_K), (128, 64, 3, 1, 1, asx.IMPL_DIRECT_K, asx.FORM_DIRECT_K)])
def test_fp32_storage(cin, cout, k, s, p, impl, form):
    spec = _spec((cin, cout, k, s, p, 17, 19, 2, 40, 2), 1)
    x, w = oracle.tf32_operand(wl.make_x(spec)), oracle.tf32_operand(wl.make_w(spec))
    b, mask = wl.make_b(spec), wl.make_layer_mask(spec)
    layer = asx.MaskedConvLayer(cin, cout, k, k, s, p)
    layer.set_mask(mask)
    y = layer.run(torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda(),
                  flags=asx.ACT_RELU | asx.F32 | impl)
    torch.cuda.synchronize()
    assert layer.last_run_form() == form
    layer.close()
    ref = oracle.masked_conv(x, w, b, mask, s, p, True, storage="fp32")
    got = y.cpu().numpy().astype(np.float64).reshape(ref.shape)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 2e-4
    assert not got.reshape(spec.M, -1)[np.tile(mask, spec.Nb) == 0].any()


@pytest.mark.parametrize("rows_hw", [(64, 64), (65, 64), (130, 127)])
def test_list_rebuilt_beside_the_convolution(rows_hw):
    """Masks of one block, one row more and several blocks of the list."""
    spec = _spec((8, 16, 1, 1, 0, *rows_hw, 1, 45, 1), 2)
    x, w, b, mask = make_problem(spec)
    layer = asx.MaskedConvLayer(8, 16, 1, 1, 1, 0)
    layer.set_mask(mask)
    layer.run(to_dev_bf16(x), to_dev_bf16(w), torch.from_numpy(b).cuda(), flags=asx.RECOMPACT | asx.IMPL_DIRECT)
    assert layer.last_run_form() == asx.FORM_DIRECT
    assert np.array_equal(layer.kept(), oracle.kept_list(mask))
    layer.close()


@pytest.mark.parametrize("impl,form", [(asx.IMPL_DIRECT, asx.FORM_DIRECT), (asx.IMPL_DIRECT_K, asx.FORM_DIRECT_K)], ids=["direct", "direct_k"])
def test_residual(impl, form):
    spec = _spec((64, 72, 1, 1, 0, 11, 13, 2, 30, 1), 3)
    x, w, b, mask = make_problem(spec)
    res = np.random.default_rng(3).standard_normal((spec.Nb, spec.Ho, spec.Wo, 72)).astype(np.float32)
    rd = to_dev_bf16(res)
    layer = asx.MaskedConvLayer(64, 72, 1, 1, 1, 0)
    layer.set_mask(mask)
    layer.set_residual(rd)
    y = layer.run(to_dev_bf16(x), to_dev_bf16(w), torch.from_numpy(b).cuda(), flags=asx.ACT_RELU | impl)
    torch.cuda.synchronize()
    assert layer.last_run_form() == form
    layer.close()
    ref = oracle.masked_conv(x, w, b, mask, 1, 0, False).reshape(spec.M, -1) + rd.float().cpu().numpy().reshape(spec.M, -1)
    ref = np.maximum(ref, 0) * np.tile(mask, spec.Nb)[:, None]
    got = y.float().cpu().numpy().reshape(spec.M, -1)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 5e-3


@pytest.mark.parametrize("impl", [0, asx.IMPL_DIRECT], ids=["default", "direct"])
@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("case", [(3, 32, 3, 2, 1, 18, 20, 2, 40, 2), (3, 64, 7, 2, 3, 32, 30, 2, 50, 4), (6, 16, 3, 1, 1, 10, 9, 2, 20, 1)],
                         ids=["3x3x3", "7x7x3", "3x3x6"])
def test_input_between_two_words(case, offset, impl):
    """Channels that are no whole 16-byte chunks: x at any 2-byte address, the word form at 4-byte ones."""
    spec = _spec(case, 5)
    x, w, b, mask = make_problem(spec)
    room = torch.zeros(x.size + 8, dtype=torch.bfloat16, device="cuda")
    xd = room[offset:offset + x.size].view(x.shape)
    xd.copy_(torch.from_numpy(x))
    assert xd.data_ptr() % 4 == 2 * (offset % 2)
    layer = asx.MaskedConvLayer(spec.C_in, spec.C_out, spec.kh, spec.kw, spec.stride, spec.pad)
    layer.set_mask(mask)
    y = layer.run(xd, to_dev_bf16(w), torch.from_numpy(b).cuda(), flags=asx.ACT_RELU | impl)
    torch.cuda.synchronize()
    assert layer.device_status() == 0
    if offset % 2:
        assert layer.last_run_form() != asx.FORM_DIRECT
    elif impl:
        assert layer.last_run_form() == asx.FORM_DIRECT
    layer.close()
    ref = oracle.masked_conv(x, w, b, mask, spec.stride, spec.pad, True)
    got = y.float().cpu().numpy().astype(np.float64).reshape(ref.shape)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 5e-3
    assert not got.reshape(spec.M, -1)[np.tile(mask, spec.Nb) == 0].any()


@pytest.mark.parametrize("C_in,W,impl", [(8, 1, asx.IMPL_DIRECT_K), (8, 1, asx.IMPL_DIRECT), (3, 2, asx.IMPL_DIRECT)], ids=["direct_k", "chunks", "words"])
def test_images_of_the_largest_height(C_in, W, impl):
    """What a group of chunks or words holds past the window stays outside an image of 32767 rows, whose windows' corners
    are rows -1 .. 32765."""
    spec = _spec((C_in, 16, 3, 2, 1, 32767, W, 1, 30, 1), 6)
    assert spec.P == 16384
    x, w, b, mask = make_problem(spec)
    mask[:3] = mask[-3:] = 1
    check_against_oracle(spec, x, w, b, mask, asx.ACT_RELU | impl, form=asx.FORM_DIRECT if impl == asx.IMPL_DIRECT else asx.FORM_DIRECT_K)


@pytest.mark.parametrize("value", [float("inf"), float("nan")], ids=["inf", "nan"])
@pytest.mark.parametrize("case,f32,impl", [
    ((3, 16, 3, 2, 1, 18, 20, 2, 20, 1), False, asx.IMPL_DIRECT), ((3, 64, 7, 2, 3, 32, 30, 2, 20, 1), False, asx.IMPL_DIRECT),
    ((4, 24, 5, 2, 2, 14, 16, 2, 20, 1), False, asx.IMPL_DIRECT), ((5, 48, 3, 2, 1, 14, 16, 2, 20, 1), False, asx.IMPL_DIRECT),
    ((3, 16, 3, 1, 1, 18, 21, 2, 20, 1), True, asx.IMPL_DIRECT), ((8, 16, 3, 1, 1, 12, 13, 2, 20, 1), False, asx.IMPL_DIRECT),
    ((24, 56, 3, 1, 1, 13, 12, 2, 20, 1), False, asx.IMPL_DIRECT), ((4, 36, 3, 1, 1, 13, 12, 2, 20, 1), True, asx.IMPL_DIRECT),
    ((8, 16, 1, 1, 0, 12, 13, 2, 20, 1), False, asx.IMPL_DIRECT), ((24, 56, 3, 1, 1, 13, 12, 2, 20, 1), False, asx.IMPL_DIRECT_K)],
    ids=lambda v: "-".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_what_is_not_finite_stays_in_its_windows(case, f32, impl, value):
    """Inf or NaN at single pixels: outputs whose window holds one become what the definition says, the others do not see it
    (filters and the other pixels are positive, so that Inf stays Inf)."""
    spec = _spec(case, 7)
    x, w, b, mask = make_problem(spec)
    x, w, b = np.abs(x) + 0.125, np.abs(w) + 0.125, np.abs(b)
    rng = np.random.default_rng(spec.C_in)
    for _ in range(3):                                      # whole pixels: every edge of every window is met
        x[rng.integers(spec.Nb), rng.integers(spec.H), rng.integers(spec.W)] = value
    x[0, spec.H // 2, spec.W // 2] = x[-1, 0, -1] = value
    layer = asx.MaskedConvLayer(spec.C_in, spec.C_out, spec.kh, spec.kw, spec.stride, spec.pad)
    layer.set_mask(mask)
    if f32:
        x, w = oracle.tf32_operand(x), oracle.tf32_operand(w)
        y = layer.run(torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda(), flags=asx.F32 | impl)
    else:
        y = layer.run(to_dev_bf16(x), to_dev_bf16(w), torch.from_numpy(b).cuda(), flags=impl)
    torch.cuda.synchronize()
    assert layer.last_run_form() == (asx.FORM_DIRECT if impl == asx.IMPL_DIRECT else asx.FORM_DIRECT_K)
    layer.close()
    got = y.double().cpu().reshape(spec.M, -1)
    # the definition in which a padding pixel is left out and not multiplied: torch's unfolded windows of a padded image
    xp = torch.nn.functional.pad(torch.from_numpy(x).double().permute(0, 3, 1, 2), (spec.pad,) * 4)
    cols = torch.nn.functional.unfold(xp, (spec.kh, spec.kw), stride=spec.stride)                    # [Nb][C kh kw][P]
    rows = cols.permute(0, 2, 1).reshape(spec.M, spec.C_in * spec.kh * spec.kw)
    wr = torch.from_numpy(w).double().permute(0, 3, 1, 2).reshape(spec.C_out, -1)
    bad = ~torch.isfinite(rows).all(1)
    ref = torch.where(bad[:, None], torch.full((1, 1), value, dtype=torch.float64), rows.nan_to_num(0, 0, 0) @ wr.t() + torch.from_numpy(b).double())
    ref = ref * torch.from_numpy(np.tile(mask, spec.Nb).astype(np.float64))[:, None].nan_to_num()
    keep = torch.from_numpy(np.tile(mask, spec.Nb) != 0)
    assert bad[keep].any() and (~bad)[keep].any()
    assert torch.equal(torch.isnan(got[keep]), torch.isnan(ref[keep])) and torch.equal(torch.isinf(got[keep]), torch.isinf(ref[keep]))
    fine = torch.isfinite(ref) & keep[:, None]
    assert ((got - ref)[fine]).norm() < 5e-3 * ref[fine].norm()
    assert not got[~keep].any()


@pytest.mark.parametrize("pad", [0, 66])
def test_wide_words_and_padding(pad):
    """Columns times channels that no longer fit 16 bits take another form."""
    spec = wl.LayerSpec("wide", 998, 8, 1, 1, 1, pad, 1, 32, 1, 50, 1, "relu", wl.BASE_SEED + 8899)
    x, w, b, mask = make_problem(spec)
    check_against_oracle(spec, x, w, b, mask, asx.ACT_RELU | asx.IMPL_DIRECT, form=asx.FORM_ROW_GATHER_COPY if pad else asx.FORM_DIRECT)
