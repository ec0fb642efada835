"""Row tiles of fewer than 128 rows (the cp.async gather levels its waves) against the oracle: one tile, a part of a
wave, a wave and a bit, tiles at the smallest height, several column tiles, fp32 storage."""
import numpy as np
import pytest
import torch

import oracle
import paper_2309_06626_b200 as asx
import workloads as wl
from gpu_util import to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [
    # C_in, C_out, k, H, W, Nb, sparsity %
    (24, 48, 3, 5, 7, 1, 0), (24, 48, 3, 31, 33, 2, 50), (40, 300, 3, 30, 31, 4, 20), (24, 32, 1, 64, 64, 1, 0),
    (24, 32, 1, 71, 67, 4, 0), (72, 520, 1, 37, 41, 7, 50), (24, 48, 3, 6, 6, 1, 97),
], ids=lambda c: "x".join(str(v) for v in c))
@pytest.mark.parametrize("f32", [False, True], ids=["bf16", "f32"])
def test_levelled_tiles(case, f32):
    cin, cout, k, H, W, Nb, sp = case
    if f32:
        cin += 4                                             # no whole number of 32-channel runs
    spec = wl.LayerSpec("level", cin, cout, k, k, 1, k // 2, H, W, Nb, sp, 1, "relu", wl.BASE_SEED + 700 + W)
    x, w, b, m = wl.make_x(spec), wl.make_w(spec), wl.make_b(spec), wl.make_layer_mask(spec)
    if f32:
        x, w = oracle.tf32_operand(x), oracle.tf32_operand(w)
        xd, wd = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
    else:
        xd, wd = to_dev_bf16(x), to_dev_bf16(w)
    ref = oracle.masked_conv(x, w, b, m, 1, k // 2, True, **({"storage": "fp32"} if f32 else {})).reshape(spec.M, cout)
    layer = asx.MaskedConvLayer(cin, cout, k, k, 1, k // 2)
    bd = torch.from_numpy(b).cuda()
    for mask in (m, torch.from_numpy(m).cuda()):             # the host knows the count, or does not
        layer.set_mask(mask)
        y = layer.run(xd, wd, bd, flags=asx.ACT_RELU | asx.IMPL_ROW_GATHER | (asx.F32 if f32 else 0))
        torch.cuda.synchronize()
        assert layer.device_status() == 0 and layer.last_run_form() == asx.FORM_ROW_GATHER_COPY
        got = y.float().cpu().numpy().astype(np.float64).reshape(spec.M, cout)
        assert np.linalg.norm(got - ref) <= (1e-4 if f32 else 5e-3) * np.linalg.norm(ref)
        assert not got[np.tile(m, Nb) == 0].any()
    layer.close()
