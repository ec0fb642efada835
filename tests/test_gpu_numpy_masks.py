"""Masks given as numpy arrays: contiguous bytes take the native path, everything else the wrapper's conversions, with the same result."""
import numpy as np
import pytest

import paper_2309_06626_b200 as asx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["bytes", "2d", "read only", "strided", "fortran", "bool", "int64", "one value"])
def test_numpy_masks(kind):
    rng = np.random.default_rng(5)
    want = (rng.random(144) < 0.5).astype(np.uint8)
    mask = {"bytes": want.copy(), "2d": want.reshape(12, 12), "read only": want.copy(), "strided": np.repeat(want, 2)[::2],
            "fortran": np.asfortranarray(want.reshape(12, 12)), "bool": want.astype(bool), "int64": want.astype(np.int64),
            "one value": np.array(1, np.uint8)}[kind]
    if kind == "read only":
        mask.setflags(write=False)
    if kind == "one value":
        want = np.ones(1, np.uint8)
    layer = asx.MaskedConvLayer(8, 8, 1, 1, 1, 0)
    layer.set_mask(mask)
    assert np.array_equal(layer.kept(), np.flatnonzero(want))
    layer.close()


def test_an_empty_mask_is_refused():
    layer = asx.MaskedConvLayer(8, 8, 1, 1, 1, 0)
    with pytest.raises(asx.AsxError):
        layer.set_mask(np.zeros(0, np.uint8))
    layer.close()
