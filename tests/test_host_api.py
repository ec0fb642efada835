"""The host side of the C ABI on a machine without a GPU: csrc/asx_api.cu against a runtime that uses host memory and
launches that only write to a log (fake_cuda.cpp)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2309_06626_b200", "csrc")
DEVICE = 1 << 62                                # an address that the fake runtime takes for device memory


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libasx_fake.so")
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", so, "-x", "c++", os.path.join(CSRC, "asx_api.cu"),
                           os.path.join(CSRC, "mask_from_scores.cpp"), os.path.join(ROOT, "tests", "fake_cuda.cpp")])
    L = ctypes.CDLL(so)
    vp, ci = ctypes.c_void_p, ctypes.c_int
    L.asx_create_layer.argtypes = [ci] * 6 + [ctypes.POINTER(vp)]
    L.asx_set_mask.argtypes = [vp, vp, ctypes.c_int64, vp]
    L.asx_set_input_mask.argtypes = [vp, vp, ctypes.c_int64, vp]
    L.asx_run.argtypes = [vp, vp, ci, ci, ci, vp, vp, vp, ci, vp]
    L.asx_destroy.argtypes = [vp]
    L.fake_log.restype = ctypes.c_char_p
    L.fake_set.argtypes = [ctypes.c_char_p, ci]
    return L


class Layer:
    def __init__(self, L, C_in, C_out, k, stride, pad):
        self.L, self.h = L, ctypes.c_void_p()
        for what, value in (("mallocs_left", -1), ("capturing", 0), ("direct_words", 0), ("patch", 0)):
            self.set(what, value)
        assert L.asx_create_layer(C_in, C_out, k, k, stride, pad, ctypes.byref(self.h)) == 0

    def set(self, what, value):
        self.L.fake_set(what.encode(), value)

    def set_mask(self, mask):
        return self.L.asx_set_mask(self.h, mask if isinstance(mask, int) else mask.ctypes.data, 64 if isinstance(mask, int) else mask.size, None)

    def run(self, Nb, H, W, x=DEVICE, flags=0):
        """Status and the launches of one asx_run."""
        self.L.fake_clear_log()
        rc = self.L.asx_run(self.h, x, Nb, H, W, DEVICE + (1 << 40), None, DEVICE + (2 << 40), flags, None)
        return rc, self.L.fake_log().decode().split("\n")[:-1]


@pytest.fixture
def layer(fake):
    made = []

    def make(*geometry):
        made.append(Layer(fake, *geometry))
        return made[-1]
    yield make
    for m in made:
        fake.asx_destroy(m.h)


IMPL_DIRECT, F32, RECOMPACT, IN_COMPACT = 512, 64, 2, 16


@pytest.mark.parametrize("flags", [0, IMPL_DIRECT])
def test_word_form_takes_word_aligned_inputs_only(layer, flags):
    """x of 3 channels may lie at any 2-byte address; the direct form reads it in 4-byte words."""
    m = layer(3, 32, 3, 2, 1)
    m.set("direct_words", 5)
    assert m.set_mask(np.ones(64, np.uint8)) == 0
    assert m.run(1, 16, 16, flags=flags) == (0, ["direct"])
    rc, launches = m.run(1, 16, 16, x=DEVICE + 2, flags=flags)
    assert rc == 0 and "direct" not in launches and launches[-1] == "row gather"
    assert m.run(1, 16, 16, x=DEVICE + 4, flags=flags) == (0, ["direct"])
    assert m.run(1, 16, 16, x=DEVICE + 4, flags=flags | F32) == (0, ["direct"])


def test_host_mask_is_refused_under_capture(layer):
    """Recorded, the copy would read the caller's memory at every replay."""
    m = layer(24, 32, 3, 1, 1)
    assert m.set_mask(np.ones(64, np.uint8)) == 0
    m.L.fake_clear_log()
    m.set("capturing", 1)
    assert m.set_mask(np.zeros(64, np.uint8)) == 7                      # ASX_ERR_CUDA
    assert m.L.asx_set_mask_random(m.h, ctypes.c_int64(64), ctypes.c_double(0.5), 1, ctypes.c_uint64(1), None) == 7
    assert m.L.fake_log() == b""
    assert m.set_mask(DEVICE) == 0                                      # stays accepted
    m.set("capturing", 0)
    assert m.set_mask(np.zeros(64, np.uint8)) == 0


@pytest.mark.parametrize("flags,first", [(0, "row gather waits for the mask"), (RECOMPACT, "row gather in order")])
def test_failed_run_leaves_the_mask_as_unsettled_as_it_was(layer, flags, first):
    """A kernel may still be writing a device mask: the next launch waits for it, also when a call failed in between."""
    m = layer(24, 32, 3, 1, 1)
    odd = layer(20, 32, 3, 1, 1)                                        # needs a padded copy, whose allocation fails
    for n in (m, odd):
        assert n.set_mask(DEVICE) == 0
    assert m.run(1, 8, 8, flags=flags)[1][-1] == first
    odd.set("mallocs_left", 0)
    assert odd.run(1, 8, 8, flags=flags) == (6, [])                     # ASX_ERR_OOM
    odd.set("mallocs_left", -1)
    assert odd.run(1, 8, 8, flags=flags)[1][-1] == first
    if not flags:                                                       # a launch that waited by itself: the next one is in order
        assert odd.run(1, 8, 8)[1][-1] == "row gather in order"
    assert odd.run(1, 8, 8, flags=flags)[1][-1] == "row gather"


def test_word_form_takes_geometries_whose_columns_fit_its_16_bits():
    """A queued row keeps ix0 * C_in in 16 bits; one that wrapped could look as if it were inside the image."""
    from paper_2309_06626_b200 import build, lib
    build.build()
    plan_direct = lib()["_ZN3asx11plan_directERKNS_8ConvGeomEiPNS_10DirectPlanE"]
    plan_direct.restype = ctypes.c_bool
    rng = np.random.default_rng(5)
    words = 0
    for i in range(4000):
        W, C_in, k, stride = int(2 ** rng.uniform(0, 14.9)), int(2 ** rng.uniform(0, 10)), int(rng.integers(1, 8)), int(rng.integers(1, 4))
        pad = int(rng.integers(0, 256)) if i % 2 else k // 2
        if W + 2 * pad < k:
            continue
        Wo = (W + 2 * pad - k) // stride + 1
        g = (ctypes.c_int * 17)(1, W, W, C_in, 16, k, k, stride, pad, Wo, Wo, stride, pad, k * k * C_in, Wo * Wo, Wo * Wo, Wo * Wo)
        plan = (ctypes.c_int * 6)()
        for elem in (2, 4):
            if not plan_direct(g, elem, plan) or plan[1] == 0:
                continue
            words += 1
            first, last = -pad * C_in, ((Wo - 1) * stride - pad) * C_in
            assert -32768 <= first and last + k * C_in <= 32767, (W, C_in, k, stride, pad)
    assert words > 200


def test_failed_set_mask_leaves_no_mask(layer):
    """A mask that outgrew the buffers took them along when their successors could not be allocated."""
    m = layer(24, 32, 3, 1, 1)
    assert m.set_mask(np.ones(64, np.uint8)) == 0
    for mallocs in range(3):
        m.set("mallocs_left", mallocs)
        assert m.set_mask(np.ones(4096, np.uint8)) == 6                 # ASX_ERR_OOM
        m.set("mallocs_left", -1)
        assert m.run(1, 8, 8) == (3, [])                                # ASX_ERR_NO_MASK
        assert m.set_mask(np.ones(64, np.uint8)) == 0
        assert m.run(1, 8, 8) == (0, ["row gather"])


def test_row_tiles_count_once_they_are_on_the_device(layer):
    """A first run that fails on the way there (no memory, or a capture, whose copies do not happen) leaves nothing behind
    that a later run takes for its tiles."""
    m = layer(64, 32, 3, 1, 1)
    m.set("patch", 1)
    mask = np.ones(256, np.uint8)
    mask[:7] = 0
    assert m.set_mask(mask) == 0
    m.set("mallocs_left", 0)
    assert m.run(1, 16, 16) == (6, [])
    m.set("mallocs_left", -1)
    tiles = (0, ["window patch, 2 tiles, the first: row 0, 128 rows"])
    assert m.run(1, 16, 16) == tiles
    assert m.set_mask(1 - mask) == 0                                    # a shorter table: the buffer stays
    m.set("capturing", 1)
    assert m.run(1, 16, 16)[0] == 7
    m.set("capturing", 0)
    assert m.run(1, 16, 16) == (0, ["window patch, 1 tiles, the first: row 0, 7 rows"])


def test_failed_set_input_mask_leaves_none(layer):
    """The rank table of the input mask before went with its buffer."""
    m = layer(24, 32, 3, 1, 1)
    assert m.set_mask(np.ones(64, np.uint8)) == 0
    assert m.run(1, 8, 8, flags=IN_COMPACT) == (3, [])                  # ASX_ERR_NO_MASK

    def set_input_mask(rows):
        mask = np.ones(rows, np.uint8)
        return m.L.asx_set_input_mask(m.h, mask.ctypes.data, rows, None)
    assert set_input_mask(64) == 0
    assert m.run(1, 8, 8, flags=IN_COMPACT) == (0, ["row gather"])
    for what, value, status in (("mallocs_left", 0, 6), ("capturing", 1, 7)):
        before = -1 if what == "mallocs_left" else 0
        m.set(what, value)
        assert set_input_mask(4096) == status
        m.set(what, before)
        assert m.run(1, 8, 8, flags=IN_COMPACT) == (3, [])
        assert set_input_mask(64) == 0
        assert m.run(1, 8, 8, flags=IN_COMPACT) == (0, ["row gather"])


def test_shared_memory_is_allowed_on_every_device(fake):
    """A kernel's limit is kept per device: each one it is launched on gets it, once, and the most any plan takes."""
    def launch(device):
        fake.fake_clear_log()
        fake.fake_set(b"device", device)
        rc = fake.fake_allow_smem(227 * 1024)
        fake.fake_set(b"device", 0)
        return rc, fake.fake_log().decode()
    fake.fake_set(b"attribute_fails", 1)
    assert launch(1) == (1, "")
    fake.fake_set(b"attribute_fails", 0)
    for device in (0, 1, 63):
        assert launch(device) == (0, f"232448 bytes on device {device}\n")
        assert launch(device) == (0, "")
    for _ in range(2):                                                  # past the devices that are remembered
        assert launch(64) == (0, "232448 bytes on device 64\n")



def test_k_blocks_are_shared_only_where_the_device_tells_its_room():
    """No device here, so no clusters are known to fit; a guess could be more than a device takes at a time."""
    import torch
    if torch.cuda.is_available():
        pytest.skip("there is a device")
    from paper_2309_06626_b200 import build, lib
    build.build()
    plan_fast = lib()["_ZN3asx9plan_fastERKNS_8ConvGeomEixibiPNS_8FastPlanE"]
    plan_fast.restype = ctypes.c_bool
    plan_fast.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong, ctypes.c_int, ctypes.c_bool, ctypes.c_int, ctypes.c_void_p]
    g = (ctypes.c_int * 17)(1, 7, 7, 512, 512, 3, 3, 1, 1, 7, 7, 1, 1, 9 * 512, 49, 49, 49)      # one row tile, 72 k-blocks
    plan = (ctypes.c_int * 12)()
    assert plan_fast(g, 148, 49, 0, True, 2, plan) and plan[5] == 1
