"""The native side of the binding (csrc/torch_binding.cpp)."""
import subprocess
import sys

import pytest

CALLS = {
    "set_mask": "layer.set_mask(t.to(torch.uint8), stream=stream)",
    "run": "layer.run(t.bfloat16().reshape(1, 2, 2, 8), torch.zeros(8, 1, 1, 8, dtype=torch.bfloat16, device=dev), stream=stream)",
    "mask_from_activation": "asx.mask_from_activation(t.bfloat16().reshape(4, 8), stream=stream)",
    "compact_mask": "asx.compact_mask(t.to(torch.uint8), stream=stream)",
}
PROGRAM = """
import torch
import paper_2309_06626_b200 as asx
class stream: cuda_stream = 0
dev = %r
layer = asx.MaskedConvLayer(8, 8, 1, 1, 1, 0)
def call(t):
    try:
        %s
    except (RuntimeError, ValueError) as e:
        print("refused", type(e).__name__)
    return t
torch.vmap(call)(torch.ones(2, 32, device=dev))
"""


def _refuses(call, dev):
    p = subprocess.run([sys.executable, "-c", PROGRAM % (dev, CALLS[call])], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "refused" in p.stdout, p.stderr[-800:]


def test_a_tensor_without_storage_raises_on_the_host():
    """torch throws for it; the exception must not leave the extension as a C++ one, which ends the process."""
    _refuses("set_mask", "cpu")


@pytest.mark.gpu
@pytest.mark.parametrize("call", CALLS)
def test_a_tensor_without_storage_raises(call):
    _refuses(call, "cuda")


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["run", "set_mask", "mask_from_activation", "compact_mask"])
def test_other_threads_run_during_a_call(call):
    """The interpreter's lock is given up around the call into the library: with switches on request only, another thread
    gets it nowhere else in this loop."""
    import threading
    import time
    import torch
    import paper_2309_06626_b200 as asx
    layer = asx.MaskedConvLayer(8, 8, 1, 1, 1, 0)
    mask = torch.ones(64, dtype=torch.uint8, device="cuda")
    layer.set_mask(mask)
    x, w = torch.ones(1, 8, 8, 8, dtype=torch.bfloat16, device="cuda"), torch.ones(8, 1, 1, 8, dtype=torch.bfloat16, device="cuda")
    y = layer.run(x, w)
    todo = {"run": lambda: layer.run(x, w, None, y), "set_mask": lambda: layer.set_mask(mask), "mask_from_activation": lambda: asx.mask_from_activation(x),
            "compact_mask": lambda: asx.compact_mask(mask)}[call]
    todo()
    turns, stop = [0], threading.Event()

    def other():
        while not stop.is_set():
            turns[0] += 1
            time.sleep(0)
    before = sys.getswitchinterval()
    thread = threading.Thread(target=other)
    sys.setswitchinterval(1000)
    try:
        thread.start()
        first = turns[0]
        for _ in range(2000):
            todo()
        got = turns[0] - first
    finally:
        sys.setswitchinterval(before)
        stop.set()
        thread.join()
    torch.cuda.synchronize()
    layer.close()
    assert got > 10, got
