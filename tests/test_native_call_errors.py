"""torch's C++ errors inside the native half of ha_la_prefill / ha_la_decode reach the caller as Python exceptions."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
import sys, torch
import paper_2609_32114_b200 as ha
from torch._subclasses.fake_tensor import FakeTensorMode
ha.binding._torch_call()     # (a missing extension is not what this is about)
with FakeTensorMode():
    e = lambda *s: torch.empty(*s, dtype=torch.bfloat16, device="cuda")
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    try:
        if sys.argv[1] == "prefill":
            ha.ha_la_prefill(e(1, 70, 2, 128), e(1, 70, 2, 128), e(1, 70, 4, 128), f(1, 70, 4), f(1, 70, 4))
        else:
            ha.ha_la_decode(e(3, 2, 128), e(3, 2, 128), e(3, 4, 128), f(3, 4), f(3, 4), f(3, 4, 128, 128))
    except Exception as x:
        print("raised", type(x).__name__)
"""


@pytest.mark.parametrize("call", ["prefill", "decode"])
def test_tensors_without_storage_or_a_driver(call):
    """CUDA tensors with nothing behind them, in a process of their own: an error, not the end of the process.  (Where there is
    no driver torch throws on the way to the current stream; where there is one the library refuses the null pointers.)"""
    r = subprocess.run([sys.executable, "-c", FAKE, call], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "raised" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])


@pytest.mark.gpu
def test_out_of_memory_keeps_its_type():
    import torch
    import paper_2609_32114_b200 as ha

    T = 8192                                               # needs 630 MB of workspace
    q = torch.nn.functional.normalize(torch.randn(1, T, 1, 128, device="cuda"), dim=-1)
    v = torch.randn(1, T, 32, 128, device="cuda")
    g, beta = -torch.rand(1, T, 32, device="cuda"), torch.rand(1, T, 32, device="cuda")
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    try:
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (400 << 20)) / total)
        with pytest.raises(torch.OutOfMemoryError):
            ha.ha_la_prefill(q, q, v, g, beta)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    o, hT, st, _ = ha.ha_la_prefill(q, q, v, g, beta)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
