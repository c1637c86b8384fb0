"""Tensors whose type, layout, size or device does not go with q are refused before anything is launched: the kernels take them
by address, and would read or write past them.  With tensors that have nothing behind them, so without a GPU, in one process of
its own."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PREFILL = {
    "h0_bf16": "h0=e(2, 4, 128, 128)", "h0_short": "h0=f(1, 4, 128, 128)", "h0_transposed": "h0=f(2, 4, 128, 128).transpose(0, 1)",
    "h0_cpu": "h0=f(2, 4, 128, 128, device='cpu')", "hT_short": "hT=f(2, 3, 128, 128)", "hT_expanded": "hT=f(1, 4, 128, 128).expand(2, 4, 128, 128)",
    "o_fp32": "o=f(2, 70, 4, 128)", "o_short": "o=e(2, 69, 4, 128)", "o_strided": "o=e(2, 70, 8, 128)[:, :, ::2]",
    "status_cpu": "status_word=torch.zeros(1, dtype=torch.int32, device='cpu')", "status_short": "status_word=torch.zeros(3, dtype=torch.uint8, device='cuda')",
    "workspace_cpu": "workspace=torch.empty(1 << 22, dtype=torch.uint8, device='cpu')",
    "workspace_strided": "workspace=torch.empty(1 << 23, dtype=torch.uint8, device='cuda')[::2]",
    "k_heads": "k=e(2, 70, 1, 128)", "k_tokens": "k=e(2, 69, 2, 128)", "k_more_tokens": "k=e(2, 71, 2, 128)", "k_rows": "k=e(1, 70, 2, 128)",
    "k_dim": "k=e(2, 70, 2, 64)", "v_tokens": "v=e(2, 60, 4, 128)", "g_heads": "g=f(2, 70, 2)", "g_per_channel_of_64": "variant='kda', g=f(2, 70, 4, 64)",
    "beta_heads": "beta=f(2, 70, 3)", "cu_strided": "cu_seqlens=torch.zeros(6, dtype=torch.int32, device='cuda')[::2], batch=1",
}
DECODE = {
    "state_bf16": "state=e(3, 4, 128, 128)", "state_short": "state=f(2, 4, 128, 128)", "state_transposed": "state=f(3, 4, 128, 128).transpose(2, 3)",
    "out_short": "state_out=f(3, 2, 128, 128)", "o_fp32": "o=f(3, 4, 128)", "o_short": "o=e(3, 3, 128)", "q_strided": "q=e(3, 4, 128)[:, ::2]",
    "q_fp16": "q=e(3, 2, 128).half()", "k_heads": "k=e(3, 1, 128)", "k_rows": "k=e(2, 2, 128)", "g_cpu": "g=f(3, 4, device='cpu')",
    "g_heads": "g=f(3, 2)", "beta_bf16": "beta=e(3, 4)", "kda_g_of_gdn": "variant='kda'",
}
CODE = """
import sys, torch
import paper_2609_32114_b200 as ha
from torch._subclasses.fake_tensor import FakeTensorMode
def e(*s, device="cuda"): return torch.empty(*s, dtype=torch.bfloat16, device=device)
def f(*s, device="cuda"): return torch.empty(*s, dtype=torch.float32, device=device)
def prefill(batch=2, **kw):
    a = dict(q=e(batch, 70, 2, 128), k=e(batch, 70, 2, 128), v=e(batch, 70, 4, 128), g=f(batch, 70, 4), beta=f(batch, 70, 4))
    a.update(kw)
    return ha.ha_la_prefill(a.pop("q"), a.pop("k"), a.pop("v"), a.pop("g"), a.pop("beta"), **a)
def decode(**kw):
    a = dict(q=e(3, 2, 128), k=e(3, 2, 128), v=e(3, 4, 128), g=f(3, 4), beta=f(3, 4), state=f(3, 4, 128, 128))
    a.update(kw)
    return ha.ha_la_decode(a.pop("q"), a.pop("k"), a.pop("v"), a.pop("g"), a.pop("beta"), a.pop("state"), **a)
with FakeTensorMode():
    for line in sys.stdin.read().splitlines():
        name, call = line.split("|")
        try:
            eval(call)
            print(name, "returned")
        except Exception as x:
            print(name, type(x).__name__, str(x).splitlines()[0][:200])
"""


@pytest.fixture(scope="module")
def outcomes():
    calls = [f"prefill.{n}|prefill({c})" for n, c in PREFILL.items()] + [f"decode.{n}|decode({c})" for n, c in DECODE.items()]
    r = subprocess.run([sys.executable, "-c", CODE], input="\n".join(calls), cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return dict(line.split(" ", 1) for line in r.stdout.splitlines())


@pytest.mark.parametrize("name", [f"prefill.{n}" for n in PREFILL] + [f"decode.{n}" for n in DECODE])
def test_refused(outcomes, name):
    what = name.split(".")[1].split("_")[0]
    what = {"out": "state_out", "status": "status_word", "cu": "cu_seqlens", "kda": "g"}.get(what, what)
    assert outcomes[name].startswith(f"ValueError {what}:"), outcomes[name]


@pytest.mark.gpu
def test_what_goes_with_q_is_taken():
    """More rows than q has in a batch of one, states and outputs of another shape with the same numbers, a longer status word, a
    pinned host state: the results of the plain call."""
    import torch
    import paper_2609_32114_b200 as ha

    gen = torch.Generator(device="cuda").manual_seed(9)
    r = lambda *s: torch.randn(s, generator=gen, device="cuda")
    u = lambda *s: torch.nn.functional.normalize(r(*s), dim=-1).bfloat16()
    q, k, v, g, beta = u(1, 90, 2, 128), u(1, 90, 2, 128), r(1, 90, 4, 128).bfloat16(), -r(1, 90, 4).abs(), torch.sigmoid(r(1, 90, 4))
    h0 = 0.1 * r(1, 4, 128, 128)
    short = lambda t: t[:, :70].contiguous()
    o, hT, _, _ = ha.ha_la_prefill(short(q), short(k), short(v), short(g), short(beta), h0=h0)
    status = torch.zeros(1, dtype=torch.int64, device="cuda")
    for kw in (dict(h0=h0), dict(h0=h0.flatten(), hT=torch.empty(5 * 16384, device="cuda")), dict(h0=h0.cpu().pin_memory(), status_word=status)):
        o2, hT2, st, _ = ha.ha_la_prefill(short(q), k, short(v), g, beta, **kw)
        torch.cuda.synchronize()
        assert int(st.item()) == 0 and torch.equal(o, o2) and torch.equal(hT.flatten(), hT2.flatten()[:65536])
