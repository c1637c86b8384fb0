"""The native call behind ha_la_prefill / ha_la_decode and binding.py's own marshalling are the same call: same results
through either, same outputs handed back when the caller brings them, same errors."""
import pytest

pytestmark = pytest.mark.gpu


def _inputs(T=70, hk=2, hv=4, d=128, kda=False):
    import torch

    g = torch.Generator(device="cuda").manual_seed(5)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    u = lambda *s: torch.nn.functional.normalize(r(*s), dim=-1).bfloat16()
    return (u(1, T, hk, d), u(1, T, hk, d), r(1, T, hv, d).bfloat16(), -r(1, T, hv, *([d] if kda else [])).abs(),
            torch.sigmoid(r(1, T, hv)))


@pytest.mark.parametrize("variant", ["gdn", "kda"])
def test_prefill_both_ways(variant):
    import torch
    import paper_2609_32114_b200 as ha

    t = _inputs(kda=variant == "kda")
    o, hT, st, ws = ha.ha_la_prefill(*t, variant=variant)
    o3, hT3, _, _ = ha.ha_la_prefill(*(x[0] for x in t), variant=variant)       # no batch dimension: marshalled in Python
    mine = dict(o=torch.zeros_like(o), hT=torch.zeros_like(hT), workspace=ws, status_word=st)
    o4, hT4, st4, ws4 = ha.ha_la_prefill(*t, variant=variant, **mine)
    assert o4 is mine["o"] and hT4 is mine["hT"] and st4 is st and ws4 is ws
    none = ha.ha_la_prefill(*t, variant=variant, want_hT=False)
    torch.cuda.synchronize()
    assert none[1] is None and int(st.item()) == 0
    assert torch.equal(o, o3.unsqueeze(0)) and torch.equal(o, o4) and torch.equal(hT, hT3) and torch.equal(hT, hT4)
    assert torch.equal(o, none[0])


def test_decode_and_errors():
    import torch
    import paper_2609_32114_b200 as ha
    from paper_2609_32114_b200 import binding

    q, k, v, g, beta = (x[0].contiguous() for x in _inputs(T=3))
    o, new = ha.ha_la_decode(q, k, v, g, beta, None)
    out = torch.empty_like(new)
    o2, new2 = ha.ha_la_decode(q, k, v, g, beta, torch.zeros_like(new), state_out=out)
    torch.cuda.synchronize()
    assert new2 is out and torch.equal(o, o2) and torch.equal(new, new2)
    with pytest.raises(ha.HaLaError) as e:
        ha.ha_la_prefill(*_inputs(d=96))
    assert e.value.status == binding.HA_LA_ERR_UNSUPPORTED
    with pytest.raises(AssertionError):
        t = _inputs()
        ha.ha_la_prefill(t[0].transpose(1, 2), *t[1:])
    with pytest.raises(ValueError):
        ha.ha_la_prefill(*(x.cpu() for x in _inputs()))


@pytest.mark.parametrize("variant,dtype,d,n,hk,hv", [("gdn", "bf16", 128, 1, 1, 1), ("kda", "fp32", 64, 3, 1, 3),
                                                     ("kda", "bf16", 128, 149, 2, 2)])
def test_decode_steps_queued_in_place(variant, dtype, d, n, hk, hv):
    """Eight steps on one state, in place and queued directly behind each other (each step is launched under the tail of
    the one before it), against the oracle's run over the same eight tokens."""
    import numpy as np
    import torch
    import paper_2609_32114_b200 as ha
    from paper_2609_32114_b200 import synth
    from tests import helpers

    steps = 8
    base = synth.WORKLOADS["gdn_varlen" if variant == "gdn" else "kda_8k"]
    w = synth.shrink(base, seq_lens=[steps] * n, hk=hk, hv=hv, dtype=dtype, dk=d, dv=d, h0_std=0.5, gate_shift=-2.0, varlen=True)
    inp = synth.make_inputs(w, seed=231)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    per_step = lambda a, t: [torch.from_numpy(np.ascontiguousarray(a.reshape(n, steps, *a.shape[1:])[:, i])).cuda().to(t)
                             for i in range(steps)]
    q, k, v = (per_step(inp[x], dt) for x in "qkv")
    g, beta = (per_step(inp[x], torch.float32) for x in ("g", "beta"))
    state = torch.from_numpy(inp["h0"]).cuda()
    torch.cuda.synchronize()
    outs = [ha.ha_la_decode(q[i], k[i], v[i], g[i], beta[i], state, variant=variant)[0] for i in range(steps)]
    torch.cuda.synchronize()
    o_ref, h_ref = helpers.run_oracle(inp)
    o = torch.stack(outs, 1).float().cpu().numpy().reshape(o_ref.shape)
    assert helpers.rel_max_err(o, o_ref) <= helpers.TOL[dtype]
    assert helpers.rel_max_err(state.cpu().numpy().astype(np.float64), h_ref) <= 1e-5


@pytest.mark.parametrize("want,given", [(1, True), (0, False), ("numpy", True), ([], False)])
def test_want_hT_is_any_true_value(want, given):
    import numpy as np
    import torch
    import paper_2609_32114_b200 as ha

    t = _inputs()
    ref = ha.ha_la_prefill(*t)
    r = ha.ha_la_prefill(*t, want_hT=np.bool_(True) if want == "numpy" else want)
    torch.cuda.synchronize()
    assert (r[1] is not None) == given and torch.equal(r[0], ref[0])
    if given:
        assert torch.equal(r[1], ref[1])


def test_want_hT_is_not_asked_of_a_call_that_brings_its_own():
    """An object without a truth value is an error where the call has to know (as it is in Python), and only there."""
    import torch
    import paper_2609_32114_b200 as ha

    class NoTruth:
        def __bool__(self):
            raise ValueError("no truth value")

    t = _inputs()
    with pytest.raises(ValueError):
        ha.ha_la_prefill(*t, want_hT=NoTruth())
    mine = torch.empty_like(ha.ha_la_prefill(*t)[1])
    assert ha.ha_la_prefill(*t, hT=mine, want_hT=NoTruth())[1] is mine
    torch.cuda.synchronize()
