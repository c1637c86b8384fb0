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
