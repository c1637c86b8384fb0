"""Calls on a stream that is not torch's current one, while the current one is behind: what the call allocates and clears goes in the
order of the call's stream."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def behind():
    """The current stream has some fifty milliseconds of waiting to do; the other stream."""
    import torch

    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)
    return side


def _inputs(lead):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(3)
    r = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    u = lambda *s: torch.nn.functional.normalize(r(*s), dim=-1).bfloat16()
    return u(*lead, 128, 1, 128), u(*lead, 128, 1, 128), r(*lead, 128, 2, 128).bfloat16(), -r(*lead, 128, 2).abs(), torch.sigmoid(r(*lead, 128, 2))


@pytest.mark.parametrize("lead", [(1,), ()], ids=["native", "marshalled"])
def test_the_status_word_is_cleared_before_the_kernels(lead, request):
    import torch
    import paper_2609_32114_b200 as ha

    q, k, v, g, beta = _inputs(lead)
    k[..., 16:32, :, :] = 60.0 * k[..., 16:17, :, :]       # far outside the stable range: reported
    g.zero_()
    beta.fill_(1.0)
    ha.ha_la_prefill(q, k, v, g, beta)                     # (the kernels are loaded: that waits for the device)
    side = request.getfixturevalue("behind")
    st = ha.ha_la_prefill(q, k, v, g, beta, stream=side.cuda_stream)[2]
    side.synchronize()
    assert not torch.cuda.current_stream().query()         # (the current stream has not come to anything queued on it)
    torch.cuda.synchronize()
    assert int(st.item()) == 6


@pytest.mark.parametrize("lead", [(1,), ()], ids=["native", "marshalled"])
def test_outputs_are_not_what_the_current_stream_is_still_writing(lead, request):
    """Freed tensors of the current stream, with a fill of theirs still queued: the call's outputs must not lie where they did."""
    import torch
    import paper_2609_32114_b200 as ha

    t = _inputs(lead)
    ref = ha.ha_la_prefill(*t)
    d = [x.reshape(-1, *x.shape[len(lead) + 1:])[:3].contiguous() for x in t]
    step = ha.ha_la_decode(*d, None)

    def leave_fills():
        for x in [torch.empty_like(x) for x in (*ref, *step)]:
            x.fill_(7)

    leave_fills()                                          # (loads what it needs: that waits for the device)
    side = request.getfixturevalue("behind")
    leave_fills()
    o, hT, st, _ = ha.ha_la_prefill(*t, stream=side.cuda_stream)
    o1, s1 = ha.ha_la_decode(*d, None, stream=side.cuda_stream)
    side.synchronize()
    assert not torch.cuda.current_stream().query()
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and torch.equal(o, ref[0]) and torch.equal(hT, ref[1])
    assert torch.equal(o1, step[0]) and torch.equal(s1, step[1])


def test_named_current_stream_and_default_stream():
    import torch
    import paper_2609_32114_b200 as ha

    t = _inputs((1,))
    ref = ha.ha_la_prefill(*t)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        here = ha.ha_la_prefill(*t, stream=side.cuda_stream)
        there = ha.ha_la_prefill(*t, stream=0)
    torch.cuda.synchronize()
    for r in (here, there):
        assert int(r[2].item()) == 0 and torch.equal(r[0], ref[0]) and torch.equal(r[1], ref[1])
    assert torch.cuda.current_stream().cuda_stream == 0
