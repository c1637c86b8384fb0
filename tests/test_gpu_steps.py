"""The tensor-core kernels against the fp64 oracle, where their indexing can go wrong: lengths around a step of 128 tokens and
a block of 16, sequences cut into runs (short ones into empty runs), more work items than work groups."""
import pytest

from paper_2609_32114_b200 import synth
from tests import helpers

pytestmark = pytest.mark.gpu
W = synth.WORKLOADS


def _inputs(variant, lens, packed, hk, hv, seed, **kw):
    base = W["gdn_varlen"] if variant == "gdn" else W["kda_8k"]
    w = synth.shrink(base, seq_lens=lens, hk=hk, hv=hv, h0_std=0.05, varlen=packed, **dict(dict(gate_shift=-1.0), **kw))
    return synth.make_inputs(w, seed=seed)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("lens,packed,hk,hv", [([1], False, 1, 1), ([127, 127], False, 1, 2), ([129], False, 2, 4),
                                               ([128, 0, 15, 257, 17], True, 2, 2), ([112] * 5, True, 1, 3)])
def test_step_edges(variant, lens, packed, hk, hv):
    helpers.check_parity(_inputs(variant, lens, packed, hk, hv, 311 + len(lens)), scale=0.5)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("runs", [1, 2, 4, 8])
def test_runs_of_a_sequence(variant, runs, monkeypatch):
    monkeypatch.setenv("HA_LA_TC_SEGMENTS", str(runs))
    helpers.check_parity(_inputs(variant, [1025], False, 1, 2, 331, gate_shift=5.0), scale=0.5)
    helpers.check_parity(_inputs(variant, [700, 0, 129, 1], True, 1, 2, 337, gate_shift=3.0))


@pytest.mark.parametrize("variant,hk,hv,lens", [("gdn", 16, 16, [2560]), ("gdn", 8, 16, [1300, 2500]), ("kda", 16, 16, [2100, 1900])])
def test_every_group_takes_several_items(variant, hk, hv, lens):
    helpers.check_parity(_inputs(variant, lens, len(lens) > 1, hk, hv, 347, gate_shift=2.0))


@pytest.mark.parametrize("log_gate", [-3.0, -9.0, -90.0, -500.0])
def test_kda_strong_decay(log_gate):
    """Channels whose decay between two block boundaries is inside, around and far outside the range that the scaled
    operands of a block hold; the last clamps the kept exponents too."""
    inp = _inputs("kda", [300], False, 1, 2, 353)
    for tok in (5, 15, 16, 37, 70, 71, 131, 200):
        inp["g"][tok, :, ::7] = log_gate
    inp["g"][140:190, :, 3::11] = log_gate
    helpers.check_parity(inp)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("runs,lens,hv", [(8, [1500, 100, 1, 0, 700, 130, 900], 8), (4, [0, 3000, 129, 1, 513], 16), (2, [5, 2000], 2)])
def test_runs_in_place(variant, runs, lens, hv, monkeypatch):
    """h0 = hT with sequences cut into runs, some shorter than the number of runs (their last runs are empty and have the end
    state at once), with more CTAs than SMs in all but the last case: the same call out of place, bit for bit, every time."""
    import torch
    import paper_2609_32114_b200 as ha

    monkeypatch.setenv("HA_LA_TC_SEGMENTS", str(runs))
    inp = _inputs(variant, lens, True, hv // 2, hv, 359)
    d = helpers.to_device(inp)
    a, keep = ha.prepare_args(d["q"], d["k"], d["v"], d["g"], d["beta"], variant=variant, h0=d["h0"],
                              cu_seqlens=d["cu_seqlens"], max_seqlen=d["max_seqlen"])
    assert ha.ha_la_prefill_num_launches(a) == 5           # plan, chunk-local, states only, start states, outputs
    assert ha.ha_la_prefill_raw(a, torch.cuda.current_stream().cuda_stream) == 0
    for _ in range(8):
        state = d["h0"].clone()
        o, hT, st, _ = ha.ha_la_prefill(d["q"], d["k"], d["v"], d["g"], d["beta"], variant=variant, h0=state, hT=state,
                                        cu_seqlens=d["cu_seqlens"], max_seqlen=d["max_seqlen"], workspace=keep["workspace"])
        torch.cuda.synchronize()
        assert hT is state and int(st.item()) == 0 and int(keep["status_word"].item()) == 0
        assert torch.equal(o, keep["o"][0]) and torch.equal(state, keep["hT"])
    helpers.check_parity(inp)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("fp32", 128)])
@pytest.mark.parametrize("seqs", [1, 2])
def test_packed_batch_without_a_token(variant, dtype, d, seqs):
    """Through the C ABI (torch has no pointers for empty tensors): a packed batch of empty sequences hands the states on.  With
    one sequence there are no chunk slots, so nothing runs between the plan kernel and the state-passing kernel."""
    import torch
    import paper_2609_32114_b200 as ha

    any_ = torch.rand(4096, device="cuda") + 1.0           # in the place of q, k, v, g, beta, o: no token of them is touched
    cu = torch.zeros(seqs + 1, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    h0 = torch.randn(4, 3, d, d, device="cuda")[:seqs]     # (room behind the states, the workspace and any_ for the numbers below)
    p = any_.data_ptr()
    for start in (h0, None):
        hT_all = torch.full((4, 3, d, d), float("nan"), device="cuda")
        hT = hT_all[:seqs]
        a = ha.make_args(variant=variant, dtype=dtype, batch=1, seqlen=0, hk=1, hv=3, dk=d, dv=d, num_seqs=seqs, q=p, k=p, v=p, g=p,
                         beta=p, o=p, h0=0 if start is None else start.data_ptr(), cu_seqlens=cu.data_ptr(), hT=hT.data_ptr(),
                         status_word=status.data_ptr())
        need = ha.ha_la_prefill_workspace_bytes(a)
        # were the tables read before they are written: sequence, token, length and slot one, which shows as a wrong state
        ws = torch.ones((need + (4 << 20)) // 4, dtype=torch.int32, device="cuda")
        a.workspace, a.workspace_bytes = (ws.data_ptr() + 255) // 256 * 256, need
        assert ha.ha_la_prefill_raw(a, torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and torch.equal(hT, torch.zeros_like(h0) if start is None else start)
        assert bool(hT_all[seqs:].isnan().all())


@pytest.mark.parametrize("hk,hv,lens", [(32, 32, [4500]), (16, 32, [4097]), (3, 9, [9000, 5, 4000])])
def test_gdn_units_of_all_groups_in_turn(hk, hv, lens):
    """Six to eight units (a step of a V-head) for every CTA of the chunk-local kernel: each of its three groups takes several, with
    both stages of tiles and both halves of tensor memory under each, alone or as one of several V-heads of a q/k head."""
    helpers.check_parity(_inputs("gdn", lens, len(lens) > 1, hk, hv, 367, gate_shift=2.0), pairs=[(0, 0), (0, hv // 2), (len(lens) - 1, hv - 1)])


@pytest.mark.parametrize("log_gate", [-3.0, -9.0, -90.0, -500.0])
def test_gdn_strong_decay(log_gate):
    """Decays between blocks of 16 tokens from moderate to far below the smallest fp32 number, at and around their edges."""
    inp = _inputs("gdn", [300], False, 1, 2, 373)
    for tok in (5, 15, 16, 37, 70, 71, 112, 131, 200):
        inp["g"][tok] = log_gate
    inp["g"][140:190] = log_gate / 8
    helpers.check_parity(inp)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("first,length", [(0, 16), (16, 40), (64, 96), (112, 128), (128, 160)])
def test_overflow_in_any_block_is_reported(variant, first, length):
    """Sixteen strongly correlated keys far outside the stable range, in one block of the solve: whichever it is, also where the
    sequence ends behind it, the status word says so."""
    import numpy as np

    inp = _inputs(variant, [length], False, 1, 1, 379, gate_shift=-6.0)
    inp["g"][:] = 0.0
    inp["k"][first:first + 16] = synth.round_to_bf16((60.0 * inp["k"][first] + 0.0 * inp["k"][first:first + 16]).astype(np.float32))
    inp["beta"][first:first + 16] = 1.0
    assert helpers.run_gpu(inp)[2] == 6


@pytest.mark.parametrize("variant,tokens", [("gdn", 6000), ("gdn", 6016), ("kda", 8200)])
def test_many_runs(variant, tokens):
    """Sequences that the rule cuts into twelve runs and more; the last run full or ragged."""
    import paper_2609_32114_b200 as ha

    inp = _inputs(variant, [tokens], False, 1, 2, 383, gate_shift=5.0)
    a = ha.make_args(variant=variant, dtype="bf16", batch=1, seqlen=tokens, hk=1, hv=2, dk=128, dv=128)
    assert ha.ha_la_prefill_num_runs(a) >= 12
    helpers.check_parity(inp)


def _four_alike(variant, length, where, size):
    """One head of `length` tokens, no decay, beta = 0 but for the tokens `where`, whose keys are alike with |k|^2 = size: the
    inverse has size (size - 1)^n between tokens n + 1 apart in that list, the identity elsewhere."""
    import numpy as np

    inp = _inputs(variant, [length], False, 1, 1, 389, gate_shift=-6.0)
    inp["g"][:] = 0.0
    inp["beta"][:] = 0.0
    inp["beta"][list(where)] = 1.0
    key = np.zeros(128, np.float32)
    key[::8] = (size / 16) ** 0.5
    inp["k"][:, :, ::8] = 0.0                              # (all others at right angles to them)
    inp["k"][list(where)] = synth.round_to_bf16(key)
    return inp


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("level", ["diagonal", "1", "2", "3", "A"])
def test_overflow_is_reported_from_every_block(variant, level):
    """The one value that leaves the fp16 range in a block of the inverse on the diagonal, next to it (level 1), two blocks from it
    (level 2), of A T between the halves (level 3), or of A itself, everything else far inside: reported whichever block it is, to
    the end of a step and where the sequence ends behind it.  With smaller keys nothing is."""
    first = lambda b: 16 * b
    if level == "diagonal":
        at = [(first(b), first(b) + 5, first(b) + 9, first(b) + 15) for b in range(8)]
    elif level == "1":
        at = [(first(b) + 2, first(b) + 9, first(b + 1) + 3, first(b + 1) + 12) for b in (0, 2, 4, 6)]
    elif level == "2":
        at = [(first(J) + 1, first(J) + 8, first(I) + 4, first(I) + 13) for h in (0, 4) for I in (h + 2, h + 3) for J in (h, h + 1)]
    elif level == "3":
        at = [(first(J) + 1, first(J) + 6, first(J) + 15, first(I) + 7) for I in range(4, 8) for J in range(4)]
    else:
        at = [(first(J) + 3, first(I) + 10) for I in range(8) for J in range(I)]
    big, small = (90000.0, 40000.0) if level == "A" else (50.0, 25.0)   # 50 49^2 = 120050 > 65504 > 25 24^2
    for where in at:
        for length in {where[-1] + 1, 128, 150}:
            assert helpers.run_gpu(_four_alike(variant, length, where, big))[2] == 6, (where, length)
            assert helpers.run_gpu(_four_alike(variant, length, where, small))[2] == 0, (where, length)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("hv,lens", [(4, [1100]), (5, [1100]), (1, [900, 0, 130, 1]), (1, [900, 0, 130, 1, 513]), (2, [900, 600])])
@pytest.mark.parametrize("runs", [2, 8])
def test_start_states_on_both_sides_of_four_pairs(variant, hv, lens, runs, monkeypatch):
    """Four (sequence, V-head) pairs and fewer have their start states from another instance than five and more."""
    monkeypatch.setenv("HA_LA_TC_SEGMENTS", str(runs))
    helpers.check_parity(_inputs(variant, lens, len(lens) > 1, 1, hv, 397, gate_shift=4.0))


@pytest.mark.parametrize("pairs", [9, 10, 18, 19])
@pytest.mark.parametrize("runs", [2, 4, 8])
def test_start_states_of_every_instance(pairs, runs, monkeypatch):
    """Both sides of the numbers of pairs where the start states' CTAs change (148 SMs: 8 columns up to 9 pairs, 16 up to 18, one group of
    warps beyond), without a product and with two and six of them, the last runs of the shorter sequence empty."""
    monkeypatch.setenv("HA_LA_TC_SEGMENTS", str(runs))
    lens = [1100] if pairs % 2 else [1100, 390]
    helpers.check_parity(_inputs("gdn", lens, len(lens) > 1, 1, pairs // len(lens), 401, gate_shift=4.0))
