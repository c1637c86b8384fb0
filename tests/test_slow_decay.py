"""What a state carries across a whole run or chunk: inputs that decay so slowly that the products with the incoming state make up much of the
result.  The kernels against the fp64 oracle on them (on a GPU); and, on the CPU, that the oracle without such a product is far outside
the tolerance on the same inputs, so that the comparison would see one that is left out."""
import numpy as np
import pytest

from paper_2609_32114_b200 import synth
from tests import helpers

W = synth.WORKLOADS
STEP, CHUNK = 128, 64                                      # tokens of a step (d = 128) and of a chunk (d = 64)


def _inputs(variant, lens, hv, d, dtype, seed, keys="unit"):
    w = synth.shrink(W["gdn_varlen"] if variant == "gdn" else W["kda_8k"], seq_lens=lens, hk=1, hv=hv, dtype=dtype, dk=d, dv=d, gate_shift=-8.0,
                     h0_std=0.05, varlen=len(lens) > 1)
    inp = synth.make_inputs(w, seed=seed)
    if keys == "unit":
        inp["beta"] *= 0.25                                # (little is erased, either)
    else:                                                  # eight keys over and over, beta |k|^2 up to 1.8
        k = (1.8 ** 0.5 * inp["k"][np.arange(inp["T"]) * 5 % 8]).astype(np.float32)
        inp["k"] = synth.round_to_bf16(k) if dtype == "bf16" else k
    return inp


def _pieces(inp, unit, per_piece):
    """Token ranges (start, end) per sequence: pieces of per_piece(number of units) units of `unit` tokens."""
    out = []
    for n, length in enumerate(inp["seq_lens"]):
        units = -(-length // unit)
        size = max(1, per_piece(units)) * unit
        out.append([(int(inp["cu_seqlens"][n]) + a, int(inp["cu_seqlens"][n]) + min(a + size, length)) for a in range(0, length, size)])
    return out


def _oracle_on(inp, ranges, h0):
    import oracle

    take = lambda a: np.concatenate([a[s:e] for s, e in ranges])
    cu = np.cumsum([0] + [e - s for s, e in ranges]).astype(np.int32)
    o, hT, _ = oracle.recurrent(take(inp["q"]), take(inp["k"]), take(inp["v"]), take(inp["g"]), take(inp["beta"]), variant=inp["workload"].variant,
                                h0=h0, cu_seqlens=cu)
    return np.split(o, cu[1:-1]), hT


def _without(inp, seqs, keep=None):
    """Per sequence, piece 1 on: how far o of the piece (all V-heads, the worst of them and the least) is off, in tolerances, where the piece
    before it handed on b (what it has from no state) plus `keep` of the state that entered it, instead of Phi h + b."""
    o_ref, _ = helpers.run_oracle(inp)
    top, tol = np.abs(o_ref).max(), helpers.TOL[inp["workload"].dtype]
    for n, ranges in enumerate(seqs):
        if len(ranges) < 3:
            continue
        zero = np.zeros((len(ranges), inp["workload"].hv, inp["workload"].dk, inp["workload"].dv), np.float32)
        _, b = _oracle_on(inp, ranges, zero)
        true, h = [], inp["h0"][n:n + 1]
        for r in ranges:                                   # the states between
            true.append(h)
            _, h = _oracle_on(inp, [r], h.astype(np.float32))
        starts = b[1:-1]                                   # of pieces 2 .. : what piece s = 1 .. has from no state
        if keep is not None:
            starts = starts + np.stack([keep(inp, ranges[s], true[s][0]) for s in range(1, len(ranges) - 1)])
        o, _ = _oracle_on(inp, ranges[2:], starts.astype(np.float32))
        for (s, e), got in zip(ranges[2:], o):
            yield np.abs(got - o_ref[s:e]).max(axis=(0, 2)) / (tol * top)


# ---- start states of runs (d = 128): h_{s+1} = Phi_s h_s + b_s.  148 SMs: 8 columns to a CTA up to 9 (sequence, V-head) pairs, 16 up to 18,
# one group of warps beyond.  `runs` forced, or None for the rule's choice, `least` runs or more, so that all three buffers of Phi are used three times (from
# 19 pairs on there are two, and six products do).
RUNS = [(9, [1900], 8, 8), (10, [1900], 8, 8), (18, [1900], 8, 8), (19, [1900], 8, 8), (5, [1900, 390], 8, 8), (10, [1000, 0, 1900], 8, 8), (19, [700], 4, 4),
        (2, [8200], None, 12), (2, [8200, 1, 130, 0, 64], None, 12)]


def _runs(inp, runs):
    return _pieces(inp, STEP, lambda steps: -(-steps // runs))


def _rule(inp, variant, hv):
    import paper_2609_32114_b200 as ha

    lens = inp["seq_lens"]
    kw = dict(batch=1, seqlen=inp["T"])
    if len(lens) > 1:
        kw.update(num_seqs=len(lens), cu_seqlens=256, max_seqlen=max(lens))
    return ha.ha_la_prefill_num_runs(ha.make_args(variant=variant, dtype="bf16", hk=1, hv=hv, dk=128, dv=128, **kw))


@pytest.mark.gpu
@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("hv,lens,runs,least", RUNS)
def test_start_states(variant, hv, lens, runs, least, monkeypatch):
    if runs:
        monkeypatch.setenv("HA_LA_TC_SEGMENTS", str(runs))
    inp = _inputs(variant, lens, hv, 128, "bf16", 409)
    assert _rule(inp, variant, hv) >= least
    helpers.check_parity(inp)


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("hv,lens,runs,least", RUNS)
def test_start_states_are_seen(variant, hv, lens, runs, least, monkeypatch):
    if runs:
        monkeypatch.setenv("HA_LA_TC_SEGMENTS", str(runs))
    inp = _inputs(variant, lens, hv, 128, "bf16", 409)
    got = _rule(inp, variant, hv)
    assert got >= least
    off = list(_without(inp, _runs(inp, got)))
    assert len(off) >= (least if runs is None else 2 * runs // 3) - 2 and min(x.min() for x in off) > 10


# ---- d = 64: a chunk's affine map h' = M h + b, o = N h + c.  Slices of 4, 8 and 16 channels in the sequential kernel (up to 9, 18 and more
# (sequence, V-head) pairs), with chunks enough that every stage is used three times.
CHUNKS = [(3, [700]), (12, [600]), (20, [450]), (10, [230, 400]), (7, [64, 0, 500])]


@pytest.mark.gpu
@pytest.mark.parametrize("keys", ["unit", "repeated"])
@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("hv,lens", CHUNKS)
def test_chunks_d64(variant, dtype, hv, lens, keys):
    helpers.check_parity(_inputs(variant, lens, hv, 64, dtype, 419, keys))


@pytest.mark.parametrize("keys", ["unit", "repeated"])
@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("hv,lens", CHUNKS)
def test_chunks_d64_are_seen(variant, dtype, hv, lens, keys):
    """... without M h, and with the decay alone for M."""
    inp = _inputs(variant, lens, hv, 64, dtype, 419, keys)
    seqs = _pieces(inp, CHUNK, lambda units: 1)

    def decay(inp, r, h):
        g = np.exp(inp["g"][r[0]:r[1]].astype(np.float64).sum(axis=0))
        return h * (g[:, None, None] if variant == "gdn" else g[:, :, None])

    for keep in (None, decay):
        off = list(_without(inp, seqs, keep))
        assert len(off) >= 5 and min(x.min() for x in off) > 1.5, keep
