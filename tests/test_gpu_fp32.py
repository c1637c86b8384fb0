"""The two-kernel fp32 path against the fp64 oracle, where its indexing can go wrong: lengths around a chunk, empty and
one-token sequences, packed and equal-length rows, both slice widths of the sequential kernel (few and many heads)."""
import pytest

from paper_2609_32114_b200 import synth
from tests import helpers

pytestmark = pytest.mark.gpu
W = synth.WORKLOADS


@pytest.mark.parametrize("variant", ["gdn", "kda"])
@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("fp32", 128), ("bf16", 64)])
@pytest.mark.parametrize("lens,packed,hk,hv", [([1], False, 1, 1), ([63, 63], False, 1, 2), ([129], False, 2, 2),
                                               ([64, 0, 65, 1, 130], True, 2, 4), ([70] * 7, True, 4, 8)])
def test_fp32_path(variant, dtype, d, lens, packed, hk, hv):
    base = W["gdn_varlen"] if variant == "gdn" else W["kda_8k"]
    w = synth.shrink(base, seq_lens=lens, hk=hk, hv=hv, dtype=dtype, dk=d, dv=d, gate_shift=-1.0, h0_std=0.05, varlen=packed)
    helpers.check_parity(synth.make_inputs(w, seed=211 + len(lens)), scale=0.5)


def test_fp32_kda_strong_decay_inside_a_block():
    """Log-gates of -90 in a few channels: the decay inside a 16-token block leaves the range of a factored product."""
    w = synth.shrink(W["kda_8k"], seq_lens=[150], hk=1, hv=2, dtype="fp32")
    inp = synth.make_inputs(w, seed=223)
    for tok in (5, 37, 70, 71):
        inp["g"][tok, :, ::7] = -90.0
    helpers.check_parity(inp)


@pytest.mark.parametrize("dtype,d,lens,hk,hv", [("fp32", 64, [65, 64, 1], 2, 4), ("bf16", 64, [100, 130], 5, 5),
                                                ("fp32", 128, [40, 70], 4, 4), ("fp32", 64, [150], 9, 9)])
def test_fp32_slice_widths(dtype, d, lens, hk, hv):
    """Numbers of heads on either side of where the sequential kernel's slices get wider."""
    w = synth.shrink(W["gdn_varlen"], seq_lens=lens, hk=hk, hv=hv, dtype=dtype, dk=d, dv=d, h0_std=0.05, varlen=len(lens) > 1)
    helpers.check_parity(synth.make_inputs(w, seed=239))


@pytest.mark.parametrize("variant,dtype", [("gdn", "fp32"), ("gdn", "bf16"), ("kda", "fp32")])
@pytest.mark.parametrize("hv,lens", [(18, [40]), (19, [64]), (37, [17]), (38, [1]), (37, [100]), (75, [63]), (9, [400]), (10, [129]), (6, [200, 0, 65])])
def test_fp32_d64_shares_and_slices(variant, dtype, hv, lens):
    """d = 64: numbers of units (chunks x V-heads: 18, 19, 37, 38, 74, 75) on both sides of where CTAs share a chunk's last product, and of heads
    (9, 10, 18, 19) where the sequential kernel's slices change; no decay in places and a decay to nothing in others."""
    w = synth.shrink(W["gdn_varlen"] if variant == "gdn" else W["kda_8k"], seq_lens=lens, hk=1, hv=hv, dtype=dtype, dk=64, dv=64, gate_shift=4.0, h0_std=0.05,
                     varlen=len(lens) > 1)
    inp = synth.make_inputs(w, seed=251 + hv)
    inp["g"][::7] = 0.0
    inp["g"][5::31] = -90.0
    helpers.check_parity(inp, scale=0.5)
