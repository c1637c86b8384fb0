"""Prints the phase time stamps of the state-passing kernel from the instrumented build.

    python -m paper_2609_32114_b200.build --profile
    python -m paper_2609_32114_b200.prof_phases [WORKLOAD]          (needs a GPU)

The instrumented library (libha_la_prof.so, -DHA_LA_PROFILE_PHASES) records clock64 of a compute warp of CTA 0 at the
phase boundaries of its steps; this script runs one workload through it and prints the cycles between them.
"""
import ctypes
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def main(argv):
    import torch

    from paper_2609_32114_b200 import binding, build, synth
    import paper_2609_32114_b200 as ha
    from tests import helpers

    if not os.path.exists(build.PROF_LIB):
        raise SystemExit("build the instrumented library first: python -m paper_2609_32114_b200.build --profile")
    binding.LIB_PATH = build.PROF_LIB
    lib = ha.load_library()
    w = synth.WORKLOADS[argv[1] if len(argv) > 1 else "gdn_layer_4k"]
    inp = synth.make_inputs(w)
    d = helpers.to_device(inp)
    a, keep = ha.prepare_args(d["q"], d["k"], d["v"], d["g"], d["beta"], variant=w.variant, h0=d["h0"],
                              cu_seqlens=d["cu_seqlens"], max_seqlen=d["max_seqlen"])
    s = torch.cuda.current_stream().cuda_stream
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(3):
        ha.ha_la_prefill_raw(a, s)
    flush.zero_()
    ha.ha_la_prefill_raw(a, s)
    torch.cuda.synchronize()

    def read(name):
        buf = (ctypes.c_longlong * 1024)()
        getattr(lib, f"ha_la_debug_read_prof_{name}")(buf)
        return np.array(buf[:], dtype=np.int64)

    t = read("walk")
    print("cycles per step: X / R / U / update operand / D2 / state / total")
    for c in range(1, min(9, (max(inp["seq_lens"]) + 127) // 128)):
        v = t[8 * c: 8 * c + 7]
        print(f"  step {c:3d}:", *(f"{x:5d}" for x in np.diff(v)), f"{v[6] - v[0]:6d}")
    print("status word:", int(keep["status_word"].item()))


if __name__ == "__main__":
    main(sys.argv)
