"""ctypes binding of libha_la.so: argument marshalling only, same names as include/ha_la.h.

Every step of the prefill runs in the library's CUDA kernels.  There is no CPU or
PyTorch fallback: if the shared library is missing, loading raises.
"""
from __future__ import annotations

import ctypes
import os
from typing import Optional, Tuple

HA_LA_GDN, HA_LA_KDA = 0, 1
HA_LA_BF16, HA_LA_FP32 = 0, 1
HA_LA_OK = 0
HA_LA_ERR_INVALID_ARG = 1
HA_LA_ERR_UNSUPPORTED = 2
HA_LA_ERR_WORKSPACE = 3
HA_LA_ERR_CUDA = 4
HA_LA_ERR_TIMEOUT = 5
HA_LA_ERR_DEVICE_CHECK = 6
HA_LA_ERR_TOO_LARGE = 7

_PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_PKG, "libha_la.so")

EXPORTS = (
    "ha_la_prefill_workspace_bytes",
    "ha_la_prefill",
    "ha_la_prefill_timed",
    "ha_la_prefill_noalloc",
    "ha_la_prefill_noalloc_scratch_bytes",
    "ha_la_prefill_path",
    "ha_la_prefill_num_launches",
    "ha_la_prefill_launch_plan",
    "ha_la_prefill_num_segments",
    "ha_la_prefill_num_runs",
    "ha_la_decode",
    "ha_la_debug_wait_timeout",
    "ha_la_status_string",
    "ha_la_version",
)


class ha_la_prefill_args(ctypes.Structure):
    _fields_ = [
        ("variant", ctypes.c_int32),
        ("dtype", ctypes.c_int32),
        ("batch", ctypes.c_int32),
        ("seqlen", ctypes.c_int32),
        ("num_qk_heads", ctypes.c_int32),
        ("num_v_heads", ctypes.c_int32),
        ("d_k", ctypes.c_int32),
        ("d_v", ctypes.c_int32),
        ("chunk", ctypes.c_int32),
        ("scale", ctypes.c_float),
        ("q", ctypes.c_void_p),
        ("k", ctypes.c_void_p),
        ("v", ctypes.c_void_p),
        ("g", ctypes.c_void_p),
        ("beta", ctypes.c_void_p),
        ("h0", ctypes.c_void_p),
        ("cu_seqlens", ctypes.c_void_p),
        ("num_seqs", ctypes.c_int32),
        ("max_seqlen", ctypes.c_int32),
        ("o", ctypes.c_void_p),
        ("hT", ctypes.c_void_p),
        ("workspace", ctypes.c_void_p),
        ("workspace_bytes", ctypes.c_size_t),
        ("status_word", ctypes.c_void_p),
    ]


class ha_la_decode_args(ctypes.Structure):
    _fields_ = [
        ("variant", ctypes.c_int32),
        ("dtype", ctypes.c_int32),
        ("num_seqs", ctypes.c_int32),
        ("num_qk_heads", ctypes.c_int32),
        ("num_v_heads", ctypes.c_int32),
        ("d_k", ctypes.c_int32),
        ("d_v", ctypes.c_int32),
        ("scale", ctypes.c_float),
        ("q", ctypes.c_void_p),
        ("k", ctypes.c_void_p),
        ("v", ctypes.c_void_p),
        ("g", ctypes.c_void_p),
        ("beta", ctypes.c_void_p),
        ("h_in", ctypes.c_void_p),
        ("h_out", ctypes.c_void_p),
        ("o", ctypes.c_void_p),
    ]


class HaLaError(RuntimeError):
    def __init__(self, status: int, what: str):
        self.status = status
        super().__init__(f"{what}: status {status} ({status_string(status)})")


_lib = None
_call = None          # the native half of ha_la_prefill / ha_la_decode (csrc/torch_call.cpp), once loaded
_call_lib = None      # ... and the library it is bound to


def load_library(path: Optional[str] = None):
    """Load libha_la.so (built in-tree by paper_2609_32114_b200.build).  Raises if it is missing."""
    global _lib
    if _lib is not None and path is None:
        return _lib
    p = path or LIB_PATH
    if not os.path.exists(p):
        raise FileNotFoundError(
            f"{p} not found: build it with `python -m paper_2609_32114_b200.build` "
            "(there is no fallback implementation)")
    lib = ctypes.CDLL(p)
    A = ctypes.POINTER(ha_la_prefill_args)
    lib.ha_la_prefill_workspace_bytes.argtypes = [A, ctypes.POINTER(ctypes.c_size_t)]
    lib.ha_la_prefill_workspace_bytes.restype = ctypes.c_int
    lib.ha_la_prefill.argtypes = [A, ctypes.c_void_p]
    lib.ha_la_prefill.restype = ctypes.c_int
    lib.ha_la_prefill_timed.argtypes = [A, ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(ctypes.c_float),
                                        ctypes.POINTER(ctypes.c_char_p), ctypes.POINTER(ctypes.c_int)]
    lib.ha_la_prefill_timed.restype = ctypes.c_int
    lib.ha_la_prefill_noalloc.argtypes = [A, ctypes.c_void_p]
    lib.ha_la_prefill_noalloc.restype = ctypes.c_int
    lib.ha_la_prefill_noalloc_scratch_bytes.argtypes = []
    lib.ha_la_prefill_noalloc_scratch_bytes.restype = ctypes.c_size_t
    lib.ha_la_prefill_path.argtypes = [A]
    lib.ha_la_prefill_path.restype = ctypes.c_char_p
    lib.ha_la_prefill_num_launches.argtypes = [A]
    lib.ha_la_prefill_num_launches.restype = ctypes.c_int
    lib.ha_la_prefill_num_segments.argtypes = [A]
    lib.ha_la_prefill_num_segments.restype = ctypes.c_int
    lib.ha_la_prefill_num_runs.argtypes = [A]
    lib.ha_la_prefill_num_runs.restype = ctypes.c_int
    lib.ha_la_prefill_launch_plan.argtypes = [A, ctypes.POINTER(ctypes.c_int), ctypes.POINTER(ctypes.c_int)]
    lib.ha_la_prefill_launch_plan.restype = ctypes.c_int
    lib.ha_la_decode.argtypes = [ctypes.POINTER(ha_la_decode_args), ctypes.c_void_p]
    lib.ha_la_decode.restype = ctypes.c_int
    lib.ha_la_debug_wait_timeout.argtypes = [A, ctypes.c_void_p, ctypes.c_uint]
    lib.ha_la_debug_wait_timeout.restype = ctypes.c_int
    lib.ha_la_status_string.argtypes = [ctypes.c_int]
    lib.ha_la_status_string.restype = ctypes.c_char_p
    lib.ha_la_version.argtypes = []
    lib.ha_la_version.restype = ctypes.c_int
    if path is None:
        _lib = lib
    return lib


def _torch_call():
    """Load ha_la_torch_call.so and bind it to the library's entry points.  Raises if it is missing."""
    global _call, _call_lib
    lib = load_library()
    if _call is None:
        import importlib.util

        import torch  # noqa: F401  (its libraries first: the extension links against them)

        path = os.path.join(_PKG, "ha_la_torch_call.so")
        if not os.path.exists(path):
            raise FileNotFoundError(f"{path} not found: build it with `python -m paper_2609_32114_b200.build`")
        spec = importlib.util.spec_from_file_location("ha_la_torch_call", path)
        mod = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(mod)
        _call = mod
    if _call_lib is not lib:
        _call.bind(*(ctypes.cast(f, ctypes.c_void_p).value
                     for f in (lib.ha_la_prefill, lib.ha_la_prefill_workspace_bytes, lib.ha_la_decode)))
        _call_lib = lib
    return _call


def status_string(status: int) -> str:
    return load_library().ha_la_status_string(int(status)).decode()


def ha_la_version() -> int:
    return load_library().ha_la_version()


def make_args(*, variant, dtype, batch, seqlen, hk, hv, dk, dv, scale=1.0, chunk=64, num_seqs=0, max_seqlen=0,
              q=0, k=0, v=0, g=0, beta=0, h0=0, cu_seqlens=0, o=0, hT=0, workspace=0, workspace_bytes=0,
              status_word=0) -> ha_la_prefill_args:
    """Fill the C struct from plain integers (device addresses) and sizes."""
    var = {"gdn": HA_LA_GDN, "kda": HA_LA_KDA}.get(variant, variant)
    dt = {"bf16": HA_LA_BF16, "fp32": HA_LA_FP32}.get(dtype, dtype)
    n = lambda p: p if p else None
    return ha_la_prefill_args(var, dt, batch, seqlen, hk, hv, dk, dv, chunk, float(scale), n(q), n(k), n(v), n(g),
                              n(beta), n(h0), n(cu_seqlens), num_seqs, max_seqlen, n(o), n(hT), n(workspace),
                              workspace_bytes, n(status_word))


def ha_la_prefill_workspace_bytes(args: ha_la_prefill_args) -> int:
    out = ctypes.c_size_t(0)
    rc = load_library().ha_la_prefill_workspace_bytes(ctypes.byref(args), ctypes.byref(out))
    if rc != HA_LA_OK:
        raise HaLaError(rc, "ha_la_prefill_workspace_bytes")
    return out.value


def ha_la_prefill_path(args: ha_la_prefill_args) -> Optional[str]:
    r = load_library().ha_la_prefill_path(ctypes.byref(args))
    return None if r is None else r.decode()


def ha_la_prefill_num_launches(args: ha_la_prefill_args) -> int:
    return load_library().ha_la_prefill_num_launches(ctypes.byref(args))


def ha_la_prefill_num_segments(args: ha_la_prefill_args) -> int:
    """Segments per sequence in the cost model of ha_la_prefill_launch_plan; what a call does is ha_la_prefill_num_runs."""
    return load_library().ha_la_prefill_num_segments(ctypes.byref(args))


def ha_la_prefill_num_runs(args: ha_la_prefill_args) -> int:
    """Runs a call cuts every sequence into, walked at the same time (1 = in order, 0 = unsupported)."""
    return load_library().ha_la_prefill_num_runs(ctypes.byref(args))


def ha_la_prefill_launch_plan(args: ha_la_prefill_args) -> Tuple[int, bool]:
    """A cost model's answer for launches in chunks of 64 tokens (see include/ha_la.h): (slice width of the sequential
    kernel or 0 on the CUDA-core path, kernels side by side?).  The kernels work in steps of 128 on whole heads."""
    nv, conc = ctypes.c_int(0), ctypes.c_int(0)
    rc = load_library().ha_la_prefill_launch_plan(ctypes.byref(args), ctypes.byref(nv), ctypes.byref(conc))
    if rc != HA_LA_OK:
        raise HaLaError(rc, "ha_la_prefill_launch_plan")
    return nv.value, bool(conc.value)


def ha_la_prefill_raw(args: ha_la_prefill_args, stream: int = 0) -> int:
    """The C call itself; returns the status code."""
    return load_library().ha_la_prefill(ctypes.byref(args), ctypes.c_void_p(stream) if stream else None)


def ha_la_prefill_noalloc(args: ha_la_prefill_args, stream: int = 0) -> int:
    """The C call for callers that cannot supply scratch memory (the workspace fields are ignored);
    returns the status code.  See include/ha_la.h for its limits and its sharing rules."""
    return load_library().ha_la_prefill_noalloc(ctypes.byref(args), ctypes.c_void_p(stream) if stream else None)


def ha_la_debug_wait_timeout(args: ha_la_prefill_args, stream: int = 0, spin_limit: int = 4096) -> int:
    """Test hook: the sequential kernel alone with its copies withheld, so that its waits run out; returns the status code."""
    return load_library().ha_la_debug_wait_timeout(ctypes.byref(args), ctypes.c_void_p(stream) if stream else None,
                                                   ctypes.c_uint(spin_limit))


def ha_la_prefill_noalloc_scratch_bytes() -> int:
    return load_library().ha_la_prefill_noalloc_scratch_bytes()


def ha_la_prefill_timed(args: ha_la_prefill_args, stream: int = 0):
    """Blocking, per-kernel device timing.  Returns [(kernel name, milliseconds), ...] in launch order."""
    ms = (ctypes.c_float * 8)()
    names = (ctypes.c_char_p * 8)()
    n = ctypes.c_int(0)
    rc = load_library().ha_la_prefill_timed(ctypes.byref(args), ctypes.c_void_p(stream) if stream else None, 8, ms,
                                            names, ctypes.byref(n))
    if rc != HA_LA_OK:
        raise HaLaError(rc, "ha_la_prefill_timed")
    return [(names[i].decode(), float(ms[i])) for i in range(n.value)]


def _aligned_part(address, nbytes):
    """What of a buffer starts on a 256-byte boundary: (address, bytes).  Nothing of one that ends before its first."""
    start = (address + 255) // 256 * 256
    return start, max(0, nbytes - (start - address))


def _reachable(t, q):
    return t.device == q.device or (t.device.type == "cpu" and t.is_pinned())


def _check_inputs(q, k, v, g, beta, kda, one_row):
    """q [rows.., HK, dk] sets the sizes of k, v [rows.., HV, dv], g [rows.., HV] (KDA: and dk) and beta [rows.., HV].  The others
    may have more rows than q where they lie one behind the other (`one_row`: of tokens, in a batch of one)."""
    lead, (hk, dk), (hv, dv) = tuple(q.shape[:-2]), q.shape[-2:], v.shape[-2:]
    for name, t, last in (("k", k, (hk, dk)), ("v", v, (hv, dv)), ("g", g, (hv, dk) if kda else (hv,)), ("beta", beta, (hv,))):
        rows, heads = tuple(t.shape[:len(lead)]), tuple(t.shape[len(lead):])
        if not (_reachable(t, q) and heads == last and len(rows) == len(lead) and rows[0] >= lead[0] and
                (rows[1:] == lead[1:] or (one_row and rows[1:] > lead[1:]))):
            raise ValueError(f"{name}: {tuple(t.shape)} on {t.device} does not go with q {tuple(q.shape)} on {q.device} and {hv} V-heads")


def _check_room(name, t, q, dtype, n):
    """A tensor (or None) that the kernels take by its address: contiguous, `n` elements of `dtype` (None: `n` bytes)."""
    if t is None:
        return
    have = t.numel() * (t.element_size() if dtype is None else 1)
    if not (_reachable(t, q) and t.is_contiguous() and (dtype is None or t.dtype == dtype) and have >= n):
        raise ValueError(f"{name}: {t.dtype} {tuple(t.shape)}, strides {tuple(t.stride())}, on {t.device}; wanted are {n} "
                         f"{'bytes' if dtype is None else dtype}, contiguous, on {q.device}")


def prepare_args(q, k, v, g, beta, *, variant="gdn", h0=None, cu_seqlens=None, max_seqlen=0, scale=1.0,
                 o=None, hT=None, want_hT=True, workspace=None, status_word=None):
    """Marshal torch CUDA tensors into ha_la_prefill_args (allocating o / hT / workspace / status word
    with torch when they are not given).  Returns (args, tensors) where `tensors` keeps them alive."""
    import torch

    if not q.is_cuda:
        raise ValueError("ha_la_prefill needs CUDA tensors (there is no CPU path)")
    packed = cu_seqlens is not None
    if q.dim() == 3:
        q, k, v, g, beta = (t.unsqueeze(0) for t in (q, k, v, g, beta))
        if o is not None:
            o = o.unsqueeze(0)
    B, T, HK, dk = q.shape
    HV, dv = v.shape[2], v.shape[3]
    dtype = {torch.bfloat16: "bf16", torch.float32: "fp32"}[q.dtype]
    for t in (q, k, v, g, beta):
        assert t.is_contiguous()
    assert k.dtype == q.dtype and v.dtype == q.dtype and g.dtype == torch.float32 and beta.dtype == torch.float32
    N = (cu_seqlens.numel() - 1) if packed else B
    if packed:
        assert cu_seqlens.dtype == torch.int32 and cu_seqlens.is_cuda and B == 1
    _check_inputs(q, k, v, g, beta, variant in ("kda", HA_LA_KDA), B == 1)
    state = N * HV * dk * dv
    for name, t, dt, n in (("h0", h0, torch.float32, state), ("hT", hT, torch.float32, state), ("o", o, q.dtype, B * T * HV * dv),
                           ("cu_seqlens", cu_seqlens, torch.int32, 0), ("workspace", workspace, None, 0), ("status_word", status_word, None, 4)):
        _check_room(name, t, q, dt, n)
    if o is None:
        o = torch.empty_like(v)
    if hT is None and want_hT:
        hT = torch.empty((N, HV, dk, dv), dtype=torch.float32, device=q.device)
    if status_word is None:
        status_word = torch.zeros(1, dtype=torch.int32, device=q.device)
    ptr = lambda t: 0 if t is None else t.data_ptr()
    args = make_args(variant=variant, dtype=dtype, batch=B, seqlen=T, hk=HK, hv=HV, dk=dk, dv=dv, scale=scale,
                     num_seqs=N if packed else 0, max_seqlen=max_seqlen, q=ptr(q), k=ptr(k), v=ptr(v), g=ptr(g),
                     beta=ptr(beta), h0=ptr(h0), cu_seqlens=ptr(cu_seqlens), o=ptr(o), hT=ptr(hT),
                     status_word=ptr(status_word))
    need = ha_la_prefill_workspace_bytes(args)
    if workspace is None:
        workspace = torch.empty(need + 256, dtype=torch.uint8, device=q.device)
    args.workspace, args.workspace_bytes = _aligned_part(workspace.data_ptr(), workspace.numel())
    keep = dict(q=q, k=k, v=v, g=g, beta=beta, h0=h0, cu_seqlens=cu_seqlens, o=o, hT=hT, workspace=workspace,
                status_word=status_word)
    return args, keep


_KDA = {"gdn": False, "kda": True}


def _prefill_call(q, k, v, g, beta, stream, *, variant="gdn", h0=None, cu_seqlens=None, max_seqlen=0, scale=1.0, o=None,
                  hT=None, want_hT=True, workspace=None, status_word=None):
    """The arguments of the native call (prepare_args' keywords and defaults, in order)."""
    return (q, k, v, g, beta, h0, cu_seqlens, max_seqlen, stream, _KDA.get(variant), scale, o, hT, want_hT, workspace,
            status_word)


def _marshal_on(stream, prepare, q, *rest, **kw):
    """prepare(q, *rest, **kw) for a call on `stream` (a cudaStream_t, None: torch's current one): what it allocates and fills is
    that stream's, and recorded on the current one (see CallStream in csrc/torch_call.cpp).  Returns (args, tensors, stream)."""
    import torch

    if stream is None:
        return *prepare(q, *rest, **kw), torch.cuda.current_stream(q.device).cuda_stream
    current = torch.cuda.current_stream(q.device if q.is_cuda else None)
    if current.cuda_stream == stream or not q.is_cuda:     # (prepare refuses the latter)
        return *prepare(q, *rest, **kw), stream
    with torch.cuda.stream(torch.cuda.ExternalStream(stream, device=q.device)):
        args, keep = prepare(q, *rest, **kw)
    for name in ("o", "hT", "workspace", "status_word", "state_out"):
        t = keep.get(name)
        if t is not None and kw.get(name) is None and all(t is not x for x in rest):
            t.record_stream(current)
    return args, keep, stream


def ha_la_prefill(q, k, v, g, beta, *, stream=None, **kw):
    """Prefill on torch CUDA tensors: prepare_args + the C call on torch's current stream.

    q, k : [B, T, HK, dk] (or [T, HK, dk])   v : [B, T, HV, dv]   bf16 or fp32
    g    : fp32 [B, T, HV] (gdn) or [B, T, HV, dk] (kda)      beta : fp32 [B, T, HV]
    h0   : fp32 [N, HV, dk, dv] or None      cu_seqlens : int32 [N+1] device tensor or None (packed, B = 1)
    Returns (o, hT, status_word, workspace); nothing is synchronised.
    """
    r = (_call if _call_lib is not None else _torch_call()).prefill(*_prefill_call(q, k, v, g, beta, stream, **kw))
    if r.__class__ is tuple:
        return r
    if r is not None:
        raise HaLaError(r, "ha_la_prefill")
    # not an entirely ordinary call: marshalled here
    squeeze = q.dim() == 3
    args, keep, stream = _marshal_on(stream, prepare_args, q, k, v, g, beta, **kw)
    rc = ha_la_prefill_raw(args, stream)
    if rc != HA_LA_OK:
        raise HaLaError(rc, "ha_la_prefill")
    o = keep["o"].squeeze(0) if squeeze else keep["o"]
    return o, keep["hT"], keep["status_word"], keep["workspace"]


def prepare_decode_args(q, k, v, g, beta, state, *, variant="gdn", scale=1.0, o=None, state_out=None):
    """Marshal torch CUDA tensors into ha_la_decode_args.  q, k: [N, HK, d]; v: [N, HV, d]; g: fp32 [N, HV] (gdn)
    or [N, HV, d] (kda); beta: fp32 [N, HV]; state: fp32 [N, HV, d, d] or None (zeros).  The new state goes to
    `state_out` (default: in place into `state`; allocated when `state` is None)."""
    import torch

    if not q.is_cuda:
        raise ValueError("ha_la_decode needs CUDA tensors (there is no CPU path)")
    N, HK, d = q.shape
    HV = v.shape[1]
    if q.dtype not in (torch.bfloat16, torch.float32):
        raise ValueError(f"q: {q.dtype}")
    _check_inputs(q, k, v, g, beta, variant != "gdn", False)
    for name, t, dt, n in (("q", q, q.dtype, 0), ("k", k, q.dtype, 0), ("v", v, q.dtype, 0), ("g", g, torch.float32, 0),
                           ("beta", beta, torch.float32, 0), ("state", state, torch.float32, N * HV * d * v.shape[2]),
                           ("state_out", state_out, torch.float32, N * HV * d * v.shape[2]), ("o", o, q.dtype, N * HV * v.shape[2])):
        _check_room(name, t, q, dt, n)
    if o is None:
        o = torch.empty_like(v)
    if state_out is None:
        state_out = state if state is not None else torch.empty(N, HV, d, d, dtype=torch.float32, device=q.device)
    ptr = lambda t: t.data_ptr() if t is not None else None
    args = ha_la_decode_args(variant=0 if variant == "gdn" else 1, dtype=0 if q.dtype == torch.bfloat16 else 1,
                             num_seqs=N, num_qk_heads=HK, num_v_heads=HV, d_k=d, d_v=v.shape[2], scale=scale,
                             q=ptr(q), k=ptr(k), v=ptr(v), g=ptr(g), beta=ptr(beta), h_in=ptr(state),
                             h_out=ptr(state_out), o=ptr(o))
    return args, dict(q=q, k=k, v=v, g=g, beta=beta, state=state, state_out=state_out, o=o)


def ha_la_decode_raw(args: ha_la_decode_args, stream: int = 0) -> int:
    return load_library().ha_la_decode(ctypes.byref(args), ctypes.c_void_p(stream))


def ha_la_decode(q, k, v, g, beta, state, *, stream=None, variant="gdn", scale=1.0, o=None, state_out=None):
    """One decoding step on torch CUDA tensors (see prepare_decode_args).  Returns (o, new_state); nothing is
    synchronised."""
    r = (_call if _call_lib is not None else _torch_call()).decode(q, k, v, g, beta, state, stream, variant != "gdn", scale,
                                                                   o, state_out)
    if r.__class__ is tuple:
        return r
    if r is not None:
        raise HaLaError(r, "ha_la_decode")
    # not an entirely ordinary call: marshalled here
    kw = dict(variant=variant, scale=scale, o=o, state_out=state_out)
    args, keep, stream = _marshal_on(stream, prepare_decode_args, q, k, v, g, beta, state, **kw)
    rc = ha_la_decode_raw(args, stream)
    if rc != HA_LA_OK:
        raise HaLaError(rc, "ha_la_decode")
    return keep["o"], keep["state_out"]
