"""AceSpec verify / sparsify / state-cache path on one GB300 GPU.

Thin Python binding of libacespec.so (declared in include/acespec.h).  The
functions below only marshal arguments: output tensors are allocated with
PyTorch on the inputs' device, pointers and the current CUDA stream are
handed to the C ABI, and every step of the computation runs in the
library's CUDA kernels.  There is no CPU fallback: calling any function
without the built library, or with host tensors, raises.

    verify(z, q, xt, u, T, top_p, k)      Sec. III-B, lossless verification
                                          fused with the sparse payload
    sparsify(z, T, top_p, k)              Sec. III-B / V-C downlink payload
    cache_build(q, xt, F)                 Sec. III-C branch cache
    cache_lookup(branch_tok, F, pi, tok)  Algorithm 1 state recovery
"""
from __future__ import annotations

import ctypes
import os
import threading

import torch

__all__ = ["load", "use_checked", "checked_violation", "checked_cache_selects", "lib_path", "workspace_bytes", "verify", "sparsify", "cache_build", "cache_lookup",
           "ROW_NONFINITE", "ROW_BAD_Q", "COUNTERS_OFFSET", "AcespecError"]

_HERE = os.path.dirname(os.path.abspath(__file__))
_LIB_PATH = os.path.join(_HERE, "libacespec.so")
_LIB_CHECKED = os.path.join(_HERE, "libacespec_checked.so")
_lock = threading.Lock()
_lib = None          # the library every function below calls
_libs = {}           # loaded libraries by path

# byte offset of the 16 path counters in a workspace (int32; after the hints
# a call leaves for the next one)
COUNTERS_OFFSET = 256

ROW_NONFINITE = 1
ROW_BAD_Q = 2
ACES_F32 = 0
ACES_BF16 = 1
_STATUS = {0: "ok", 1: "invalid argument", 2: "unsupported argument", 3: "CUDA launch error"}


class AcespecError(RuntimeError):
    def __init__(self, fn, code):
        super().__init__(f"{fn} failed: {_STATUS.get(code, code)} (status {code})")
        self.code = code


def lib_path() -> str:
    return _LIB_PATH


def load():
    """Load libacespec.so (built by __graft_entry__.build() or build.py)."""
    global _lib
    lib = _lib
    if lib is not None:
        return lib
    with _lock:
        if _lib is None:
            _lib = _open(_LIB_PATH)
        return _lib


def use_checked(on: bool = True):
    """Route every call of this module to the checked test build,
    libacespec_checked.so (built with build.build(checked=True)), or back to
    the product library.  Returns the library now in use."""
    global _lib
    with _lock:
        _lib = _open(_LIB_CHECKED if on else _LIB_PATH)
        return _lib


def checked_violation():
    """(site, index, bound) of the first out-of-range index the checked
    build met since the last call, or None; clears the record."""
    lib = load()
    if not hasattr(lib, "aces_checked_violation"):
        raise RuntimeError("the product library has no index checks: call use_checked() first")
    out = (ctypes.c_ulonglong * 3)()
    _check("aces_checked_violation", lib.aces_checked_violation(out))
    return None if out[0] == 0 else (int(out[0]), int(out[1]), int(out[2]))


def checked_cache_selects():
    """Rows of q that the checked build's cache_build read again since the
    last call (their first read's candidates were not enough); clears the count."""
    lib = load()
    if not hasattr(lib, "aces_checked_cache_selects"):
        raise RuntimeError("the product library counts nothing: call use_checked() first")
    n = ctypes.c_uint(0)
    _check("aces_checked_cache_selects", lib.aces_checked_cache_selects(ctypes.byref(n)))
    return int(n.value)


def _open(path):
    if path in _libs:
        return _libs[path]
    if not os.path.exists(path):
        raise RuntimeError(f"{path} is missing: build it with `python -m paper_2609_02514_gb300.build`")
    lib = ctypes.CDLL(path)
    P, I, F, S = ctypes.c_void_p, ctypes.c_int, ctypes.c_float, ctypes.c_size_t
    lib.aces_workspace_bytes.argtypes = [I, I, I, I]
    lib.aces_workspace_bytes.restype = S
    lib.aces_verify.argtypes = [P, I, P, P, P, I, I, I, F, F, P, P, I, P, P, P, P, P, S, P]
    lib.aces_verify_exact.argtypes = lib.aces_verify.argtypes
    lib.aces_sparsify.argtypes = [P, I, I, I, F, F, I, P, P, P, P, P, S, P]
    lib.aces_cache_build.argtypes = [P, P, P, I, I, I, P, P, P]
    lib.aces_cloud_step.argtypes = [P, I, P, P, P, I, I, I, F, F, P, P, I, P, P, P, P, P, P, P, P, S, P]
    lib.aces_cache_lookup.argtypes = [P, P, I, I, P, P, P, P]
    lib.aces_resample_sparse.argtypes = [P, P, P, P, P, P, P, I, I, I, I, P, P, P]
    lib.aces_compact_kv.argtypes = [P, I, I, I, I, I, I, P, P, P, I, I, P, P]
    lib.aces_tree_tokens.argtypes = [P, I, I]
    lib.aces_tree_tokens.restype = I
    lib.aces_tree_mask.argtypes = [P, I, I, P, P, P]
    lib.aces_tree_budget.argtypes = [P, I, ctypes.c_double, ctypes.c_double, I, P]
    lib.aces_branch_alloc.argtypes = [I, I, ctypes.c_double, ctypes.c_double, P]
    lib.aces_status_string.argtypes = [I]
    lib.aces_status_string.restype = ctypes.c_char_p
    for f in (lib.aces_verify, lib.aces_verify_exact, lib.aces_sparsify, lib.aces_cache_build,
              lib.aces_cache_lookup, lib.aces_resample_sparse, lib.aces_tree_budget, lib.aces_branch_alloc,
              lib.aces_compact_kv, lib.aces_tree_mask):
        f.restype = I
    if hasattr(lib, "aces_checked_violation"):
        lib.aces_checked_violation.argtypes = [P]
        lib.aces_checked_violation.restype = I
        lib.aces_checked_cache_selects.argtypes = [P]
        lib.aces_checked_cache_selects.restype = I
    _libs[path] = lib
    return lib


def _check(fn, code):
    if code != 0:
        raise AcespecError(fn, code)


# A small call is bound by the host, so the marshalling below allocates only the
# outputs it was not given and hands plain integers to ctypes (its argtypes make
# the pointers): a verify() call took 34 us of host time on a Grace core and
# takes 28, of which the C call is 6 and the six allocations 9.
def _cuda(t: torch.Tensor, name: str) -> torch.Tensor:
    if not isinstance(t, torch.Tensor) or not t.is_cuda:
        raise ValueError(f"{name} must be a CUDA tensor")
    if not t.is_contiguous():
        raise ValueError(f"{name} must be contiguous")
    return t


def _ptr(o, key):
    t = o.get(key)
    return None if t is None else t.data_ptr()


_raw_stream = torch._C._cuda_getCurrentRawStream if hasattr(torch._C, "_cuda_getCurrentRawStream") else None


def _stream(dev) -> int:
    """The current CUDA stream of the device."""
    if _raw_stream is not None and dev.index is not None:
        return _raw_stream(dev.index)
    return torch.cuda.current_stream(dev).cuda_stream


_empty = torch.empty
_I32, _F32 = torch.int32, torch.float32
_DTYPES = {torch.float32: ACES_F32, torch.bfloat16: ACES_BF16}


def _dtype_code(t: torch.Tensor) -> int:
    code = _DTYPES.get(t.dtype)
    if code is None:
        raise ValueError(f"target logits must be float32 or bfloat16, got {t.dtype}")
    return code


def _outputs(out, dev, *specs):
    """out's tensors, and new ones for the (key, shape, dtype) it lacks."""
    if out is None:
        return {key: _empty(shape, dtype=dtype, device=dev) for key, shape, dtype in specs}
    o = dict(out)
    for key, shape, dtype in specs:
        if key not in o:
            o[key] = _empty(shape, dtype=dtype, device=dev)
    return o


def _verify_outputs(out, dev, B, R, k):
    rest = () if k <= 0 else (("topk_ids", (B, R, k), _I32), ("topk_probs", (B, R, k), _F32), ("tail_mass", (B, R), _F32))
    return _outputs(out, dev, ("accept_len", (B,), _I32), ("out_token", (B,), _I32), ("row_status", (B, R), _I32), *rest)


def _workspace(workspace, dev, B, K, V, k):
    if workspace is not None:
        return workspace
    return torch.empty(max(workspace_bytes(B, K, V, k), 16), dtype=torch.uint8, device=dev)


def workspace_bytes(B: int, K: int, V: int, k: int) -> int:
    return int(load().aces_workspace_bytes(int(B), int(K), int(V), int(k)))


def verify(target_logits, draft_probs, draft_tokens, uniforms, T: float, top_p: float, k: int = 0,
           out: dict | None = None, workspace: torch.Tensor | None = None, exact: bool = False):
    """Lossless verification of B drafted chains (+ sparse payload when k > 0).

    target_logits [B, K+1, V] float32/bfloat16, draft_probs [B, K, V] float32,
    draft_tokens [B, K] int32, uniforms [B, K+1] float32.
    Returns a dict of device tensors: accept_len [B], out_token [B],
    row_status [B, K+1] and, when k > 0, topk_ids / topk_probs [B, K+1, k],
    tail_mass [B, K+1].  `out` may supply preallocated outputs (same keys).
    exact=True calls aces_verify_exact (every row on the exact general
    kernel; same results, slower).
    """
    lib = load()
    z = _cuda(target_logits, "target_logits")
    q = _cuda(draft_probs, "draft_probs")
    xt = _cuda(draft_tokens, "draft_tokens")
    u = _cuda(uniforms, "uniforms")
    if z.dim() != 3:
        raise ValueError("target_logits must be [B, K+1, V]")
    B, R, V = z.shape
    K = R - 1
    if q.dtype != _F32 or q.shape != (B, K, V):
        raise ValueError("draft_probs must be float32 [B, K, V]")
    if xt.dtype != _I32 or xt.shape != (B, K):
        raise ValueError("draft_tokens must be int32 [B, K]")
    if u.dtype != _F32 or u.shape != (B, R):
        raise ValueError("uniforms must be float32 [B, K+1]")
    dev = z.device
    o = _verify_outputs(out, dev, B, R, k)
    ws = _workspace(workspace, dev, B, K, V, k)
    fn = lib.aces_verify_exact if exact else lib.aces_verify
    code = fn(z.data_ptr(), _dtype_code(z), q.data_ptr(), xt.data_ptr(), u.data_ptr(), B, K, V, float(T),
              float(top_p), _ptr(o, "accept_len"), _ptr(o, "out_token"), int(k), _ptr(o, "topk_ids"), _ptr(o, "topk_probs"),
              _ptr(o, "tail_mass"), _ptr(o, "row_status"), ws.data_ptr(), ws.numel(), _stream(dev))
    if code != 0:
        _check("aces_verify_exact" if exact else "aces_verify", code)
    return o


def sparsify(target_logits, T: float, top_p: float, k: int, out: dict | None = None,
             workspace: torch.Tensor | None = None):
    """Sparse top-k payload of every row of target_logits [rows, V] (or [..., V])."""
    lib = load()
    z = _cuda(target_logits, "target_logits")
    V = z.shape[-1]
    rows = z.numel() // V
    dev = z.device
    lead = tuple(z.shape[:-1])
    o = _outputs(out, dev, ("topk_ids", (*lead, k), torch.int32), ("topk_probs", (*lead, k), torch.float32),
                 ("tail_mass", lead, torch.float32), ("row_status", lead, torch.int32))
    ws = _workspace(workspace, dev, rows, 0, V, k)
    code = lib.aces_sparsify(z.data_ptr(), _dtype_code(z), rows, V, float(T), float(top_p), int(k),
                             _ptr(o, "topk_ids"), _ptr(o, "topk_probs"), _ptr(o, "tail_mass"), _ptr(o, "row_status"), ws.data_ptr(),
                             ws.numel(), _stream(dev))
    if code != 0:
        _check("aces_sparsify", code)
    return o


def _f_host(F):
    return (ctypes.c_int32 * len(F))(*map(int, F))


def cache_build(draft_probs, draft_tokens, F, out: dict | None = None):
    """Branch cache: q [B,K,V] float32, x~ [B,K] int32, F (K ints) ->
    branch_tok [B, sum F] int32, branch_prob [B, sum F] float32."""
    lib = load()
    q = _cuda(draft_probs, "draft_probs")
    xt = _cuda(draft_tokens, "draft_tokens")
    B, K, V = q.shape
    if len(F) != K:
        raise ValueError("F must have K entries")
    Fh = _f_host(F)
    tot = sum(Fh)
    dev = q.device
    o = _outputs(out, dev, ("branch_tok", (B, tot), torch.int32), ("branch_prob", (B, tot), torch.float32))
    code = lib.aces_cache_build(q.data_ptr(), xt.data_ptr(), Fh, B, K, V, _ptr(o, "branch_tok"),
                                _ptr(o, "branch_prob"), _stream(dev))
    if code != 0:
        _check("aces_cache_build", code)
    return o


def cloud_step(target_logits, draft_probs, draft_tokens, uniforms, T: float, top_p: float, k: int, F,
               out: dict | None = None, workspace: torch.Tensor | None = None):
    """verify() and cache_build() of the same batch in one call (the cache
    build runs concurrently on the library's own stream).  Returns the keys of
    both: accept_len, out_token, row_status, the payload when k > 0,
    branch_tok and branch_prob."""
    lib = load()
    z = _cuda(target_logits, "target_logits")
    q = _cuda(draft_probs, "draft_probs")
    xt = _cuda(draft_tokens, "draft_tokens")
    u = _cuda(uniforms, "uniforms")
    if z.dim() != 3:
        raise ValueError("target_logits must be [B, K+1, V]")
    B, R, V = z.shape
    K = R - 1
    if q.dtype != _F32 or q.shape != (B, K, V):
        raise ValueError("draft_probs must be float32 [B, K, V]")
    if xt.dtype != _I32 or xt.shape != (B, K):
        raise ValueError("draft_tokens must be int32 [B, K]")
    if u.dtype != _F32 or u.shape != (B, R):
        raise ValueError("uniforms must be float32 [B, K+1]")
    if len(F) != K:
        raise ValueError("F must have K entries")
    Fh = _f_host(F)
    tot = sum(Fh)
    dev = z.device
    o = _verify_outputs(out, dev, B, R, k)
    if "branch_tok" not in o or "branch_prob" not in o:
        o = _outputs(o, dev, ("branch_tok", (B, tot), torch.int32), ("branch_prob", (B, tot), torch.float32))
    ws = _workspace(workspace, dev, B, K, V, k)
    code = lib.aces_cloud_step(z.data_ptr(), _dtype_code(z), q.data_ptr(), xt.data_ptr(), u.data_ptr(), B, K, V, float(T),
                               float(top_p), _ptr(o, "accept_len"), _ptr(o, "out_token"), int(k), _ptr(o, "topk_ids"),
                               _ptr(o, "topk_probs"), _ptr(o, "tail_mass"), _ptr(o, "row_status"), Fh,
                               _ptr(o, "branch_tok"), _ptr(o, "branch_prob"), ws.data_ptr(), ws.numel(), _stream(dev))
    if code != 0:
        _check("aces_cloud_step", code)
    return o


def cache_lookup(branch_tok, F, accept_len, token, out: torch.Tensor | None = None):
    """slot [B] int32: off_pi + j on a hit, -1 on a miss, -2 when pi == K."""
    lib = load()
    bt = _cuda(branch_tok, "branch_tok")
    al = _cuda(accept_len, "accept_len")
    tk = _cuda(token, "token")
    B = al.shape[0]
    K = len(F)
    slot = out if out is not None else torch.empty(B, dtype=torch.int32, device=al.device)
    code = lib.aces_cache_lookup(bt.data_ptr(), _f_host(F), B, K, al.data_ptr(), tk.data_ptr(), slot.data_ptr(),
                                 _stream(al.device))
    if code != 0:
        _check("aces_cache_lookup", code)
    return slot


def resample_sparse(accept_len, topk_ids, topk_probs, tail_mass, row_status, draft_probs, uniforms,
                    out: dict | None = None):
    """Edge-side draw from the sparse payload of row pi (Alg. 1 RESAMPLE).

    accept_len [B], topk_ids / topk_probs [B,K+1,k], tail_mass / row_status
    [B,K+1] (as written by verify), draft_probs [B,K,V] float32, uniforms
    [B,K+1] float32 -> token [B] int32, status [B] int32.
    """
    lib = load()
    al = _cuda(accept_len, "accept_len")
    ids = _cuda(topk_ids, "topk_ids")
    pr = _cuda(topk_probs, "topk_probs")
    tl = _cuda(tail_mass, "tail_mass")
    st = _cuda(row_status, "row_status")
    q = _cuda(draft_probs, "draft_probs")
    u = _cuda(uniforms, "uniforms")
    B, K, V = q.shape
    k = ids.shape[-1]
    dev = q.device
    o = _outputs(out, dev, ("token", (B,), torch.int32), ("status", (B,), torch.int32))
    code = lib.aces_resample_sparse(al.data_ptr(), ids.data_ptr(), pr.data_ptr(), tl.data_ptr(), st.data_ptr(),
                                    q.data_ptr(), u.data_ptr(), B, K, V, k, _ptr(o, "token"), _ptr(o, "status"),
                                    _stream(dev))
    if code != 0:
        _check("aces_resample_sparse", code)
    return o


def tree_budget(draft_latency_s, rtt_s: float, verify_s: float, B_max: int) -> int:
    """Network-aware budget B* (Sec. IV-B) from the drafting times of tree sizes 1..n."""
    lib = load()
    n = len(draft_latency_s)
    arr = (ctypes.c_double * n)(*[float(t) for t in draft_latency_s])
    out = ctypes.c_int(0)
    _check("aces_tree_budget", lib.aces_tree_budget(arr, n, float(rtt_s), float(verify_s), int(B_max),
                                                    ctypes.byref(out)))
    return int(out.value)


def branch_alloc(B_alloc: int, gamma: int, alpha: float, beta: float) -> list:
    """Integer branch counts F_0..F_{gamma-1} of the geometric-decay allocation (Sec. IV-C)."""
    lib = load()
    F = (ctypes.c_int32 * int(gamma))()
    _check("aces_branch_alloc", lib.aces_branch_alloc(int(B_alloc), int(gamma), float(alpha), float(beta), F))
    return [int(f) for f in F]


def compact_kv(kv, prefix_len, accept_len, slot, K: int, branch_len: int, new_len: torch.Tensor | None = None):
    """COMPACT_KV / ROLLBACK_KV (Alg. 1) in place on kv [planes, B, H, S, D];
    returns new_len [B] int32."""
    lib = load()
    kv = _cuda(kv, "kv")
    t = _cuda(prefix_len, "prefix_len")
    al = _cuda(accept_len, "accept_len")
    sl = _cuda(slot, "slot")
    planes, B, H, S, D = kv.shape
    out = new_len if new_len is not None else torch.empty(B, dtype=torch.int32, device=kv.device)
    code = lib.aces_compact_kv(kv.data_ptr(), kv.element_size(), planes, B, H, S, D, t.data_ptr(), al.data_ptr(),
                               sl.data_ptr(), int(K), int(branch_len), out.data_ptr(), _stream(kv.device))
    if code != 0:
        _check("aces_compact_kv", code)
    return out


def tree_mask(F, branch_len: int, device=None):
    """Tree attention mask (Sec. III-C): mask [n, ceil(n/32)] int32 words (bit
    j of word w: key 32 w + j allowed) and depth [n] int32 on the device."""
    lib = load()
    K = len(F)
    Fh = _f_host(F)
    n = int(lib.aces_tree_tokens(Fh, K, int(branch_len)))
    if n < 0:
        raise ValueError("invalid tree shape")
    dev = torch.device("cuda") if device is None else torch.device(device)
    mask = torch.empty(n, (n + 31) // 32, dtype=torch.int32, device=dev)
    depth = torch.empty(n, dtype=torch.int32, device=dev)
    _check("aces_tree_mask", lib.aces_tree_mask(Fh, K, int(branch_len), mask.data_ptr(), depth.data_ptr(),
                                                _stream(mask.device)))
    return mask, depth
