"""ctypes binding of include/grass.h: same names, torch tensors in place of pointers.

Argument marshalling only.  Every function enqueues on torch's current CUDA
stream and raises GrassError on a non-zero status; nothing here computes.
"""
from __future__ import annotations

import ctypes
import importlib.util
import os
from ctypes import c_double, c_int, c_int32, c_int64, c_size_t, c_uint32, c_uint64, c_void_p

import torch

F32, BF16 = 0, 1
SEL_TOPR, SEL_MULTINOMIAL_NORM = 0, 1
SEL_MULTINOMIAL_NORM2, SEL_UNIFORM = 2, 3
SEL_MULTINOMIAL_NORM_NR, SEL_MULTINOMIAL_NORM2_NR, SEL_UNIFORM_NR = 4, 5, 6

_HERE = os.path.dirname(os.path.abspath(__file__))
_LIB = None


class GrassError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {grass_status_string(status)} (status {status})")


def library_path() -> str:
    return os.path.join(_HERE, "libgrass_b200.so")


_SIGNATURES = {
    "grass_row_norms": (c_int, [c_void_p, c_int, c_int64, c_int64, c_int64, c_void_p, c_void_p]),
    "grass_select_workspace_bytes": (c_size_t, [c_int64, c_int32, c_int]),
    "grass_select": (c_int, [c_void_p, c_int64, c_int32, c_int, c_uint64, c_uint32, c_uint32,
                             c_void_p, c_void_p, c_void_p, c_size_t, c_void_p]),
    "grass_select_static": (c_int, [c_void_p, c_int64, c_int32, c_int, c_uint64, c_uint32, c_uint32,
                                    c_void_p, c_void_p, c_void_p]),
    "grass_project_workspace_bytes": (c_size_t, [c_int64, c_int64, c_int64, c_int32, c_int]),
    "grass_project_grad": (c_int, [c_void_p, c_int64, c_void_p, c_int64, c_int, c_int64, c_int64,
                                   c_int64, c_void_p, c_void_p, c_int32, c_void_p, c_int64,
                                   c_void_p, c_size_t, c_void_p]),
    "grass_grad_row_norms_workspace_bytes": (c_size_t, [c_int64, c_int64, c_int64, c_int]),
    "grass_grad_row_norms": (c_int, [c_void_p, c_int64, c_void_p, c_int64, c_int, c_int64, c_int64,
                                     c_int64, c_void_p, c_void_p, c_size_t, c_void_p]),
    "grass_subspace_adam": (c_int, [c_void_p, c_int64, c_void_p, c_void_p, c_void_p, c_int64,
                                    c_int32, c_int64, c_double, c_double, c_double, c_double,
                                    c_int32, c_void_p]),
    "grass_scatter_update": (c_int, [c_void_p, c_int, c_int64, c_int64, c_int64, c_void_p, c_int64,
                                     c_void_p, c_void_p, c_int32, c_double, c_void_p]),
    "grass_adam_scatter": (c_int, [c_void_p, c_int64, c_void_p, c_void_p, c_void_p, c_int64, c_void_p,
                                   c_int, c_int64, c_int64, c_int64, c_void_p, c_void_p, c_int32,
                                   c_double, c_double, c_double, c_double, c_int32, c_double,
                                   c_void_p]),
    "grass_scatter_update_cols": (c_int, [c_void_p, c_int, c_int64, c_int64, c_int64, c_void_p,
                                          c_int64, c_void_p, c_void_p, c_int32, c_double, c_void_p]),
    "grass_device_status": (c_int, [c_void_p, ctypes.POINTER(c_int32)]),
    "grass_status_string": (ctypes.c_char_p, [c_int]),
    "grass_selftest_bounded_wait": (c_int, [c_int64, c_void_p]),
    "grass_profile_begin": (c_int, [c_int32]),
    "grass_profile_end": (c_int, [ctypes.POINTER(c_int32), ctypes.POINTER(ctypes.c_float),
                                  ctypes.POINTER(c_int32)]),
    "grass_profile_end_timeline": (c_int, [ctypes.POINTER(c_int32), ctypes.POINTER(ctypes.c_float),
                                           ctypes.POINTER(ctypes.c_float), ctypes.POINTER(c_int32)]),
}

KERNEL_NAMES = ["row_norms", "select", "gather", "project_tc", "splitk_reduce", "project_fp32",
                "adam", "scatter", "adam_scatter", "project_tc_dense"]


def load_library():
    """Load libgrass_b200.so (once).  There is no fallback: a missing library is an error."""
    global _LIB
    if _LIB is None:
        path = library_path()
        if not os.path.exists(path):
            raise RuntimeError(
                f"{path} is missing: build it with `python -m paper_2406_17660_b200.build` "
                "(needs nvcc); this package has no other execution path")
        lib = ctypes.CDLL(path)
        for name, (res, args) in _SIGNATURES.items():
            fn = getattr(lib, name)
            fn.restype, fn.argtypes = res, args
        _LIB = lib
    return _LIB


def exported_symbols():
    return sorted(_SIGNATURES)


def grass_status_string(status: int) -> str:
    return load_library().grass_status_string(int(status)).decode()


def _dtype_code(t: torch.Tensor) -> int:
    if t.dtype == torch.float32:
        return F32
    if t.dtype == torch.bfloat16:
        return BF16
    raise TypeError(f"unsupported dtype {t.dtype}")


def _ptr(t):
    return None if t is None else c_void_p(t.data_ptr())


def _ld(t: torch.Tensor) -> int:
    if t.dim() != 2 or t.stride(1) != 1:
        raise ValueError("expected a 2-D tensor with unit inner stride")
    return t.stride(0) if t.shape[0] > 1 else max(t.stride(0), t.shape[1])


def _stream():
    """torch's current stream on the current device, as a pointer."""
    return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice())


def _check(status: int, where: str):
    if status != 0:
        raise GrassError(status, where)


def _require(t, dtype, name):
    if t.dtype != dtype or not t.is_cuda:
        raise TypeError(f"{name} must be a CUDA tensor of {dtype}")


def grass_row_norms(G: torch.Tensor, norms: torch.Tensor) -> None:
    m, n = G.shape
    _require(norms, torch.float32, "norms")
    _check(load_library().grass_row_norms(_ptr(G), _dtype_code(G), m, n, _ld(G), _ptr(norms),
                                          _stream()), "grass_row_norms")


def grass_select_workspace_bytes(m: int, r: int, method: int) -> int:
    return int(load_library().grass_select_workspace_bytes(m, r, method))


def grass_select(norms, r, method, seed, layer_id, epoch, idx, rho, ws) -> None:
    _require(norms, torch.float32, "norms")
    _require(idx, torch.int32, "idx")
    _require(rho, torch.float32, "rho")
    ws_bytes = 0 if ws is None else ws.numel() * ws.element_size()
    _check(load_library().grass_select(_ptr(norms), norms.numel(), r, method, seed, layer_id, epoch,
                                       _ptr(idx), _ptr(rho), _ptr(ws), ws_bytes, _stream()),
           "grass_select")


def grass_select_static(norms, r, method, seed, layer_id, epoch, idx, rho) -> None:
    """grass_select with the library's built-in scratch: no workspace argument, nothing is
    allocated.  For callers that have tensors but no way to get device memory at this point
    (see include/grass.h for the size limit and the sharing rules)."""
    _require(norms, torch.float32, "norms")
    _require(idx, torch.int32, "idx")
    _require(rho, torch.float32, "rho")
    _check(load_library().grass_select_static(_ptr(norms), norms.numel(), r, method, seed, layer_id,
                                              epoch, _ptr(idx), _ptr(rho), _stream()),
           "grass_select_static")


def grass_project_workspace_bytes(T: int, m: int, n: int, r: int, dt: int) -> int:
    return int(load_library().grass_project_workspace_bytes(T, m, n, r, dt))


def grass_project_grad(dY, X, idx, rho, r, Gc, ws) -> None:
    T, m = dY.shape
    T2, n = X.shape
    if T2 != T or dY.dtype != X.dtype:
        raise ValueError("dY and X must share the token dimension and dtype")
    _require(Gc, torch.float32, "Gc")
    if idx is not None:
        _require(idx, torch.int32, "idx")
    if rho is not None:
        _require(rho, torch.float32, "rho")
    ws_bytes = 0 if ws is None else ws.numel() * ws.element_size()
    _check(load_library().grass_project_grad(_ptr(dY), _ld(dY), _ptr(X), _ld(X), _dtype_code(X), T,
                                             m, n, _ptr(idx), _ptr(rho), r, _ptr(Gc), _ld(Gc),
                                             _ptr(ws), ws_bytes, _stream()), "grass_project_grad")


def grass_grad_row_norms_workspace_bytes(T: int, m: int, n: int, dt: int) -> int:
    return int(load_library().grass_grad_row_norms_workspace_bytes(T, m, n, dt))


def grass_grad_row_norms(dY, X, norms, ws) -> None:
    T, m = dY.shape
    T2, n = X.shape
    if T2 != T or dY.dtype != X.dtype:
        raise ValueError("dY and X must share the token dimension and dtype")
    _require(norms, torch.float32, "norms")
    ws_bytes = 0 if ws is None else ws.numel() * ws.element_size()
    _check(load_library().grass_grad_row_norms(_ptr(dY), _ld(dY), _ptr(X), _ld(X), _dtype_code(X),
                                               T, m, n, _ptr(norms), _ptr(ws), ws_bytes, _stream()),
           "grass_grad_row_norms")


def grass_subspace_adam(Gc, M, V, U, lr, beta1, beta2, eps, step) -> None:
    r, n = M.shape
    for t, name in ((Gc, "Gc"), (M, "M"), (V, "V"), (U, "U")):
        _require(t, torch.float32, name)
    if _ld(V) != _ld(M) or _ld(U) != _ld(M):
        raise ValueError("M, V and U must share one row pitch")
    _check(load_library().grass_subspace_adam(_ptr(Gc), _ld(Gc), _ptr(M), _ptr(V), _ptr(U), _ld(M),
                                              r, n, lr, beta1, beta2, eps, step, _stream()),
           "grass_subspace_adam")


def grass_scatter_update(W, U, idx, rho, alpha) -> None:
    m, n = W.shape
    r = idx.numel()
    _require(U, torch.float32, "U")
    _require(idx, torch.int32, "idx")
    if rho is not None:
        _require(rho, torch.float32, "rho")
    _check(load_library().grass_scatter_update(_ptr(W), _dtype_code(W), m, n, _ld(W), _ptr(U),
                                               _ld(U), _ptr(idx), _ptr(rho), r, alpha, _stream()),
           "grass_scatter_update")


def grass_adam_scatter(Gc, M, V, U, W, idx, rho, lr, beta1, beta2, eps, step, alpha) -> None:
    """Adam on the r x n state and the row-sparse apply in one kernel; U may be None."""
    r, n = M.shape
    m = W.shape[0]
    for t, name in ((Gc, "Gc"), (M, "M"), (V, "V")):
        _require(t, torch.float32, name)
    if U is not None:
        _require(U, torch.float32, "U")
        if _ld(U) != _ld(M):
            raise ValueError("M, V and U must share one row pitch")
    if _ld(V) != _ld(M):
        raise ValueError("M and V must share one row pitch")
    _require(idx, torch.int32, "idx")
    _check(load_library().grass_adam_scatter(_ptr(Gc), _ld(Gc), _ptr(M), _ptr(V), _ptr(U), _ld(M),
                                             _ptr(W), _dtype_code(W), m, n, _ld(W), _ptr(idx),
                                             _ptr(rho), r, lr, beta1, beta2, eps, step, alpha,
                                             _stream()), "grass_adam_scatter")


def grass_scatter_update_cols(W, U, idx, rho, alpha) -> None:
    m, n = W.shape
    r = idx.numel()
    _require(U, torch.float32, "U")
    _require(idx, torch.int32, "idx")
    if rho is not None:
        _require(rho, torch.float32, "rho")
    _check(load_library().grass_scatter_update_cols(_ptr(W), _dtype_code(W), m, n, _ld(W), _ptr(U),
                                                    _ld(U), _ptr(idx), _ptr(rho), r, alpha,
                                                    _stream()), "grass_scatter_update_cols")


def grass_device_status(raise_on_error: bool = True):
    """Synchronise the current stream and return (status, detail) of the device status word."""
    detail = c_int32(0)
    status = load_library().grass_device_status(_stream(), ctypes.byref(detail))
    if status != 0 and raise_on_error:
        raise GrassError(status, f"device status (detail {detail.value})")
    return status, detail.value


def grass_profile_end_timeline():
    """Returns (launches_seen, [(kernel_name, start_ms, ms), ...]); start_ms counts from the start
    of the first recorded launch, across streams."""
    cap = grass_profile_begin.cap
    kid = (c_int32 * cap)()
    ms = (ctypes.c_float * cap)()
    st = (ctypes.c_float * cap)()
    n = c_int32(0)
    _check(load_library().grass_profile_end_timeline(kid, ms, st, ctypes.byref(n)),
           "grass_profile_end_timeline")
    timed = min(n.value, cap)
    return n.value, [(KERNEL_NAMES[kid[i]], float(st[i]), float(ms[i])) for i in range(timed)]


def grass_selftest_bounded_wait(limit_cycles: int) -> None:
    _check(load_library().grass_selftest_bounded_wait(limit_cycles, _stream()),
           "grass_selftest_bounded_wait")


def grass_profile_begin(max_launches: int) -> None:
    _check(load_library().grass_profile_begin(max_launches), "grass_profile_begin")
    grass_profile_begin.cap = max_launches


def grass_profile_end():
    """Returns (launches_seen, [(kernel_name, ms), ...]) for the launches that were timed."""
    cap = grass_profile_begin.cap
    kid = (c_int32 * cap)()
    ms = (ctypes.c_float * cap)()
    n = c_int32(0)
    _check(load_library().grass_profile_end(kid, ms, ctypes.byref(n)), "grass_profile_end")
    timed = min(n.value, cap)
    return n.value, [(KERNEL_NAMES[kid[i]], float(ms[i])) for i in range(timed)]


# ---- batched calls: `count` layers of one shape per launch ----
_SIGNATURES_BATCHED = {
    "grass_project_batched_workspace_bytes": (c_size_t, [c_int32, c_int64, c_int64, c_int64, c_int32]),
    "grass_project_grad_batched": (c_int, [c_int32, c_void_p, c_int64, c_void_p, c_int64, c_int64,
                                           c_int64, c_int64, c_void_p, c_void_p, c_int32, c_void_p,
                                           c_int64, c_void_p, c_size_t, c_void_p]),
    "grass_adam_scatter_batched": (c_int, [c_int32, c_void_p, c_int64, c_void_p, c_void_p, c_void_p,
                                           c_int64, c_void_p, c_int, c_int64, c_int64, c_int64,
                                           c_void_p, c_void_p, c_int32, c_double, c_double, c_double,
                                           c_double, c_int32, c_double, c_void_p]),
}
_SIGNATURES.update(_SIGNATURES_BATCHED)

GATHER_AUTO, GATHER_PREPASS, GATHER_IN_CTA, GATHER_COOPERATIVE = 0, 1, 2, 3
PAIR_AUTO, PAIR_NEVER, PAIR_ALWAYS = 0, 1, 2


class ProjectOpts(ctypes.Structure):
    """grass_project_opts_t: 0 in a field keeps the library's own choice."""
    _fields_ = [("gather", c_int32), ("n_blocks_per_cta", c_int32), ("cta_pair", c_int32),
                ("token_slices", c_int32), ("gather_warps", c_int32)]


class ProjectPlan(ctypes.Structure):
    """grass_project_plan_t."""
    _fields_ = [("gather", c_int32), ("rows_per_tile", c_int32), ("row_blocks", c_int32),
                ("n_blocks_per_cta", c_int32), ("ctas_per_slice", c_int32), ("cta_pair", c_int32),
                ("token_slices", c_int32), ("short_slices", c_int32), ("long_slice_tokens", c_int32),
                ("tokens_per_stage", c_int32), ("stages", c_int32),
                ("workspace_bytes", c_size_t)]


_SIGNATURES.update({
    "grass_project_plan": (c_int, [c_int32, c_int64, c_int64, c_int64, c_int32,
                                   ctypes.POINTER(ProjectOpts), ctypes.POINTER(ProjectPlan)]),
    "grass_plan_searches": (c_int64, []),
    "grass_step_plan": (c_int, [c_int32, c_int64, c_int64, c_int64, c_int32, ctypes.POINTER(ProjectPlan)]),
    "grass_project_grad_ex": (c_int, [c_int32, c_void_p, c_int64, c_void_p, c_int64, c_int64, c_int64,
                                      c_int64, c_void_p, c_void_p, c_int32, c_void_p, c_int64,
                                      c_void_p, c_size_t, ctypes.POINTER(ProjectOpts), c_void_p]),
})


def _opts(opts):
    if opts is None:
        return None
    if isinstance(opts, ProjectOpts):
        return ctypes.byref(opts)
    return ctypes.byref(ProjectOpts(**opts))


def grass_project_plan(count: int, T: int, m: int, n: int, r: int, opts=None) -> dict:
    """What grass_project_grad_ex would do for these arguments (host only, no GPU needed)."""
    plan = ProjectPlan()
    _check(load_library().grass_project_plan(count, T, m, n, r, _opts(opts), ctypes.byref(plan)),
           "grass_project_plan")
    return {name: int(getattr(plan, name)) for name, _ in ProjectPlan._fields_}


def grass_step_plan(count: int, T: int, m: int, n: int, r: int) -> dict:
    """What grass_layer_step does for bf16 layers of this shape on a regular iteration (host only)."""
    plan = ProjectPlan()
    _check(load_library().grass_step_plan(count, T, m, n, r, ctypes.byref(plan)), "grass_step_plan")
    return {name: int(getattr(plan, name)) for name, _ in ProjectPlan._fields_}


def grass_plan_searches() -> int:
    """How many plans the calling thread has searched for."""
    return int(load_library().grass_plan_searches())


def grass_project_grad_ex(dYs, Xs, idxs, rhos, r, Gcs, ws, opts=None) -> None:
    count = len(dYs)
    T, m = dYs[0].shape
    n = Xs[0].shape[1]
    for t in Gcs:
        _require(t, torch.float32, "Gc")
    for t in idxs:
        _require(t, torch.int32, "idx")
    keep = (_ptr_array(dYs), _ptr_array(Xs), _ptr_array(idxs), _ptr_array(rhos), _ptr_array(Gcs))
    ws_bytes = 0 if ws is None else ws.numel() * ws.element_size()
    _check(load_library().grass_project_grad_ex(
        count, keep[0], _ld(dYs[0]), keep[1], _ld(Xs[0]), T, m, n, keep[2], keep[3], r, keep[4],
        _ld(Gcs[0]), _ptr(ws), ws_bytes, _opts(opts), _stream()), "grass_project_grad_ex")


def _ptr_array(tensors):
    """Host array of device pointers (None entries become NULL); None -> NULL array."""
    if tensors is None:
        return None
    arr = (c_void_p * len(tensors))(*[None if t is None else t.data_ptr() for t in tensors])
    return arr


def grass_project_batched_workspace_bytes(count: int, T: int, m: int, n: int, r: int) -> int:
    return int(load_library().grass_project_batched_workspace_bytes(count, T, m, n, r))


def grass_project_grad_batched(dYs, Xs, idxs, rhos, r, Gcs, ws) -> None:
    count = len(dYs)
    T, m = dYs[0].shape
    n = Xs[0].shape[1]
    for t in Gcs:
        _require(t, torch.float32, "Gc")
    for t in idxs:
        _require(t, torch.int32, "idx")
    keep = (_ptr_array(dYs), _ptr_array(Xs), _ptr_array(idxs), _ptr_array(rhos), _ptr_array(Gcs))
    ws_bytes = 0 if ws is None else ws.numel() * ws.element_size()
    _check(load_library().grass_project_grad_batched(
        count, keep[0], _ld(dYs[0]), keep[1], _ld(Xs[0]), T, m, n, keep[2], keep[3], r, keep[4],
        _ld(Gcs[0]), _ptr(ws), ws_bytes, _stream()), "grass_project_grad_batched")


def grass_adam_scatter_batched(Gcs, Ms, Vs, Us, Ws, idxs, rhos, lr, beta1, beta2, eps, step,
                               alpha) -> None:
    count = len(Gcs)
    r, n = Ms[0].shape
    m = Ws[0].shape[0]
    keep = (_ptr_array(Gcs), _ptr_array(Ms), _ptr_array(Vs), _ptr_array(Us), _ptr_array(Ws),
            _ptr_array(idxs), _ptr_array(rhos))
    _check(load_library().grass_adam_scatter_batched(
        count, keep[0], _ld(Gcs[0]), keep[1], keep[2], keep[3], _ld(Ms[0]), keep[4],
        _dtype_code(Ws[0]), m, n, _ld(Ws[0]), keep[5], keep[6], r, lr, beta1, beta2, eps, step,
        alpha, _stream()), "grass_adam_scatter_batched")


# ---- one call per layer-step ----
MAX_GROUP = 8
_PtrArray = c_void_p * MAX_GROUP


class LayerStep(ctypes.Structure):
    """grass_step_t: the arguments of grass_layer_step."""
    _fields_ = [("count", c_int32), ("dt", c_int32), ("wdt", c_int32), ("r", c_int32),
                ("side", c_int32), ("T", c_int64), ("m", c_int64), ("n", c_int64),
                ("lddy", c_int64), ("ldx", c_int64), ("ldgc", c_int64), ("ldstate", c_int64),
                ("ldw", c_int64),
                ("dY", _PtrArray), ("X", _PtrArray), ("idx", _PtrArray), ("rho", _PtrArray),
                ("Gc", _PtrArray), ("M", _PtrArray), ("V", _PtrArray), ("U", _PtrArray),
                ("W", _PtrArray),
                ("lr", c_double), ("beta1", c_double), ("beta2", c_double), ("eps", c_double),
                ("alpha", c_double), ("step", c_int32), ("ws", c_void_p), ("ws_bytes", c_size_t)]


_SIGNATURES["grass_layer_step"] = (c_int, [ctypes.POINTER(LayerStep), c_void_p])


class Refresh(ctypes.Structure):
    """grass_refresh_t: what grass_refresh_step takes beside a grass_step_t."""
    _fields_ = [("method", c_int32), ("layer_id", c_uint32), ("epoch", c_uint32),
                ("reset_state", c_int32), ("seed", c_uint64), ("norms", c_void_p),
                ("norm_ws", c_void_p), ("norm_ws_bytes", c_size_t),
                ("select_ws", c_void_p), ("select_ws_bytes", c_size_t)]


_SIGNATURES["grass_refresh_step"] = (c_int, [ctypes.POINTER(LayerStep), ctypes.POINTER(Refresh), c_void_p])
_SIGNATURES["grass_refresh_workspace_bytes"] = (c_size_t, [c_int64, c_int64, c_int64, c_int32, c_int])
_SIGNATURES["grass_refresh_keeps_gradient"] = (c_int, [c_int64, c_int64, c_int64, c_int32, c_int])


def grass_refresh_workspace_bytes(T: int, m: int, n: int, r: int, dt: int) -> int:
    return int(load_library().grass_refresh_workspace_bytes(T, m, n, r, dt))


def grass_refresh_keeps_gradient(T: int, m: int, n: int, r: int, dt: int) -> bool:
    return bool(load_library().grass_refresh_keeps_gradient(T, m, n, r, dt))


_F32, _I32 = torch.float32, torch.int32
_CODES = {torch.float32: F32, torch.bfloat16: BF16}


_SCAN = None


def _accepted():
    """accepted() of the module that is built for this torch and this Python (csrc/scan.cpp)."""
    global _SCAN
    if _SCAN is None:
        from .build import scan_path
        path = scan_path()
        if not os.path.exists(path):
            raise RuntimeError(f"{path} is missing: build it with `python -m paper_2406_17660_b200.build`")
        spec = importlib.util.spec_from_file_location(f"{__package__}._scan", path)
        module = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(module)
        _SCAN = module.accepted
    return _SCAN


class LayerStepCall:
    """A grass_step_t and what fills it: state() for the buffers a layer owns, inputs() for what
    arrives anew with every call.  Both look at everything each time they are called; a step of a small layer takes
    the GPU no longer than that takes the host.  So a native scan goes first: tensors that are alike in all but
    their addresses to the ones that the checks let through last need only their addresses put in place (state()
    of a layer 2.7 -> 0.2 us, inputs() 1.2 -> 0.1)."""

    def __init__(self):
        self.args = a = LayerStep()
        self._ref = ctypes.byref(a)
        self._slots = (a.dY, a.X, a.idx, a.rho, a.Gc, a.M, a.V, a.U, a.W)
        self._refresh = f = Refresh()
        self._refresh_ref = ctypes.byref(f)
        lib = load_library()
        self._launch, self._launch_refresh = lib.grass_layer_step, lib.grass_refresh_step
        self._now = None
        self._accepted = _accepted()
        self._at = ctypes.addressof(a) + LayerStep.dY.offset     # of the pointers: nine fields of MAX_GROUP each
        self._forget()

    def _forget(self):
        """What the checks let through last, as the scan describes it: per layer with and without cols, and inputs."""
        self._alike = ([None] * MAX_GROUP, [None] * MAX_GROUP)
        self._alike_inputs = None

    def __reduce__(self):
        return (LayerStepCall, ())       # a copied layer marshals its own buffers anew

    def state(self, g, idx, rho, Gc, M, V, U, W, cols=False):
        """Layer g's selection, state and weights; layer 0 sets sizes, pitches and W's dtype.
        cols: idx selects columns of W, whose rows the state runs along."""
        k = 1 if cols else 0
        seen = self._accepted(self._at + 8 * (2 * MAX_GROUP + g), self._alike[k][g], idx, rho, Gc, M, V, U, W)
        if seen is True:
            return
        if not (M.dtype is _F32 and V.dtype is _F32 and Gc.dtype is _F32 and idx.dtype is _I32
                and (rho is None or rho.dtype is _F32) and (U is None or U.dtype is _F32)):
            raise TypeError("Gc, M, V, U and rho must be float32 and idx int32")
        if not (M.is_cuda and V.is_cuda and Gc.is_cuda and W.is_cuda and idx.is_cuda
                and (rho is None or rho.is_cuda) and (U is None or U.is_cuda)):
            raise TypeError("a layer step takes CUDA tensors")
        shape, stride, wshape, wstride = M.shape, M.stride(), W.shape, W.stride()
        r, n = shape
        if V.shape != shape or Gc.shape != shape or len(wshape) != 2 or wshape[1 - k] != n or \
                (U is not None and U.shape != shape):
            raise ValueError("Gc, M, V and U must be r x n and W m x n")
        if idx.numel() < r or not idx.is_contiguous() or \
                (rho is not None and (rho.numel() < r or not rho.is_contiguous())):
            raise ValueError("idx and rho must hold one value per selected row, next to one another")
        if stride[1] != 1 or wstride[1] != 1:
            raise ValueError("expected a 2-D tensor with unit inner stride")
        ldm = stride[0] if r > 1 else max(stride[0], n)
        ldw = wstride[0] if wshape[0] > 1 else max(wstride[0], wshape[1])
        if (V.stride() != stride and _ld(V) != ldm) or \
                (U is not None and U.stride() != stride and _ld(U) != ldm):
            raise ValueError("M, V and U must share one row pitch")
        code = _CODES.get(W.dtype)
        if code is None:
            raise TypeError(f"unsupported dtype {W.dtype}")
        own = (r, n, wshape[k], code, ldm if Gc.stride() == stride else _ld(Gc), ldm, ldw, k)
        if g == 0:
            self._forget()                 # the other layers and the inputs are compared with layer 0
            a = self.args
            self._own = own
            a.r, a.n, a.m, a.wdt, a.ldgc, a.ldstate, a.ldw, a.side = own
        elif own != self._own:
            raise ValueError("the layers of a call must share shapes, pitches and dtypes")
        _, _, si, sr, sg, sm, sv, su, sw = self._slots
        si[g] = idx.data_ptr()
        sr[g] = None if rho is None else rho.data_ptr()
        sg[g], sm[g], sv[g], sw[g] = Gc.data_ptr(), M.data_ptr(), V.data_ptr(), W.data_ptr()
        su[g] = None if U is None else U.data_ptr()
        self._alike[k][g] = seen

    def inputs(self, g, dY, X):
        """Layer g's dY (T x m) and X (T x n); after state(0, ..)."""
        seen = self._accepted(self._at + 8 * g, self._alike_inputs, dY, X)
        if seen is True:
            return
        if not (dY.is_cuda and X.is_cuda):
            raise TypeError("a layer step takes CUDA tensors")
        now = (dY.shape, X.shape, dY.stride(), X.stride(), dY.dtype, X.dtype)
        if g == 0:
            yshape, xshape, ystride, xstride, dt, dt2 = now
            if len(yshape) != 2 or len(xshape) != 2:
                raise ValueError("expected a 2-D tensor with unit inner stride")
            if yshape[0] != xshape[0] or dt is not dt2:
                raise ValueError("dY and X must share the token dimension and dtype")
            _, n, m = self._own[:3]
            if yshape[1] != m or xshape[1] != n:
                raise ValueError("dY must be T x m and X T x n for an m x n layer")
            code = _CODES.get(dt)
            if code is None:
                raise TypeError(f"unsupported dtype {dt}")
            if ystride[1] != 1 or xstride[1] != 1:
                raise ValueError("expected a 2-D tensor with unit inner stride")
            a, T = self.args, xshape[0]
            a.T, a.dt = T, code
            a.lddy, a.ldx = (ystride[0], xstride[0]) if T > 1 else (max(ystride[0], m), max(xstride[0], n))
            self._now, self._alike_inputs = now, seen     # one record: a refused pair leaves neither
        elif now != self._now and not (             # (one token has no pitch)
                now[0][0] == 1 and now[:2] == self._now[:2] and now[4:] == self._now[4:]
                and now[2][1] == now[3][1] == 1):
            raise ValueError("the layers of a call must share shapes, pitches and dtypes")
        s = self._slots
        s[0][g], s[1][g] = dY.data_ptr(), X.data_ptr()

    def _scalars(self, count, ws, hyper, step):
        a = self.args
        a.count, a.step = count, step
        a.lr, a.beta1, a.beta2, a.eps, a.alpha = hyper
        a.ws, a.ws_bytes = (None, 0) if ws is None else (ws.data_ptr(), ws.nbytes)

    def launch(self, count, ws, lr, beta1, beta2, eps, step, alpha) -> None:
        self._scalars(count, ws, (lr, beta1, beta2, eps, alpha), step)
        status = self._launch(self._ref, _stream())
        if status != 0:
            raise GrassError(status, "grass_layer_step")

    def refresh(self, ws, lr, beta1, beta2, eps, step, alpha, method, seed, layer_id, epoch, reset_state,
                norms, norm_ws, select_ws) -> None:
        """grass_refresh_step on layer 0."""
        self._scalars(1, ws, (lr, beta1, beta2, eps, alpha), step)
        if norms.dtype is not _F32 or not norms.is_cuda:
            raise TypeError("norms must be a CUDA tensor of torch.float32")
        if norms.numel() < self.args.m:
            raise ValueError("norms must hold one value per row")
        f = self._refresh
        f.method, f.layer_id, f.epoch, f.reset_state, f.seed = method, layer_id, epoch, 1 if reset_state else 0, seed
        f.norms, f.norm_ws, f.norm_ws_bytes = norms.data_ptr(), norm_ws.data_ptr(), norm_ws.nbytes
        f.select_ws, f.select_ws_bytes = (None, 0) if select_ws is None else (select_ws.data_ptr(), select_ws.nbytes)
        status = self._launch_refresh(self._ref, self._refresh_ref, _stream())
        if status != 0:
            raise GrassError(status, "grass_refresh_step")


def grass_layer_step(dYs, Xs, idxs, rhos, Gcs, Ms, Vs, Us, Ws, ws, lr, beta1, beta2, eps, step,
                     alpha) -> None:
    """Projection, Adam and row-sparse apply of up to 8 same-shaped layers in one call.  rhos and
    Us, or entries of them, may be None."""
    none = [None] * len(dYs)
    call = LayerStepCall()
    for g, own in enumerate(zip(idxs, rhos or none, Gcs, Ms, Vs, Us or none, Ws)):
        call.state(g, *own)
        call.inputs(g, dYs[g], Xs[g])
    call.launch(len(dYs), ws, lr, beta1, beta2, eps, step, alpha)
