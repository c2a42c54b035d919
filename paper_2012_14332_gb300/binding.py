"""Python binding of the C ABI in ``include/abc_gb300.h`` (ctypes).

Argument marshalling only: host arrays are passed as pointers, device buffers
are torch CUDA tensors (PyTorch supplies device memory and the current
stream); every step of the method runs in the CUDA library. The library must
be built (``paper_2012_14332_gb300.build.build()``); there is no fallback.
"""
import ctypes
import math
import os
import threading

import numpy as np
import torch

from . import build as _build

ABC_EXACT, ABC_FAST, ABC_VARIANCE_LITERAL = 0, 1, 4
ABC_OK, ABC_ERR_INVALID_ARG, ABC_ERR_CAPACITY, ABC_ERR_CUDA, ABC_ERR_TIMEOUT, ABC_ERR_NOMEM = range(6)
ABC_T_MAX = 4096

PAPER_LO = (0.0,) * 8
PAPER_HI = (1.0, 100.0, 2.0, 1.0, 1.0, 1.0, 1.0, 2.0)   # Sec. 2.1, Eq. 2

EXPORTED = ("abc_sample", "abc_distances", "abc_simulate", "abc_step", "abc_kth_smallest", "abc_select_below",
            "abc_sample_quantile", "abc_strerror",
            "abc_last_error", "abc_version", "abc_last_simulated_days", "abc_sample_noalloc", "abc_plan_create",
            "abc_plan_reset", "abc_plan_run", "abc_plan_run_graph", "abc_plan_tune", "abc_plan_results",
            "abc_plan_copy_results", "abc_plan_set_region", "abc_plan_set_shape", "abc_plan_destroy", "abc_maf_create",
            "abc_maf_init_random", "abc_maf_param_count", "abc_maf_set_params", "abc_maf_get_params", "abc_maf_sample", "abc_maf_log_q",
            "abc_maf_gradient", "abc_maf_adam_step", "abc_maf_train", "abc_maf_destroy", "abc_smc_run", "abc_project", "abc_pmc_run", "abc_pmc_propose",
            "abc_pmc_weights")
ABC_MAX_REGIONS = 32
ABC_NOALLOC_T_MAX = 1024


class AbcPriorBox(ctypes.Structure):
    _fields_ = [("lo", ctypes.c_float * 8), ("hi", ctypes.c_float * 8)]


class AbcRegion(ctypes.Structure):
    _fields_ = [("observed", ctypes.c_void_p), ("T", ctypes.c_int32), ("N_pop", ctypes.c_int64),
                ("eps", ctypes.c_double), ("n_samples", ctypes.c_uint64), ("first_index", ctypes.c_uint64),
                ("stream", ctypes.c_uint32), ("capacity", ctypes.c_uint64), ("theta_in", ctypes.c_void_p)]


class AbcLaunchShape(ctypes.Structure):
    _fields_ = [("block_threads", ctypes.c_int32), ("pairs_per_iteration", ctypes.c_int32),
                ("blocks_per_sm", ctypes.c_int32), ("lean", ctypes.c_int32), ("ms", ctypes.c_float)]


class AbcSmcConfig(ctypes.Structure):
    _fields_ = [("rounds", ctypes.c_int32), ("sims_per_round", ctypes.c_uint64), ("eps0", ctypes.c_double),
                ("eps_factor", ctypes.c_double), ("ess_min", ctypes.c_double), ("flow_blocks", ctypes.c_int32),
                ("flow_hidden", ctypes.c_int32), ("train_steps", ctypes.c_int32), ("train_batch", ctypes.c_int32),
                ("train_lr", ctypes.c_float), ("seed", ctypes.c_uint64), ("capacity", ctypes.c_uint64),
                ("mode", ctypes.c_int), ("defensive", ctypes.c_double), ("val_fraction", ctypes.c_double),
                ("train_weight_power", ctypes.c_double), ("fresh_init", ctypes.c_int32),
                ("proposal_scale", ctypes.c_double), ("fallback_rule", ctypes.c_int32)]


class AbcSmcRound(ctypes.Structure):
    _fields_ = [("eps", ctypes.c_double), ("proposal", ctypes.c_int32), ("n_sims", ctypes.c_uint64),
                ("n_accepted", ctypes.c_uint64), ("simulated_days", ctypes.c_uint64),
                ("ess_fraction", ctypes.c_double), ("train_loss", ctypes.c_float), ("ms_propose", ctypes.c_float),
                ("ms_simulate", ctypes.c_float), ("ms_train", ctypes.c_float), ("n_defensive", ctypes.c_uint64),
                ("n_defensive_accepted", ctypes.c_uint64)]


class AbcSmcRegion(ctypes.Structure):
    _fields_ = [("observed", ctypes.c_void_p), ("T", ctypes.c_int32), ("N_pop", ctypes.c_int64),
                ("eps", ctypes.c_double), ("theta_out", ctypes.c_void_p), ("weight_out", ctypes.c_void_p),
                ("dist_out", ctypes.c_void_p), ("capacity", ctypes.c_uint64), ("n_pooled", ctypes.c_uint64),
                ("n_out", ctypes.c_uint64)]


class AbcSmcStreamConfig(ctypes.Structure):
    _fields_ = [("base", AbcSmcConfig), ("shrink_rounds", ctypes.c_int32), ("train_steps_warm", ctypes.c_int32)]


class AbcPmcConfig(ctypes.Structure):
    _fields_ = [("rounds", ctypes.c_int32), ("n_particles", ctypes.c_uint64), ("batch", ctypes.c_uint64),
                ("max_batches", ctypes.c_int32), ("eps0", ctypes.c_double), ("eps_factor", ctypes.c_double),
                ("seed", ctypes.c_uint64), ("capacity", ctypes.c_uint64), ("mode", ctypes.c_int)]


class AbcPmcRound(ctypes.Structure):
    _fields_ = [("eps", ctypes.c_double), ("n_sims", ctypes.c_uint64), ("n_accepted", ctypes.c_uint64),
                ("ess_fraction", ctypes.c_double), ("ms", ctypes.c_float)]


class AbcError(RuntimeError):
    def __init__(self, status, message):
        super().__init__("%s: %s" % (_strerror(status), message))
        self.status = status
        self.message = message


_lock = threading.Lock()
_lib = None


def library_path():
    return _build.LIB


def load(path=None):
    """Load the CUDA library (raises if it has not been built)."""
    global _lib
    with _lock:
        if _lib is not None and path is None:
            return _lib
        p = path or _build.LIB
        if not os.path.exists(p):
            raise ImportError("CUDA library %s is not built; run paper_2012_14332_gb300.build.build()" % p)
        L = ctypes.CDLL(p)
        vp, u64, i32, i64, u32 = ctypes.c_void_p, ctypes.c_uint64, ctypes.c_int32, ctypes.c_int64, ctypes.c_uint32
        box = ctypes.POINTER(AbcPriorBox)
        L.abc_sample.argtypes = [box, vp, i32, i64, ctypes.c_double, u64, u64, u32, ctypes.c_int, u64, vp, vp, vp,
                                 u64, ctypes.POINTER(ctypes.c_uint64), vp]
        L.abc_sample_noalloc.argtypes = list(L.abc_sample.argtypes)
        L.abc_distances.argtypes = [box, vp, i32, i64, u64, u64, u32, ctypes.c_int, u64, vp, vp, vp]
        L.abc_simulate.argtypes = [vp, vp, u64, vp, i32, i64, u64, u32, ctypes.c_int, vp, vp]
        L.abc_step.argtypes = [vp, vp, vp, vp, u64, i64, u64, u32, ctypes.c_int, vp, vp, vp]
        L.abc_kth_smallest.argtypes = [vp, u64, u64, ctypes.POINTER(ctypes.c_double), vp]
        L.abc_select_below.argtypes = [vp, vp, u64, ctypes.c_double, u64, vp, vp, vp, u64,
                                       ctypes.POINTER(ctypes.c_uint64), vp]
        L.abc_sample_quantile.argtypes = [box, vp, i32, i64, u64, u64, u64, u32, ctypes.c_int, u64, vp, vp, vp, u64,
                                          ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_uint64), vp]
        L.abc_observed_create.argtypes = [vp, i32, i64, ctypes.POINTER(ctypes.c_void_p)]
        L.abc_observed_destroy.argtypes = [vp]
        L.abc_sample_async.argtypes = [box, vp, ctypes.c_double, u64, u64, u32, ctypes.c_int, u64, vp, vp, vp, u64,
                                       vp, vp]
        L.abc_sample_until.argtypes = [box, vp, ctypes.c_double, u64, u64, u64, u64, u32, ctypes.c_int, u64, vp, vp,
                                       vp, u64, ctypes.POINTER(ctypes.c_uint64), ctypes.POINTER(ctypes.c_uint64), vp]
        for nm in ("abc_sample", "abc_sample_noalloc", "abc_distances", "abc_simulate", "abc_step",
                   "abc_kth_smallest", "abc_select_below", "abc_sample_quantile", "abc_observed_create",
                   "abc_observed_destroy", "abc_sample_async", "abc_sample_until"):
            getattr(L, nm).restype = ctypes.c_int
        L.abc_strerror.argtypes = [ctypes.c_int]
        L.abc_strerror.restype = ctypes.c_char_p
        L.abc_last_error.argtypes = []
        L.abc_last_error.restype = ctypes.c_char_p
        L.abc_version.restype = ctypes.c_int
        pp = ctypes.c_void_p
        L.abc_plan_create.argtypes = [box, ctypes.POINTER(AbcRegion), i32, u64, ctypes.c_int, ctypes.POINTER(pp)]
        L.abc_plan_reset.argtypes = [pp, vp]
        L.abc_plan_run.argtypes = [pp, vp]
        L.abc_plan_run_graph.argtypes = [pp, i32, vp]
        L.abc_plan_tune.argtypes = [pp, vp, ctypes.POINTER(AbcLaunchShape), i32, ctypes.POINTER(ctypes.c_int32),
                                    ctypes.POINTER(AbcLaunchShape)]
        L.abc_plan_results.argtypes = [pp, i32, ctypes.POINTER(ctypes.c_uint64), ctypes.POINTER(ctypes.c_uint64),
                                       vp, vp, vp, vp]
        L.abc_plan_copy_results.argtypes = [pp, i32, vp, vp, vp, u64, ctypes.POINTER(ctypes.c_uint64), vp]
        L.abc_plan_set_region.argtypes = [pp, i32, vp, u64]
        L.abc_plan_destroy.argtypes = [pp]
        for nm in ("abc_plan_create", "abc_plan_reset", "abc_plan_run", "abc_plan_run_graph", "abc_plan_tune",
                   "abc_plan_results", "abc_plan_copy_results", "abc_plan_set_region", "abc_plan_destroy"):
            getattr(L, nm).restype = ctypes.c_int
        L.abc_maf_create.argtypes = [i32, i32, box, ctypes.POINTER(pp)]
        L.abc_maf_init_random.argtypes = [pp, u64, ctypes.c_float]
        L.abc_maf_init_random.restype = ctypes.c_int
        L.abc_maf_param_count.argtypes = [pp]
        L.abc_maf_param_count.restype = ctypes.c_int64
        L.abc_maf_set_params.argtypes = [pp, vp]
        L.abc_maf_get_params.argtypes = [pp, vp]
        L.abc_maf_sample.argtypes = [pp, u64, vp, u64, u32, u64, vp, vp, vp]
        L.abc_maf_log_q.argtypes = [pp, u64, vp, vp, vp]
        L.abc_maf_gradient.argtypes = [pp, u64, vp, vp, ctypes.POINTER(ctypes.c_float), vp, vp]
        L.abc_maf_adam_step.argtypes = [pp, ctypes.c_float, ctypes.c_float, ctypes.c_float, ctypes.c_float, vp]
        L.abc_maf_train.argtypes = [pp, u64, vp, vp, i32, i32, ctypes.c_float, u64, ctypes.POINTER(ctypes.c_float),
                                    vp]
        L.abc_maf_destroy.argtypes = [pp]
        L.abc_maf_create_multi.argtypes = [i32, i32, i32, box, ctypes.POINTER(pp)]
        L.abc_maf_flow_count.argtypes = [pp]
        L.abc_maf_flow_count.restype = ctypes.c_int32
        L.abc_maf_set_proposal_scale.argtypes = [pp, ctypes.c_float]
        L.abc_maf_set_proposal_scale.restype = ctypes.c_int
        L.abc_maf_test_hold_products.argtypes = [pp, ctypes.c_int32]
        L.abc_maf_test_hold_products.restype = ctypes.c_int
        L.abc_maf_check.argtypes = [pp, vp]
        L.abc_maf_check.restype = ctypes.c_int
        L.abc_maf_sample_at.argtypes = [pp, i32, u64, vp, u64, u32, u64, vp, vp, vp]
        L.abc_maf_log_q_at.argtypes = [pp, i32, u64, vp, vp, vp]
        L.abc_maf_train_flows.argtypes = [pp, vp, vp, vp, i32, i32, ctypes.c_float, u64, ctypes.c_float, vp, vp]
        for nm in ("abc_maf_create_multi", "abc_maf_sample_at", "abc_maf_log_q_at", "abc_maf_train_flows"):
            getattr(L, nm).restype = ctypes.c_int
        for nm in ("abc_maf_create", "abc_maf_set_params", "abc_maf_get_params", "abc_maf_sample", "abc_maf_log_q",
                   "abc_maf_gradient", "abc_maf_adam_step", "abc_maf_train", "abc_maf_destroy", "abc_smc_run", "abc_project", "abc_pmc_run", "abc_pmc_propose",
            "abc_pmc_weights"):
            getattr(L, nm).restype = ctypes.c_int
        L.abc_project.argtypes = [vp, vp, u64, vp, i32, i64, u64, u32, ctypes.c_int, vp, i32, vp, vp]
        L.abc_project.restype = ctypes.c_int
        L.abc_pmc_run.argtypes = [box, vp, i32, i64, ctypes.POINTER(AbcPmcConfig), ctypes.POINTER(AbcPmcRound), vp, vp,
                                  vp, ctypes.POINTER(ctypes.c_uint64), vp]
        L.abc_pmc_propose.argtypes = [box, vp, vp, u64, vp, u64, u64, u64, vp, vp]
        L.abc_pmc_weights.argtypes = [vp, u64, vp, vp, u64, vp, vp, vp]
        for nm in ("abc_pmc_run", "abc_pmc_propose", "abc_pmc_weights"):
            getattr(L, nm).restype = ctypes.c_int
        L.abc_smc_run.argtypes = [box, vp, i32, i64, ctypes.POINTER(AbcSmcConfig), ctypes.POINTER(AbcSmcRound), vp, vp,
                                  vp, ctypes.POINTER(ctypes.c_uint64), vp]
        L.abc_smc_run.restype = ctypes.c_int
        L.abc_smc_run_regions.argtypes = [box, ctypes.POINTER(AbcSmcRegion), i32, ctypes.POINTER(AbcSmcStreamConfig),
                                          ctypes.POINTER(AbcSmcRound), vp]
        L.abc_smc_run_regions.restype = ctypes.c_int
        L.abc_plan_set_eps.argtypes = [pp, i32, ctypes.c_double]
        L.abc_plan_set_eps.restype = ctypes.c_int
        L.abc_plan_set_shape.argtypes = [pp, ctypes.POINTER(AbcLaunchShape)]
        L.abc_plan_set_shape.restype = ctypes.c_int
        L.abc_last_simulated_days.argtypes = []
        L.abc_last_simulated_days.restype = ctypes.c_uint64
        if path is None:
            _lib = L
        return L


def _strerror(status):
    try:
        return load().abc_strerror(int(status)).decode()
    except ImportError:
        return "status %d" % status


def _check(L, status, allow=()):
    if status != ABC_OK and status not in allow:
        raise AbcError(status, L.abc_last_error().decode())
    return status


_MODES = {"exact": 0, "fast": 1, "exact_literal": 4, "fast_literal": 5}


def _mode(mode):
    """'exact' or 'fast', with '_literal' for the literal-variance model
    variant (ABC_VARIANCE_LITERAL), or the ABI's integer value."""
    if isinstance(mode, str) and mode in _MODES:
        return _MODES[mode]
    if isinstance(mode, int) and mode in _MODES.values():
        return mode
    raise ValueError("mode must be one of %s" % ", ".join(_MODES))


def prior_box(lo=PAPER_LO, hi=PAPER_HI):
    b = AbcPriorBox()
    lo = np.asarray(lo, dtype=np.float32).reshape(8)
    hi = np.asarray(hi, dtype=np.float32).reshape(8)
    for j in range(8):
        b.lo[j] = float(lo[j])
        b.hi[j] = float(hi[j])
    return b


# The helpers below run on every call; a call of a few samples takes some 30 us
# on the device, so each argument is marshalled in well under a microsecond:
# addresses are plain integers, sizes are multiplied without numpy, and the
# default prior box (immutable tuples) is laid out once.
_PAPER_BOX = prior_box()


def _box(lo, hi):
    return ctypes.byref(_PAPER_BOX if lo is PAPER_LO and hi is PAPER_HI else prior_box(lo, hi))


def _host_i32(a):
    a = np.ascontiguousarray(a, dtype=np.int32)
    return a, a.__array_interface__["data"][0]


def _stream(cuda_stream):
    if cuda_stream is None:
        return torch._C._cuda_getCurrentRawStream(torch.cuda.current_device())
    if isinstance(cuda_stream, torch.cuda.Stream):
        return cuda_stream.cuda_stream
    return int(cuda_stream)


def _dev(t, dtype, shape):
    assert t.is_cuda and t.dtype == dtype and t.is_contiguous(), (t.device, t.dtype)
    assert t.numel() >= math.prod(shape), (t.shape, shape)
    return t.data_ptr()


def _first(t, m):
    """t[:m], and t itself where that is all of it."""
    return t if t.shape[0] == m else t[:m]


def abc_sample(observed, N_pop, eps, n_samples, seed, stream=0, mode="fast", first_index=0, lo=PAPER_LO,
               hi=PAPER_HI, capacity=None, out=None, cuda_stream=None, allow_overflow=False):
    """ABC rejection over [first_index, first_index + n_samples).

    observed: host int32 [3, T+1] (rows A, R, D). Returns
    (theta [m, 8] f32, dist [m] f64, idx [m] u64 (as int64 storage), n_accepted)
    as CUDA tensors, m = min(n_accepted, capacity), in unspecified order.
    """
    L = load()
    obs, obs_p = _host_i32(observed)
    T = obs.shape[1] - 1
    if capacity is None:
        capacity = max(1024, int(n_samples) // 100)
    dev = torch.device("cuda", torch.cuda.current_device())
    if out is None:
        theta = torch.empty((capacity, 8), dtype=torch.float32, device=dev)
        dist = torch.empty((capacity,), dtype=torch.float64, device=dev)
        idx = torch.empty((capacity,), dtype=torch.int64, device=dev)
    else:
        theta, dist, idx = out
    nacc = ctypes.c_uint64(0)
    b = _box(lo, hi)
    st = L.abc_sample(b, obs_p, T, int(N_pop), float(eps), int(n_samples), int(seed), int(stream),
                      _mode(mode), int(first_index), _dev(theta, torch.float32, (capacity, 8)),
                      _dev(dist, torch.float64, (capacity,)), _dev(idx, torch.int64, (capacity,)), int(capacity),
                      ctypes.byref(nacc), _stream(cuda_stream))
    _check(L, st, allow=(ABC_ERR_CAPACITY,) if allow_overflow else ())
    n = int(nacc.value)
    m = min(n, capacity)
    return _first(theta, m), _first(dist, m), _first(idx, m), n


class Observed:
    """A region's observed series (host int32 [3, T+1]) uploaded once to the
    current device, for abc_sample_async."""

    def __init__(self, observed, N_pop):
        L = load()
        obs, obs_p = _host_i32(observed)
        self.T = obs.shape[1] - 1
        self.N_pop = int(N_pop)
        h = ctypes.c_void_p()
        _check(L, L.abc_observed_create(obs_p, self.T, self.N_pop, ctypes.byref(h)))
        self._h = h

    @property
    def handle(self):
        if self._h is None:
            raise ValueError("observed series handle is closed")
        return self._h

    def close(self):
        if self._h is not None:
            _check(load(), load().abc_observed_destroy(self._h))
            self._h = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def abc_observed_create(observed, N_pop):
    """The observed series uploaded to the current device (an Observed)."""
    return Observed(observed, N_pop)


def abc_observed_destroy(obs):
    obs.close()


def abc_sample_async(obs, eps, n_samples, seed, out, counters, stream=0, mode="fast", first_index=0, lo=PAPER_LO,
                     hi=PAPER_HI, cuda_stream=None):
    """Enqueue ABC rejection for one chunk without waiting for it: obs is an
    Observed, out = (theta [cap, 8] f32, dist [cap] f64, idx [cap] int64) and
    counters a CUDA int64 tensor of >= 3 entries, all on the current device.
    When the stream gets there, counters[0] = accepted (may exceed cap),
    counters[1] = the claim counter (>= n_samples), counters[2] = simulated days."""
    L = load()
    theta, dist, idx = out
    capacity = theta.shape[0]
    if counters.dtype != torch.int64 or not counters.is_cuda or counters.numel() < 3 or not counters.is_contiguous():
        raise ValueError("counters must be a contiguous CUDA int64 tensor of >= 3 entries")
    b = _box(lo, hi)
    _check(L, L.abc_sample_async(b, obs.handle, float(eps), int(n_samples), int(seed), int(stream),
                                 _mode(mode), int(first_index), _dev(theta, torch.float32, (capacity, 8)),
                                 _dev(dist, torch.float64, (capacity,)), _dev(idx, torch.int64, (capacity,)),
                                 int(capacity), counters.data_ptr(), _stream(cuda_stream)))


def abc_sample_until(obs, eps, n_target, seed, batch=1 << 22, max_samples=1 << 40, stream=0, mode="fast",
                     first_index=0, capacity=None, out=None, lo=PAPER_LO, hi=PAPER_HI, cuda_stream=None,
                     allow_overflow=False):
    """ABC rejection in batches of `batch` indices from first_index on until
    n_target samples are accepted (or max_samples indices are used). obs is an
    Observed. Returns (theta [m, 8] f32, dist [m] f64, idx [m] int64,
    n_accepted, n_used) as CUDA tensors, m = min(n_accepted, capacity): every
    sample accepted among [first_index, first_index + n_used)."""
    L = load()
    if capacity is None:
        capacity = max(4 * int(n_target), 1024)
    dev = torch.device("cuda", torch.cuda.current_device())
    if out is None:
        theta = torch.empty((capacity, 8), dtype=torch.float32, device=dev)
        dist = torch.empty((capacity,), dtype=torch.float64, device=dev)
        idx = torch.empty((capacity,), dtype=torch.int64, device=dev)
    else:
        theta, dist, idx = out
        capacity = theta.shape[0]
    nacc, used = ctypes.c_uint64(0), ctypes.c_uint64(0)
    b = _box(lo, hi)
    st = L.abc_sample_until(b, obs.handle, float(eps), int(n_target), int(batch), int(max_samples),
                            int(seed), int(stream), _mode(mode), int(first_index),
                            _dev(theta, torch.float32, (capacity, 8)), _dev(dist, torch.float64, (capacity,)),
                            _dev(idx, torch.int64, (capacity,)), int(capacity), ctypes.byref(nacc), ctypes.byref(used),
                            _stream(cuda_stream))
    _check(L, st, allow=(ABC_ERR_CAPACITY,) if allow_overflow else ())
    n = int(nacc.value)
    m = min(n, capacity)
    return _first(theta, m), _first(dist, m), _first(idx, m), n, int(used.value)


def abc_sample_noalloc(observed, N_pop, eps, n_samples, seed, out, stream=0, mode="fast", first_index=0,
                       lo=PAPER_LO, hi=PAPER_HI, cuda_stream=None, allow_overflow=False):
    """abc_sample for callers that cannot allocate device memory while sampling:
    the library allocates nothing (its scratch is a fixed device array) and the
    caller passes the output buffers out = (theta [cap, 8] f32, dist [cap] f64,
    idx [cap] int64) it allocated up front. T <= ABC_NOALLOC_T_MAX; calls that
    overlap on the GPU race on the shared scratch and must be serialized.
    Returns (theta, dist, idx, n_accepted) views like abc_sample."""
    L = load()
    obs, obs_p = _host_i32(observed)
    T = obs.shape[1] - 1
    theta, dist, idx = out
    capacity = theta.shape[0]
    nacc = ctypes.c_uint64(0)
    b = _box(lo, hi)
    st = L.abc_sample_noalloc(b, obs_p, T, int(N_pop), float(eps), int(n_samples), int(seed),
                              int(stream), _mode(mode), int(first_index), _dev(theta, torch.float32, (capacity, 8)),
                              _dev(dist, torch.float64, (capacity,)), _dev(idx, torch.int64, (capacity,)),
                              int(capacity), ctypes.byref(nacc), _stream(cuda_stream))
    _check(L, st, allow=(ABC_ERR_CAPACITY,) if allow_overflow else ())
    n = int(nacc.value)
    m = min(n, capacity)
    return _first(theta, m), _first(dist, m), _first(idx, m), n


def abc_distances(observed, N_pop, n_samples, seed, stream=0, mode="fast", first_index=0, lo=PAPER_LO, hi=PAPER_HI,
                  want_theta=False, out=None, cuda_stream=None):
    """Distances of every sample (and optionally the prior draws): dist [n] f64 (, theta [n, 8])."""
    L = load()
    obs, obs_p = _host_i32(observed)
    T = obs.shape[1] - 1
    dev = torch.device("cuda", torch.cuda.current_device())
    if out is None:
        dist = torch.empty((n_samples,), dtype=torch.float64, device=dev)
        theta = torch.empty((n_samples, 8), dtype=torch.float32, device=dev) if want_theta else None
    else:
        dist, theta = out
    b = _box(lo, hi)
    st = L.abc_distances(b, obs_p, T, int(N_pop), int(n_samples), int(seed), int(stream), _mode(mode),
                         int(first_index), _dev(dist, torch.float64, (n_samples,)),
                         _dev(theta, torch.float32, (n_samples, 8)) if theta is not None else None,
                         _stream(cuda_stream))
    _check(L, st)
    return (dist, theta) if want_theta else dist


def abc_simulate(theta, sample_index, init_ard, T, N_pop, seed, stream=0, mode="exact", cuda_stream=None):
    """Trajectories [B, T+1, 6] (S, I, A, R, D, Ru) for theta [B, 8] (CUDA f32) and sample_index [B] (CUDA int64)."""
    L = load()
    B = theta.shape[0]
    traj = torch.empty((B, T + 1, 6), dtype=torch.int32, device=theta.device)
    a, a_p = _host_i32(init_ard)
    st = L.abc_simulate(_dev(theta, torch.float32, (B, 8)), _dev(sample_index, torch.int64, (B,)), B, a_p, int(T),
                        int(N_pop), int(seed), int(stream), _mode(mode), _dev(traj, torch.int32, (B, T + 1, 6)),
                        _stream(cuda_stream))
    _check(L, st)
    return traj


def abc_step(theta, state_in, sample_index, day, N_pop, seed, stream=0, mode="exact", cuda_stream=None):
    """One day for B states: returns (state_out [B, 6] int32, counts [B, 5] int32)."""
    L = load()
    B = theta.shape[0]
    state_out = torch.empty((B, 6), dtype=torch.int32, device=theta.device)
    counts = torch.empty((B, 5), dtype=torch.int32, device=theta.device)
    st = L.abc_step(_dev(theta, torch.float32, (B, 8)), _dev(state_in, torch.int32, (B, 6)),
                    _dev(sample_index, torch.int64, (B,)), _dev(day, torch.int32, (B,)), B, int(N_pop), int(seed),
                    int(stream), _mode(mode), _dev(state_out, torch.int32, (B, 6)), _dev(counts, torch.int32, (B, 5)),
                    _stream(cuda_stream))
    _check(L, st)
    return state_out, counts


def abc_kth_smallest(dist, k, cuda_stream=None):
    """k-th smallest (1-based) of a CUDA f64 tensor of non-negative distances."""
    L = load()
    out = ctypes.c_double(0)
    st = L.abc_kth_smallest(_dev(dist, torch.float64, (dist.numel(),)), dist.numel(), int(k), ctypes.byref(out),
                            _stream(cuda_stream))
    _check(L, st)
    return out.value


def abc_select_below(dist, eps, first_index=0, theta=None, capacity=1 << 16, out=None, cuda_stream=None):
    """Samples accepted at eps from distances already computed (dist: CUDA f64
    [n], theta: CUDA f32 [n, 8] or None, sample j has index first_index + j):
    (theta [m, 8] or None, dist [m], idx [m], m), unsorted, m = the number
    with dist <= eps. Raises AbcError when m > capacity."""
    L = load()
    n = dist.numel()
    dev = dist.device
    if out is None:
        outs = (torch.empty((capacity, 8), dtype=torch.float32, device=dev) if theta is not None else None,
                torch.empty((capacity,), dtype=torch.float64, device=dev),
                torch.empty((capacity,), dtype=torch.int64, device=dev))
    else:
        outs = out
        capacity = outs[1].shape[0]
    m = ctypes.c_uint64(0)
    st = L.abc_select_below(_dev(dist, torch.float64, (n,)), _dev(theta, torch.float32, (n, 8)) if theta is not None
                            else None, n, float(eps), int(first_index),
                            _dev(outs[0], torch.float32, (capacity, 8)) if theta is not None else None,
                            _dev(outs[1], torch.float64, (capacity,)), _dev(outs[2], torch.int64, (capacity,)),
                            capacity, ctypes.byref(m), _stream(cuda_stream))
    _check(L, st)
    k = int(m.value)
    return (outs[0][:k] if theta is not None else None), outs[1][:k], outs[2][:k], k


def abc_sample_quantile(observed, N_pop, n_samples, k, seed, stream=0, mode="fast", first_index=0, lo=PAPER_LO,
                        hi=PAPER_HI, capacity=None, out=None, cuda_stream=None):
    """ABC rejection over [first_index, first_index + n_samples) with eps the
    k-th smallest distance, in one call. observed: host int32 [3, T+1].
    Returns (theta [m, 8] f32, dist [m] f64, idx [m] (int64 storage),
    n_accepted, eps) with the accepted samples as CUDA tensors in unspecified
    order. Raises AbcError when more than capacity samples are accepted."""
    L = load()
    obs, obs_p = _host_i32(observed)
    T = obs.shape[1] - 1
    dev = torch.device("cuda", torch.cuda.current_device())
    if out is None:
        if capacity is None:
            capacity = max(1024, 2 * int(k))
        theta = torch.empty((capacity, 8), dtype=torch.float32, device=dev)
        dist = torch.empty((capacity,), dtype=torch.float64, device=dev)
        idx = torch.empty((capacity,), dtype=torch.int64, device=dev)
    else:
        theta, dist, idx = out
        capacity = dist.shape[0]
    nacc = ctypes.c_uint64(0)
    eps = ctypes.c_double(0.0)
    b = _box(lo, hi)
    st = L.abc_sample_quantile(b, obs_p, T, int(N_pop), int(n_samples), int(k), int(seed), int(stream),
                               _mode(mode), int(first_index), _dev(theta, torch.float32, (capacity, 8)),
                               _dev(dist, torch.float64, (capacity,)), _dev(idx, torch.int64, (capacity,)),
                               int(capacity), ctypes.byref(eps), ctypes.byref(nacc), _stream(cuda_stream))
    _check(L, st)
    n = int(nacc.value)
    return theta[:n], dist[:n], idx[:n], n, float(eps.value)


def abc_strerror(status):
    return _strerror(status)


def abc_version():
    return load().abc_version()


def abc_last_simulated_days():
    """Model days simulated by the last abc_sample call on this thread."""
    return int(load().abc_last_simulated_days())


class Plan:
    """Batched regions in one launch (C ABI abc_plan_*). regions: list of dicts
    with keys observed (host int32 [3, T+1]), N_pop, eps, n_samples and optional
    first_index, stream, capacity, theta_in (CUDA f32 [n_samples, 8])."""

    def __init__(self, regions, seed, mode="fast", lo=PAPER_LO, hi=PAPER_HI):
        L = load()
        self._L = L
        self._obs = [np.ascontiguousarray(np.asarray(r["observed"], dtype=np.int32)) for r in regions]
        arr = (AbcRegion * len(regions))()
        for j, r in enumerate(regions):
            o = self._obs[j]
            th = r.get("theta_in")
            arr[j] = AbcRegion(o.ctypes.data, o.shape[1] - 1, int(r["N_pop"]), float(r["eps"]), int(r["n_samples"]),
                               int(r.get("first_index", 0)), int(r.get("stream", j)), int(r.get("capacity", 4096)),
                               th.data_ptr() if th is not None else None)
        self.capacity = [int(r.get("capacity", 4096)) for r in regions]
        self.n_regions = len(regions)
        b = _box(lo, hi)
        h = ctypes.c_void_p()
        _check(L, L.abc_plan_create(b, arr, len(regions), int(seed), _mode(mode), ctypes.byref(h)))
        self._h = h

    def reset(self, cuda_stream=None):
        _check(self._L, self._L.abc_plan_reset(self._h, _stream(cuda_stream)))

    def run(self, cuda_stream=None):
        _check(self._L, self._L.abc_plan_run(self._h, _stream(cuda_stream)))

    def run_graph(self, n_runs, cuda_stream=None):
        _check(self._L, self._L.abc_plan_run_graph(self._h, int(n_runs), _stream(cuda_stream)))

    def tune(self, cuda_stream=None):
        shapes = (AbcLaunchShape * 32)()
        n = ctypes.c_int32()
        best = AbcLaunchShape()
        _check(self._L, self._L.abc_plan_tune(self._h, _stream(cuda_stream), shapes, 32, ctypes.byref(n),
                                              ctypes.byref(best)))
        as_dict = lambda s: dict(block_threads=s.block_threads, pairs_per_iteration=s.pairs_per_iteration,
                                 blocks_per_sm=s.blocks_per_sm, lean=s.lean, ms=s.ms)
        return as_dict(best), [as_dict(shapes[j]) for j in range(n.value)]

    def set_shape(self, shape):
        """Pin a compiled launch shape (a dict as tune() returns) without tuning."""
        sh = AbcLaunchShape(int(shape["block_threads"]), int(shape["pairs_per_iteration"]),
                            int(shape["blocks_per_sm"]), int(shape.get("lean", 0)), 0.0)
        _check(self._L, self._L.abc_plan_set_shape(self._h, ctypes.byref(sh)))

    def counts(self, region, cuda_stream=None):
        n, d = ctypes.c_uint64(), ctypes.c_uint64()
        _check(self._L, self._L.abc_plan_results(self._h, int(region), ctypes.byref(n), ctypes.byref(d), None, None,
                                                 None, _stream(cuda_stream)))
        return int(n.value), int(d.value)

    def results(self, region, cuda_stream=None):
        """(theta [m, 8], dist [m], idx [m], n_accepted, simulated_days) as CUDA tensors."""
        n_acc, days = self.counts(region, cuda_stream)
        m = min(n_acc, self.capacity[region])
        dev = torch.device("cuda", torch.cuda.current_device())
        theta = torch.empty((max(m, 1), 8), dtype=torch.float32, device=dev)
        dist = torch.empty((max(m, 1),), dtype=torch.float64, device=dev)
        idx = torch.empty((max(m, 1),), dtype=torch.int64, device=dev)
        got = ctypes.c_uint64()
        _check(self._L, self._L.abc_plan_copy_results(self._h, int(region), theta.data_ptr(), dist.data_ptr(),
                                                      idx.data_ptr(), m, ctypes.byref(got), _stream(cuda_stream)))
        torch.cuda.current_stream().synchronize() if cuda_stream is None else None
        return theta[:m], dist[:m], idx[:m], n_acc, days

    def set_region(self, region, theta_in=None, first_index=0):
        _check(self._L, self._L.abc_plan_set_region(self._h, int(region),
                                                    theta_in.data_ptr() if theta_in is not None else None,
                                                    int(first_index)))

    def set_eps(self, region, eps):
        _check(self._L, self._L.abc_plan_set_eps(self._h, int(region), float(eps)))

    def close(self):
        if getattr(self, "_h", None):
            self._L.abc_plan_destroy(self._h)
            self._h = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


abc_plan_create = Plan


def abc_plan_reset(plan, cuda_stream=None):
    plan.reset(cuda_stream)


def abc_plan_run(plan, cuda_stream=None):
    plan.run(cuda_stream)


def abc_plan_run_graph(plan, n_runs, cuda_stream=None):
    plan.run_graph(n_runs, cuda_stream)


def abc_plan_tune(plan, cuda_stream=None):
    return plan.tune(cuda_stream)


def abc_plan_results(plan, region, cuda_stream=None):
    return plan.counts(region, cuda_stream)


def abc_plan_copy_results(plan, region, cuda_stream=None):
    return plan.results(region, cuda_stream)


def abc_plan_set_region(plan, region, theta_in=None, first_index=0):
    plan.set_region(region, theta_in, first_index)


def abc_plan_set_eps(plan, region, eps):
    plan.set_eps(region, eps)


def abc_plan_set_shape(plan, shape):
    plan.set_shape(shape)


def abc_plan_destroy(plan):
    plan.close()



class Flow:
    """Masked autoregressive flow proposal on the prior box (C ABI abc_maf_*);
    n_flows > 1 holds that many independent flows of the same shape."""

    def __init__(self, n_blocks=3, hidden=256, lo=PAPER_LO, hi=PAPER_HI, n_flows=1):
        L = load()
        self._L = L
        h = ctypes.c_void_p()
        b = _box(lo, hi)
        _check(L, L.abc_maf_create_multi(int(n_flows), int(n_blocks), int(hidden), b, ctypes.byref(h)))
        self._h = h
        self.n_blocks, self.hidden, self.n_flows = int(n_blocks), int(hidden), int(n_flows)
        self.n_params = int(L.abc_maf_param_count(h))

    def init_random(self, seed=0, scale=0.3):
        _check(self._L, self._L.abc_maf_init_random(self._h, int(seed), float(scale)))

    def set_proposal_scale(self, tau):
        """Sample and evaluate with the base broadened by tau (training is unaffected)."""
        _check(self._L, self._L.abc_maf_set_proposal_scale(self._h, float(tau)))

    def test_hold_products(self, hold):
        """Testing hook: the kernels issue no tensor-core products, so their
        bounded waits run out: gradient/training raise ABC_ERR_TIMEOUT, sample
        and log_q give NaN and check raises."""
        _check(self._L, self._L.abc_maf_test_hold_products(self._h, int(bool(hold))))

    def check(self, cuda_stream=None):
        """Synchronise the stream and raise AbcError (ABC_ERR_TIMEOUT) if a wait
        of a sample or log_q launch ran out since the last check; its rows are
        NaN."""
        _check(self._L, self._L.abc_maf_check(self._h, _stream(cuda_stream)))

    def set_params(self, params):
        """params: [n_params] (one flow) or [n_flows, n_params]."""
        v = np.ascontiguousarray(np.asarray(params, dtype=np.float32).ravel())
        assert v.size == self.n_params * self.n_flows
        _check(self._L, self._L.abc_maf_set_params(self._h, v.ctypes.data))

    def get_params(self):
        v = np.empty(self.n_params * self.n_flows, dtype=np.float32)
        _check(self._L, self._L.abc_maf_get_params(self._h, v.ctypes.data))
        return v if self.n_flows == 1 else v.reshape(self.n_flows, self.n_params)

    def train_flows(self, thetas, weights=None, n_steps=500, batch=1024, lr=1e-3, seed=0, val_fraction=0.0,
                    cuda_stream=None):
        """Train every flow on its own data in the same launches: thetas is a
        list of n_flows CUDA f32 [n_r, 8] tensors (None or empty = leave that
        flow as it is), weights a matching list or None; val_fraction > 0 holds
        out that share of each flow's points for early stopping. Returns the
        losses."""
        R = self.n_flows
        th = (ctypes.c_void_p * R)()
        wt = (ctypes.c_void_p * R)()
        nn = (ctypes.c_uint64 * R)()
        for r in range(R):
            t = thetas[r]
            if t is not None and t.shape[0] > 0:
                th[r] = t.data_ptr()
                nn[r] = t.shape[0]
                if weights is not None and weights[r] is not None:
                    wt[r] = weights[r].data_ptr()
        loss = (ctypes.c_float * R)()
        s = cuda_stream if cuda_stream is not None else torch.cuda.Stream()
        torch.cuda.current_stream().synchronize()
        _check(self._L, self._L.abc_maf_train_flows(self._h, ctypes.cast(th, ctypes.c_void_p),
                                                    ctypes.cast(wt, ctypes.c_void_p) if weights is not None else None,
                                                    ctypes.cast(nn, ctypes.c_void_p), int(n_steps), int(batch),
                                                    float(lr), int(seed), float(val_fraction),
                                                    ctypes.cast(loss, ctypes.c_void_p), _stream(s)))
        return np.array(loss[:], dtype=np.float64)

    def sample(self, n, seed=0, stream=0, first_index=0, base=None, want_logq=True, out=None,
               cuda_stream=None, flow=0):
        dev = torch.device("cuda", torch.cuda.current_device())
        if out is None:
            theta = torch.empty((n, 8), dtype=torch.float32, device=dev)
            logq = torch.empty((n,), dtype=torch.float32, device=dev) if want_logq else None
        else:
            theta, logq = out
        u = base.data_ptr() if base is not None else None
        _check(self._L, self._L.abc_maf_sample_at(self._h, int(flow), int(n), u, int(seed), int(stream),
                                                  int(first_index), theta.data_ptr(),
                                                  logq.data_ptr() if logq is not None else None, _stream(cuda_stream)))
        return theta, logq

    def log_q(self, theta, cuda_stream=None, flow=0):
        n = theta.shape[0]
        out = torch.empty((n,), dtype=torch.float32, device=theta.device)
        _check(self._L, self._L.abc_maf_log_q_at(self._h, int(flow), n, theta.data_ptr(), out.data_ptr(),
                                                 _stream(cuda_stream)))
        return out

    def gradient(self, theta, weights=None, cuda_stream=None):
        """(loss, gradient as a float32 numpy vector in the parameter order)."""
        loss = ctypes.c_float()
        g = np.empty(self.n_params, dtype=np.float32)
        _check(self._L, self._L.abc_maf_gradient(self._h, theta.shape[0], theta.data_ptr(),
                                                 weights.data_ptr() if weights is not None else None,
                                                 ctypes.byref(loss), g.ctypes.data, _stream(cuda_stream)))
        return float(loss.value), g

    def adam_step(self, lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, cuda_stream=None):
        _check(self._L, self._L.abc_maf_adam_step(self._h, lr, beta1, beta2, eps, _stream(cuda_stream)))

    def train(self, theta, weights=None, n_steps=500, batch=1024, lr=1e-3, seed=0, cuda_stream=None):
        s = cuda_stream if cuda_stream is not None else torch.cuda.Stream()
        torch.cuda.current_stream().synchronize()
        loss = ctypes.c_float()
        _check(self._L, self._L.abc_maf_train(self._h, theta.shape[0], theta.data_ptr(),
                                              weights.data_ptr() if weights is not None else None, int(n_steps),
                                              int(batch), float(lr), int(seed), ctypes.byref(loss), _stream(s)))
        return float(loss.value)

    def close(self):
        if getattr(self, "_h", None):
            self._L.abc_maf_destroy(self._h)
            self._h = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


abc_maf_create = Flow


def abc_maf_create_multi(n_flows, n_blocks=3, hidden=256, lo=PAPER_LO, hi=PAPER_HI):
    return Flow(n_blocks, hidden, lo, hi, n_flows=n_flows)


def abc_maf_init_random(flow, seed=0, scale=0.3):
    flow.init_random(seed, scale)


def abc_maf_param_count(flow):
    return flow.n_params


def abc_maf_set_params(flow, params):
    flow.set_params(params)


def abc_maf_get_params(flow):
    return flow.get_params()


def abc_maf_sample(flow, n, **kw):
    return flow.sample(n, **kw)


def abc_maf_log_q(flow, theta, cuda_stream=None):
    return flow.log_q(theta, cuda_stream)


def abc_maf_gradient(flow, theta, weights=None, cuda_stream=None):
    return flow.gradient(theta, weights, cuda_stream)


def abc_maf_adam_step(flow, **kw):
    flow.adam_step(**kw)


def abc_maf_train(flow, theta, weights=None, **kw):
    return flow.train(theta, weights, **kw)


def abc_maf_destroy(flow):
    flow.close()


def abc_maf_flow_count(flow):
    return flow.n_flows


def abc_maf_set_proposal_scale(flow, tau):
    flow.set_proposal_scale(tau)


def abc_maf_test_hold_products(flow, hold):
    flow.test_hold_products(hold)


def abc_maf_check(flow, cuda_stream=None):
    flow.check(cuda_stream)


def abc_maf_sample_at(flow, r, n, **kw):
    return flow.sample(n, flow=r, **kw)


def abc_maf_log_q_at(flow, r, theta, cuda_stream=None):
    return flow.log_q(theta, cuda_stream, flow=r)


def abc_maf_train_flows(flow, thetas, weights=None, **kw):
    return flow.train_flows(thetas, weights, **kw)



ABC_FALLBACK_EFFICIENCY, ABC_FALLBACK_ESS = 0, 1
_FALLBACK = {"efficiency": ABC_FALLBACK_EFFICIENCY, "ess": ABC_FALLBACK_ESS}


def _fallback(rule):
    if rule not in _FALLBACK:
        raise ValueError("fallback must be one of %s" % sorted(_FALLBACK))
    return _FALLBACK[rule]


def abc_smc_run(observed, N_pop, eps0, rounds=5, sims_per_round=1 << 22, eps_factor=0.7, ess_min=0.1,
                flow_blocks=3, flow_hidden=256, train_steps=500, train_batch=1024, train_lr=1e-3, seed=0,
                capacity=None, mode="fast", defensive=0.1, val_fraction=0.1, train_weight_power=0.8, fresh_init=False,
                proposal_scale=1.25, fallback="efficiency", lo=PAPER_LO, hi=PAPER_HI, cuda_stream=None):
    """Sequential ABC with the learned flow proposal. Returns (rounds: list of
    dicts, theta [m, 8], weights [m] (f64, sum 1), dist [m]) of the last round.
    The defaults proposal_scale=1.25 (proposals from the flow with its base
    broadened by 1.25) and train_weight_power=0.8 (training weights w^0.8)
    trade some acceptance for proposals that cover the posterior's tails: on
    the P = 6e7, T = 100 workload they gave the highest median and worst-case
    effective samples per second over six seeds among the settings tried
    (scale 1 to 1.7, power 0.7 to 1)."""
    L = load()
    obs, obs_p = _host_i32(observed)
    T = obs.shape[1] - 1
    if capacity is None:
        capacity = sims_per_round
    cfg = AbcSmcConfig(int(rounds), int(sims_per_round), float(eps0), float(eps_factor), float(ess_min),
                       int(flow_blocks), int(flow_hidden), int(train_steps), int(train_batch), float(train_lr),
                       int(seed), int(capacity), _mode(mode), float(defensive), float(val_fraction),
                       float(train_weight_power), int(bool(fresh_init)), float(proposal_scale), _fallback(fallback))
    rr = (AbcSmcRound * int(rounds))()
    dev = torch.device("cuda", torch.cuda.current_device())
    theta = torch.empty((capacity, 8), dtype=torch.float32, device=dev)
    w = torch.empty((capacity,), dtype=torch.float64, device=dev)
    dist = torch.empty((capacity,), dtype=torch.float64, device=dev)
    n = ctypes.c_uint64()
    s = cuda_stream if cuda_stream is not None else torch.cuda.Stream()
    torch.cuda.current_stream().synchronize()
    b = _box(lo, hi)
    _check(L, L.abc_smc_run(b, obs_p, T, int(N_pop), ctypes.byref(cfg), rr, theta.data_ptr(),
                            w.data_ptr(), dist.data_ptr(), ctypes.byref(n), _stream(s)))
    out = [dict((f, getattr(r, f)) for f, _ in AbcSmcRound._fields_) for r in rr]
    m = int(n.value)
    return out, theta[:m], w[:m], dist[:m]



def abc_smc_run_regions(regions, rounds=16, shrink_rounds=4, sims_per_round=1 << 20, eps_factor=0.7, ess_min=0.1,
                        flow_blocks=3, flow_hidden=256, train_steps=500, train_steps_warm=100, train_batch=1024,
                        train_lr=1e-3, seed=0, capacity=None, mode="fast", defensive=0.1, val_fraction=0.1,
                        train_weight_power=0.8, proposal_scale=1.25, fallback="efficiency", lo=PAPER_LO, hi=PAPER_HI,
                        cuda_stream=None):
    """Sequential ABC with one flow proposal per region, all regions in one
    batched launch per round. regions: list of dicts with observed (host int32
    [3, T+1]), N_pop, eps (final) and pool (samples kept at the final eps).
    Returns (rounds [rounds][n_regions] of dicts, per region a tuple
    (theta [m, 8], weights [m] f64 (a round's normalised weights times its
    ESS), dist [m], n_pooled))."""
    L = load()
    R = len(regions)
    if capacity is None:
        capacity = sims_per_round
    dev = torch.device("cuda", torch.cuda.current_device())
    keep, outs = [], []
    arr = (AbcSmcRegion * R)()
    for g, reg in enumerate(regions):
        obs, obs_p = _host_i32(reg["observed"])
        keep.append(obs)
        pool = int(reg.get("pool", 1 << 16))
        th = torch.empty((max(pool, 1), 8), dtype=torch.float32, device=dev)
        w = torch.empty((max(pool, 1),), dtype=torch.float64, device=dev)
        d = torch.empty((max(pool, 1),), dtype=torch.float64, device=dev)
        outs.append((th, w, d))
        arr[g] = AbcSmcRegion(obs_p, obs.shape[1] - 1, int(reg["N_pop"]),
                              float(reg["eps"]), th.data_ptr(), w.data_ptr(), d.data_ptr(), pool, 0, 0)
    base = AbcSmcConfig(int(rounds), int(sims_per_round), 0.0, float(eps_factor), float(ess_min), int(flow_blocks),
                        int(flow_hidden), int(train_steps), int(train_batch), float(train_lr), int(seed),
                        int(capacity), _mode(mode), float(defensive), float(val_fraction),
                        float(train_weight_power), 0, float(proposal_scale), _fallback(fallback))
    cfg = AbcSmcStreamConfig(base, int(shrink_rounds), int(train_steps_warm))
    rr = (AbcSmcRound * (int(rounds) * R))()
    s = cuda_stream if cuda_stream is not None else torch.cuda.Stream()
    torch.cuda.current_stream().synchronize()
    b = _box(lo, hi)
    _check(L, L.abc_smc_run_regions(b, arr, R, ctypes.byref(cfg), rr, _stream(s)))
    info = [[dict((f, getattr(rr[r * R + g], f)) for f, _ in AbcSmcRound._fields_) for g in range(R)]
            for r in range(int(rounds))]
    res = []
    for g in range(R):
        m = int(arr[g].n_out)
        th, w, d = outs[g]
        res.append((th[:m], w[:m], d[:m], int(arr[g].n_pooled)))
    return info, res


def abc_project(theta, sample_index, init_ard, T, N_pop, seed, quantiles=(0.05, 0.5, 0.95), stream=0, mode="fast",
                cuda_stream=None):
    """Quantile bands [n_q, T+1, 3] (A, R, D) of trajectories simulated from
    theta [B, 8] (CUDA f32) with sample_index [B] (CUDA int64). On a cuda_stream
    other than the current one the call returns when the bands are complete."""
    L = load()
    B = theta.shape[0]
    q = np.ascontiguousarray(np.asarray(quantiles, dtype=np.float64))
    bands = torch.empty((len(q), T + 1, 3), dtype=torch.float32, device=theta.device)
    a, a_p = _host_i32(init_ard)
    raw = _stream(cuda_stream)
    _check(L, L.abc_project(_dev(theta, torch.float32, (B, 8)), _dev(sample_index, torch.int64, (B,)), B, a_p,
                            int(T), int(N_pop), int(seed), int(stream), _mode(mode), q.ctypes.data, len(q),
                            bands.data_ptr(), raw))
    if raw != _stream(None):
        # the caller reads the bands, and gives the inputs' memory back, on the current stream
        (torch.cuda.ExternalStream(raw) if raw else torch.cuda.default_stream()).synchronize()
    return bands



def abc_pmc_run(observed, N_pop, eps0, rounds=4, n_particles=4096, batch=1 << 20, max_batches=64, eps_factor=0.7,
                seed=0, capacity=1 << 17, mode="fast", lo=PAPER_LO, hi=PAPER_HI, cuda_stream=None):
    """Population Monte Carlo ABC. Returns (rounds: list of dicts, theta [m, 8],
    weights [m] (f64, sum 1), dist [m]) of the last population."""
    L = load()
    obs, obs_p = _host_i32(observed)
    T = obs.shape[1] - 1
    cfg = AbcPmcConfig(int(rounds), int(n_particles), int(batch), int(max_batches), float(eps0), float(eps_factor),
                       int(seed), int(capacity), _mode(mode))
    rr = (AbcPmcRound * int(rounds))()
    dev = torch.device("cuda", torch.cuda.current_device())
    theta = torch.empty((capacity, 8), dtype=torch.float32, device=dev)
    w = torch.empty((capacity,), dtype=torch.float64, device=dev)
    dist = torch.empty((capacity,), dtype=torch.float64, device=dev)
    n = ctypes.c_uint64()
    s = cuda_stream if cuda_stream is not None else torch.cuda.Stream()
    torch.cuda.current_stream().synchronize()
    b = _box(lo, hi)
    _check(L, L.abc_pmc_run(b, obs_p, T, int(N_pop), ctypes.byref(cfg), rr, theta.data_ptr(),
                            w.data_ptr(), dist.data_ptr(), ctypes.byref(n), _stream(s)))
    out = [dict((f, getattr(r, f)) for f, _ in AbcPmcRound._fields_) for r in rr]
    m = int(n.value)
    return out, theta[:m], w[:m], dist[:m]


def abc_pmc_propose(theta_old, w_old, Lmat, n, seed=0, first_index=0, lo=PAPER_LO, hi=PAPER_HI, cuda_stream=None):
    """n proposals from a weighted population (CUDA f32 [m, 8], CUDA f64 [m]) and
    the host lower-triangular L [8, 8]; NaN first coordinate = outside the box."""
    L = load()
    Lh = np.ascontiguousarray(np.asarray(Lmat, dtype=np.float32).reshape(8, 8))
    out = torch.empty((n, 8), dtype=torch.float32, device=theta_old.device)
    b = _box(lo, hi)
    _check(L, L.abc_pmc_propose(b, theta_old.data_ptr(), w_old.data_ptr(), theta_old.shape[0],
                                Lh.ctypes.data, int(seed), int(first_index), int(n), out.data_ptr(),
                                _stream(cuda_stream)))
    return out


def abc_pmc_weights(theta_new, theta_old, w_old, Lmat, cuda_stream=None):
    """Unnormalised population Monte Carlo weights of theta_new (CUDA f64 [n])."""
    L = load()
    Lh = np.ascontiguousarray(np.asarray(Lmat, dtype=np.float32).reshape(8, 8))
    out = torch.empty((theta_new.shape[0],), dtype=torch.float64, device=theta_new.device)
    _check(L, L.abc_pmc_weights(theta_new.data_ptr(), theta_new.shape[0], theta_old.data_ptr(), w_old.data_ptr(),
                                theta_old.shape[0], Lh.ctypes.data, out.data_ptr(), _stream(cuda_stream)))
    return out
