"""ctypes binding of the C ABI in ``include/svip.h``: argument marshalling only.

Every method of :class:`Context` has the name and the argument order of the C
function it calls.  Device buffers may be given as ``torch`` CUDA tensors (their
``data_ptr()`` is passed) or as integer device addresses; ``stream`` may be a
``torch.cuda.Stream``, an integer ``cudaStream_t`` or ``None`` (the legacy
default stream).  Nothing here computes: if the compiled library is missing the
import of a symbol fails with :class:`SvipError`.

The library is loaded with ctypes.  The entry points that are called per token or per round
have their arguments converted by a small extension (csrc/native_calls.cpp), because for the
smallest launches the conversion took longer than the GPU; an interpreter it was not built for
falls back to ctypes, with the same conversions.
"""
from __future__ import annotations

import ctypes as C
import importlib.machinery
import importlib.util
import os
import sysconfig

SVIP_F32 = 0
SVIP_BF16 = 1
SVIP_Q_PACKED = -1
SVIP_STATUS_NONFINITE_ROW = 1
SVIP_STATUS_BAD_DRAFT_LEN = 2
SVIP_STATUS_WAIT_TIMEOUT = 4
SVIP_STATUS_BAD_TREE = 8
SVIP_STATUS_LOOP_OVERLAP = 32

_HERE = os.path.dirname(os.path.abspath(__file__))
# SVIP_LIBRARY in the environment points at another build of the same ABI (a debug build, say)
_LIB_PATH = os.environ.get("SVIP_LIBRARY") or os.path.join(_HERE, "csrc", "libsvip.so")
_lib = None
_calls = None       # the per-token and per-round entry points: f(handle, *arguments) -> status
_CALL_NAMES = ("draft_step", "draft_step_masked", "draft_step_at", "draft_step_filtered", "draft_step_truncated",
               "row_threshold", "policy_advance", "policy_update", "pack_ragged", "verify", "verify_early_exit",
               "verify_filtered", "verify_tree", "vp_partial", "vp_combine", "vp_locate", "pair_stats", "pair_stats_given",
               "graph_launch")


class SvipError(RuntimeError):
    def __init__(self, code: int, text: str):
        super().__init__("svip: %s (status %d)" % (text, code))
        self.code = code


def library_path() -> str:
    return _LIB_PATH


def library():
    """Loads csrc/libsvip.so (built by ``python -m paper_2411_18462_b200.build``)."""
    global _lib, _calls
    if _lib is not None:
        return _lib
    if not os.path.exists(_LIB_PATH):
        raise SvipError(-100, "CUDA library %s is not built; run python -m paper_2411_18462_b200.build"
                        % _LIB_PATH)
    L = C.CDLL(_LIB_PATH)
    vp, i32, lng, f32 = C.c_void_p, C.c_int, C.c_long, C.c_float
    L.svip_strerror.restype = C.c_char_p
    L.svip_strerror.argtypes = [i32]
    L.svip_version.restype = i32
    L.svip_version.argtypes = []
    L.svip_last_cuda_error.restype = i32
    L.svip_last_cuda_error.argtypes = [vp]
    L.svip_create.restype = i32
    L.svip_create.argtypes = [C.POINTER(vp), i32, i32]
    L.svip_destroy.restype = i32
    L.svip_destroy.argtypes = [vp]
    L.svip_set_cluster_size.restype = i32
    L.svip_set_cluster_size.argtypes = [vp, i32]
    L.svip_launch_count.restype = lng
    L.svip_launch_count.argtypes = [vp]
    L.svip_read_status.restype = i32
    L.svip_read_status.argtypes = [vp, C.POINTER(C.c_uint), vp]
    L.svip_draft_step.restype = i32
    L.svip_draft_step.argtypes = [vp, vp, i32, i32, i32, lng, f32, f32, vp, vp, vp, vp, vp, vp]
    L.svip_pack_ragged.restype = i32
    L.svip_pack_ragged.argtypes = [vp, vp, i32, i32, vp, vp, vp, vp]
    L.svip_verify.restype = i32
    L.svip_verify.argtypes = [vp, vp, vp, lng, vp, lng, lng, vp, lng, i32, vp, i32, i32, i32, i32, f32,
                              vp, vp, vp, vp]
    L.svip_verify_early_exit.restype = i32
    L.svip_verify_early_exit.argtypes = [vp, vp, vp, lng, vp, lng, lng, vp, lng, i32, vp, i32, i32, i32, i32, f32,
                              vp, vp, vp, vp]
    L.svip_profile_enable.restype = i32
    L.svip_profile_enable.argtypes = [vp, i32]
    L.svip_profile_read.restype = i32
    L.svip_profile_read.argtypes = [vp, C.POINTER(C.c_double), C.POINTER(C.c_long)]
    L.svip_pair_stats_given.restype = i32
    L.svip_pair_stats_given.argtypes = [vp, vp, lng, vp, vp, lng, vp, i32, i32, i32, f32, f32, vp, vp]
    L.svip_verify_tree.restype = i32
    L.svip_verify_tree.argtypes = [vp, vp, vp, vp, lng, vp, vp, lng, i32, i32, i32, i32, f32, vp, vp, vp, vp, vp]
    L.svip_selftest_wait_timeout.restype = i32
    L.svip_selftest_wait_timeout.argtypes = [vp, lng, vp]
    L.svip_draft_step_masked.restype = i32
    L.svip_draft_step_masked.argtypes = [vp, vp, i32, i32, i32, lng, f32, f32, vp, vp, vp, vp, vp, vp, vp]
    L.svip_draft_step_at.restype = i32
    L.svip_draft_step_at.argtypes = [vp, vp, i32, i32, i32, lng, lng, vp, lng, f32, f32, vp, vp, vp, vp, vp, vp, vp]
    L.svip_graph_loop_begin.restype = i32
    L.svip_graph_loop_begin.argtypes = [vp, vp, vp, i32, C.POINTER(vp)]
    L.svip_graph_loop_end.restype = i32
    L.svip_graph_loop_end.argtypes = [vp]
    L.svip_row_threshold.restype = i32
    L.svip_row_threshold.argtypes = [vp, vp, i32, i32, i32, lng, f32, i32, f32, vp, vp, vp]
    L.svip_draft_step_filtered.restype = i32
    L.svip_draft_step_filtered.argtypes = [vp, vp, i32, i32, i32, lng, f32, f32, vp, vp, vp, vp, vp, vp, vp, vp]
    L.svip_draft_step_truncated.restype = i32
    L.svip_draft_step_truncated.argtypes = [vp, vp, i32, i32, i32, lng, f32, f32, i32, f32, vp, vp, vp, vp, vp, vp, vp, vp]
    L.svip_verify_filtered.restype = i32
    L.svip_verify_filtered.argtypes = [vp, vp, vp, lng, vp, vp, lng, lng, vp, lng, vp, vp, i32, vp, i32, i32, i32,
                                       i32, f32, vp, vp, vp, vp]
    L.svip_policy_advance.restype = i32
    L.svip_policy_advance.argtypes = [vp, i32, vp, vp, vp, vp, i32, i32, vp, vp]
    L.svip_policy_update.restype = i32
    L.svip_policy_update.argtypes = [vp, i32, vp, vp, vp, vp, i32, i32, vp]
    L.svip_vp_partial.restype = i32
    L.svip_vp_partial.argtypes = [vp, vp, i32, i32, i32, lng, f32, i32, vp, vp]
    L.svip_vp_combine.restype = i32
    L.svip_vp_combine.argtypes = [vp, vp, i32, i32, i32, f32, f32, vp, vp, vp, vp, vp, vp, vp, vp]
    L.svip_vp_locate.restype = i32
    L.svip_vp_locate.argtypes = [vp, vp, i32, i32, i32, lng, f32, vp, vp, i32, vp, vp]
    L.svip_pair_stats.restype = i32
    L.svip_pair_stats.argtypes = [vp, vp, lng, vp, lng, i32, i32, i32, f32, f32, vp, vp]
    L.svip_verify_noalloc.restype = i32
    L.svip_verify_noalloc.argtypes = [i32, vp, vp, lng, vp, lng, lng, vp, lng, i32, vp, i32, i32, i32, i32, f32,
                                      vp, vp, vp, vp, vp]
    L.svip_graph_begin.restype = i32
    L.svip_graph_begin.argtypes = [vp, vp]
    L.svip_graph_end.restype = i32
    L.svip_graph_end.argtypes = [vp, vp, C.POINTER(vp)]
    L.svip_graph_launch.restype = i32
    L.svip_graph_launch.argtypes = [vp, vp]
    L.svip_graph_destroy.restype = i32
    L.svip_graph_destroy.argtypes = [vp]
    _lib, _calls = L, _load_calls(L)
    return L


def native_calls_path() -> str:
    return os.path.join(_HERE, "csrc", "native_calls" + sysconfig.get_config_var("EXT_SUFFIX"))


def _load_calls(L):
    path = native_calls_path()
    if not os.path.exists(path):
        return _CtypesCalls(L)
    loader = importlib.machinery.ExtensionFileLoader("native_calls", path)
    native = importlib.util.module_from_spec(importlib.util.spec_from_file_location("native_calls", path, loader=loader))
    loader.exec_module(native)
    # an extension of another header would call the library with shifted arguments (without the header beside the package
    # there is nothing to compare, and nothing that could have changed)
    from . import build
    if os.path.exists(os.path.join(build.INCLUDE, "svip.h")) and \
            getattr(native, "abi_fingerprint", "") != build.abi_fingerprint():
        return _CtypesCalls(L)
    native.load({n: C.cast(getattr(L, "svip_" + n), C.c_void_p).value for n in _CALL_NAMES})
    return native


class _CtypesCalls:
    """The functions of the extension, through ctypes."""

    def __init__(self, L):
        for name in _CALL_NAMES:
            setattr(self, name, self._wrap(getattr(L, "svip_" + name)))

    @staticmethod
    def _wrap(fn):
        def call(*args):
            if len(args) != len(fn.argtypes):
                raise TypeError("%s takes %d arguments, %d given" % (fn.__name__, len(fn.argtypes), len(args)))
            return fn(*[_convert(a, t) for a, t in zip(args, fn.argtypes)])
        return call


def _ptr(x):
    if x is None:
        return None
    if isinstance(x, int):
        return x
    return x.data_ptr()


def _stream(s):
    if s is None:
        return None
    if isinstance(s, int):
        return s
    return s.cuda_stream


def _convert(a, t):
    """What ctypes needs for one argument of type t."""
    if t is C.c_void_p:
        return _ptr(a) if not hasattr(a, "cuda_stream") else a.cuda_stream
    return float(a) if t is C.c_float else int(a)


def _check(code: int, ctx=None):
    if code != 0:
        text = library().svip_strerror(code).decode()
        if code == -4 and ctx is not None:
            text += " (cudaError %d)" % library().svip_last_cuda_error(ctx)
        raise SvipError(code, text)


def verify_noalloc(device, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                   target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                   n_accepted, next_token, status=None, stream=None):
    """``svip_verify_noalloc``: the verify round without a context and without any allocation."""
    _check(library().svip_verify_noalloc(int(device), _ptr(draft_tokens), _ptr(q_logits), int(q_row_stride),
                                         _ptr(q_stats), int(q_seq_stride), int(q_pos_stride),
                                         _ptr(target_logits), int(t_row_stride), int(dtype), _ptr(cu_rows),
                                         int(B), int(K), int(n_target_rows), int(V), float(T), _ptr(uniforms),
                                         _ptr(n_accepted), _ptr(next_token), _ptr(status), _stream(stream)))


class Graph:
    def __init__(self, handle):
        self._h = handle
        self._hv = handle.value        # what the calls are given

    def launch(self, stream=None):
        rc = _calls.graph_launch(self._hv, stream)
        if rc:
            _check(rc)

    def destroy(self):
        if self._h:
            library().svip_graph_destroy(self._h)
            self._h, self._hv = None, 0


class Context:
    """Owns an ``svip_ctx``; methods mirror the C functions one to one."""

    def __init__(self, device: int = 0, max_rows: int = 1 << 15):
        self._h = C.c_void_p()
        _check(library().svip_create(C.byref(self._h), int(device), int(max_rows)))
        self._hv = self._h.value       # what the calls are given

    def destroy(self):
        if self._h:
            library().svip_destroy(self._h)
            self._h, self._hv = C.c_void_p(), 0

    def __del__(self):
        try:
            self.destroy()
        except Exception:
            pass

    def set_cluster_size(self, cluster_size: int):
        _check(library().svip_set_cluster_size(self._h, int(cluster_size)))

    def launch_count(self) -> int:
        return int(library().svip_launch_count(self._h))

    def read_status(self, stream=None) -> int:
        flags = C.c_uint(0)
        _check(library().svip_read_status(self._h, C.byref(flags), _stream(stream)), self._h)
        return int(flags.value)

    def draft_step(self, logits, dtype, B, V, row_stride, T, thresh, uniforms, token, entropy, stop,
                   row_stats=None, stream=None):
        rc = _calls.draft_step(self._hv, logits, dtype, B, V, row_stride, T, thresh, uniforms, token, entropy, stop,
                               row_stats, stream)
        if rc:
            _check(rc, self._h)

    def draft_step_masked(self, logits, dtype, B, V, row_stride, T, thresh, uniforms, active, token, entropy, stop,
                          row_stats=None, stream=None):
        rc = _calls.draft_step_masked(self._hv, logits, dtype, B, V, row_stride, T, thresh, uniforms, active, token,
                                      entropy, stop, row_stats, stream)
        if rc:
            _check(rc, self._h)

    def draft_step_at(self, logits, dtype, B, V, row_stride, pos_stride, pos, slot_stride, T, thresh, uniforms,
                      active, token, entropy, stop, row_stats=None, stream=None):
        rc = _calls.draft_step_at(self._hv, logits, dtype, B, V, row_stride, pos_stride, pos, slot_stride, T, thresh,
                                  uniforms, active, token, entropy, stop, row_stats, stream)
        if rc:
            _check(rc, self._h)

    def row_threshold(self, logits, dtype, n_rows, V, row_stride, T, top_k, top_p, thr, stats=None, stream=None):
        rc = _calls.row_threshold(self._hv, logits, dtype, n_rows, V, row_stride, T, top_k, top_p, thr, stats, stream)
        if rc:
            _check(rc, self._h)

    def draft_step_filtered(self, logits, dtype, B, V, row_stride, T, thresh, uniforms, active, thr, token, entropy,
                            stop, row_stats=None, stream=None):
        rc = _calls.draft_step_filtered(self._hv, logits, dtype, B, V, row_stride, T, thresh, uniforms, active, thr,
                                        token, entropy, stop, row_stats, stream)
        if rc:
            _check(rc, self._h)

    def draft_step_truncated(self, logits, dtype, B, V, row_stride, T, thresh, top_k, top_p, uniforms, active, thr,
                             token, entropy, stop, row_stats=None, stream=None):
        rc = _calls.draft_step_truncated(self._hv, logits, dtype, B, V, row_stride, T, thresh, top_k, top_p, uniforms,
                                         active, thr, token, entropy, stop, row_stats, stream)
        if rc:
            _check(rc, self._h)

    def verify_filtered(self, draft_tokens, q_logits, q_row_stride, q_stats, q_thr, q_seq_stride, q_pos_stride,
                        target_logits, t_row_stride, p_thr, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                        n_accepted, next_token, p_stats=None, stream=None):
        rc = _calls.verify_filtered(self._hv, draft_tokens, q_logits, q_row_stride, q_stats, q_thr, q_seq_stride,
                                    q_pos_stride, target_logits, t_row_stride, p_thr, p_stats, dtype, cu_rows, B, K,
                                    n_target_rows, V, T, uniforms, n_accepted, next_token, stream)
        if rc:
            _check(rc, self._h)

    def policy_advance(self, policy, stop, gamma, draft_len, active, B, K_cap, n_active=None, stream=None):
        rc = _calls.policy_advance(self._hv, policy, stop, gamma, draft_len, active, B, K_cap, n_active, stream)
        if rc:
            _check(rc, self._h)

    def policy_update(self, policy, n_accepted, draft_len, gamma, active, B, K_cap, stream=None):
        rc = _calls.policy_update(self._hv, policy, n_accepted, draft_len, gamma, active, B, K_cap, stream)
        if rc:
            _check(rc, self._h)

    def pack_ragged(self, draft_len, B, K_max, cu_rows, row_seq=None, row_pos=None, stream=None):
        rc = _calls.pack_ragged(self._hv, draft_len, B, K_max, cu_rows, row_seq, row_pos, stream)
        if rc:
            _check(rc, self._h)

    def verify(self, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
               target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
               n_accepted, next_token, stream=None):
        rc = _calls.verify(self._hv, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                           target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                           n_accepted, next_token, stream)
        if rc:
            _check(rc, self._h)

    def verify_early_exit(self, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                          target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                          n_accepted, next_token, stream=None):
        rc = _calls.verify_early_exit(self._hv, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride,
                                      q_pos_stride, target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows,
                                      V, T, uniforms, n_accepted, next_token, stream)
        if rc:
            _check(rc, self._h)

    def vp_partial(self, logits, dtype, B, V_shard, row_stride, T, vocab_offset, partial, stream=None):
        rc = _calls.vp_partial(self._hv, logits, dtype, B, V_shard, row_stride, T, vocab_offset, partial, stream)
        if rc:
            _check(rc, self._h)

    def vp_combine(self, partials, G, rank, B, T, thresh, uniforms, entropy, stop, token, owner, local_target,
                   active, stream=None):
        rc = _calls.vp_combine(self._hv, partials, G, rank, B, T, thresh, uniforms, entropy, stop, token, owner,
                               local_target, active, stream)
        if rc:
            _check(rc, self._h)

    def vp_locate(self, logits, dtype, B, V_shard, row_stride, T, local_target, active, vocab_offset, token,
                  stream=None):
        rc = _calls.vp_locate(self._hv, logits, dtype, B, V_shard, row_stride, T, local_target, active, vocab_offset,
                              token, stream)
        if rc:
            _check(rc, self._h)

    def pair_stats(self, q_logits, q_row_stride, target_logits, t_row_stride, dtype, n_pairs, V, T, c_bound, out,
                   stream=None):
        rc = _calls.pair_stats(self._hv, q_logits, q_row_stride, target_logits, t_row_stride, dtype, n_pairs, V, T,
                               c_bound, out, stream)
        if rc:
            _check(rc, self._h)

    def verify_tree(self, tokens, parent, q_logits, q_row_stride, q_stats, target_logits, t_row_stride, dtype, B, N, V,
                    T, uniforms, n_accepted, path, next_token, stream=None):
        rc = _calls.verify_tree(self._hv, tokens, parent, q_logits, q_row_stride, q_stats, target_logits, t_row_stride,
                                dtype, B, N, V, T, uniforms, n_accepted, path, next_token, stream)
        if rc:
            _check(rc, self._h)

    def pair_stats_given(self, q_logits, q_row_stride, q_stats, target_logits, t_row_stride, p_stats, dtype, n_pairs, V, T,
                         c_bound, out, stream=None):
        rc = _calls.pair_stats_given(self._hv, q_logits, q_row_stride, q_stats, target_logits, t_row_stride, p_stats,
                                     dtype, n_pairs, V, T, c_bound, out, stream)
        if rc:
            _check(rc, self._h)

    def selftest_wait_timeout(self, wait_ns: int, stream=None):
        _check(library().svip_selftest_wait_timeout(self._h, int(wait_ns), _stream(stream)), self._h)

    def profile_enable(self, on: bool):
        _check(library().svip_profile_enable(self._h, 1 if on else 0), self._h)

    def profile_read(self):
        ms = C.c_double(0.0)
        n = C.c_long(0)
        _check(library().svip_profile_read(self._h, C.byref(ms), C.byref(n)), self._h)
        return float(ms.value), int(n.value)

    def bind(self, name: str, *args):
        """Pre-marshals one call: returns a zero-argument callable that runs ``svip_<name>(ctx, *args)``
        and raises on a non-zero status.  Saves the per-call conversion cost in launch-bound loops."""
        entry = getattr(library(), "svip_" + name)
        argtypes = entry.argtypes
        if len(args) != len(argtypes) - 1:
            raise TypeError("svip_%s takes %d arguments after the context, %d given" % (name, len(argtypes) - 1, len(args)))
        # through the ctypes types, which take no fraction for an integer and no text for a number
        conv = tuple(t(_convert(a, t) if t is C.c_void_p else a).value for a, t in zip(args, argtypes[1:]))
        fn, h, hv = getattr(_calls, name, entry), self._h, self._hv

        def call():
            rc = fn(hv, *conv)
            if rc:
                _check(rc, h)
        return call

    def graph_begin(self, stream):
        _check(library().svip_graph_begin(self._h, _stream(stream)), self._h)

    def graph_loop_begin(self, stream, n_active, max_iters) -> int:
        """Opens the loop body; returns the raw stream handle on which the body is recorded."""
        body = C.c_void_p()
        _check(library().svip_graph_loop_begin(self._h, _stream(stream), _ptr(n_active), int(max_iters),
                                               C.byref(body)), self._h)
        return int(body.value)

    def graph_loop_end(self):
        _check(library().svip_graph_loop_end(self._h), self._h)

    def graph_end(self, stream) -> Graph:
        g = C.c_void_p()
        _check(library().svip_graph_end(self._h, _stream(stream), C.byref(g)), self._h)
        return Graph(g)
