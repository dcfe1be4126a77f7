"""Binding of ``librac.so`` -- argument marshalling only.

Every function has the name and the argument order of its C entry point in
``include/rac.h``.  Arguments are either raw addresses (int) or torch tensors
living where the C function expects them (device pointers for the ``rac_*``
calls); the binding checks dtype, contiguity and device, takes the tensor's
address and the current CUDA stream (or ``stream``: a ``torch.cuda.Stream`` or
an address), calls the library and raises on a non-zero return code.  The launching calls are marshalled by the extension module
``_native`` (``csrc/rac_py.cpp``), the others and the plain library by ctypes.
No arithmetic of the method happens here and there is no fallback: if the
library cannot be loaded, importing callers get an error.
"""
from __future__ import annotations

import ctypes as C
import os
from typing import Optional

import torch  # noqa: F401  (the extension module needs its libraries in the process)

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "librac.so")

RAC_OK = 0
STATUS_REF_RANGE = 1
STATUS_RESERVED_CODE = 2
STATUS_NONFINITE = 4
STATUS_TIMEOUT = 8
STATUS_OUTLIER_RANGE = 16

EXPORTS = [
    "rac_version", "rac_strerror", "rac_record_bytes", "rac_payload_bytes", "rac_header_write", "rac_header_parse",
    "rac_match_workspace_bytes", "rac_match_spans", "rac_spans_to_rows",
    "rac_match_spans_static",
    "rac_index_bytes", "rac_index_reset", "rac_index_append", "rac_index_query_workspace_bytes", "rac_index_query",
    "rac_index_query_live",
    "rac_encode_workspace_bytes", "rac_encode", "rac_encode_reconstruct", "rac_decode_reconstruct",
    "rac_sender_reconstruct",
    "rac_split_waves", "rac_encode_reconstruct_list", "rac_decode_reconstruct_list",
    "rac_fit_segments_workspace_bytes", "rac_fit_segments", "rac_spans_to_segments",
    "rac_calibrate_workspace_bytes", "rac_calibrate_steps", "rac_calibrate_steps_shared",
    "rac_recon_error_workspace_bytes", "rac_recon_error",
    "rac_selftest_bounded_wait",
]


class RacError(RuntimeError):
    def __init__(self, fn: str, code: int, msg: str):
        super().__init__(f"{fn} failed: {code} ({msg})")
        self.code = code


class CodecCfg(C.Structure):
    """Mirror of ``rac_codec_cfg``."""
    _fields_ = [(n, C.c_int32) for n in ("d", "group", "bits", "topk", "coef_fmt", "scale_mode", "flags",
                                         "qgroup", "topk_group")]

    def __init__(self, d: int, group: int, bits: int, topk: int = 0, scale_mode: int = 0, qgroup: int = 0,
                 topk_group: int = 0, coef_fmt: int = 0):
        super().__init__(d, group, bits, topk, coef_fmt, scale_mode, 0, qgroup, topk_group)

    def __repr__(self):
        return (f"CodecCfg(d={self.d}, group={self.group}, bits={self.bits}, topk={self.topk}, "
                f"scale_mode={self.scale_mode}, qgroup={self.qgroup}, topk_group={self.topk_group})")


class IndexCfg(C.Structure):
    """Mirror of ``rac_index_cfg``."""
    _fields_ = [("capacity", C.c_int64), ("min_ngram", C.c_int32), ("max_hits", C.c_int32)]

    def __init__(self, capacity: int, min_ngram: int = 4, max_hits: int = 8):
        super().__init__(capacity, min_ngram, max_hits)


_lib: Optional[C.CDLL] = None


class _Recorder:
    """Stands in for the extension module while `prepare` runs a wrapper once: calls are recorded instead of made."""

    def __init__(self, native):
        self._native = native
        self.calls = []

    def __getattr__(self, name):
        entry = getattr(self._native, name)

        def record(*args):
            self.calls.append((entry, args))
        return record


_native = None        # the extension module, or the recorder while a call is prepared


def prepare(wrapper, *args, **kwargs):
    """Marshals the arguments of one call ONCE and returns a function without arguments that repeats the call.

    ``wrapper`` is one of the functions of this module that launch work (``rac_encode_reconstruct``,
    ``rac_decode_reconstruct``, ...), ``args`` what it would be given.  Tensor addresses, sizes and the stream
    (``stream=`` or the current one at the time of this call) are fixed here; the tensors must stay alive and in
    place.  For loops that issue the same small call many times (a decode step per token), where looking at a dozen
    tensors takes a share of the call.  Not thread safe while it prepares."""
    global _native
    load()
    native = _native
    rec = _Recorder(native)
    _native = rec
    try:
        wrapper(*args, **kwargs)
    finally:
        _native = native
    if len(rec.calls) != 1:
        raise ValueError("prepare() wants a wrapper that makes exactly one library call")
    entry, cargs = rec.calls[0]
    # the tensors (and the configuration struct the pointers refer to) stay referenced
    return native.prepare(entry, cargs, (args, kwargs))


def load():
    """Load the C-ABI library.  Raises if it has not been built (``__graft_entry__.build()``)."""
    global _lib, _native
    if _lib is not None:
        return _lib
    if not os.path.exists(LIB_PATH):
        raise RuntimeError(f"{LIB_PATH} is missing: build it with `python -m paper_2608_04991_b200.build` "
                           "(there is no CPU fallback)")
    l = C.CDLL(LIB_PATH)
    # (the launching calls below go through `_native`; their signatures are for callers who use the library returned here)
    vp, i64, i32, sz = C.c_void_p, C.c_int64, C.c_int32, C.c_size_t
    cfgp = C.POINTER(CodecCfg)
    l.rac_version.restype = C.c_char_p
    l.rac_version.argtypes = []
    l.rac_strerror.restype = C.c_char_p
    l.rac_strerror.argtypes = [C.c_int]
    l.rac_record_bytes.restype = sz
    l.rac_record_bytes.argtypes = [cfgp]
    l.rac_payload_bytes.restype = sz
    l.rac_payload_bytes.argtypes = [cfgp, i64]
    l.rac_header_write.restype = C.c_int
    l.rac_header_write.argtypes = [cfgp, i64, vp]
    l.rac_header_parse.restype = C.c_int
    l.rac_header_parse.argtypes = [vp, cfgp, C.POINTER(i64)]
    l.rac_match_workspace_bytes.restype = sz
    l.rac_match_workspace_bytes.argtypes = [i64, i64, i32]
    l.rac_match_spans.restype = C.c_int
    l.rac_match_spans.argtypes = [vp, i64, vp, i64, i32, i32, vp, vp, vp, vp, sz, vp]
    l.rac_match_spans_static.restype = C.c_int
    l.rac_match_spans_static.argtypes = [vp, i64, vp, i64, i32, i32, vp, vp, vp, vp]
    icfgp = C.POINTER(IndexCfg)
    l.rac_index_bytes.restype = sz
    l.rac_index_bytes.argtypes = [icfgp]
    l.rac_index_reset.restype = C.c_int
    l.rac_index_reset.argtypes = [icfgp, vp, sz, vp]
    l.rac_index_append.restype = C.c_int
    l.rac_index_append.argtypes = [icfgp, vp, sz, vp, i64, i64, vp]
    l.rac_index_query_workspace_bytes.restype = sz
    l.rac_index_query_workspace_bytes.argtypes = [i64]
    l.rac_index_query.restype = C.c_int
    l.rac_index_query.argtypes = [icfgp, vp, sz, vp, i64, vp, i64, i32, vp, vp, vp, vp, sz, vp]
    l.rac_index_query_live.restype = C.c_int
    l.rac_index_query_live.argtypes = [icfgp, vp, sz, vp, i64, i64, vp, i64, i32, vp, vp, vp, vp, sz, vp]
    l.rac_spans_to_rows.restype = C.c_int
    l.rac_spans_to_rows.argtypes = [vp, vp, i64, vp, vp]
    l.rac_encode.restype = C.c_int
    l.rac_encode_workspace_bytes.restype = sz
    l.rac_encode_workspace_bytes.argtypes = [cfgp, i64]
    l.rac_encode.argtypes = [cfgp, vp, i64, vp, i64, vp, vp, vp, vp, vp, vp, sz, vp, sz, vp, vp]
    l.rac_encode_reconstruct.restype = C.c_int
    l.rac_encode_reconstruct.argtypes = [cfgp, vp, i64, vp, i64, vp, vp, vp, vp, vp, vp, sz, vp, vp, sz, vp, vp]
    for name in ("rac_decode_reconstruct", "rac_sender_reconstruct"):
        f = getattr(l, name)
        f.restype = C.c_int
        f.argtypes = [cfgp, vp, i64, vp, i64, vp, vp, vp, vp, vp, vp, vp]
    l.rac_selftest_bounded_wait.restype = C.c_int
    l.rac_selftest_bounded_wait.argtypes = [cfgp, i32, vp, i64, vp, i64, vp, vp, vp, sz, vp, sz, vp, vp]
    l.rac_split_waves.restype = C.c_int
    l.rac_split_waves.argtypes = [vp, i64, i64, vp, vp, vp, vp]
    l.rac_encode_reconstruct_list.restype = C.c_int
    l.rac_encode_reconstruct_list.argtypes = [cfgp, vp, i64, vp, vp, vp, i64, vp, vp, i64, vp, vp, vp, vp, vp, vp, vp, sz,
                                              vp, vp, sz, vp, vp]
    l.rac_decode_reconstruct_list.restype = C.c_int
    l.rac_decode_reconstruct_list.argtypes = [cfgp, vp, i64, vp, vp, vp, i64, vp, vp, i64, vp, vp, vp, vp, vp, vp, vp, vp]
    l.rac_spans_to_segments.restype = C.c_int
    l.rac_spans_to_segments.argtypes = [vp, vp, i64, i64, vp, vp, vp]
    l.rac_fit_segments_workspace_bytes.restype = sz
    l.rac_fit_segments_workspace_bytes.argtypes = [cfgp, i64]
    l.rac_fit_segments.restype = C.c_int
    l.rac_fit_segments.argtypes = [cfgp, vp, i64, vp, i64, vp, vp, vp, vp, i64, vp, vp, vp, sz, vp, vp]
    l.rac_recon_error_workspace_bytes.restype = sz
    l.rac_recon_error_workspace_bytes.argtypes = []
    l.rac_recon_error.restype = C.c_int
    l.rac_recon_error.argtypes = [vp, vp, i64, i32, vp, vp, sz, vp]
    l.rac_calibrate_workspace_bytes.restype = sz
    l.rac_calibrate_workspace_bytes.argtypes = [cfgp]
    l.rac_calibrate_steps.restype = C.c_int
    l.rac_calibrate_steps.argtypes = [cfgp, vp, i64, vp, i64, vp, vp, vp, C.c_float, vp, vp, vp, sz, vp, vp]
    l.rac_calibrate_steps_shared.restype = C.c_int
    l.rac_calibrate_steps_shared.argtypes = [cfgp, vp, i64, vp, i64, vp, vp, vp, vp, vp, C.c_float, vp, vp, vp, sz, vp, vp]
    from . import _native as native
    native.setup(_check, _stream_address, CodecCfg, IndexCfg)
    _native = native
    _lib = l
    return l


def _calls():
    """Where launching calls go: the extension module (loaded on first use)."""
    if _native is None:
        load()
    return _native


def _check(fn: str, rc: int) -> None:
    if rc != RAC_OK:
        raise RacError(fn, rc, load().rac_strerror(rc).decode())


def _stream_address(stream) -> int:
    """Address of a stream that is neither None nor an integer: a ``torch.cuda.Stream``, a ``c_void_p``, whatever else
    ctypes passes as a pointer."""
    return C.cast(stream, C.c_void_p).value or 0


# ----------------------------------------------------------------------------- plain queries
def rac_version() -> str:
    return load().rac_version().decode()


def rac_strerror(code: int) -> str:
    return load().rac_strerror(int(code)).decode()


def rac_record_bytes(cfg: CodecCfg) -> int:
    return int(load().rac_record_bytes(C.byref(cfg)))


def rac_payload_bytes(cfg: CodecCfg, T: int) -> int:
    return int(load().rac_payload_bytes(C.byref(cfg), int(T)))


HEADER_BYTES = 64


def rac_header_write(cfg: CodecCfg, T: int) -> bytes:
    """The 64-byte header of a serialised payload of T records (host work only)."""
    buf = C.create_string_buffer(HEADER_BYTES)
    _check("rac_header_write", load().rac_header_write(C.byref(cfg), int(T), buf))
    return buf.raw


def rac_header_parse(header: bytes):
    """(CodecCfg, T) of a header written by rac_header_write; raises RacError when it does not check out."""
    if len(header) < HEADER_BYTES:
        raise ValueError("a header is 64 bytes")
    buf = C.create_string_buffer(bytes(header[:HEADER_BYTES]), HEADER_BYTES)
    cfg, T = CodecCfg(64, 32, 4, 0), C.c_int64(0)
    _check("rac_header_parse", load().rac_header_parse(buf, C.byref(cfg), C.byref(T)))
    return cfg, int(T.value)


def rac_match_workspace_bytes(n_hist: int, n_query: int, max_hits: int) -> int:
    return int(load().rac_match_workspace_bytes(int(n_hist), int(n_query), int(max_hits)))


def rac_encode_workspace_bytes(cfg: CodecCfg, T: int) -> int:
    return int(load().rac_encode_workspace_bytes(C.byref(cfg), int(T)))


def rac_split_waves(ref_row, T, first_intra_row, wave1, wave2, wave_count, stream=None) -> None:
    _calls().rac_split_waves(ref_row, T, first_intra_row, wave1, wave2, wave_count, stream)


def rac_encode_reconstruct_list(cfg, X, T, tok_list, tok_count, ref_base, ref_rows, ref_row, intra_base, intra_rows,
                                ref_gain, ref_bias, step, inv_step, payload, payload_cap, X_hat, workspace,
                                workspace_bytes, dev_status, stream=None, coef_seg=None, seg_of=None) -> None:
    _calls().rac_encode_reconstruct_list(cfg, X, T, tok_list, tok_count, ref_base, ref_rows, ref_row, intra_base,
                                         intra_rows, coef_seg, seg_of, ref_gain, ref_bias, step, inv_step, payload,
                                         payload_cap, X_hat, workspace, workspace_bytes, dev_status, stream)


def rac_decode_reconstruct_list(cfg, payload, T, tok_list, tok_count, ref_base, ref_rows, ref_row, intra_base,
                                intra_rows, ref_gain, ref_bias, step, X_hat, dev_status, stream=None, coef_seg=None,
                                seg_of=None) -> None:
    _calls().rac_decode_reconstruct_list(cfg, payload, T, tok_list, tok_count, ref_base, ref_rows, ref_row, intra_base,
                                         intra_rows, coef_seg, seg_of, ref_gain, ref_bias, step, X_hat, dev_status,
                                         stream)


def rac_spans_to_segments(spans, n_spans, T, max_seg, seg_off, n_seg, stream=None) -> None:
    _calls().rac_spans_to_segments(spans, n_spans, T, max_seg, seg_off, n_seg, stream)


def rac_fit_segments_workspace_bytes(cfg: CodecCfg, T: int) -> int:
    return int(load().rac_fit_segments_workspace_bytes(C.byref(cfg), int(T)))


def rac_fit_segments(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, seg_off, n_seg, coef_seg, seg_of,
                     workspace, workspace_bytes, dev_status, stream=None) -> None:
    """Eq. 6 over several fitting positions; ``coef_seg`` is an int32 tensor [n_seg, J] holding the u32 words."""
    _calls().rac_fit_segments(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, seg_off, n_seg, coef_seg,
                              seg_of, workspace, workspace_bytes, dev_status, stream)


def rac_recon_error_workspace_bytes() -> int:
    return int(load().rac_recon_error_workspace_bytes())


def rac_recon_error(X, X_hat, T, d, out, workspace, workspace_bytes, stream=None) -> None:
    _calls().rac_recon_error(X, X_hat, T, d, out, workspace, workspace_bytes, stream)


def rac_calibrate_workspace_bytes(cfg: CodecCfg) -> int:
    return int(load().rac_calibrate_workspace_bytes(C.byref(cfg)))


# ----------------------------------------------------------------------------- device calls
def rac_match_spans(hist_tok, n_hist, query_tok, n_query, min_ngram, max_hits, ref_row, spans, n_spans, workspace,
                    workspace_bytes, stream=None) -> None:
    _calls().rac_match_spans(hist_tok, n_hist, query_tok, n_query, min_ngram, max_hits, ref_row, spans, n_spans,
                             workspace, workspace_bytes, stream)


MATCH_STATIC_BYTES = 3 << 20  # RAC_MATCH_STATIC_BYTES in rac.h


def rac_match_spans_static(hist_tok, n_hist, query_tok, n_query, min_ngram, max_hits, ref_row, spans, n_spans,
                           stream=None) -> None:
    """Span retrieval on the library's built-in 3 MiB scratch: for callers that may not allocate device memory.
    Calls on one device must not overlap on the GPU (they share the scratch)."""
    _calls().rac_match_spans_static(hist_tok, n_hist, query_tok, n_query, min_ngram, max_hits, ref_row, spans, n_spans,
                                    stream)


def rac_index_bytes(cfg: IndexCfg) -> int:
    return int(load().rac_index_bytes(C.byref(cfg)))


def rac_index_query_workspace_bytes(n_query: int) -> int:
    return int(load().rac_index_query_workspace_bytes(int(n_query)))


def rac_index_reset(cfg, index, index_bytes, stream=None) -> None:
    _calls().rac_index_reset(cfg, index, index_bytes, stream)


def rac_index_append(cfg, index, index_bytes, hist_tok, n_before, n_after, stream=None) -> None:
    _calls().rac_index_append(cfg, index, index_bytes, hist_tok, n_before, n_after, stream)


def rac_index_query_live(cfg, index, index_bytes, hist_tok, n_hist, first_live, query_tok, n_query, intra, ref_row,
                         spans, n_spans, workspace, workspace_bytes, stream=None) -> None:
    _calls().rac_index_query_live(cfg, index, index_bytes, hist_tok, n_hist, first_live, query_tok, n_query, intra,
                                  ref_row, spans, n_spans, workspace, workspace_bytes, stream)


def rac_index_query(cfg, index, index_bytes, hist_tok, n_hist, query_tok, n_query, intra, ref_row, spans, n_spans,
                    workspace, workspace_bytes, stream=None) -> None:
    _calls().rac_index_query(cfg, index, index_bytes, hist_tok, n_hist, query_tok, n_query, intra, ref_row, spans,
                             n_spans, workspace, workspace_bytes, stream)


def rac_spans_to_rows(spans, n_spans, n_query, ref_row, stream=None) -> None:
    _calls().rac_spans_to_rows(spans, n_spans, n_query, ref_row, stream)


def rac_encode(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step, payload, payload_cap,
               workspace, workspace_bytes, dev_status, stream=None) -> None:
    _calls().rac_encode(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step, payload,
                        payload_cap, workspace, workspace_bytes, dev_status, stream)


def rac_encode_reconstruct(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step, payload,
                           payload_cap, X_hat, workspace, workspace_bytes, dev_status, stream=None) -> None:
    _calls().rac_encode_reconstruct(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step,
                                    payload, payload_cap, X_hat, workspace, workspace_bytes, dev_status, stream)


def rac_decode_reconstruct(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat, dev_status,
                           stream=None) -> None:
    _calls().rac_decode_reconstruct(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat,
                                    dev_status, stream)


def rac_sender_reconstruct(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat, dev_status,
                           stream=None) -> None:
    _calls().rac_sender_reconstruct(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat,
                                    dev_status, stream)


def rac_selftest_bounded_wait(cfg, which, inp, T, ref_base, ref_rows, step, inv_step, out, out_cap, workspace,
                              workspace_bytes, dev_status, stream=None) -> None:
    """Runs the encode (which=0), reconstruction (1) or encode-and-reconstruct (2) kernels with waits that cannot complete; see rac.h."""
    _calls().rac_selftest_bounded_wait(cfg, which, inp, T, ref_base, ref_rows, step, inv_step, out, out_cap, workspace,
                                       workspace_bytes, dev_status, stream)


def rac_calibrate_steps(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, clip_sigmas, step, inv_step,
                        workspace, workspace_bytes, dev_status, stream=None) -> None:
    _calls().rac_calibrate_steps(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, clip_sigmas, step,
                                 inv_step, workspace, workspace_bytes, dev_status, stream)


def rac_calibrate_steps_shared(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, coef_seg, seg_of,
                               clip_sigmas, step, inv_step, workspace, workspace_bytes, dev_status, stream=None) -> None:
    _calls().rac_calibrate_steps_shared(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, coef_seg, seg_of,
                                        clip_sigmas, step, inv_step, workspace, workspace_bytes, dev_status, stream)