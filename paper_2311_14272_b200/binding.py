"""ctypes binding of libcrisp's C ABI (see include/crisp.h).

Argument marshalling only: every step of the path runs in the CUDA kernels of
``libcrisp.so``.  PyTorch supplies device buffers and streams.  There is no CPU or
PyTorch fallback: if the shared library is missing, loading raises.
"""
from __future__ import annotations

import ctypes as C
import os
import re
import sys
from array import array
from typing import Optional

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libcrisp.so")

OK, INVALID_ARG, UNSUPPORTED, BAD_SHAPE, BUFFER_TOO_SMALL, CUDA_ERROR, TIMEOUT = range(7)
PATH_DIRECT, PATH_DENSE, PATH_SPARSE, PATH_SPARSE2 = 0, 1, 2, 3
PATH_NAMES = {0: "direct", 1: "dense_tcgen05", 2: "sparse_tcgen05", 3: "sparse_tcgen05_two_addends"}


class LayerDesc(C.Structure):
    _fields_ = [("rows", C.c_int32), ("k", C.c_int32), ("n", C.c_int32), ("m", C.c_int32),
                ("block_rows", C.c_int32), ("block_k", C.c_int32), ("keep_ratio", C.c_double),
                ("score_mode", C.c_int32)]


class RankLayer(C.Structure):
    _fields_ = [("d_scores", C.c_void_p), ("d_max_key", C.c_void_p), ("nrt", C.c_int32), ("nblk", C.c_int32),
                ("block_elems", C.c_int64), ("min_keep", C.c_int32), ("reserved", C.c_int32)]


class PruneLayer(C.Structure):
    _fields_ = [("desc", LayerDesc), ("d_w_bf16", C.c_void_p), ("ld_w", C.c_int64), ("d_grads", C.c_void_p),
                ("ld_grads", C.c_void_p), ("grad_dtypes", C.c_void_p), ("samples", C.c_int32), ("d_saliency", C.c_void_p),
                ("ld_s", C.c_int64), ("d_mask_buf", C.c_void_p), ("d_workspace", C.c_void_p), ("kkeep", C.c_int32),
                ("d_canonical_buf", C.c_void_p), ("d_exec_buf", C.c_void_p)]


class ConvDesc(C.Structure):
    _fields_ = [("batch", C.c_int32), ("height", C.c_int32), ("width", C.c_int32), ("channels", C.c_int32),
                ("kernel_h", C.c_int32), ("kernel_w", C.c_int32), ("pad", C.c_int32), ("y_layout", C.c_int32)]


class LaunchInfo(C.Structure):
    _fields_ = [("path", C.c_int32), ("tile_cols", C.c_int32), ("accumulators", C.c_int32), ("stack", C.c_int32),
                ("epilogue_warps", C.c_int32), ("stages", C.c_int32), ("ctas", C.c_int32), ("conv", C.c_int32),
                ("stage_blocks", C.c_int32)]

    def as_dict(self):
        return {f: int(getattr(self, f)) for f, _ in self._fields_}


class BytesModel(C.Structure):
    _fields_ = [("nnz", C.c_int64), ("vals_bytes", C.c_int64), ("idx_bytes", C.c_int64),
                ("blk_col_bytes", C.c_int64), ("x_bytes", C.c_int64), ("y_bytes", C.c_int64),
                ("useful_macs", C.c_int64), ("slot_macs", C.c_int64), ("path", C.c_int32)]

    def as_dict(self):
        return {f: int(getattr(self, f)) for f, _ in self._fields_}


class CrispError(RuntimeError):
    def __init__(self, code: int, where: str):
        self.code = code
        msg = crisp_status_string(code) if _lib is not None else str(code)
        super().__init__(f"{where}: {msg} (status {code})")


_lib = None
_native = None                                            # the hot ones of the same calls on plain integers (csrc/calls.cpp)
_network = None                                           # what goes over all tensors of a network (csrc/network.cpp); False: not built


def _bind_network():
    """csrc/network.cpp for the library that is loaded, or False in a tree where it could not be built (it needs torch's headers) or was built for
    another torch or Python."""
    global _network
    lib = load()
    if _network is not False:
        import torch                                      # (the module's libraries)
        release = ".".join(re.findall(r"\d+", torch.__version__)[:3])
        try:
            from . import _network as module
            if getattr(module, "built_for", None) == "%s %d.%d" % (release, *sys.version_info[:2]):
                module.bind(C.cast(lib.crisp_decode, C.c_void_p).value)
                _network = module
            else:
                _network = False
        except ImportError:
            _network = False
    return _network


class _CtypesCalls:
    """The calls of csrc/calls.cpp through ctypes: the same arguments and results, 1.5 us slower each.  For a tree where that
    module could not be built (it needs Python's headers)."""

    def __init__(self, lib):
        self._lib = lib
        self.spmm, self.decode = lib.crisp_spmm, lib.crisp_decode

    def spmm_conv(self, handle, activation, *rest):
        *conv, y, ldy, y_dtype, stream = rest
        if any(v != C.c_int32(v).value for v in conv):
            return BAD_SHAPE
        return self._lib.crisp_spmm_conv(handle, activation, ConvDesc(*conv), y, ldy, y_dtype, stream)

    def build_mask(self, saliency, ld, desc, mask_buf, workspace, stream, replaced):
        self._lib.crisp_mask_destroy(replaced)
        mask = C.c_void_p()
        code = self._lib.crisp_build_mask(saliency, ld, LayerDesc.from_address(desc), mask_buf, workspace, stream, C.byref(mask))
        return code, mask.value or 0

    def encode_sizes(self, mask):
        canonical, execution = C.c_size_t(), C.c_size_t()
        code = self._lib.crisp_encode_sizes(mask, C.byref(canonical), C.byref(execution))
        return code, canonical.value, execution.value

    def encode(self, w, ld, mask, canonical_buf, exec_buf, stream, replaced):
        self._lib.crisp_destroy(replaced)
        handle = C.c_void_p()
        code = self._lib.crisp_encode(w, ld, mask, canonical_buf, exec_buf, stream, C.byref(handle))
        return code, handle.value or 0


def load(path: Optional[str] = None):
    """Load libcrisp.so (built in-tree by ``paper_2311_14272_b200.build``)."""
    global _lib, _native
    if _lib is not None and path is None:
        return _lib
    p = path or LIB_PATH
    if not os.path.exists(p):
        raise FileNotFoundError(
            f"{p} not found: build it with `python -m paper_2311_14272_b200.build` "
            "(there is no fallback implementation)")
    lib = C.CDLL(p)
    vp, i32, i64, sz = C.c_void_p, C.c_int32, C.c_int64, C.c_size_t
    P = C.POINTER
    sig = {
        "crisp_keep_count": [P(LayerDesc), P(i32), P(i32)],
        "crisp_mask_sizes": [P(LayerDesc), P(sz), P(sz)],
        "crisp_build_mask": [vp, i64, P(LayerDesc), vp, vp, vp, P(vp)],
        "crisp_build_mask_static": [vp, i64, P(LayerDesc), vp, vp, P(vp)],
        "crisp_mask_export": [vp, vp, vp, vp],
        "crisp_mask_info": [vp, P(LayerDesc), P(i32), P(i32), P(i32)],
        "crisp_encode_sizes": [vp, P(sz), P(sz)],
        "crisp_encode": [vp, i64, vp, vp, vp, vp, P(vp)],
        "crisp_encoded_counts": [vp, P(i64), P(i64), P(i64)],
        "crisp_export": [vp, vp, vp, vp, vp],
        "crisp_decode": [vp, vp, i64, vp],
        "crisp_spmm": [vp, vp, i64, i64, vp, i64, i32, vp],
        "crisp_spmm_conv": [vp, vp, P(ConvDesc), vp, i64, i32, vp],
        "crisp_saliency_accumulate": [vp, i32, i64, i32, i32, vp, i64, i32, vp],
        "crisp_saliency_finish": [vp, i64, vp, i64, i32, i32, i32, vp, i64, vp],
        "crisp_saliency_finish_max": [vp, i64, vp, i64, i32, i32, i32, vp, i64, vp, vp],
        "crisp_build_mask_ex": [vp, i64, P(LayerDesc), vp, vp, C.c_uint32, vp, P(vp)],
        "crisp_mask_reselect": [vp, i32, vp, vp],
        "crisp_prune_fraction": [C.c_double, i32, i32, P(C.c_double)],
        "crisp_keep_ratio_for_count": [P(LayerDesc), i32, P(C.c_double)],
        "crisp_set_path": [vp, i32],
        "crisp_set_epilogue": [vp, vp, i32],
        "crisp_device_status": [vp, vp, P(i32)],
        "crisp_last_launch": [vp, P(LaunchInfo)],
        "crisp_last_resident_bytes": [vp, P(i64)],
        "crisp_set_tuning": [vp, i32, C.c_uint64, i32],
        "crisp_set_stage_blocks": [vp, i32],
        "crisp_reset_status": [vp, vp],
        "crisp_bytes_model": [vp, i64, i32, P(BytesModel)],
        "crisp_mask_scores": [P(LayerDesc), vp, P(vp), P(vp)],
        "crisp_global_rank_sizes": [i32, P(RankLayer), P(sz)],
        "crisp_prune_score": [i32, P(PruneLayer), vp],
        "crisp_prune_encode_sizes": [i32, P(PruneLayer), P(sz), P(sz)],
        "crisp_prune_encode": [i32, P(PruneLayer), vp, P(vp), P(vp)],
        "crisp_destroy_layers": [i32, P(vp), P(vp)],
        "crisp_global_rank": [i32, P(RankLayer), C.c_double, vp, vp, vp],
    }
    for name, args in sig.items():
        fn = getattr(lib, name)
        fn.argtypes = args
        fn.restype = C.c_int
    lib.crisp_mask_destroy.argtypes = [vp]
    lib.crisp_mask_destroy.restype = None
    lib.crisp_destroy.argtypes = [vp]
    lib.crisp_destroy.restype = None
    lib.crisp_status_string.argtypes = [C.c_int]
    lib.crisp_status_string.restype = C.c_char_p
    try:
        from . import _calls as native
        native.bind(*[C.cast(getattr(lib, "crisp_" + name), vp).value for name in
                      ("spmm", "spmm_conv", "decode", "build_mask", "encode_sizes", "encode", "mask_destroy", "destroy")])
    except ImportError:
        native = _CtypesCalls(lib)
    _lib, _native = lib, native
    if _network:
        _bind_network()
    return lib


def crisp_status_string(code: int) -> str:
    return load().crisp_status_string(code).decode()


status_string = crisp_status_string


def _check(code: int, where: str):
    if code != OK:
        raise CrispError(code, where)


def _ptr(t) -> int:
    """Device (or host) address of a torch tensor / numpy array / int."""
    if t is None:
        return 0
    if isinstance(t, int):
        return t
    if hasattr(t, "data_ptr"):
        return t.data_ptr()
    return t.ctypes.data


def _bind_current_stream():
    """The address of torch's current stream on the current device.  torch.cuda.current_stream() builds a Stream object on
    every call, 3.2 us of the 9.6 us that a small product used to spend on the host; the two C functions it asks in the
    end take 0.2 us.  They are not public: without them the public call stays."""
    global _current_stream
    import torch
    torch.cuda.current_stream()                  # initialises CUDA, or says why it cannot
    device, raw = getattr(torch._C, "_cuda_getDevice", None), getattr(torch._C, "_cuda_getCurrentRawStream", None)
    if device is not None and raw is not None:
        _current_stream = lambda: raw(device())
    else:
        _current_stream = lambda: torch.cuda.current_stream().cuda_stream
    return _current_stream()


_current_stream = _bind_current_stream


def _stream(stream) -> int:
    if stream is None:
        return _current_stream()
    if isinstance(stream, int):
        return stream
    return stream.cuda_stream


def make_desc(rows, k, n, m, block_rows, block_k, keep_ratio, score_mode=0) -> LayerDesc:
    return LayerDesc(rows, k, n, m, block_rows, block_k, float(keep_ratio), score_mode)


# ------------------------------------------------------------------ raw entry points

def crisp_keep_count(desc: LayerDesc):
    nblk, kkeep = C.c_int32(), C.c_int32()
    _check(load().crisp_keep_count(C.byref(desc), C.byref(nblk), C.byref(kkeep)), "crisp_keep_count")
    return nblk.value, kkeep.value


def crisp_mask_sizes(desc: LayerDesc):
    a, b = C.c_size_t(), C.c_size_t()
    _check(load().crisp_mask_sizes(C.byref(desc), C.byref(a), C.byref(b)), "crisp_mask_sizes")
    return a.value, b.value


def crisp_saliency_accumulate(d_grad, grad_dtype: int, ld_g: int, rows: int, k: int, d_acc, ld_acc: int, first: bool,
                              stream=None):
    _check(load().crisp_saliency_accumulate(_ptr(d_grad), grad_dtype, ld_g, rows, k, _ptr(d_acc), ld_acc,
                                            1 if first else 0, _stream(stream)), "crisp_saliency_accumulate")


def crisp_saliency_finish(d_acc, ld_acc: int, d_w, ld_w: int, rows: int, k: int, samples: int, d_saliency, ld_s: int,
                          stream=None):
    _check(load().crisp_saliency_finish(_ptr(d_acc), ld_acc, _ptr(d_w), ld_w, rows, k, samples, _ptr(d_saliency), ld_s,
                                        _stream(stream)), "crisp_saliency_finish")


def crisp_saliency_finish_max(d_acc, ld_acc: int, d_w, ld_w: int, rows: int, k: int, samples: int, d_saliency, ld_s: int,
                              d_mask_workspace, stream=None):
    _check(load().crisp_saliency_finish_max(_ptr(d_acc), ld_acc, _ptr(d_w), ld_w, rows, k, samples, _ptr(d_saliency),
                                            ld_s, _ptr(d_mask_workspace), _stream(stream)), "crisp_saliency_finish_max")


MASK_MAX_KNOWN = 1


def crisp_build_mask_ex(d_saliency, ld_s: int, desc: LayerDesc, d_mask_buf, d_workspace, flags: int, stream=None) -> int:
    out = C.c_void_p()
    _check(load().crisp_build_mask_ex(_ptr(d_saliency), ld_s, C.byref(desc), _ptr(d_mask_buf), _ptr(d_workspace),
                                      flags, _stream(stream), C.byref(out)), "crisp_build_mask_ex")
    return out.value


def crisp_mask_reselect(mask: int, kkeep: int, d_workspace, stream=None):
    _check(load().crisp_mask_reselect(mask, kkeep, _ptr(d_workspace), _stream(stream)), "crisp_mask_reselect")


def crisp_prune_fraction(kappa: float, n: int, m: int) -> float:
    out = C.c_double()
    _check(load().crisp_prune_fraction(float(kappa), n, m, C.byref(out)), "crisp_prune_fraction")
    return out.value


def crisp_keep_ratio_for_count(desc: LayerDesc, kkeep: int) -> float:
    out = C.c_double()
    _check(load().crisp_keep_ratio_for_count(C.byref(desc), kkeep, C.byref(out)), "crisp_keep_ratio_for_count")
    return out.value


def crisp_mask_scores(desc: LayerDesc, d_workspace):
    """-> (address of the [nrt, nblk] uint64 block scores, address of the max-key word) inside a workspace
    that crisp_build_mask has filled."""
    a, b = C.c_void_p(), C.c_void_p()
    _check(load().crisp_mask_scores(C.byref(desc), _ptr(d_workspace), C.byref(a), C.byref(b)), "crisp_mask_scores")
    return a.value, b.value


def make_rank_layers(layers):
    """layers: iterable of (d_scores, d_max_key, nrt, nblk, block_elems, min_keep) -> ctypes array."""
    layers = list(layers)
    arr = (RankLayer * len(layers))()
    for i, (sc, mk, nrt, nblk, be, keep) in enumerate(layers):
        arr[i] = RankLayer(_ptr(sc), _ptr(mk), nrt, nblk, be, keep, 0)
    return arr


def crisp_global_rank_sizes(rank_layers) -> int:
    out = C.c_size_t()
    _check(load().crisp_global_rank_sizes(len(rank_layers), rank_layers, C.byref(out)), "crisp_global_rank_sizes")
    return out.value


def crisp_global_rank(rank_layers, prune_fraction: float, d_workspace, d_kkeep, stream=None):
    _check(load().crisp_global_rank(len(rank_layers), rank_layers, float(prune_fraction), _ptr(d_workspace),
                                    _ptr(d_kkeep), _stream(stream)), "crisp_global_rank")


def crisp_prune_score(layers, stream=None):
    """layers: ctypes array of PruneLayer."""
    _check(load().crisp_prune_score(len(layers), layers, _stream(stream)), "crisp_prune_score")


def crisp_prune_encode_sizes(layers):
    """-> (canonical bytes, execution bytes) of every layer, for the kept counts in the array."""
    a, b = (C.c_size_t * len(layers))(), (C.c_size_t * len(layers))()
    _check(load().crisp_prune_encode_sizes(len(layers), layers, a, b), "crisp_prune_encode_sizes")
    return list(a), list(b)


def crisp_prune_encode(layers, stream=None):
    """-> (masks, handles)"""
    m, h = (C.c_void_p * len(layers))(), (C.c_void_p * len(layers))()
    _check(load().crisp_prune_encode(len(layers), layers, _stream(stream), m, h), "crisp_prune_encode")
    return list(m), list(h)


def crisp_build_mask(d_saliency, ld_s: int, desc: LayerDesc, d_mask_buf, d_workspace, stream=None) -> int:
    out = C.c_void_p()
    _check(load().crisp_build_mask(_ptr(d_saliency), ld_s, C.byref(desc), _ptr(d_mask_buf), _ptr(d_workspace),
                                   _stream(stream), C.byref(out)), "crisp_build_mask")
    return out.value


STATIC_SCRATCH_BYTES = 256 * 1024


def crisp_build_mask_static(d_saliency, ld_s: int, desc: LayerDesc, d_mask_buf, stream=None) -> int:
    """crisp_build_mask without a caller-provided workspace: the scratch is a fixed array inside
    the library, for callers that may not allocate device memory.  Layers whose workspace exceeds
    STATIC_SCRATCH_BYTES raise CrispError(BUFFER_TOO_SMALL).  Calls share that array, so they must
    not overlap on the GPU."""
    out = C.c_void_p()
    _check(load().crisp_build_mask_static(_ptr(d_saliency), ld_s, C.byref(desc), _ptr(d_mask_buf),
                                          _stream(stream), C.byref(out)), "crisp_build_mask_static")
    return out.value


def crisp_mask_info(mask: int):
    d, a, b, c = LayerDesc(), C.c_int32(), C.c_int32(), C.c_int32()
    _check(load().crisp_mask_info(mask, C.byref(d), C.byref(a), C.byref(b), C.byref(c)), "crisp_mask_info")
    return d, a.value, b.value, c.value


def crisp_mask_export(mask: int, h_blk_col, h_nm_bits, stream=None):
    _check(load().crisp_mask_export(mask, _ptr(h_blk_col), _ptr(h_nm_bits), _stream(stream)), "crisp_mask_export")


def crisp_encode_sizes(mask: int):
    a, b = C.c_size_t(), C.c_size_t()
    _check(load().crisp_encode_sizes(mask, C.byref(a), C.byref(b)), "crisp_encode_sizes")
    return a.value, b.value


def crisp_encode(d_w, ld_w: int, mask: int, d_canonical, d_exec, stream=None) -> int:
    out = C.c_void_p()
    _check(load().crisp_encode(_ptr(d_w), ld_w, mask, _ptr(d_canonical), _ptr(d_exec), _stream(stream),
                               C.byref(out)), "crisp_encode")
    return out.value


def crisp_encoded_counts(handle: int):
    a, b, c = C.c_int64(), C.c_int64(), C.c_int64()
    _check(load().crisp_encoded_counts(handle, C.byref(a), C.byref(b), C.byref(c)), "crisp_encoded_counts")
    return a.value, b.value, c.value


def crisp_export(handle: int, h_blk_col, h_vals, h_idx, stream=None):
    _check(load().crisp_export(handle, _ptr(h_blk_col), _ptr(h_vals), _ptr(h_idx), _stream(stream)), "crisp_export")


def crisp_decode(handle: int, d_w_dense, ld: int, stream=None):
    _check(load().crisp_decode(handle, _ptr(d_w_dense), ld, _stream(stream)), "crisp_decode")


def crisp_spmm(handle: int, d_x, ldx: int, ncols: int, d_y, ldy: int, y_dtype: int = 0, stream=None):
    _check(load().crisp_spmm(handle, _ptr(d_x), ldx, ncols, _ptr(d_y), ldy, y_dtype, _stream(stream)), "crisp_spmm")


def crisp_spmm_conv(handle: int, d_act_nhwc, conv: ConvDesc, d_y, ldy: int, y_dtype: int = 0, stream=None):
    _check(load().crisp_spmm_conv(handle, _ptr(d_act_nhwc), C.byref(conv), _ptr(d_y), ldy, y_dtype, _stream(stream)),
           "crisp_spmm_conv")


def crisp_set_epilogue(handle: int, d_bias_f32, relu: int):
    _check(load().crisp_set_epilogue(handle, _ptr(d_bias_f32), int(relu)), "crisp_set_epilogue")


def crisp_set_path(handle: int, path: int):
    _check(load().crisp_set_path(handle, path), "crisp_set_path")


def crisp_device_status(handle: int, stream=None) -> int:
    s = C.c_int32()
    _check(load().crisp_device_status(handle, _stream(stream), C.byref(s)), "crisp_device_status")
    return s.value


def crisp_last_launch(handle: int) -> dict:
    """Kernel family (`path`) and tile configuration of the last product launched through the handle."""
    info = LaunchInfo()
    _check(load().crisp_last_launch(handle, C.byref(info)), "crisp_last_launch")
    return info.as_dict()


def crisp_last_resident_bytes(handle: int) -> int:
    """Bytes of weight tiles that the last product's CTAs kept in shared memory for all of their tiles."""
    out = C.c_int64()
    _check(load().crisp_last_resident_bytes(handle, C.byref(out)), "crisp_last_resident_bytes")
    return out.value


def crisp_set_tuning(handle: int, tile_boxes: int = 0, wait_limit_cycles: int = 0, skip_fill: int = -1):
    _check(load().crisp_set_tuning(handle, tile_boxes, wait_limit_cycles, skip_fill), "crisp_set_tuning")


def crisp_set_stage_blocks(handle: int, max_blocks: int = 0):
    """Most kept blocks one pipeline stage may take (1, 2, 4; 0 = chosen by the library)."""
    _check(load().crisp_set_stage_blocks(handle, max_blocks), "crisp_set_stage_blocks")


def crisp_reset_status(handle: int, stream=None):
    _check(load().crisp_reset_status(handle, _stream(stream)), "crisp_reset_status")


def crisp_bytes_model(handle: int, ncols: int, y_dtype: int = 0) -> dict:
    b = BytesModel()
    _check(load().crisp_bytes_model(handle, ncols, y_dtype, C.byref(b)), "crisp_bytes_model")
    return b.as_dict()


def crisp_destroy_layers(masks, handles):
    """masks, handles: ctypes arrays of c_void_p of one length (nulls are skipped)."""
    _check(load().crisp_destroy_layers(len(masks), masks, handles), "crisp_destroy_layers")


def crisp_mask_destroy(mask: int):
    if mask:
        load().crisp_mask_destroy(mask)


def crisp_destroy(handle: int):
    if handle:
        load().crisp_destroy(handle)


# -------------------------------------------------- buffer-owning convenience wrapper

class HybridLayer:
    """Owns the device buffers of one pruned layer and forwards to the C ABI.

    ``build_mask`` -> ``encode`` -> ``spmm`` mirror crisp_build_mask / crisp_encode /
    crisp_spmm; tensors are torch CUDA tensors (bf16 tensors or their int16/uint16 views).
    """

    def __init__(self, rows, k, n, m, block_rows, block_k, keep_ratio, score_mode=0, device="cuda"):
        import torch
        self.torch = torch
        self.device = torch.device(device)
        self.desc = make_desc(rows, k, n, m, block_rows, block_k, keep_ratio, score_mode)
        self.nblk, self.kkeep = crisp_keep_count(self.desc)
        self.nrt = (rows + block_rows - 1) // block_rows
        mask_bytes, ws_bytes = crisp_mask_sizes(self.desc)
        self.mask_buf = torch.empty(mask_bytes, dtype=torch.uint8, device=self.device)
        self.workspace = torch.empty(ws_bytes, dtype=torch.uint8, device=self.device)
        self.device = self.mask_buf.device                   # with its index: results lie beside the buffers, whatever device is current by then
        self.mask = 0
        self.handle = 0
        self.canonical_buf = None
        self.exec_buf = None
        self._gpu = self.device.index if (_network or _bind_network()) else None       # (decode makes its tensors through it)

    # build_mask, encode, decode, spmm and spmm_conv are made once per layer and pass; for small layers their host time is the
    # time of the pass, so they hand plain integers to the library (and ask a tensor for all its strides at once, which is cheaper
    # than for one).
    def build_mask(self, saliency, stream=None):
        strides = saliency.stride()
        assert saliency.is_cuda and saliency.dtype == self.torch.float32 and strides[1] == 1
        old, self.mask = self.mask, 0
        code, self.mask = _native.build_mask(saliency.data_ptr(), strides[0], C.addressof(self.desc), self.mask_buf.data_ptr(),
                                             self.workspace.data_ptr(), _stream(stream), old)
        if code:
            raise CrispError(code, "crisp_build_mask")
        return self

    def rank_layer(self, min_keep=0):
        """This layer's entry for crisp_global_rank (valid after build_mask, until the workspace is reused)."""
        sc, mk = crisp_mask_scores(self.desc, self.workspace)
        return (sc, mk, self.nrt, self.nblk, self.desc.block_rows * self.desc.block_k, min_keep)

    def set_kkeep(self, kkeep: int):
        """Keep ratio that makes the next build_mask keep exactly `kkeep` blocks per row tile."""
        self.desc.keep_ratio = crisp_keep_ratio_for_count(self.desc, kkeep)
        self.nblk, self.kkeep = crisp_keep_count(self.desc)
        assert self.kkeep == kkeep
        mask_bytes, ws_bytes = crisp_mask_sizes(self.desc)
        if self.mask_buf.numel() < mask_bytes:
            self.mask_buf = self.torch.empty(mask_bytes, dtype=self.torch.uint8, device=self.device)
        return self

    def build_mask_max_known(self, saliency, stream=None):
        """build_mask when the workspace already holds the layer maximum (crisp_saliency_finish_max wrote it)."""
        assert saliency.is_cuda and saliency.dtype == self.torch.float32 and saliency.stride(1) == 1
        crisp_mask_destroy(self.mask)
        self.mask = crisp_build_mask_ex(saliency, saliency.stride(0), self.desc, self.mask_buf, self.workspace,
                                        MASK_MAX_KNOWN, stream)
        return self

    def reselect(self, kkeep: int, stream=None):
        """Keep only the `kkeep` best blocks per row tile of the mask just built (no pass over the saliency)."""
        crisp_mask_reselect(self.mask, kkeep, self.workspace, stream)
        self.desc.keep_ratio = crisp_keep_ratio_for_count(self.desc, kkeep)
        self.kkeep = kkeep
        return self

    def export_mask(self, stream=None):
        import numpy as np
        wpr = self.nblk * self.desc.block_k // 32
        blk_col = np.zeros((self.nrt, self.kkeep), dtype=np.int32)
        nm_bits = np.zeros((self.nrt * self.desc.block_rows, wpr), dtype=np.uint32)
        crisp_mask_export(self.mask, blk_col, nm_bits, stream)
        return blk_col, nm_bits

    def encode(self, w, stream=None):
        strides = w.stride()
        assert w.is_cuda and w.element_size() == 2 and strides[1] == 1
        code, canonical_bytes, exec_bytes = _native.encode_sizes(self.mask)
        if code:
            raise CrispError(code, "crisp_encode_sizes")
        self._reserve(canonical_bytes, exec_bytes)
        old, self.handle = self.handle, 0
        code, self.handle = _native.encode(w.data_ptr(), strides[0], self.mask, self.canonical_buf.data_ptr(), self.exec_buf.data_ptr(),
                                           _stream(stream), old)
        if code:
            raise CrispError(code, "crisp_encode")
        return self

    def _reserve(self, canonical_bytes, exec_bytes):
        if self.canonical_buf is None or self.canonical_buf.numel() < canonical_bytes:
            self.canonical_buf = self.torch.empty(canonical_bytes, dtype=self.torch.uint8, device=self.device)
        if self.exec_buf is None or self.exec_buf.numel() < exec_bytes:
            self.exec_buf = self.torch.empty(exec_bytes, dtype=self.torch.uint8, device=self.device)

    def export(self, stream=None):
        import numpy as np
        nb, nv, nw = crisp_encoded_counts(self.handle)
        blk_col = np.zeros(nb, dtype=np.int32)
        vals = np.zeros(nv, dtype=np.uint16)
        idx = np.zeros(nw, dtype=np.uint32)
        crisp_export(self.handle, blk_col, vals, idx, stream)
        return blk_col.reshape(self.nrt, self.kkeep), vals, idx

    # (of the calls in Python empty_strided is the cheapest that allocates: 1.1 us against 3.2 for new_empty and 4.2 for empty)
    def decode(self, stream=None):
        desc, torch = self.desc, self.torch
        k = desc.k
        if self._gpu is not None:
            code, w = _network.decode(self.handle, desc.rows, k, self._gpu, _stream(stream))
            if code:
                raise CrispError(code, "crisp_decode")
            return w
        w = torch.empty_strided((desc.rows, k), (k, 1), dtype=torch.bfloat16, device=self.device)
        code = _native.decode(self.handle, w.data_ptr(), k, _stream(stream))
        if code:
            raise CrispError(code, "crisp_decode")
        return w

    def spmm(self, x, y=None, y_dtype=0, stream=None):
        shape, strides = x.shape, x.stride()
        assert x.is_cuda and x.element_size() == 2 and strides[1] == 1 and shape[0] == self.desc.k
        ncols = shape[1]
        if y is None:
            y = self.torch.empty_strided((self.desc.rows, ncols), (ncols, 1), device=self.device,
                                         dtype=self.torch.float32 if y_dtype else self.torch.bfloat16)
        code = _native.spmm(self.handle, x.data_ptr(), strides[0], ncols, y.data_ptr(), y.stride()[0], y_dtype, _stream(stream))
        if code:
            raise CrispError(code, "crisp_spmm")
        return y

    def spmm_conv(self, act_nhwc, kernel_h, kernel_w, pad, y=None, y_dtype=0, stream=None, nhwc_out=False):
        """Convolution (stride 1) of an NHWC bf16 activation with this layer's weights, without an X matrix.
        nhwc_out: Y is [batch, ho, wo, rows] (the next convolution's activation) instead of [rows, batch*ho*wo]."""
        assert act_nhwc.is_cuda and act_nhwc.element_size() == 2 and act_nhwc.is_contiguous() and act_nhwc.dim() == 4
        b, h, w, c = act_nhwc.shape
        if y is None:
            ho, wo = h + 2 * pad - kernel_h + 1, w + 2 * pad - kernel_w + 1
            dt = self.torch.float32 if y_dtype else self.torch.bfloat16
            y = self.torch.empty((b, ho, wo, self.desc.rows) if nhwc_out else (self.desc.rows, b * ho * wo), dtype=dt, device=self.device)
        ldy = y.stride()[2 if nhwc_out else 0]
        code = _native.spmm_conv(self.handle, act_nhwc.data_ptr(), b, h, w, c, kernel_h, kernel_w, pad, 1 if nhwc_out else 0,
                                 y.data_ptr(), ldy, y_dtype, _stream(stream))
        if code:
            raise CrispError(code, "crisp_spmm_conv")
        return y

    def set_epilogue(self, bias=None, relu=False):
        """Y = act(W X + bias) for later products; `bias` is an fp32 CUDA tensor [rows] that this object keeps."""
        if bias is not None:
            assert bias.is_cuda and bias.dtype == self.torch.float32 and bias.numel() == self.desc.rows
        self._bias = bias
        crisp_set_epilogue(self.handle, bias, 1 if relu else 0)
        return self

    def set_path(self, path: int):
        crisp_set_path(self.handle, path)

    def device_status(self, stream=None) -> int:
        return crisp_device_status(self.handle, stream)

    def last_launch(self) -> dict:
        return crisp_last_launch(self.handle)

    def last_resident_bytes(self) -> int:
        return crisp_last_resident_bytes(self.handle)

    def set_tuning(self, tile_boxes=0, wait_limit_cycles=0, skip_fill=-1):
        crisp_set_tuning(self.handle, tile_boxes, wait_limit_cycles, skip_fill)
        return self

    def set_stage_blocks(self, max_blocks=0):
        crisp_set_stage_blocks(self.handle, max_blocks)
        return self

    def reset_status(self, stream=None):
        crisp_reset_status(self.handle, stream)

    def bytes_model(self, ncols, y_dtype=0):
        return crisp_bytes_model(self.handle, ncols, y_dtype)

    def close(self):
        crisp_destroy(self.handle)
        crisp_mask_destroy(self.mask)
        self.handle = 0
        self.mask = 0

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def _holds_rows(t, rows, k):
    """Whether `rows` rows of k elements lie at the tensor's address, its first stride apart: a matrix of at least that size whose columns are
    consecutive, or more dimensions where those behind the first are dense in any order (a convolution's weights, channels last or not)."""
    shape, strides = t.shape, t.stride()
    if not shape or shape[0] < rows or 0 in shape:
        return False
    run = 1
    for step, size in sorted((step, size) for step, size in zip(strides[1:], shape[1:]) if size != 1):
        if step != run:
            return k == 1
        run *= size
    return run >= k


class PruningNetwork:
    """One pruning iteration of Algorithm 1 over all layers of a network, without the fine-tuning that follows it:

        network     saliency of Eq. 1 from the caller's gradients, N:M step, block scores   crisp_prune_score
        network     rank-column sums, global order, selection                              crisp_global_rank
        network     keep the selected number of blocks per layer, compress                 crisp_prune_encode

    This class only owns buffers and issues those calls in that order; every number is computed by the library.
    `shapes` is a list of (rows, k); the pattern (n:m, block shape) is shared by the layers.
    """

    def __init__(self, shapes, n, m, block_rows, block_k, min_keep=1, device="cuda"):
        import torch
        self.torch = torch
        self.device = torch.device(device)
        self.n, self.m = n, m
        self.min_keep = min_keep
        self.layers = [HybridLayer(r, k, n, m, block_rows, block_k, 1.0, device=device) for (r, k) in shapes]
        self.sal = [torch.empty((r, k), dtype=torch.float32, device=self.device) for (r, k) in shapes]
        self._acc = None
        self.rank_arr = make_rank_layers([L.rank_layer(min_keep) for L in self.layers])
        self.rank_ws = torch.empty(crisp_global_rank_sizes(self.rank_arr), dtype=torch.uint8, device=self.device)
        self.d_kkeep = torch.zeros(len(shapes), dtype=torch.int32, device=self.device)
        self._h_kkeep = torch.zeros(len(shapes), dtype=torch.int32, pin_memory=True)
        self._blocks = (C.c_int32 * len(shapes))(*[L.nblk for L in self.layers])

    @property
    def acc(self):
        """The running gradient sums of layers whose gradients come in turn (allocated when first used)."""
        if self._acc is None:
            self._acc = [self.torch.empty_like(s) for s in self.sal]
        return self._acc

    def _score_in_turn(self, weights, grads, stream):
        """crisp_prune_score in the calls it replaces, one gradient tensor at a time; the number of layers."""
        count = 0
        for L, w, gs, acc, s in zip(self.layers, weights, grads, self.acc, self.sal):
            rows, k = L.desc.rows, L.desc.k
            for i, g in enumerate(gs):
                self._check_gradient(g, L)
                crisp_saliency_accumulate(g, 0 if g.dtype == self.torch.bfloat16 else 1, g.stride(0), rows, k, acc, k, i == 0,
                                          stream)
            crisp_saliency_finish_max(acc, k, w, w.stride(0), rows, k, len(gs), s, k, L.workspace, stream)
            L.desc.keep_ratio = 1.0
            L.nblk, L.kkeep = crisp_keep_count(L.desc)
            L.build_mask_max_known(s, stream)
            count += 1
        return count

    def _check_gradient(self, g, layer):
        """The library gets an address and a pitch: what is no bf16 or fp32 matrix of the layer's size on a GPU would be read beyond its end, or as
        something else.  (What only has a tensor's methods answers for itself.)"""
        torch = self.torch
        if isinstance(g, torch.Tensor):
            assert g.is_cuda and g.dtype in (torch.bfloat16, torch.float32) and _holds_rows(g, layer.desc.rows, layer.desc.k), \
                "a gradient is a bf16 or fp32 CUDA tensor of its layer's shape"

    def _table(self, arr, layers, weights, grads):
        """Fills in the table of the layers: one host array each for what there is per gradient (returned; the entries point into them),
        and one struct per layer."""
        for L, gs in zip(layers, grads):
            for g in gs:
                self._check_gradient(g, L)
        flat = [g for gs in grads for g in gs]
        ptrs = array("Q", [g.data_ptr() for g in flat])
        lds = array("q", [g.stride()[0] for g in flat])
        dts = array("i", [0 if g.dtype is self.torch.bfloat16 else 1 for g in flat])
        p0, l0, d0, at = ptrs.buffer_info()[0], lds.buffer_info()[0], dts.buffer_info()[0], 0
        for P, L, w, gs, s in zip(arr, layers, weights, grads, self.sal):
            P.desc, P.d_w_bf16, P.ld_w = L.desc, w.data_ptr(), w.stride()[0]
            n = len(gs)
            P.d_grads, P.ld_grads, P.grad_dtypes, P.samples = p0 + 8 * at, l0 + 8 * at, d0 + 4 * at, n
            P.d_saliency, P.ld_s = s.data_ptr(), s.stride()[0]
            P.d_mask_buf, P.d_workspace = L.mask_buf.data_ptr(), L.workspace.data_ptr()
            at += n
        return ptrs, lds, dts, flat

    def step(self, weights, grads, kappa, stream=None):
        """weights[l]: bf16 CUDA tensor [rows, k]; grads[l]: list of H gradient tensors (bf16 or fp32) of that shape;
        kappa: overall sparsity target of this iteration.  Returns the kept-block count of every layer; the layers'
        masks and handles (self.layers[l]) hold the result.

        Lists and tuples (or stacked tensors) of gradients are taken for all layers at once.  Anything else that can be iterated over (a generator
        that makes one layer's gradients after the other, say) is read layer by layer and gradient by gradient, and each
        gradient's kernel is on the stream before the next one is asked for."""
        torch = self.torch
        weights = list(weights)
        # every gradient exists, and none is changed by asking for the next
        held = (list, tuple, torch.Tensor)
        at_once = isinstance(grads, held) and (set(map(type, grads)) <= {list, tuple} or all(isinstance(gs, held) for gs in grads))
        count = min(len(self.layers), len(weights), len(grads) if at_once else len(weights))
        weights, layers = weights[:count], self.layers[:count]
        arr, table = (PruneLayer * count)(), None
        if at_once and _network:
            gradients = [gs if type(gs) in (list, tuple) else list(gs) for gs in grads[:count]]
            table = _network.table(layers, weights, gradients, self.sal, C.addressof(arr))
        if table is None:
            assert all(w.is_cuda and w.element_size() == 2 and w.stride()[1] == 1 and (not isinstance(w, torch.Tensor) or _holds_rows(w, L.desc.rows, L.desc.k))
                       for w, L in zip(weights, layers))
            if not at_once:
                count = self._score_in_turn(weights, grads, stream)
                arr, layers = (PruneLayer * count)(), layers[:count]
            table = self._table(arr, layers, weights, grads[:count] if at_once else [()] * count)
        if at_once:
            crisp_prune_score(arr, stream)
        crisp_global_rank(self.rank_arr, crisp_prune_fraction(kappa, self.n, self.m), self.rank_ws, self.d_kkeep, stream)
        # While the device scores and ranks: what the encodings need whatever the counts are, and the masks and handles that
        # they will take the place of.
        old_masks, old_handles, masks, handles = [(C.c_void_p * count)() for _ in range(4)]
        canonical_bytes, exec_bytes, have_c, have_e = [(C.c_size_t * count)() for _ in range(4)]
        if not (_network and _network.encodings(layers, *map(C.addressof, (arr, have_c, have_e, old_masks, old_handles)))):
            for i, (P, L) in enumerate(zip(arr, layers)):
                if L.canonical_buf is not None:
                    P.d_canonical_buf, P.d_exec_buf = L.canonical_buf.data_ptr(), L.exec_buf.data_ptr()
                    have_c[i], have_e[i] = L.canonical_buf.numel(), L.exec_buf.numel()
                old_masks[i], old_handles[i] = L.mask, L.handle
        # (a copy into pinned memory and a wait for the stream: 10 us less than a copy into pageable memory)
        with torch.cuda.stream(stream):                      # (None: the current one)
            self._h_kkeep.copy_(self.d_kkeep, non_blocking=True)
            torch.cuda.current_stream(self.d_kkeep.device).synchronize()
        kk = self._h_kkeep.tolist()
        for P, c in zip(arr, kk):
            P.kkeep = c
        _check(_lib.crisp_prune_encode_sizes(count, arr, canonical_bytes, exec_bytes), "crisp_prune_encode_sizes")
        for i, (cb, eb) in enumerate(zip(canonical_bytes, exec_bytes)):
            if cb > have_c[i] or eb > have_e[i]:
                P, L = arr[i], layers[i]
                L._reserve(cb, eb)
                P.d_canonical_buf, P.d_exec_buf = L.canonical_buf.data_ptr(), L.exec_buf.data_ptr()
        _check(_lib.crisp_prune_encode(count, arr, _stream(stream), masks, handles), "crisp_prune_encode")
        if _network:
            _network.encoded(layers, kk, *map(C.addressof, (self._blocks, masks, handles)))
        else:
            for L, c, mask, handle in zip(layers, kk, masks, handles):
                L.mask, L.handle, L.kkeep = mask, handle, c
                L.desc.keep_ratio = c / L.nblk               # floor(ratio * nblk + 0.5) gives the count back
        crisp_destroy_layers(old_masks, old_handles)
        return kk

    def close(self):
        for L in self.layers:
            L.close()
