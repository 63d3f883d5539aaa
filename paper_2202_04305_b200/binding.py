"""Thin ctypes binding over libsp.so: argument marshalling only.

Every function has the name and the meaning of the C entry point in
``include/sp.h``; torch supplies device memory and the current stream.
There is no fallback: if the library is missing, importing fails.
"""
from __future__ import annotations

import ctypes as C
import os

import torch

DENSE, COMPRESSED = 0, 1
MAX_RANK = 5
DUP_SUM, DUP_ERROR = 0, 1

_HERE = os.path.dirname(os.path.abspath(__file__))
# SP_DEBUG_BOUNDS=1 in the environment selects the bounds-checking build of the same library (every
# index derived from stored positions / coordinates is checked on the device; a bad one makes the call
# return SP_ERR_OUT_OF_RANGE instead of reading or writing out of bounds).  Much slower; for debugging.
DEBUG_BOUNDS = os.environ.get("SP_DEBUG_BOUNDS", "") not in ("", "0")
_LIB_PATH = os.path.join(_HERE, "libsp_debug_bounds.so" if DEBUG_BOUNDS else "libsp.so")
_TORCH_LIB_PATH = os.path.join(_HERE, "libsp_torch.so")

SYMBOLS = ["sp_status_string", "sp_set_allocator", "sp_pack", "sp_free", "sp_info", "sp_positions",
           "sp_coordinates", "sp_values", "sp_unpack", "sp_spmv", "sp_spmm", "sp_sddmm", "sp_mttkrp",
           "sp_launch_count", "sp_spmv_static", "sp_mttkrp_mode", "sp_spmspm", "sp_convert", "sp_scale", "sp_vec_dot"]
SPMV_STATIC_MAX_ITEMS = 134217728


class SpError(RuntimeError):
    def __init__(self, code: int, where: str):
        self.code = code
        super().__init__(f"{where}: {_lib.sp_status_string(code).decode()} (status {code})")


def _load():
    for path in (_LIB_PATH, _TORCH_LIB_PATH):
        if not os.path.exists(path):
            raise ImportError(f"{path} not found: build it with `python -m paper_2202_04305_b200.build"
                              f"{' --debug-bounds' if DEBUG_BOUNDS else ''}` (there is no CPU fallback)")
    lib = C.CDLL(_LIB_PATH)
    lib.sp_status_string.restype = C.c_char_p
    lib.sp_status_string.argtypes = [C.c_int]
    for name in SYMBOLS[1:]:
        getattr(lib, name).restype = C.c_int
    lib.sp_launch_count.restype = C.c_int64
    # argument types stated once: plain integers are then converted in C, without an object per argument
    p, n, i = C.c_void_p, C.c_int64, C.c_int
    for name, args in {"sp_pack": [i, p, n, p, i, p, p, p, i, i, C.c_uint, p, p], "sp_free": [p], "sp_info": [p] * 7,
                       "sp_positions": [p, i, p, p], "sp_coordinates": [p, i, p, p], "sp_values": [p, p, p],
                       "sp_unpack": [p] * 5, "sp_spmv": [p] * 4, "sp_spmv_static": [p] * 4, "sp_spmm": [p, p, n, n, p, n, p],
                       "sp_sddmm": [p, p, n, p, n, n, p, p], "sp_mttkrp": [p, p, p, n, p, p], "sp_mttkrp_mode": [p, i, p, n, p, p],
                       "sp_spmspm": [p, p, i, i, p, p], "sp_convert": [p, p, p, i, i, p, p], "sp_scale": [p, C.c_double, p],
                       "sp_vec_dot": [p] * 4}.items():
        getattr(lib, name).argtypes = args
    side = C.PyDLL(_TORCH_LIB_PATH)
    side.sp_torch_alloc.restype, side.sp_torch_alloc.argtypes = p, [C.c_size_t, p, p]
    side.sp_torch_free.restype, side.sp_torch_free.argtypes = None, [p, p, p]
    side.sp_torch_view.restype, side.sp_torch_view.argtypes = C.py_object, [p, n, i, C.py_object]
    return lib, side


_lib, _torch_lib = _load()

_ALLOC_T = C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
_FREE_T = C.CFUNCTYPE(None, C.c_void_p, C.c_void_p, C.c_void_p)
_torch_alloc, _torch_free = _torch_lib.sp_torch_alloc, _torch_lib.sp_torch_free
_alloc_cb, _free_cb = C.cast(_torch_alloc, C.c_void_p), C.cast(_torch_free, C.c_void_p)
_allocator_set = False


def use_torch_allocator():
    """Route the library's allocations through torch's caching allocator."""
    global _allocator_set
    if not _allocator_set:
        _check(_lib.sp_set_allocator(_alloc_cb, _free_cb, None), "sp_set_allocator")
        _allocator_set = True


def _check(code, where):
    if code != 0:
        raise SpError(code, where)


_current_device = torch._C._cuda_getDevice
_current_stream = torch._C._cuda_getCurrentRawStream


def _stream():
    return _current_stream(_current_device())


def _dptr(t):
    return t.data_ptr() if t is not None else 0        # 0 for an empty tensor too


def _f64(t, name):
    if t.dtype is not torch.float64 or not t.is_cuda:
        raise TypeError(f"{name} must be a CUDA float64 tensor")
    return t


def _view(ptr, n, code, owner):
    """Zero-copy tensor over library-owned device memory that keeps its owner alive."""
    v = _torch_lib.sp_torch_view(ptr, n, code, owner)
    return v if v.get_device() == _current_device() else v.to("cuda")


_WIDTH_DTYPE = {8: torch.uint8, 16: torch.uint16, 32: torch.int32, 64: torch.int64}


def _encoding(rank, dimLevelType, dimOrdering):
    """The level types and the level order as C arrays (no order = None) and as tuples."""
    lt = (C.c_int * rank)(*map(int, dimLevelType))
    if dimOrdering is None:
        return lt, None, tuple(lt), tuple(range(rank))
    od = (C.c_int * rank)(*map(int, dimOrdering))
    return lt, od, tuple(lt), tuple(od)


class SpTensor:
    """Owner of an sp_tensor handle."""

    def __init__(self, handle, known=None):
        """known: (dims, lt, ord, posBits, crdBits) where the caller has just stated them; asked for otherwise."""
        self._h = handle
        if known is None:
            rank = C.c_int()
            dims, lt, od = (C.c_int64 * MAX_RANK)(), (C.c_int * MAX_RANK)(), (C.c_int * MAX_RANK)()
            pb, cb = C.c_int(), C.c_int()
            _check(_lib.sp_info(handle, C.byref(rank), dims, lt, od, C.byref(pb), C.byref(cb)), "sp_info")
            r = rank.value
            known = tuple(dims[:r]), tuple(lt[:r]), tuple(od[:r]), pb.value, cb.value
        self.dims, self.lt, self.ord, self.pos_bits, self.crd_bits = known
        self.rank = len(self.dims)

    def _arr(self, fn, level, bits):
        p, n = C.c_void_p(), C.c_int64()
        _check(fn(self._h, level, C.byref(p), C.byref(n)), fn.__name__)
        if n.value == 0 or not p.value:
            return torch.empty(0, dtype=_WIDTH_DTYPE[bits], device="cuda")
        return _view(p.value, n.value, bits // 8, self)

    def positions(self, level):
        """pos[level] as a view of the device array (empty at dense levels): uint8 / uint16 for the
        narrow widths, a signed view of the unsigned words for 32 and 64 bits."""
        return self._arr(_lib.sp_positions, level, self.pos_bits)

    def coordinates(self, level):
        return self._arr(_lib.sp_coordinates, level, self.crd_bits)

    def values(self):
        p, n = C.c_void_p(), C.c_int64()
        _check(_lib.sp_values(self._h, C.byref(p), C.byref(n)), "sp_values")
        if n.value == 0:
            return torch.empty(0, dtype=torch.float64, device="cuda")
        return _view(p.value, n.value, 0, self)

    @property
    def nval(self):
        p, n = C.c_void_p(), C.c_int64()
        _check(_lib.sp_values(self._h, C.byref(p), C.byref(n)), "sp_values")
        return n.value

    def free(self):
        if self._h:
            _lib.sp_free(self._h)
            self._h = None

    def __del__(self):
        try:
            self.free()
        except Exception:
            pass


def sp_pack(dims, coords, vals, dimLevelType, dimOrdering=None, posBits=32, crdBits=32, flags=DUP_SUM) -> SpTensor:
    """coords: one CUDA int32/int64 tensor per logical dimension; vals: CUDA float64."""
    use_torch_allocator()
    rank = len(dims)
    nnz = int(vals.numel())
    _f64(vals, "vals")
    bits = 64
    if rank and len(coords):
        bits = 32 if coords[0].dtype == torch.int32 else 64
    for c in coords:
        if not c.is_cuda or c.dtype not in (torch.int32, torch.int64) or (32 if c.dtype == torch.int32 else 64) != bits:
            raise TypeError("coords must be CUDA tensors of one integer type (int32 or int64)")
        if c.numel() != nnz or not c.is_contiguous():
            raise ValueError("each coords tensor must be contiguous with nnz entries")
    h = C.c_void_p()
    c_lt, c_od, lt, od = _encoding(rank, dimLevelType, dimOrdering)
    c_dims = (C.c_int64 * rank)(*map(int, dims))
    cptrs = (C.c_void_p * max(rank, 1))(*[c.data_ptr() if nnz else 0 for c in coords])
    _check(_lib.sp_pack(rank, c_dims, nnz, cptrs, bits, vals.data_ptr(), c_lt, c_od, posBits, crdBits, flags, _stream(),
                        C.byref(h)), "sp_pack")
    return SpTensor(h, (tuple(c_dims), lt, od, posBits or 64, crdBits or 64))


def sp_unpack(t: SpTensor):
    n = t.nval
    outs = [torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(t.rank)]
    vals = torch.empty(n, dtype=torch.float64, device="cuda")
    cnt = C.c_int64()
    ptrs = (C.c_void_p * t.rank)(*[o.data_ptr() if n else 0 for o in outs])
    if n == 0:
        return outs, vals
    _check(_lib.sp_unpack(t._h, ptrs, _dptr(vals), C.byref(cnt), _stream()), "sp_unpack")
    return outs, vals


def sp_spmv(A: SpTensor, x, y=None):
    _f64(x, "x")
    if y is None:
        y = torch.empty(A.dims[0], dtype=torch.float64, device="cuda")
    _check(_lib.sp_spmv(A._h, _dptr(x), _dptr(y), _stream()), "sp_spmv")
    return y


def sp_spmv_static(A: SpTensor, x, y):
    """sp_spmv for callers that may not allocate: the library's scratch is a fixed device array.

    y must be supplied (this wrapper allocates nothing either).  Calls share that one array, so
    do not let two of them overlap on the GPU; see include/sp.h for the capacity and the rules."""
    _f64(x, "x"); _f64(y, "y")
    _check(_lib.sp_spmv_static(A._h, _dptr(x), _dptr(y), _stream()), "sp_spmv_static")
    return y


def sp_spmm(A: SpTensor, B, C_out=None):
    _f64(B, "B")
    N = B.shape[1]
    if C_out is None:
        C_out = torch.empty((A.dims[0], N), dtype=torch.float64, device="cuda")
    _check(_lib.sp_spmm(A._h, _dptr(B), N, B.stride(0), _dptr(C_out), C_out.stride(0),
                        _stream()), "sp_spmm")
    return C_out


def sp_sddmm(S: SpTensor, A, B, x_vals=None):
    _f64(A, "A"); _f64(B, "B")
    if x_vals is None:
        x_vals = torch.empty(S.nval, dtype=torch.float64, device="cuda")
    _check(_lib.sp_sddmm(S._h, _dptr(A), A.stride(0), _dptr(B), B.stride(0), A.shape[1], _dptr(x_vals), _stream()), "sp_sddmm")
    return x_vals


def sp_mttkrp(T: SpTensor, B, Cf, M=None):
    _f64(B, "B"); _f64(Cf, "C")
    if not (B.is_contiguous() and Cf.is_contiguous()):
        raise ValueError("factor matrices must be contiguous")
    R = B.shape[1]
    if M is None:
        M = torch.empty((T.dims[0], R), dtype=torch.float64, device="cuda")
    _check(_lib.sp_mttkrp(T._h, _dptr(B), _dptr(Cf), R, _dptr(M), _stream()), "sp_mttkrp")
    return M


def sp_launch_count() -> int:
    return int(_lib.sp_launch_count())


def sp_mttkrp_mode(T: SpTensor, mode: int, factors, M=None):
    """factors: three CUDA float64 matrices (factors[mode] may be None); T stores dimension `mode` at level 0."""
    use = [f for d, f in enumerate(factors) if d != mode]
    for f in use:
        _f64(f, "factor")
        if not f.is_contiguous():
            raise ValueError("factor matrices must be contiguous")
    R = use[0].shape[1]
    if M is None:
        M = torch.empty((T.dims[mode], R), dtype=torch.float64, device="cuda")
    ptrs = (C.c_void_p * 3)(*[f.data_ptr() if (f is not None and d != mode) else 0 for d, f in enumerate(factors)])
    _check(_lib.sp_mttkrp_mode(T._h, mode, ptrs, R, _dptr(M), _stream()), "sp_mttkrp_mode")
    return M


def sp_spmspm(A: SpTensor, B: SpTensor, posBits=32, crdBits=32) -> SpTensor:
    """C = A * B with A, B, C all CSR; returns a new handle."""
    use_torch_allocator()
    h = C.c_void_p()
    _check(_lib.sp_spmspm(A._h, B._h, posBits, crdBits, _stream(), C.byref(h)), "sp_spmspm")
    return SpTensor(h)


def sp_convert(t: SpTensor, dimLevelType, dimOrdering=None, posBits=32, crdBits=32) -> SpTensor:
    """Re-encode a tensor through coordinates (unpack + pack on the device)."""
    use_torch_allocator()
    h = C.c_void_p()
    c_lt, c_od, lt, od = _encoding(t.rank, dimLevelType, dimOrdering)
    _check(_lib.sp_convert(t._h, c_lt, c_od, posBits, crdBits, _stream(), C.byref(h)), "sp_convert")
    return SpTensor(h, (t.dims, lt, od, posBits or 64, crdBits or 64))


def sp_scale(x: SpTensor, c: float):
    _check(_lib.sp_scale(x._h, c, _stream()), "sp_scale")
    return x


def sp_vec_dot(a: SpTensor, b: SpTensor):
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    _check(_lib.sp_vec_dot(a._h, b._h, _dptr(out), _stream()), "sp_vec_dot")
    return out
