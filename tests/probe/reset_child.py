"""Child process of test_native_calls: the forward through the C library alone (no torch), before and after a cudaDeviceReset,
which takes every kernel's attributes with it.  Prints the calls' statuses."""
import ctypes
import os

LIB = os.path.join(os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__)))), "paper_2605_05838_b200", "libmdn.so")


class Params(ctypes.Structure):   # mdn_params of include/mdn.h
    _fields_ = [(n, ctypes.c_int32) for n in ("B", "T", "H", "dk", "dv", "chunk", "num_seqs", "io_dtype", "o_dtype", "path")] + \
               [("scale", ctypes.c_float), ("segments", ctypes.c_int32)]


def forward(rt, mdn, io_dtype):
    p = Params(1, 70, 2, 128, 128, 64, 0, io_dtype, io_dtype, 0, 0.1, 0)
    mdn.mdn_chunk_fwd_workspace_bytes.restype = ctypes.c_size_t
    need = ctypes.c_size_t(mdn.mdn_chunk_fwd_workspace_bytes(ctypes.byref(p)))

    def buf(n):
        d = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(d), n) == 0 and rt.cudaMemset(d, 0, n) == 0
        return d
    q, k, v, g, o, S, M = (buf(ctypes.c_size_t(1 << 20)) for _ in range(7))
    st = mdn.mdn_chunk_fwd(ctypes.byref(p), q, k, v, g, g, g, g, None, None, None, o, S, M, buf(need), need, None)
    assert rt.cudaDeviceSynchronize() == 0
    return st


if __name__ == "__main__":
    mdn, rt = ctypes.CDLL(LIB), ctypes.CDLL("libcudart.so.12")
    res = []
    for _ in range(2):
        res += [forward(rt, mdn, io_dtype) for io_dtype in (0, 1)]
        assert rt.cudaDeviceReset() == 0
    print(res)
