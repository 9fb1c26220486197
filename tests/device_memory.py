"""Device memory taken away for a test, by allocations that are given back."""
import contextlib
import ctypes
import glob


def _cudart():
    for name in ("libcudart.so.13", "libcudart.so", *sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*"))):
        try:
            return ctypes.CDLL(name)
        except OSError:
            continue
    raise RuntimeError("no CUDA runtime library")


@contextlib.contextmanager
def all_but(leave):
    """Leaves between leave and leave + 2 MB of the device's memory free."""
    rt = _cudart()
    held, free, total = [], ctypes.c_size_t(), ctypes.c_size_t()
    try:
        for block in (1 << 38, 1 << 36, 1 << 34, 1 << 32, 1 << 30, 1 << 28, 1 << 26, 1 << 24, 1 << 22, 1 << 21):
            while True:
                assert rt.cudaMemGetInfo(ctypes.byref(free), ctypes.byref(total)) == 0
                if free.value < leave + block:
                    break
                p = ctypes.c_void_p()
                if rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(block)) != 0:
                    rt.cudaGetLastError()
                    break
                held.append(p)
        yield free.value
    finally:
        for p in held:
            rt.cudaFree(p)
