"""A device memory pool of limited size in place of the device's default one (CUDA's stream-ordered
allocator): what the library holds at most, and what it does when there is no more."""
import ctypes as C

import torch


class _Location(C.Structure):
    _fields_ = [("type", C.c_int), ("id", C.c_int)]


class _Props(C.Structure):
    _fields_ = [("allocType", C.c_int), ("handleTypes", C.c_int), ("location", _Location),
                ("win32SecurityAttributes", C.c_void_p), ("maxSize", C.c_size_t),
                ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]


PINNED, DEVICE, USED_HIGH = 1, 1, 8  # cudaMemAllocationTypePinned, cudaMemLocationTypeDevice, ...


def _cudart():
    """The runtime that the library is linked with (loaded already)."""
    for line in open("/proc/self/maps"):
        path = line.split()[-1]
        if "libcudart.so" in path:
            return C.CDLL(path)
    raise RuntimeError("no CUDA runtime is loaded")


class MemPool:
    """`with MemPool(limit) as pool`: allocations of device 0 come from a pool of at most `limit` bytes
    (0: no limit).  Everything allocated inside has to be freed inside."""

    def __init__(self, limit=0):
        self.limit = int(limit)

    def _do(self, what, *args):
        rc = getattr(self.rt, what)(*args)
        assert rc == 0, (what, rc)

    def __enter__(self):
        torch.cuda.init()
        torch.cuda.synchronize()
        self.rt = _cudart()
        self.old, self.pool = C.c_void_p(), C.c_void_p()
        self._do("cudaDeviceGetMemPool", C.byref(self.old), 0)
        props = _Props(allocType=PINNED, location=_Location(DEVICE, 0), maxSize=self.limit)
        self._do("cudaMemPoolCreate", C.byref(self.pool), C.byref(props))
        self._do("cudaDeviceSetMemPool", 0, self.pool)
        return self

    def high(self):
        """Most bytes in use at one time so far."""
        torch.cuda.synchronize()
        v = C.c_uint64()
        self._do("cudaMemPoolGetAttribute", self.pool, USED_HIGH, C.byref(v))
        return v.value

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        self._do("cudaDeviceSetMemPool", 0, self.old)
        self._do("cudaMemPoolDestroy", self.pool)
        return False
