"""Device memory taken away for a test, through the driver's own allocator (no caching in between)."""
import contextlib
import ctypes

MB = 1 << 20


@contextlib.contextmanager
def only(leave: int):
    """Inside the block `leave` bytes of device memory can be allocated: the rest is held."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    cu = ctypes.CDLL("libcuda.so.1")
    held = []

    def take(size):
        p = ctypes.c_uint64()
        if cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(size)) != 0:
            return False
        held.append(p)
        return True

    try:
        assert take(leave)
        size = torch.cuda.mem_get_info()[0]
        while size >= 2 * MB:
            if not take(size):
                size //= 2
        cu.cuMemFree_v2(held.pop(0))
        yield
    finally:
        torch.cuda.synchronize()
        for p in held:
            cu.cuMemFree_v2(p)
