"""Device memory held back in a test, so that a call has only so much left."""
import contextlib

import torch


@contextlib.contextmanager
def free_bytes(keep: int):
    """Takes all of the device's free memory but about `keep` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    for piece in (1 << 36, 1 << 33, 1 << 30, 1 << 27, 1 << 24):
        while torch.cuda.mem_get_info()[0] - keep >= piece:
            held.append(torch.cuda.caching_allocator_alloc(piece))
    try:
        yield
    finally:
        torch.cuda.synchronize()
        for p in held:
            torch.cuda.caching_allocator_delete(p)
        torch.cuda.empty_cache()
