"""A context whose device memory comes from an allocator that the test can look
into: every live allocation by address, refusals of chosen requests, a budget,
and addresses that are aligned to 8 bytes only."""
import ctypes
from contextlib import contextmanager

import torch


class Recorder:
    def __init__(self, grx, refuse=(), budget=None, skew=0):
        self.live = {}                   # address -> (tensor, bytes asked for)
        self.asked = 0                   # requests so far
        self.refuse = set(refuse)        # requests (by number) that get NULL
        self.budget = budget             # bytes that may be live at once
        self.refused = 0
        self.skew = skew
        self.device = torch.cuda.current_device()

        def alloc(nbytes, stream, user):
            k, self.asked = self.asked, self.asked + 1
            if k in self.refuse or (self.budget is not None and self.used() + nbytes > self.budget):
                self.refused += 1
                return None
            t = torch.zeros(int(nbytes) + 16, dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr() + self.skew] = (t, int(nbytes))
            return t.data_ptr() + self.skew

        def free(ptr, nbytes, stream, user):
            t, n = self.live.pop(ptr)
            assert n == nbytes

        self._fns = grx._ALLOC_FN(alloc), grx._FREE_FN(free)
        self._allocator = grx.grx_allocator(*self._fns, None)
        self.handle = ctypes.c_void_p()
        assert grx.lib().grx_ctx_create(ctypes.byref(self._allocator), ctypes.byref(self.handle)) == grx.GRX_OK

    def used(self):
        return sum(n for _, n in self.live.values())

    def words(self, ptr, count):
        """The first `count` 32-bit words of the allocation at ptr."""
        t, _ = self.live[ptr]
        return t[self.skew:self.skew + 4 * count].clone().view(torch.int32)


@contextmanager
def recorded(grx, **kw):
    """Graphs loaded inside take their memory from the Recorder."""
    r = Recorder(grx, **kw)
    ctx, grx._ctx = grx._ctx, lambda device=None: r
    try:
        yield r
    finally:
        grx._ctx = ctx
