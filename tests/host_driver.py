"""Runs in a process with the fake CUDA runtime preloaded: the library's entry points
over host memory, and the fake's controls."""
import ctypes
import os

import numpy as np

from paper_1601_05725_gb300 import basker

OK, OOM, TIMEOUT, NOT_FACTORED = 0, 6, 7, 9
#: 32-bit words of the kernels' status: room ran out, a wait gave up, rejected pivots, moved pivots
CAPACITY, GAVE_UP, REJECTED, MOVED = 2, 3, 4, 8

fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
fake.fake_held.restype = ctypes.c_int64
fake.fake_cap.argtypes = [ctypes.c_int64]
fake.fake_ints.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int]
fake.fake_launched.restype = ctypes.c_char_p


def launched():
    return fake.fake_launched().decode()


class Host:
    def __init__(self, p, **options):
        self.L = basker.load()
        o = basker.default_options()
        for k, v in options.items():
            setattr(o, k, v)
        nd = p.nd_node_ptr if p.nd_block >= 0 else np.zeros(1, np.int32)
        arrs = [basker._i32(a) for a in (p.colptr, p.rowind, p.P, p.Q, p.block_ptr, nd)]
        self.p, self.h = p, ctypes.c_void_p()
        self.status = self.L.basker_symbolic(p.n, *[basker._np_ptr(a) for a in arrs[:4]], len(arrs[4]) - 1,
                                             basker._np_ptr(arrs[4]), p.nd_block, p.nd_leaves, basker._np_ptr(arrs[5]),
                                             ctypes.byref(o), ctypes.byref(self.h))
        self.x = np.zeros(p.n)

    def factor(self):
        return self.L.basker_factor(self.h, basker._np_ptr(self.p.values), None)

    def refactor(self):
        return self.L.basker_refactor(self.h, basker._np_ptr(self.p.values), None)

    def solve(self):
        b = np.ones(self.p.n)
        return self.L.basker_solve(self.h, 1, basker._np_ptr(b), self.p.n, basker._np_ptr(self.x), self.p.n, None)

    def free(self):
        self.L.basker_free(self.h)
