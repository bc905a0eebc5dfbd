"""A run's state into host memory goes through the batch's page-locked buffer: the
same values as into device memory, into either part alone, and with several
threads reading at once."""
import ctypes
import threading

import numpy as np
import pytest

from helpers import CHEB, TRIG
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_readback_into_host_and_device_memory():
    spec = [(500, 5, 4, CHEB, 33, 1), (900, 16, 10, TRIG, 257, 2), (1, 1, 1, CHEB, 4, 3)]
    runs = []
    for M, N, d, basis, P, seed in spec:
        pr = dg.regression(M + N, M, N, min(d, 4), 0.05, degree=d, basis=basis)
        runs.append((pr.X, pr.y, d, basis, P, seed))
    with game.Batch(runs, autotune=False) as b:
        b.generation()
        want = []
        for r, (_, _, K, P) in enumerate(b.shapes):
            pop = torch.empty(P, K, device="cuda")
            fit = torch.empty(P, dtype=torch.float64, device="cuda")
            p, f = ctypes.c_void_p(pop.data_ptr()), ctypes.c_void_p(fit.data_ptr())
            assert game.load().game_batch_get_run(b.h, r, p, f, None) == 0
            b.sync()
            want.append((pop.cpu().numpy(), fit.cpu().numpy()))
            only_fit = np.zeros(P)
            only_pop = np.zeros((P, K), dtype=np.float32)
            ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
            assert game.load().game_batch_get_run(b.h, r, None, ptr(only_fit), None) == 0
            assert game.load().game_batch_get_run(b.h, r, ptr(only_pop), None, None) == 0
            assert np.array_equal(only_pop, want[r][0]) and np.array_equal(only_fit, want[r][1])
        wrong = []

        def read(first):
            for k in range(30):
                r = (first + k) % b.R
                pop, fit, gen = b.run(r)
                if gen != 1 or not (np.array_equal(pop, want[r][0])
                                    and np.array_equal(fit, want[r][1])):
                    wrong.append(r)

        threads = [threading.Thread(target=read, args=(t,)) for t in range(4)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert not wrong
