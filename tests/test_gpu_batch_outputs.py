"""A run's state into every kind of memory: warm, fresh and page-locked host memory,
each part alone, one part on the device and one on the host, a population whose
fitness is larger than the batch's page-locked buffer, guard bytes on both sides;
and threads that read and wait on one batch at once."""
import ctypes
import mmap
import threading

import numpy as np
import pytest

from helpers import CHEB
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def batch():
    runs = []
    for r, (M, N, d, P) in enumerate([(300, 4, 2, 33), (700, 16, 8, 512), (200, 2, 1, 9001),
                                      (100, 1, 1, 4)]):
        pr = dg.regression(r, M, N, 2, 0.05, degree=d, basis=CHEB)
        runs.append((pr.X, pr.y, d, CHEB, P, r))
    return game.Batch(runs, autotune=False)


def get(b, r, pop, fit):
    ptr = lambda a: None if a is None else ctypes.c_void_p(
        a.data_ptr() if torch.is_tensor(a) else a.ctypes.data)
    assert game.load().game_batch_get_run(b.h, r, ptr(pop), ptr(fit), None) == 0
    b.sync()
    return [None if a is None else (a.cpu().numpy() if torch.is_tensor(a) else a)
            for a in (pop, fit)]


def fresh(shape, dtype):
    n = int(np.prod(shape)) * np.dtype(dtype).itemsize
    return np.frombuffer(mmap.mmap(-1, n), dtype, count=int(np.prod(shape))).reshape(shape)


def guarded(shape, dtype):
    n = int(np.prod(shape))
    whole = np.full(n + 64, 7, dtype=dtype)
    return whole, whole[32:32 + n].reshape(shape)


MAKE = {
    "warm": lambda s, d: np.ones(s, dtype=d),
    "fresh": fresh,
    "pinned": lambda s, d: torch.empty(s, dtype=getattr(torch, np.dtype(d).name), pin_memory=True),
    "device": lambda s, d: torch.empty(s, dtype=getattr(torch, np.dtype(d).name), device="cuda"),
    "none": lambda s, d: None,
}


@pytest.mark.parametrize("genes", sorted(MAKE))
@pytest.mark.parametrize("fitness", sorted(MAKE))
def test_every_kind_of_memory(genes, fitness):
    with batch() as b:
        b.generation()
        for r, (_, _, K, P) in enumerate(b.shapes):
            want = get(b, r, MAKE["device"]((P, K), np.float32), MAKE["device"](P, np.float64))
            got = get(b, r, MAKE[genes]((P, K), np.float32), MAKE[fitness](P, np.float64))
            for g, w in zip(got, want):
                assert g is None or np.array_equal(g, w)
            (gw, gp), (fw, fp) = guarded((P, K), np.float32), guarded(P, np.float64)
            get(b, r, gp, fp)
            assert np.array_equal(gp, want[0]) and np.array_equal(fp, want[1])
            for w in (gw, fw):
                assert np.all(w[:32] == 7) and np.all(w[-32:] == 7)


def test_threads_read_and_wait():
    with batch() as b:
        b.generation()
        want = [b.run(r)[:2] for r in range(b.R)]
        wrong = []

        def work(t):
            try:
                for k in range(40):
                    r = (t + k) % b.R
                    if t % 2:
                        b.sync()
                    pop, fit, _ = b.run(r)
                    if not (np.array_equal(pop, want[r][0]) and np.array_equal(fit, want[r][1])):
                        wrong.append(r)
            except Exception as e:   # noqa: BLE001
                wrong.append(e)

        threads = [threading.Thread(target=work, args=(t,)) for t in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert not wrong
