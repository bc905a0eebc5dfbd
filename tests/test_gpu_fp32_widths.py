"""The plain FP32 form at each CTA width its plan picks (64, 128 and 256
chromosomes) and at the edges of its tiles, against the FP64 oracle within the
form's stated tolerance; every degree of both bases (1 to 10 stream whole
features, beyond them column runs)."""
import numpy as np
import pytest

import oracle
from helpers import CHEB, TRIG, fp32_tol
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

def check(M, N, d, basis, P):
    pr = dg.regression(M + N + d, M, N, min(d, 4), 0.05, degree=d, basis=basis)
    pop = dg.random_population(5 + P, P, pr.K)
    ref = oracle.fitness(pr.X, pr.y, pop, d, basis)
    with game.Game(pr.X, pr.y, d, basis, P=max(P, 4)) as g:
        got = g.eval_fitness(pop)
    assert np.all(np.abs(got - ref) <= fp32_tol(ref, pr.y)), np.max(np.abs(got - ref) / ref)


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 13])
@pytest.mark.parametrize("basis", [CHEB, TRIG])
def test_degrees(basis, d):
    check(260, 11, d, basis, 70)
    check(129, 1, d, basis, 1)


@pytest.mark.parametrize("M", [1, 127, 128, 20001])
@pytest.mark.parametrize("P", [1, 64, 65, 128, 129, 257, 513])
def test_widths(M, P):
    check(M, 5, 4, CHEB, P)


def test_many_tiles_per_cta():
    check(60_011, 8, 8, CHEB, 256)   # 256 chromosomes per CTA, several tiles each


def test_absolute_error():
    pr = dg.regression(3, 1001, 7, 4, 0.05, degree=5, basis=TRIG)
    pop = dg.random_population(6, 130, pr.K)
    ref = oracle.fitness(pr.X, pr.y, pop, 5, TRIG, oracle.ERR_MAE)
    with game.Game(pr.X, pr.y, 5, TRIG, P=130, error=game.GAME_ERR_MAE, rescore_top=0) as g:
        got = g.eval_fitness(pop)
    assert np.all(np.abs(got - ref) <= fp32_tol(ref, pr.y))
