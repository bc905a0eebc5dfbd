"""The Gram form where its kernels change: the re-scoring on both sides of the sizes
and candidate counts that spread it over the GPU, and evaluations up to the longest
contraction, against the quadratic form of the handle's own G, b and y.y in numpy,
within tests/helpers.quad_bound's rounding bound."""
import numpy as np
import pytest

from helpers import CHEB, U64
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
M = 300


def quad(G, b, yy, pop):
    """The fitness and quad_bound's bound (its triple sum as products of matrices)."""
    A = pop.astype(np.float64)
    B = np.abs(A)
    want = np.maximum((yy - 2 * A @ b + ((A @ G) * A).sum(1)) / M, 0)
    mag = yy + 2 * B @ np.abs(b) + ((B @ np.abs(G)) * B).sum(1)
    return want, 4 * (A.shape[1] + 8) * U64 * mag / M


def problem(N, d):
    return dg.regression(N + d, M, N, min(d, 4), 0.05, degree=d, basis=CHEB)


# K = 49 and 64 (pair list, spread up to 8 candidates), 48 and 65 beside them; 1899
# and 1901, 3897 and 3901 on both sides of the long rules; the longest
@pytest.mark.parametrize("N,d", [(47, 1), (12, 4), (63, 1), (8, 8), (146, 13), (100, 19),
                                 (487, 8), (130, 30), (128, 32)])
@pytest.mark.parametrize("n", [1, 8, 9, 16])
def test_rescoring(N, d, n):
    pr = problem(N, d)
    pop = dg.random_population(7, 20, pr.K)
    fit = np.random.default_rng(N + n).random(20)
    with game.Game(pr.X, pr.y, d, CHEB, P=4, error=game.GAME_ERR_MSE) as g:
        G, b, yy = g.gram()
        got, idx = g.rescore_top(pop, fit, n)
    assert np.array_equal(idx, np.argsort(fit, kind="stable")[:n])
    rest = np.setdiff1d(np.arange(20), idx)
    assert np.array_equal(got[rest], fit[rest])
    want, bound = quad(G, b, yy, pop[idx])
    assert np.all(np.abs(got[idx] - want) <= bound)


def test_rescoring_the_root():
    pr = problem(128, 10)
    pop = dg.random_population(7, 20, pr.K)
    fit = np.random.default_rng(1).random(20)
    with game.Game(pr.X, pr.y, 10, CHEB, P=4, error=game.GAME_ERR_RMSE) as g:
        G, b, yy = g.gram()
        got, idx = g.rescore_top(pop, fit, 16)
    want, bound = quad(G, b, yy, pop[idx])
    assert np.all(np.abs(got[idx] ** 2 - want) <= 1.01 * bound)


@pytest.mark.parametrize("N,d", [(100, 10), (100, 20), (128, 32)])
@pytest.mark.parametrize("P", [1, 5, 304])
def test_long_forms(N, d, P):
    pr = problem(N, d)
    pop = dg.random_population(P, P, pr.K)
    with game.Game(pr.X, pr.y, d, CHEB, P=8, precision=game.GAME_PREC_GRAM) as g:
        G, b, yy = g.gram()
        got = g.eval_fitness(pop)
    want, bound = quad(G, b, yy, pop)
    assert np.all(np.abs(got - want) <= bound)


# 4 chromosomes share the entries of G from 153 on, one each below
@pytest.mark.parametrize("N,d", [(8, 8), (13, 5), (32, 8), (61, 10)])
def test_a_value_does_not_depend_on_its_population(N, d):
    pr = problem(N, d)
    pop = dg.random_population(3, 700, pr.K)
    with game.Game(pr.X, pr.y, d, CHEB, P=8, precision=game.GAME_PREC_GRAM) as g:
        whole = g.eval_fitness(pop)
        for lo, hi in ((0, 1), (5, 12), (100, 700), (301, 605), (699, 700)):
            part = g.eval_fitness(pop[lo:hi])
            assert np.array_equal(part, whole[lo:hi])
