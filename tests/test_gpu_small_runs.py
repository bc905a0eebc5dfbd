"""The Gram form's quadratic forms at the edges of their splits, and small runs
whose generations run in one launch against the same generations by the
separate kernels (stage timing selects those)."""
import numpy as np
import pytest

from helpers import CHEB, TRIG, quad_bound
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# K = 2 ... 64 take the pair list, 65 and more the row blocks (32 rows each)
@pytest.mark.parametrize("N,d", [(1, 1), (8, 4), (9, 7), (64, 1), (12, 8), (32, 8), (61, 10)])
@pytest.mark.parametrize("P", [4, 16, 131, 700])
def test_quadratic_forms(N, d, P):
    pr = dg.regression(N + d, 700, N, min(d, 4), 0.05, degree=d, basis=CHEB)
    pop = dg.random_population(P, P, pr.K)
    with game.Game(pr.X, pr.y, d, CHEB, P=P, precision=game.GAME_PREC_GRAM) as g:
        G, b, yy = g.gram()
        got = g.eval_fitness(pop)
    A = pop.astype(np.float64)
    want = (yy - 2 * A @ b + np.einsum("pk,kl,pl->p", A, G, A)) / 700
    assert np.all(np.abs(got - np.maximum(want, 0)) <= quad_bound(G, b, yy, pop, 700))


def run_both(gens, setup, **prm):
    pr = dg.small_classification(M=300)
    out = []
    for separate in (False, True):
        with game.Game(pr.X, pr.y, setup["d"], setup["basis"], precision=game.GAME_PREC_GRAM,
                       seed=11, **prm) as g:
            g.set_timing(separate)
            ran = g.train(gens)
            g.generation(5)
            out.append((ran,) + g.population())
    return out


@pytest.mark.parametrize("selection", [game.GAME_SEL_TOURNAMENT, game.GAME_SEL_RANKING,
                                       game.GAME_SEL_ROULETTE])
@pytest.mark.parametrize("P,d,tied,error", [(19, 8, 1, game.GAME_ERR_MSE),
                                            (64, 3, 0, game.GAME_ERR_RMSE),
                                            (300, 1, 1, game.GAME_ERR_MSE)])
def test_whole_generations(selection, P, d, tied, error):
    a, b = run_both(23, dict(d=d, basis=TRIG), P=P, tied=tied, selection=selection, pm=0.2,
                    error=error, immigrants=3, elitism=3)
    assert a[0] == b[0] == 23 and a[3] == b[3]
    assert np.array_equal(a[1].view(np.uint32), b[1].view(np.uint32))
    assert np.array_equal(a[2].view(np.uint64), b[2].view(np.uint64))


def test_stop_rule_on_the_device():
    a, b = run_both(400, dict(d=2, basis=CHEB), P=40, mse_threshold=0.75, check_every=7)
    assert a[0] == b[0] and 0 < a[0] < 400 and a[0] % 7 == 0
    assert np.array_equal(a[1].view(np.uint32), b[1].view(np.uint32))


@pytest.mark.parametrize("P", [16, 33, 2048, 2049, 16384, 16385])
def test_candidate_selection(P):
    """The candidates' order (fitness, index, NaN last) at the edges of the
    selection's key chunks and on both of its kernels."""
    pr = dg.regression(3, 50, 1, 1, 0.05, degree=1, basis=CHEB)
    pop = dg.random_population(P, P, pr.K)
    rng = np.random.default_rng(P)
    fit = rng.integers(0, max(4, P // 8), P).astype(np.float64)   # many ties
    fit[rng.integers(0, P, 3)] = np.nan
    fit[rng.integers(0, P, 2)] = -0.0
    order = np.lexsort((np.arange(P), np.where(np.isnan(fit), np.inf, fit)))
    with game.Game(pr.X, pr.y, 1, CHEB, P=P, precision=game.GAME_PREC_BF16) as g:
        for n in (1, 16):
            _, idx = g.rescore_top(pop, fit, n)
            assert np.array_equal(idx, order[:n])


@pytest.mark.parametrize("P,oversample", [(18, 8), (130, 3), (1026, 8), (2048, 8)])
def test_screening_keeps_the_best_predictions(P, oversample):
    """Once trusted, the screening keeps the smallest predictions, ties by slot,
    at child counts off and on the selection's warp ranges."""
    pr = dg.regression(9, 3000, 6, 2, 0.05, degree=2, basis=CHEB)
    with game.Game(pr.X, pr.y, 2, CHEB, P=P, precision=game.GAME_PREC_BF16, surrogate=1,
                   oversample=oversample, seed=4) as g:
        seen = 0
        for _ in range(12):
            g.generation(4)
            pred, keep, trusted, _ = g.surrogate_last()
            want = np.zeros(len(pred), dtype=np.int32)
            n_keep = P - 2
            want[np.argsort(pred, kind="stable")[:n_keep] if trusted else slice(0, n_keep)] = 1
            assert np.array_equal(keep, want)
            seen += trusted
        assert seen, "the surrogate was never trusted"
