"""The elites of a generation on both sides of the rule that finds them by counting
or by one arg-min each (P^2 against 8000 per elite, at most 512 chromosomes), with
ties and NaN at the ranks in question: the whole generation bit for bit the oracle's,
as one run and as a run of a batch."""
import numpy as np
import pytest

from helpers import CHEB
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(20, 0), (89, 1), (90, 1), (126, 2), (127, 2), (252, 8), (253, 8), (512, 32), (512, 33),
         (512, 256), (513, 33), (600, 256)]


@pytest.mark.parametrize("selection", [game.GAME_SEL_TOURNAMENT, game.GAME_SEL_ROULETTE])
@pytest.mark.parametrize("P,E", SIZES)
def test_elites(orc, P, E, selection):
    pr = dg.regression(2, 100, 2, 1, 0.05, degree=1, basis=CHEB)
    rng = np.random.default_rng(P + E)
    pop = dg.random_population(P, P, pr.K)
    fit = rng.integers(0, max(2, P // 3), P).astype(np.float64)
    fit[rng.integers(0, P, 2)] = np.nan
    fit[rng.integers(0, P, 2)] = -0.0
    prm = orc.ga_params(elitism=E, selection=selection)
    with game.Game(pr.X, pr.y, 1, CHEB, P=P, elitism=E, selection=selection) as g:
        g.set_state(pop, fit, 3)
        g.generation(11)
        nxt, _, _ = g.population()
    want = orc.generation(pop, fit, 11, 3, prm)
    assert np.array_equal(nxt.view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("E", [0, 2, 40])
def test_elites_of_a_batch(orc, E):
    runs = []
    for r, P in enumerate((64, 126, 127, 512, 513)):
        pr = dg.regression(r, 200 + r, 2, 1, 0.05, degree=2, basis=CHEB)
        runs.append((pr.X, pr.y, 2, CHEB, P, 9 + r))
    prm = orc.ga_params(elitism=E)
    with game.Batch(runs, autotune=False, elitism=E) as b:
        states = [b.run(r)[:2] for r in range(b.R)]
        b.generation()
        for r, (pop, fit) in enumerate(states):
            want = orc.generation(pop, fit, 9 + r, 0, prm)
            assert np.array_equal(b.run(r)[0].view(np.uint32), want.view(np.uint32))
