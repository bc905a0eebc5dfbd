"""Training of small Gram-form runs, whose generations run up to 1000 to a launch, over
the ends of those launches: against the same training by the separate kernels (stage
timing selects those), bit for bit in genes, fitness and generations run."""
import numpy as np
import pytest

from helpers import CHEB
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def handle(separate, P=24, **prm):
    pr = dg.regression(5, 400, 4, 4, 0.05, degree=3, basis=CHEB)
    g = game.Game(pr.X, pr.y, 3, CHEB, P=P, precision=game.GAME_PREC_GRAM, seed=11, sigma=0.02,
                  **prm)
    g.set_timing(separate)
    return g


def train(separate, steps, **prm):
    """What each train call returns, and the state after it and one generation more."""
    out = []
    with handle(separate, **prm) as g:
        for n in steps:
            out.append(g.train(n))
            pop, fit, gen = g.population()
            out += [pop.view(np.uint32), fit.view(np.uint64), gen]
        g.generation(3)
        pop, fit, gen = g.population()
        out += [pop.view(np.uint32), fit.view(np.uint64), gen]
    return out


def same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def best_after(gens):
    out = {}
    with handle(True) as g:
        for n in sorted(gens):
            g.train(n - g.population()[2])
            out[n] = g.population()[1].min()
    return out


@pytest.mark.parametrize("P", [96, 97])   # the largest population of the path, the next
def test_at_the_population_limit(P):
    same(train(False, [40, 1], P=P), train(True, [40, 1], P=P))


@pytest.mark.parametrize("prm", [{}, dict(mse_threshold=1e-9, check_every=7)])
def test_over_several_launches(prm):
    a = train(False, [999, 2, 2300], **prm)
    assert a[0] == 999 and a[4] == 2 and a[8] == 2300 and a[-1] == 3302
    same(a, train(True, [999, 2, 2300], **prm))


def test_stop_where_a_launch_ends():
    best = best_after([1000])[1000]
    prm = dict(mse_threshold=best * (1 + 1e-12), check_every=1000)
    a = train(False, [2500, 30], **prm)
    assert a[0] == 1000 and a[4] == 0      # the second launch and the second call run none
    same(a, train(True, [2500, 30], **prm))


def test_stop_phase_carried_over_a_launch():
    best = best_after([900, 1200])
    assert best[1200] < best[900]
    prm = dict(mse_threshold=best[1200] * (1 + 1e-12), check_every=300)
    a = train(False, [2500], **prm)
    assert a[0] == 1200
    same(a, train(True, [2500], **prm))


def test_threshold_already_met():
    prm = dict(mse_threshold=1e9, check_every=5)
    a = train(False, [50], **prm)
    assert a[0] == 0 and a[3] == 0
    same(a, train(True, [50], **prm))
