"""More handles at once than the process's page-locked block has units: those beyond it
use ordinary host memory, with the same results, timeouts and readbacks, and units
that were given back serve again."""
import numpy as np
import pytest

from helpers import CHEB
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_beyond_the_page_locked_block():
    pr = dg.regression(3, 64, 2, 1, 0.05, degree=2)
    pop = dg.random_population(1, 40, pr.K)
    make = lambda: game.Game(pr.X, pr.y, 2, CHEB, P=8, seed=4)
    run = (pr.X, pr.y, 2, CHEB, 600, 5)

    def all_of(g, b):
        p, f, _ = g.population()
        return [g.eval_fitness(pop), p, f, *b.run(0)[:2]]

    with make() as g, game.Batch([run], autotune=False) as b:
        want = all_of(g, b)
    handles = [make() for _ in range(4150)]
    try:
        late = game.Batch([run], autotune=False)
        with late as b:
            for g in (handles[0], handles[-1]):
                for x, y in zip(all_of(g, b), want):
                    assert np.array_equal(x, y)
        g = handles[-1]
        game.game_test_hook(game.GAME_HOOK_STALL_NS, 20_000_000)
        try:
            with pytest.raises(game.GameError) as ei:
                g.eval_fitness(pop, game.GAME_PREC_BF16)
        finally:
            game.game_test_hook(game.GAME_HOOK_STALL_NS, 0)
        assert ei.value.code == game.GAME_ETIMEOUT
        assert np.array_equal(g.eval_fitness(pop), want[0])
        for k in range(0, 4150, 2):
            handles[k].close()
        with make() as g, game.Batch([run], autotune=False) as b:
            for x, y in zip(all_of(g, b), want):
                assert np.array_equal(x, y)
    finally:
        for g in handles:
            g.close()
