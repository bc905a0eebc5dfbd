"""The BF16 kernels with features read from global memory (Chebyshev runs of 8
degrees), whose two expansion warpgroups take the K-blocks in turn, and the
epilogue that finishes each accumulator's sum during the next one: several tiles
per CTA, odd and single K-block counts, one and several chromosome tiles, a ragged
last tile, against the CPU model of the form (tests/emulation.py; the tolerance
is the model's own)."""
import numpy as np
import pytest

from emulation import model
from helpers import CHEB
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,d,P", [
    (90_001, 3, 8, 5),       # one K-block, one chromosome tile
    (90_001, 17, 8, 130),    # three, two tiles
    (120_031, 5, 16, 20),    # two, degree 16: two chunks per feature
    (50_000, 40, 8, 140),    # five: SM pairs
    (50_000, 47, 8, 20),     # six: 128-pattern tiles
])
def test_features_from_l2(M, N, d, P):
    pr = dg.regression(M + N + d, M, N, 4, 0.05, degree=d, basis=CHEB)
    pop = dg.random_population(11 + P, P, pr.K)
    want, tol = model("bf16", pr.X, pr.y, pop, d, CHEB)
    with game.Game(pr.X, pr.y, d, CHEB, P=P, precision=game.GAME_PREC_BF16) as g:
        assert not g.plan()["staged"]
        got = g.eval_fitness(pop)
    assert np.all(np.abs(got - want) <= tol), np.max(np.abs(got - want) / tol)
