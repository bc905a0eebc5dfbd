"""The tensor-core forms at degrees of 32 and beyond (a chunk of 8 columns may start at
any degree), one feature with the longest run included, single problems on one SM, SM
pairs and a batch, against the CPU model of each form (tests/emulation.py; the
tolerance is the model's own)."""
import numpy as np
import pytest

from emulation import model
from helpers import CHEB, TRIG, fp32_tol
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PREC = {"bf16": game.GAME_PREC_BF16, "bf16x3": game.GAME_PREC_BF16X3,
        "fp8": game.GAME_PREC_FP8}


def problem(N, d, basis, P):
    pr = dg.regression(N + d, 300, N, 4, 0.05, degree=d, basis=basis)
    return pr, dg.random_population(P, P, pr.K)


@pytest.mark.parametrize("N,d,P", [(4, 31, 5), (4, 32, 140), (3, 33, 5), (5, 40, 140), (2, 100, 20),
                                   (1, 257, 9), (1, 300, 130)])
@pytest.mark.parametrize("basis", [CHEB, TRIG])
@pytest.mark.parametrize("form", sorted(PREC))
def test_high_degrees(form, basis, N, d, P):
    pr, pop = problem(N, d, basis, P)
    want, tol = model(form, pr.X, pr.y, pop, d, basis)
    with game.Game(pr.X, pr.y, d, basis, P=max(P, 4), precision=PREC[form]) as g:
        got = g.eval_fitness(pop)
    assert np.all(np.abs(got - want) <= tol), np.max(np.abs(got - want) / tol)


@pytest.mark.parametrize("N,d", [(10, 37), (9, 40)])   # read staged and from L2
def test_high_degrees_on_pairs(N, d):
    pr, pop = problem(N, d, CHEB, 300)
    want, tol = model("bf16", pr.X, pr.y, pop, d, CHEB)
    with game.Game(pr.X, pr.y, d, CHEB, P=300, precision=game.GAME_PREC_BF16) as g:
        assert g.plan()["kernel"] == "fitness_tc2_kernel"
        got = g.eval_fitness(pop)
    assert np.all(np.abs(got - want) <= tol), np.max(np.abs(got - want) / tol)


def test_high_degrees_in_a_batch():
    runs, want = [], []
    for r, (N, d, basis) in enumerate([(3, 33, CHEB), (2, 40, TRIG), (1, 200, CHEB)]):
        pr, _ = problem(N, d, basis, 4)
        runs.append((pr.X, pr.y, d, basis, 40, 5 + r))
    with game.Batch(runs, autotune=False) as b:
        for r, (X, y, d, basis, _, _) in enumerate(runs):
            pop, fit, _ = b.run(r)
            want, tol = model("bf16", X, y, pop, d, basis)
            assert np.all(np.abs(fit - want) <= tol)


# runs of degrees that end in every place of a 16-column chunk, one feature, columns
# past the last feature
@pytest.mark.parametrize("d", [11, 12, 14, 15, 16, 17, 19, 24, 31, 33])
@pytest.mark.parametrize("basis", [CHEB, TRIG])
def test_plain_fp32(orc, basis, d):
    for N, P in ((1, 5), (3, 64), (5, 130), (7, 257)):
        pr, pop = problem(N, d, basis, P)
        ref = orc.fitness(pr.X, pr.y, pop, d, basis)
        with game.Game(pr.X, pr.y, d, basis, P=max(P, 4)) as g:
            got = g.eval_fitness(pop)
        assert np.all(np.abs(got - ref) <= fp32_tol(ref, pr.y))
