"""The streaming expansion of the tensor-core forms (degrees 1 to 10, whole
features at a time) against the CPU model of each form (tests/emulation.py):
every degree of both bases, feature counts that leave a partly filled last
group, a single feature, and shapes that reach the narrower pattern tiles, where
several threads share a row. The tolerance is the model's own (operand roundings
and FP32 summation order)."""
import numpy as np
import pytest

from emulation import model
from helpers import CHEB, TRIG
from paper_1211_5481_gb300 import datagen as dg
from paper_1211_5481_gb300 import game

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PREC = {"bf16": game.GAME_PREC_BF16, "bf16x3": game.GAME_PREC_BF16X3,
        "fp8": game.GAME_PREC_FP8}


def check(form, M, N, d, basis, P):
    pr = dg.regression(M + N + d, M, N, min(d, 4), 0.05, degree=d, basis=basis)
    pop = dg.random_population(11 + P, P, pr.K)
    want, tol = model(form, pr.X, pr.y, pop, d, basis)
    with game.Game(pr.X, pr.y, d, basis, P=max(P, 4), precision=PREC[form]) as g:
        got = g.eval_fitness(pop)
    assert np.all(np.abs(got - want) <= tol), np.max(np.abs(got - want) / tol)


@pytest.mark.parametrize("d", range(1, 11))
@pytest.mark.parametrize("basis", [CHEB, TRIG])
@pytest.mark.parametrize("form", ["bf16", "bf16x3", "fp8"])
def test_every_degree(form, basis, d):
    check(form, 300, 17, d, basis, 70)   # 17 features: a partly filled last group
    check(form, 257, 1, d, basis, 5)     # one feature, one pattern past a tile


@pytest.mark.parametrize("form,M,N,d,basis,P", [
    ("bf16", 400, 39, 6, CHEB, 90),      # 192-pattern tiles: three rows per thread
    ("bf16", 400, 31, 8, CHEB, 90),      # the same, degree 8 staged
    ("bf16", 400, 39, 5, TRIG, 90),      # 128-pattern tiles: two threads per row
    ("bf16", 400, 61, 5, TRIG, 90),      # 64: four threads per row
    ("bf16", 400, 66, 10, TRIG, 90),     # 32
    ("bf16", 700, 39, 6, TRIG, 300),     # SM pairs
    ("bf16x3", 400, 61, 9, TRIG, 40),    # 32
    ("fp8", 400, 61, 7, TRIG, 140),      # 128
    ("fp8", 400, 61, 10, TRIG, 40),      # 64
])
def test_tile_widths(form, M, N, d, basis, P):
    check(form, M, N, d, basis, P)
