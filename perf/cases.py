"""Performance cases of the GAME library: the calls a user of it makes, over the
sizes they are made at.

A case is a dict of plain values. Its "op" says which call one pass is:

  eval        Game.eval_fitness of a caller's population on a handle of the
              case's precision form; "host": the population and the fitness are
              numpy arrays (the binding's default), else CUDA tensors.
  train       Game.train for "gens" generations, then Game.population.
  generation  Game.generation, then the population and fitness into CUDA tensors.
  surrogate   the same on a handle that screens oversampled offspring; the MLP's
              parameters, which every generation trains, come back too.
  batch       "gens" Batch.generation of "R" uneven runs, then every run's state.
  predict     Game.predict of one chromosome on new patterns (row-major CUDA tensor).

Sizes: M patterns, N features, basis degree d (K = B N d + 1 genes, B = 2 for the
trigonometric basis), P chromosomes.
"""
import math

import numpy as np
import torch

from paper_1211_5481_gb300 import game

CHEB, TRIG = game.GAME_BASIS_CHEB, game.GAME_BASIS_TRIG
FORMS = {"fp32": game.GAME_PREC_FP32, "bf16": game.GAME_PREC_BF16,
         "bf16x3": game.GAME_PREC_BF16X3, "fp8": game.GAME_PREC_FP8,
         "gram": game.GAME_PREC_GRAM}
ERRORS = {"mse": game.GAME_ERR_MSE, "rmse": game.GAME_ERR_RMSE, "mae": game.GAME_ERR_MAE}
SELECTIONS = {"tournament": game.GAME_SEL_TOURNAMENT, "ranking": game.GAME_SEL_RANKING,
              "roulette": game.GAME_SEL_ROULETTE}
SEED = 7          # the GA's own seed, fixed as in a user's script


def _case(name, op, form, M, N, basis, d, P, **more):
    c = {"op": op, "form": form, "M": M, "N": N, "basis": basis, "d": d, "P": P,
         "target": "poly", "error": "mse", "host": False, "gens": 1,
         "selection": "tournament", "tied": False, "R": 1}
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # The small regression of the tests and the README, trained as a whole:
        # the smallest calls, where launches and latency count.
        _case("small_fp32_train", "train", "fp32", 2000, 8, "cheb", 4, 64, gens=10),
        # The paper's own experiment: Globular-Cluster shape, trigonometric basis
        # with shared genes, P = 2 N + 1, ranking selection, the MSE stop rule.
        _case("paper_grid_train", "train", "gram", 2100, 9, "trig", 8, 19, gens=100,
              target="class", selection="ranking", tied=True),
        # One generation of the benchmark's classification workload (BF16, the 16
        # best re-scored): what a long training run repeats.
        _case("cls_bf16_generation", "generation", "bf16", 1_000_000, 32, "cheb", 8, 1024,
              target="class"),
        # The same workload's fitness in the plain FP32 form, the form at its full
        # accuracy and the default precision of a handle.
        _case("cls_fp32_eval", "eval", "fp32", 1_000_000, 32, "cheb", 8, 1024, target="class"),
        # ... and in the FP8 form, the cheapest operands.
        _case("cls_fp8_eval", "eval", "fp8", 1_000_000, 32, "cheb", 8, 1024, target="class"),
        # Split products (near-FP32 accuracy on the tensor cores) at odd sizes:
        # a ragged last pattern tile, a ragged last K-block, a partly empty
        # chromosome tile.
        _case("ragged_bf16x3_eval", "eval", "bf16x3", 150_001, 17, "trig", 5, 300,
              error="rmse"),
        # The FP64 Gram form: independent of M once the handle exists, for runs of
        # many generations under the MSE.
        _case("cls_gram_eval", "eval", "gram", 200_000, 32, "cheb", 8, 1024, target="class"),
        # A mid-sized call of a script that keeps its population in numpy: the
        # copies and the call itself weigh as much as the kernel.
        _case("host_bf16_eval", "eval", "bf16", 30_011, 11, "trig", 7, 100, host=True,
              error="mae"),
        # The longest contraction of the batched workload's range (64 features,
        # trigonometric degree 10) as a single problem.
        _case("wide_bf16_eval", "eval", "bf16", 50_000, 64, "trig", 10, 512),
        # The 4-million-pattern regression with surrogate screening: the largest
        # training set, with the MLP trained on line.
        _case("surrogate_generation", "surrogate", "bf16", 4_000_000, 48, "cheb", 6, 2048),
        # Independent runs of uneven shape in one launch per generation: M from
        # 1,000 to 200,000, N from 4 to 64, degree 2 to 10, P from 32 to 512.
        _case("batch_24_runs", "batch", "bf16", 200_000, 64, "mixed", 10, 512, R=24, gens=4),
        # A trained model applied to new data: FP64 outputs of one chromosome.
        _case("predict_rows", "predict", "fp32", 1_000_000, 32, "cheb", 8, 64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["train", "eval", "eval", "eval", "eval", "generation", "surrogate", "batch",
                     "predict"])
    basis = rng.choice(["cheb", "trig"])
    N, d = rng.randint(4, 64), rng.randint(2, 10)
    if op == "train":
        tied = rng.random() < 0.3
        form = rng.choice(["fp32", "bf16", "gram"])
        return _case(None, op, form, _log(rng, 1000, 20_000), rng.randint(4, 16), basis,
                     rng.randint(2, 8), _log(rng, 16, 128), gens=rng.choice([10, 20]),
                     target=rng.choice(["poly", "class"]),
                     selection=rng.choice(sorted(SELECTIONS)), tied=tied)
    if op == "generation":
        return _capped(_case(None, op, "bf16", _log(rng, 100_000, 1_000_000), N, basis, d,
                             _log(rng, 128, 2048), target=rng.choice(["poly", "class"])), 2.6e11)
    if op == "surrogate":
        return _capped(_case(None, op, "bf16", _log(rng, 100_000, 4_000_000),
                             rng.randint(8, 48), "cheb", rng.randint(3, 8),
                             _log(rng, 256, 2048)), 1.2e12)
    if op == "batch":
        return _case(None, op, "bf16", _log(rng, 20_000, 200_000), N, "mixed", d,
                     _log(rng, 64, 512), R=rng.randint(8, 24), gens=rng.randint(1, 4))
    if op == "predict":
        return _case(None, op, "fp32", _log(rng, 10_000, 1_000_000), min(N, 32), basis, min(d, 8),
                     64)
    form = rng.choice(["fp32", "bf16", "bf16", "bf16x3", "fp8", "gram"])
    # the direct forms take any error, the Gram form no absolute one
    error = rng.choice(["mse", "mse", "rmse"] + ([] if form == "gram" else ["mae"]))
    if form == "bf16x3" and basis == "trig":
        d = min(d, 8)   # its contraction is limited to about 1,200 columns
    return _capped(_case(None, op, form, _log(rng, 1000, 1_000_000), N, basis, d,
                         _log(rng, 32, 2048), error=error, host=rng.random() < 0.25,
                         target=rng.choice(["poly", "class"])),
                   1e11 if form in ("fp32", "bf16x3") else 2.6e11)


def _capped(c, most):
    """The case with its patterns cut so that M P K is at most `most`."""
    c["M"] = max(1000, min(c["M"], int(most / (c["P"] * _genes(c)))))
    return c


def _basis(c):
    return TRIG if c["basis"] == "trig" else CHEB


def _genes(c):
    return (2 if c["basis"] == "trig" else 1) * c["N"] * c["d"] + 1


def _generator(seed, tag):
    return torch.Generator(device="cuda").manual_seed(seed * 1_000_003 + tag)


def _features(g, M, N, correlated):
    """Uniform features in [-1, 1], or correlated Gaussian ones scaled into it."""
    if not correlated:
        return torch.rand(M, N, generator=g, device="cuda") * 2 - 1
    W = torch.randn(N, N, generator=g, device="cuda").double().cpu().numpy()
    L = np.linalg.cholesky(W @ W.T / N + 0.1 * np.eye(N)).astype(np.float32)
    X = torch.randn(M, N, generator=g, device="cuda") @ torch.from_numpy(L).cuda().T
    lo, hi = X.amin(0), X.amax(0)
    return (2 * (X - lo) / (hi - lo) - 1).clamp(-1, 1).contiguous()


def _targets(g, X, D, label):
    """An additive Chebyshev polynomial of degree D with noise 0.05, or its sign
    with 5% of the labels flipped."""
    M, N = X.shape
    coef = torch.rand(D, N, generator=g, device="cuda") * 2 - 1
    t = torch.rand(1, generator=g, device="cuda") * 2 - 1
    tm, tc = torch.ones_like(X), X
    for j in range(D):
        t = t + tc @ coef[j]
        tm, tc = tc, 2 * X * tc - tm
    if not label:
        return t + 0.05 * torch.randn(M, generator=g, device="cuda")
    lab = torch.where(t >= 0, 1.0, -1.0)
    flip = torch.rand(M, generator=g, device="cuda") < 0.05
    return torch.where(flip, -lab, lab).contiguous()


def _population(g, P, K):
    """Half of it uniform, as a run begins; half mutated copies of one parent, as
    it looks later on."""
    pop = torch.rand(P, K, generator=g, device="cuda") * 2 - 1
    kids = P // 2
    step = 0.1 * torch.randn(kids, K, generator=g, device="cuda")
    step *= torch.rand(kids, K, generator=g, device="cuda") < 0.1
    pop[:kids] = (pop[-1] + step).clamp(-1, 1)
    return pop


def _data(case, seed):
    g = _generator(seed, 1)
    label = case["target"] == "class"
    X = _features(g, case["M"], case["N"], label and case["M"] > 10_000)
    y = _targets(g, X, min(case["d"], 8), label)
    return X, y


def _params(case):
    prm = dict(P=case["P"], seed=SEED, precision=FORMS[case["form"]],
               error=ERRORS[case["error"]], selection=SELECTIONS[case["selection"]],
               tied=int(case["tied"]))
    if case["op"] == "eval":
        prm["rescore_top"] = 0
    if case["op"] == "train" and case["target"] == "class":
        prm.update(pm=0.2, mse_threshold=0.001)
    if case["op"] == "surrogate":
        prm["surrogate"] = 1
    return prm


def _runs(case, seed):
    """R problems of uneven shape up to the case's sizes; the shapes are the
    case's, the data the seed's."""
    r = np.random.Generator(np.random.Philox(key=[11, case["R"]]))
    runs = []
    for k in range(case["R"]):
        M = int(round(math.exp(r.uniform(math.log(1000), math.log(case["M"])))))
        N = int(r.integers(4, case["N"] + 1))
        basis = int(r.integers(0, 2))
        d = int(r.integers(2, case["d"] + 1))
        P = int(round(math.exp(r.uniform(math.log(32), math.log(case["P"])))))
        runs.append((M, N, basis, d, P))
    if seed is None:
        return runs
    out = []
    for k, (M, N, basis, d, P) in enumerate(runs):
        g = _generator(seed, 100 + k)
        X = _features(g, M, N, False)
        out.append((X, _targets(g, X, 4, False), d, basis, P, SEED + k))
    return out


def prepare(case, seed):
    op = case["op"]
    state = {"op": op, "gens": case["gens"]}
    if op == "batch":
        # given widths keep a batch reproducible: no autotuning
        state["batch"] = game.Batch(_runs(case, seed), autotune=False)
        return state
    X, y = _data(case, seed)
    if op == "predict":
        # the model was trained on a small set; the patterns are new
        n = min(case["M"], 4096)
        state["game"] = game.Game(X[:n].contiguous(), y[:n].contiguous(), case["d"],
                                  _basis(case), **_params(case))
        state["chrom"] = _population(_generator(seed, 2), 2, _genes(case))[1].contiguous()
        state["X"] = X
        return state
    h = state["game"] = game.Game(X, y, case["d"], _basis(case), **_params(case))
    if op == "eval":
        pop = _population(_generator(seed, 2), case["P"], h.K)
        state["pop"] = pop.cpu().numpy() if case["host"] else pop
    elif op in ("generation", "surrogate"):
        state["out"] = (torch.empty(h.P, h.K, device="cuda"),
                        torch.empty(h.P, device="cuda", dtype=torch.float64))
    return state


def run(state):
    op = state["op"]
    if op == "batch":
        b = state["batch"]
        for _ in range(state["gens"]):
            b.generation()
        return [b.run(r)[:2] for r in range(b.R)]
    h = state["game"]
    if op == "eval":
        return h.eval_fitness(state["pop"])
    if op == "predict":
        return h.predict(state["chrom"], state["X"])
    if op == "train":
        h.train(state["gens"])
        return h.population()
    h.generation(SEED)
    pop, fit = state["out"]
    game.game_get_population(h.h, pop, fit)
    if op == "surrogate":
        return pop, fit, h.surrogate_params()
    return pop, fit


def work(case):
    op = case["op"]
    if op == "batch":
        nbytes = flops = 0
        for M, N, basis, d, P in _runs(case, None):
            K = (2 if basis else 1) * N * d + 1
            flops += case["gens"] * M * P * (2 * (K - 1) + 3)
            nbytes += case["gens"] * (4 * M * (N + 1) + 8 * P * K + 8 * P)
        return {"bytes": nbytes, "flops": flops}
    M, N, P, K = case["M"], case["N"], case["P"], _genes(case)
    if op == "predict":
        return {"bytes": 4 * M * N + 8 * M + 4 * K, "flops": 4 * M * (K - 1)}
    Kg = (K - 1) // N + 1 if case["tied"] else K
    # fitness of one population: the patterns once, the genes once
    if case["form"] == "gram":
        nbytes, flops = 8 * Kg * (Kg + 1) // 2, P * Kg * (Kg + 1)
    else:
        nbytes, flops = 4 * M * (N + 1), M * P * (2 * (K - 1) + 3)
    nbytes += 4 * P * Kg + 8 * P
    if op != "eval":
        nbytes += 4 * P * Kg   # the next population
    if op == "surrogate":
        # 8 (P - 2) children bred and predicted, 16 training steps of P pairs
        # (forward and backward), the Adam state
        mac = 256 * Kg + 256 * 256 + 256
        flops += 2 * mac * 8 * (P - 2) + 6 * mac * 16 * P
        nbytes += 4 * Kg * 8 * (P - 2) + 24 * mac
    return {"bytes": nbytes * case["gens"], "flops": flops * case["gens"]}


def _design(X, d, basis):
    """[M][K - 1] expansion in FP64, columns in gene order."""
    x = X.double()
    if basis == TRIG:
        j = torch.arange(1, d + 1, device=x.device, dtype=torch.float64)
        ang = x[:, :, None] * j
        cols = torch.cat([torch.cos(ang), torch.sin(ang)], dim=2)
    else:
        t = [torch.ones_like(x), x]
        for _ in range(d - 1):
            t.append(2 * x * t[-1] - t[-2])
        cols = torch.stack(t[1:], dim=2)
    return cols.reshape(x.shape[0], -1)


def exact(case, seed):
    op = case["op"]
    if op not in ("eval", "predict"):
        return None   # populations the operators bred, and what follows from them
    X, y = _data(case, seed)
    g = _generator(seed, 2)
    step = max(256, (1 << 25) // _genes(case))
    if op == "predict":
        a = _population(g, 2, _genes(case))[1].double()
        return torch.cat([_design(x, case["d"], _basis(case)) @ a[1:] + a[0]
                          for x in X.split(step)])
    a = _population(g, case["P"], _genes(case)).double()
    total = torch.zeros(case["P"], device="cuda", dtype=torch.float64)
    for x, t in zip(X.split(step), y.double().split(step)):
        r = t[:, None] - a[:, 0] - _design(x, case["d"], _basis(case)) @ a[:, 1:].T
        total += r.abs().sum(0) if case["error"] == "mae" else r.square().sum(0)
    total /= case["M"]
    total = total.sqrt() if case["error"] == "rmse" else total
    return total.cpu().numpy() if case["host"] else total
