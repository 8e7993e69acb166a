"""What this library is used for, as cases to be timed.

A pass is what a pruning program does with one weight matrix (or one layer's matrices): it hands a
score matrix to the solver on the device and gets the transposable N:M mask back.  Sizes and value
distributions are those of the benchmark's configurations (``synth.py``, ``bench.py``), drawn on
the device: the paper's LLaMA-3 matrices are not available.

A case is a dict:
  kind    abs        |W|, tsenor_solve
          wanda      |W_ij| a_j, a_j lognormal(0, 1), tsenor_solve_scores
          admm       (W + V / rho)^2 and the keep-previous-mask safeguard: one D-update of ADMM
          sparsegpt  |W_ij / d_j| on a column group of one block column
          ablation   Algorithm 1 to the log-plan, then the three roundings of it, and what they retain
  flow    True: the program also chooses tau from the largest score, and verifies the mask
          (feasibility, and the retained score of |W|); False: tau is in hand
  rows, cols, N, M, iters; bf16 (weights in bfloat16, else float32); eps > 0: the stopping-test mode
  pad     columns of the surrounding matrix that are not part of the one that is pruned
  dist    gauss N(0, std^2), student Student-t(3), outlier N(0, std^2) with 0.1 % of columns x20
  layer   True: the seven linear shapes of one Llama-3-8B layer instead of rows x cols
"""
import math

import torch

from paper_2505_23949_b200 import binding as ts
from paper_2505_23949_b200 import synth

ITERS = 300      # T of the paper and of every configuration
RHO = 0.3        # ADMM penalty of the benchmark's D-update


def _case(name, kind, rows, cols, N, M, dist="gauss", bf16=False, flow=False, eps=0.0, pad=0, layer=False, std=0.02):
    c = {"kind": kind, "rows": rows, "cols": cols, "N": N, "M": M, "dist": dist, "bf16": bf16, "flow": flow,
         "eps": eps, "pad": pad, "layer": layer, "std": std, "iters": ITERS}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest matrices one prunes, with a last mask word that is not full: launch and latency
        _case("tiny-2:4", "abs", 256, 264, 2, 4, dist="outlier"),
        # a small matrix (configuration 1): 4,096 blocks, less than one wave of the GPU
        _case("small-4:8", "abs", 512, 512, 4, 8, std=1.0),
        # a sub-matrix of a larger one whose rows are not aligned, N other than M / 2, an odd number
        # of blocks; the program picks tau and checks what it got
        _case("ragged-3:8", "abs", 1000, 2056, 3, 8, dist="student", flow=True, pad=5),
        # one attention projection (configuration 2): 1,048,576 of the smallest blocks
        _case("proj-2:4", "abs", 4096, 4096, 2, 4),
        # Wanda on bf16 weights (configuration 3) from the activation norms to a checked mask
        _case("wanda-8:16", "wanda", 4096, 4096, 8, 16, bf16=True, flow=True),
        # one D-update of ADMM on a small layer: called once per ADMM iteration
        _case("admm-8:16", "admm", 1024, 1024, 8, 16),
        # one column group of SparseGPT: called once per group of every matrix
        _case("sparsegpt-16:32", "sparsegpt", 14336, 32, 16, 32),
        # the MLP's up-projection (configuration 4, the headline workload)
        _case("up-16:32", "abs", 14336, 4096, 16, 32, dist="student"),
        # the MLP's down-projection handed over in bf16
        _case("down-bf16-16:32", "wanda", 4096, 14336, 16, 32, dist="outlier", bf16=True),
        # one layer of an 8B model, all seven linears (configuration 5): the largest
        _case("layer-4:8", "abs", 0, 0, 4, 8, dist="outlier", layer=True),
        # the rounding study: plan, simple rounding, greedy alone, greedy and local search
        _case("ablation-8:16", "ablation", 2048, 2048, 8, 16),
        # the stopping-test mode on the headline matrix
        _case("stopping-16:32", "abs", 14336, 4096, 16, 32, dist="student", eps=1e-3),
    ]


def draw(rng):
    kind = rng.choice(["abs", "abs", "abs", "wanda", "admm", "sparsegpt", "ablation"])
    M = rng.choice([4, 8, 16, 32])
    N = M // 2 if rng.random() < 0.7 else rng.randint(1, M - 1)
    dist = rng.choice(["gauss", "student", "outlier"])
    if kind == "sparsegpt":      # a column group: one block column, any number of block rows
        rows, cols = M * round(2 ** rng.uniform(math.log2(4), math.log2(65536 // M))), M
    else:                        # 2^14 .. 2^26 scores (2^23 for the study), one to sixteen times as long as wide
        n, r = 2 ** rng.uniform(14, 23 if kind == "ablation" else 26), 2 ** rng.uniform(-2, 2)
        rows, cols = (max(1, round(x / M)) * M for x in (math.sqrt(n * r), math.sqrt(n / r)))
    return _case(None, kind, rows, cols, N, M, dist=dist, bf16=kind != "ablation" and rng.random() < 0.3,
                 flow=kind in ("abs", "wanda") and rng.random() < 0.3,
                 eps=1e-3 if kind in ("abs", "wanda") and rng.random() < 0.15 else 0.0,
                 pad=rng.choice([0, 0, 0, 4, 5]))


def _shapes(case):
    return list(synth.LLAMA3_8B_LAYER_SHAPES.values()) if case["layer"] else [(case["rows"], case["cols"])]


def _weights(gen, case, rows, cols, std):
    """rows x cols weights of the case's distribution inside a matrix of cols + pad columns."""
    shape = (rows, cols + case["pad"])
    w = torch.randn(shape, generator=gen, device="cuda")
    if case["dist"] == "student":        # t(3), scaled to standard deviation 1
        chi = sum(torch.randn(shape, generator=gen, device="cuda").square_() for _ in range(3))
        w /= chi.sqrt_()
    elif case["dist"] == "outlier":
        k = max(1, round(1e-3 * cols))
        w[:, torch.randperm(shape[1], generator=gen, device="cuda")[:k]] *= 20.0
    w *= std
    if case["bf16"]:
        w = w.to(torch.bfloat16)
    return w[:, case["pad"]:]


class _Matrix:
    """One matrix and what the program keeps for it: score source, mask and status buffers, tau."""

    def __init__(self, gen, case, rows, cols):
        self.rows, self.cols = rows, cols
        self.w = _weights(gen, case, rows, cols, case["std"])
        self.mask = ts.new_mask(rows, cols, self.w.device)
        self.status = ts.new_status(self.w.device)
        kind, opt = case["kind"], {"early_exit_eps": case["eps"]}
        if kind == "wanda":
            a = torch.randn(cols, generator=gen, device="cuda").exp_()
            self.src = ts.Scores(ts.SCORES_COLMUL, self.w, colvec=a, **opt)
        elif kind == "sparsegpt":
            d = torch.randn(cols, generator=gen, device="cuda").abs_() + 0.05
            self.src = ts.Scores(ts.SCORES_COLDIV, self.w, colvec=d, **opt)
        elif kind == "admm":
            v = torch.randn((rows, cols), generator=gen, device="cuda") * (0.2 * case["std"])
            self.src = ts.Scores(ts.SCORES_ADMM, self.w, v=v, scalar=1.0 / RHO, **opt)
        else:
            self.src = ts.Scores(ts.SCORES_ABS, self.w, **opt)
        self.plain = kind in ("abs", "ablation") and not case["bf16"] and not case["eps"]
        self.tau = synth.default_tau(ts.scores_max(self.src).item())
        if kind == "admm":               # the mask of the ADMM iteration before: half of it up to date
            self.prev = ts.solve_scores(ts.Scores(ts.SCORES_ABS, self.w), case["N"], case["M"], self.tau, 50)
            self.prev[: rows // 2] = ts.solve_scores(self.src, case["N"], case["M"], self.tau, 50)[: rows // 2]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {"case": case, "mats": [_Matrix(gen, case, r, c) for r, c in _shapes(case)]}


def _solve(m, c, tau):
    if m.plain:
        return ts.solve(m.w, c["N"], c["M"], tau, c["iters"], -1, mask_out=m.mask, status=m.status)
    return ts.solve_scores(m.src, c["N"], c["M"], tau, c["iters"], -1, mask_out=m.mask, status=m.status)


def run(state):
    c, out = state["case"], []
    N, M = c["N"], c["M"]
    for m in state["mats"]:
        if c["kind"] == "ablation":
            plan = ts.dykstra(m.w, N, M, m.tau, c["iters"], plan_is_log=True, status=m.status)
            masks = [ts.simple_round(plan, N, M), ts.round_plan(plan, m.w, N, M, ls_steps=0),
                     ts.round_plan(plan, m.w, N, M, ls_steps=-1)]
            out += [plan, *masks, *[ts.objective(m.w, k) for k in masks]]
        elif c["kind"] == "admm":
            mask = _solve(m, c, m.tau)
            out += [ts.keep_better(m.src, m.prev, mask), mask]
        elif c["flow"]:
            top = ts.max_abs(m.w) if m.plain else ts.scores_max(m.src)
            tau = synth.default_tau(top.item())
            mask = _solve(m, c, tau)
            out += [mask, ts.check(mask, m.rows, m.cols, N, M)]
            if m.plain:
                out.append(ts.objective(m.w, mask))
        else:
            out.append(_solve(m, c, m.tau))
    return out


def exact(case, seed):
    """The rounding study's log-plan by Algorithm 1 in its printed log-domain form, in fp64.  The masks
    are picks, not computed numbers, and what they retain follows them."""
    if case["kind"] != "ablation":
        return None
    m, M, N = prepare(case, seed)["mats"][0], case["M"], case["N"]
    tau = torch.tensor(m.tau, dtype=torch.float32).double().item()     # the interface takes tau in fp32
    x = m.w.double().abs_().mul_(tau).view(m.rows // M, M, m.cols // M, M).transpose(1, 2)
    x, q = x.contiguous(), torch.zeros((), dtype=torch.float64, device="cuda")
    for _ in range(case["iters"]):
        x = x - torch.logsumexp(x, -1, keepdim=True) + math.log(N)
        x = x - torch.logsumexp(x, -2, keepdim=True) + math.log(N)
        y = x + q
        x = y.clamp(max=0.0)
        q = y - x
    return [x.transpose(1, 2).reshape(m.rows, m.cols)] + [None] * 6


def work(case):
    """Scores read once per call that needs them, masks (and the study's plan) written once; four
    fp32 operations per entry and iteration: clip, row sum, column sum, scaling.  The operations of
    the stopping-test mode are not known beforehand and are left out."""
    n = sum(r * c for r, c in _shapes(case))
    read = 2 if case["bf16"] else 4
    if case["kind"] == "admm":
        read += 4
    calls = {"admm": 2, "ablation": 1}.get(case["kind"], 1) + (1 if case["flow"] else 0)
    b = n * (read * calls + 1 / 8)
    if case["kind"] == "ablation":
        b += n * (4 + 3 * 4 + 3 * 4)     # the plan written, read by three roundings; |W| by the objectives
    return {"bytes": b, "flops": 0 if case["eps"] else 4 * n * case["iters"]}


def tolerance(case):
    """Measured on these cases and two dozen drawn ones, against the fp64 oracle on up to 2,048 blocks
    and against the kernel itself with its sums in another order (the other register layout): mask words
    differ in up to 8e-4 (M = 32) and 1e-5 (M < 32) of all words, by greedy picks between entries of the
    plan that agree to rounding; a small matrix may hold one such block.  The log-plan differs by up to
    2e-6 (2-norm) and 7e-5 (largest entry).  The retained score moves with the masks."""
    n = sum(r * ((c + 31) // 32) for r, c in _shapes(case))
    differ = max(3e-3 if case["M"] == 32 else 1e-4, min(0.01, case["M"] / n))
    return {"rel": 8e-6, "max": 3e-4, "differ": differ}
