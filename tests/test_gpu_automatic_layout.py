"""What the automatic choice of the register layout picks between a lone warp per scheduler and a full
GPU, where the dispatch has builds that no fixed layout reaches, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_23949_b200 import binding as ts
from paper_2505_23949_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (M, N, rows, cols, iterations), by warps per SM of 148
CASES = [
    (4, 2, 512, 516, 20), (4, 1, 384, 388, 300), (4, 3, 520, 516, 100),           # latency, latency, throughput
    (8, 4, 640, 648, 60), (8, 3, 768, 776, 60), (8, 5, 776, 768, 300),            # latency, spread, throughput
    (16, 8, 496, 528, 60), (16, 5, 640, 656, 60), (16, 8, 880, 912, 300),         # latency, spread, spread
    (16, 8, 1024, 1024, 300), (16, 11, 1040, 1008, 300), (16, 9, 768, 784, 300),  # spread
    (16, 8, 16 * 7104, 16, 60), (8, 2, 8 * 9000, 8, 60),                          # slabs: spread, spread
    (32, 16, 1280, 1248, 60),                                                     # latency
]


@pytest.mark.parametrize("M,N,rows,cols,iters", CASES)
def test_plan_and_mask_against_the_oracle(M, N, rows, cols, iters):
    W = synth.student_t_abs(rows, cols, 0.02, seed=M + rows)
    Wd = torch.from_numpy(W).to(DEV)
    tau = synth.default_tau(float(W.max()))
    st = ts.new_status(DEV)
    plan = ts.dykstra(Wd, N, M, tau, iters, plan_is_log=True, status=st)
    ref = oracle.dykstra(W, N, M, tau, iters)
    # the plan's parity bound: fp32 rounding of t0 (ulp(288) in base-2 units) and of the potentials
    assert np.abs(np.exp(plan.cpu().numpy().astype(np.float64)) - ref).max() <= 1e-4
    got = ts.round_plan(plan, Wd, N, M, status=st).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, oracle.round_plan(plan.cpu().numpy(), W, N, M))    # rounding: bit for bit
    # the whole method rounds the same plan in base-2 units, a positive multiple of the keys: only products
    # by ln 2 that round to one key may order differently, in a few blocks at most
    mask = ts.solve(Wd, N, M, tau, iters, mask_out=ts.new_mask(rows, cols, DEV).fill_(-1), status=st)
    assert np.mean(mask.cpu().numpy().view(np.uint32) != got) <= 1e-4
    assert int(ts.check(mask, rows, cols, N, M).item()) == 0
    assert int(st.item()) == 0


@pytest.mark.parametrize("M,N,rows,cols", [(8, 4, 768, 776), (16, 8, 640, 656), (16, 3, 880, 912)])
def test_stopping_test_in_the_spread_layout(M, N, rows, cols):
    """Iterations at 5, 9, 13, ...; the plan of a block is that of some tested iteration whose violation is below
    eps, so it is as close to the fixed-count plan as eps allows; every mask is feasible."""
    W = synth.student_t_abs(rows, cols, 0.02, seed=M + rows)
    Wd = torch.from_numpy(W).to(DEV)
    tau = synth.default_tau(float(W.max()))
    nblk = (rows // M) * (cols // M)
    ran = torch.zeros(1, dtype=torch.int64, device=DEV)
    src = ts.Scores(ts.SCORES_ABS, Wd, early_exit_eps=1e-3, iters_out=ran)
    mask = ts.solve_scores(src, N, M, tau, 300)
    assert int(ts.check(mask, rows, cols, N, M).item()) == 0
    # a warp stops when all its blocks pass: no fewer iterations than block by block, and no more than 300
    _, alone = oracle.dykstra_earlyexit(W, N, M, tau, 300, 1e-3, check_every=4)
    assert int(alone.sum()) - 4 * nblk // 100 <= int(ran.item()) <= 300 * nblk
    full = ts.solve(Wd, N, M, tau, 300)
    a, b = float(ts.objective(Wd, mask).item()), float(ts.objective(Wd, full).item())
    assert abs(a - b) <= 1e-3 * b


@pytest.mark.parametrize("M,N,rows,cols", [(8, 3, 768, 776), (16, 8, 640, 656)])
@pytest.mark.parametrize("kind", ["abs", "mul", "div", "admm"])
@pytest.mark.parametrize("bf16,pad", [(False, 0), (False, 5), (True, 4)])
def test_spread_layout_on_every_source(M, N, rows, cols, kind, bf16, pad):
    """Described scores give what their materialised fp32 copy gives, and a block's own tau what the oracle says."""
    g = torch.Generator(device=DEV).manual_seed(M)
    big = torch.randn((rows, cols + pad), generator=g, device=DEV)
    w = (big.to(torch.bfloat16) if bf16 else big)[:, pad:]
    v = torch.randn((rows, cols), generator=g, device=DEV)
    a = torch.randn(cols, generator=g, device=DEV).abs_() + 0.1

    def source(**opt):
        return {"abs": lambda: ts.Scores(ts.SCORES_ABS, w, **opt),
                "mul": lambda: ts.Scores(ts.SCORES_COLMUL, w, colvec=a, **opt),
                "div": lambda: ts.Scores(ts.SCORES_COLDIV, w, colvec=a, **opt),
                "admm": lambda: ts.Scores(ts.SCORES_ADMM, w, v=v, scalar=0.5, **opt)}[kind]()

    src = source()
    plain = ts.scores_materialize(src)
    tau = 200.0 / float(ts.scores_max(src).item())
    assert torch.equal(ts.solve_scores(src, N, M, tau, 40), ts.solve(plain, N, M, tau, 40))
    assert torch.equal(ts.dykstra_scores(src, N, M, tau, 40), ts.dykstra(plain, N, M, tau, 40))
    got = ts.dykstra_scores(source(per_block_tau=True), N, M, 200.0, 40).cpu().numpy().astype(np.float64)
    assert np.abs(got - oracle.dykstra(plain.cpu().numpy(), N, M, 200.0, 40, per_block_tau=True)).max() <= 1e-4
