"""Calls with host arguments captured into a CUDA graph: the graph keeps the
arguments of the captured call.  Many later calls with other and larger
arguments reuse (and regrow) every staging slot of the thread before the
replay, which still gives the captured call's results, and none of them
fails."""
import numpy as np
import pytest

from paper_1508_02766_gb300 import kde
from paper_1508_02766_gb300 import learned as Lm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI, M = [-5.0, -5.0], [5.0, 5.0], (64, 64)


def _bandwidths(seed, count):
    rng = np.random.default_rng(seed)
    R = np.zeros((count, 2, 2))
    R[:, 0, 0], R[:, 1, 1] = np.exp(rng.uniform(-3.0, -1.2, size=(2, count)))
    R[:, 1, 0] = rng.uniform(-0.3, 0.3, size=count)
    return R @ R.transpose(0, 2, 1)


def _plan():
    return kde.Plan(M, LO, HI, 0.01 * np.eye(2), P_min=(128, 128))


def _multi(plan, seed, count):
    c = torch.arange(64 * 64, device="cuda").reshape(64, 64) << 20
    H = _bandwidths(seed, count)
    out = torch.zeros(count, *M, device="cuda")
    ws = torch.empty(kde.kde_fft_eval_multi_workspace_bytes(plan), dtype=torch.uint8, device="cuda")
    return lambda: kde.kde_fft_eval_multi(plan, 100, H, c, density=out, workspace=ws), out


def _autocorr(plan, seed, count):
    R = torch.rand(*plan.info.P, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))
    H = _bandwidths(seed, count)
    out = torch.zeros(count, dtype=torch.float64, device="cuda")
    ws = torch.empty(kde.kde_lscv_autocorr_workspace_bytes(plan), dtype=torch.uint8, device="cuda")
    return lambda: kde.kde_lscv_autocorr(plan, 100 + seed, H, R, lscv=out, workspace=ws), out


def _theta(plan, seed, count):
    g = torch.Generator(device="cuda").manual_seed(seed)
    nsets = max(2, count // 8)
    R, th = torch.rand(nsets, *plan.info.P, device="cuda", generator=g), torch.rand(nsets, 3, device="cuda", generator=g) - 2
    ns = np.arange(nsets) + 50 + seed
    offs = 0.5 * Lm.NEIGHBOUR_OFFSETS * Lm.STEP + 0.01 * seed
    lscv = torch.zeros(nsets, 28, dtype=torch.float64, device="cuda")
    out = torch.zeros(nsets, 6, dtype=torch.float64, device="cuda")
    ws = torch.empty(kde.lscv_theta_select_workspace_bytes(plan, nsets, 27), dtype=torch.uint8, device="cuda")
    return lambda: kde.kde_lscv_theta_select(plan, ns, th, [-9.0] * 3, [9.0] * 3, offs, Lm.normal_reference_thetas(ns),
                                             R, lscv=lscv, out=out, workspace=ws), lscv


def _cands(plan, seed, count):
    cands = kde.LscvCands(plan, _bandwidths(3, 20))
    R = torch.rand(count, *plan.info.P, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))
    ns = np.arange(count) + 50 + seed
    out = torch.zeros(count, 20, dtype=torch.float64, device="cuda")
    ws = torch.empty(max(256, cands.batch_workspace_bytes(count)), dtype=torch.uint8, device="cuda")
    return lambda: cands.score_batch(ns, R, lscv=out, workspace=ws), out


# counts below and above one kernel's worth of arguments, and above a slot's first size
@pytest.mark.parametrize("make,count,later", [(_multi, 5, 1500), (_multi, 700, 40), (_autocorr, 37, 1000),
                                              (_theta, 24, 80), (_cands, 9, 300)])
def test_graph_keeps_the_captured_arguments(make, count, later):
    plan = _plan()
    run, out = make(plan, 1, count)
    run()
    torch.cuda.synchronize()
    ref = out.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        run()
    other, out2 = make(plan, 2, later)
    other()
    torch.cuda.synchronize()
    ref2 = out2.clone()
    for i in range(20):
        (other if i % 3 else make(plan, 4 + i, count)[0])()
    torch.cuda.synchronize()
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and torch.equal(out2, ref2)
    other()
    torch.cuda.synchronize()
    assert torch.equal(out2, ref2)
