"""Width of the FP32 lag sums: with a bandwidth so wide that every kernel value
is exactly 1, and an autocorrelation of ones in row 0 and 2^-25 elsewhere (too
small to change a 1 in FP32), the pair sums still hold every term.  One chain
over several rows, or FP32 additions across rows or windows, would lose them.
All four forms: one dataset, a prepared set, many datasets, candidates built
on the device."""
import math

import numpy as np
import pytest

from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TINY = 2.0 ** -25


def _case(M, P_min, nsets):
    """Plan, autocorrelations (different by powers of two) and their exact half-plane sums."""
    lo, hi = [0.0, 0.0], [M[0] - 1.0, M[1] - 1.0]
    plan = kde.Plan(M, lo, hi, np.eye(2), P_min=P_min)
    P = plan.info.P
    R = np.full((nsets,) + tuple(P), TINY, dtype=np.float32)
    R[:, 0, :] = 1.0
    # row 0: ones in the lags' first window, tiny terms from the next on
    R[:, 0, 64:P[1] - 63] = TINY
    R *= 2.0 ** np.arange(nsets)[:, None, None]
    L0, L1 = M[0] - 1, M[1] - 1
    ones, tiny = min(L1, 63), max(0, L1 - 63)
    half = 0.5 + ones + tiny * TINY + L0 * (2 * L1 + 1) * TINY
    return plan, torch.from_numpy(R).cuda(), 2.0 * half * 2.0 ** np.arange(nsets)


def _norm(det):
    return float(np.float32(1.0 / (2.0 * math.pi) / math.sqrt(det)))


@pytest.mark.parametrize("M,P_min", [((9, 33), (17, 65)), ((40, 60), (79, 119)), ((70, 200), (139, 399)),
                                     ((5, 700), (9, 1399))])
@pytest.mark.parametrize("nsets", [1, 9, 17])
def test_no_term_is_lost(M, P_min, nsets):
    plan, R, want = _case(M, P_min, nsets)
    h = 2.0 ** 60                              # exponents above -2^-30: every 2^x rounds to 1
    H = np.array([h * np.eye(2), 4.0 * h * np.eye(2), h * np.eye(2)])
    cands = kde.LscvCands(plan, H)
    norm = np.array([[_norm(h * h * s * s), _norm(4.0 * h * h * s * s)] for s in (1.0, 4.0, 1.0)])
    S = torch.empty(nsets, 3, 2, dtype=torch.float64, device="cuda")
    cands.score_batch([100] * nsets, R, pair_sums=S)
    # pairs of FP32 lose less than 2^-44 a sum
    assert np.allclose(S.cpu().numpy(), want[:, None, None] * norm, rtol=1e-12, atol=0.0)
    for i in (0, nsets - 1):
        S1 = torch.empty(3, 2, dtype=torch.float64, device="cuda")
        cands.score(100, R[i], pair_sums=S1)
        assert torch.equal(S1, S[i])
        kde.kde_lscv_autocorr(plan, 100, H, R[i], pair_sums=S1)
        assert torch.equal(S1, S[i])


@pytest.mark.parametrize("nsets", [1, 5])
def test_no_term_is_lost_in_device_built_candidates(nsets):
    M = (40, 60)
    plan, R, want = _case(M, (79, 119), nsets)
    a = math.log(2.0 ** 30)                    # H = 2^60 I
    offs = np.zeros((3, 3))
    refs = np.tile([a, 0.0, a], (nsets, 1))
    th = torch.tensor(refs, dtype=torch.float32, device="cuda")
    lscv = torch.empty(nsets, 4, dtype=torch.float64, device="cuda")
    n = 100.0
    kde.kde_lscv_theta_select(plan, [int(n)] * nsets, th, [-50.0] * 3, [50.0] * 3, offs, refs, R, lscv=lscv)
    # the reference candidate: LSCV = S(2H)/n^2 - 2 (S(H) - n K_H(0)) / (n (n-1))
    h = math.exp(a) ** 2
    S1, S2 = want * _norm(h * h), want * _norm(4.0 * h * h)
    ref = S2 / n ** 2 - 2.0 * (S1 - n / (2.0 * math.pi * h)) / (n * (n - 1.0))
    # the normalisation is rounded to FP32 on both sides from FP64 values that
    # can differ in the last bit: at most one FP32 step, but the same for every set
    got = lscv.cpu().numpy()[:, 3]
    assert np.allclose(got, ref, rtol=3e-7, atol=0.0)
    assert np.allclose((got - got[0]) * (want[-1] - want[0]), (got[-1] - got[0]) * (want - want[0]),
                       rtol=1e-11, atol=1e-11 * abs(got).max() * want.max())
