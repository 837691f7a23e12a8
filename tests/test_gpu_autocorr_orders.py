"""The counts' autocorrelation on every entry against a 64-bit FFT: splits
above 2048 points on either axis, with what else feeds on such a plan (the
evaluation that leaves the counts zeroed, the power spectrum behind the
spectrum-dot LSCV), and odd and even padded lengths with one and several
datasets (the output rows store their mirrors)."""
import os
import re

import numpy as np
import pytest

from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = os.path.join(os.path.dirname(kde.__file__), "csrc", "fx_pairs.h")
BODY = open(SRC).read().split("#define KDE_FX_LONG_TRIPLES")[1].split("\n\n")[0]
SPLITS = [tuple(int(v) for v in m.split(",")) for m in re.findall(r"X\(([\d,\s]+)\)", BODY)]


def _reference(counts, P):
    F = torch.fft.rfft2(counts.double() * 2.0 ** -32, s=tuple(P))
    return torch.fft.irfft2(F.abs() ** 2, s=tuple(P))


def _counts(M, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.rand(*M, device="cuda", generator=g).pow(4) * 2.0 ** 36).long()


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("split", SPLITS)
def test_long_lines(split, axis):
    P = int(np.prod(split))
    M, P_min = [14, 13], [401, 401]
    M[axis], P_min[axis] = P - 600, P
    lo, hi = [0.0, 0.0], [M[0] - 1.0, M[1] - 1.0]
    H = np.array([[2.0, 0.5], [0.5, 3.0]])
    plan = kde.Plan(M, lo, hi, H, P_min=P_min)
    assert plan.info.engine == "two_phase" and plan.info.P[axis] == P
    c = _counts(M, P)
    ref = _reference(c, plan.info.P)
    R = kde.kde_autocorrelation(plan, c)
    assert float((R.double() - ref).abs().max()) <= 1e-5 * float(ref.max())
    n = int(c.double().sum().item() * 2.0 ** -32)
    K = kde.kde_kernel_grid(plan, n)
    dens = kde.kde_fft_eval(plan, c, K)
    left = c.clone()
    assert torch.equal(kde.kde_fft_eval(plan, left, K, consume=True), dens) and not left.any()
    W = kde.kde_power_spectrum(plan, c)
    a, b = (torch.empty(2, 2, dtype=torch.float64, device="cuda") for _ in range(2))
    Hs = np.stack([0.3 * H, 0.5 * H])
    kde.kde_lscv(plan, n, Hs, W, pair_sums=a)
    kde.kde_lscv_autocorr(plan, n, Hs, R, pair_sums=b)
    assert float(((a - b) / b).abs().max()) <= 2e-5


@pytest.mark.parametrize("P", [(35, 64), (63, 49), (81, 81), (135, 96), (80, 105), (400, 64)])
@pytest.mark.parametrize("nsets", [1, 2, 5])
def test_odd_and_even_lengths_of_several_datasets(P, nsets):
    M = (32, 32)
    plan = kde.Plan(M, [-5.0, -5.0], [5.0, 5.0], 1e-3 * np.eye(2), P_min=P)
    assert plan.info.engine == "two_phase" and tuple(plan.info.P) == P
    n = 500
    X = torch.randn(nsets * n, 2, device="cuda", generator=torch.Generator(device="cuda").manual_seed(nsets))
    prep = kde.BatchPrep(plan, nsets, nsets * n)
    F = torch.empty(nsets, kde.FEAT_DIM, device="cuda")
    R = torch.full((nsets,) + P, float("nan"), device="cuda")
    prep.run(X, np.arange(nsets + 1) * n, F, R)
    for i in range(nsets):
        ref = _reference(prep.counts[i], P)
        assert float((R[i].double() - ref).abs().max()) <= 1e-5 * float(ref.max())
        assert torch.equal(kde.kde_autocorrelation(plan, prep.counts[i].contiguous()), R[i])
