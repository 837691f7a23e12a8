"""One-dimensional plans on the cluster and cosine-sum kernels: lengths either
side of the one-block switch, odd and even factors (a column without a
partner, a middle row), supports from a few lags to the whole grid and either
side of the switch of the spectrum, both layouts and precisions, every node
against the oracle."""
import numpy as np
import pytest

from oracle import kde_oracle as O
from paper_1508_02766_gb300 import kde
from paper_1508_02766_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-12, "f32": 1e-5}


def _need(P):
    """M, tau giving the padded length P when L is a tenth of it."""
    L = max(1, P // 10)
    return P - L, L


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("P", [250, 256, 270, 343, 486, 625, 1024, 2100, 2401, 3125, 4096])
def test_lengths(P, prec):
    M, L = _need(P)
    w = W.small_case(P, 1, (M,), n=4000, precision=prec)
    w.tau = (L - 0.5) * (w.hi[0] - w.lo[0]) / (M - 1) / np.sqrt(w.H[0, 0])
    _check(w, L)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("M,L", [(1500, 1), (1500, 31), (1500, 32), (1500, 33), (1600, 1024), (1600, 1025),
                                 (1600, 1599)])
def test_supports(M, L, prec):
    w = W.small_case(M + L, 1, (M,), n=4000, precision=prec)
    w.tau = (L - 0.5) * (w.hi[0] - w.lo[0]) / (M - 1) / np.sqrt(w.H[0, 0])
    _check(w, L)
    _check(w, L, layout="wand")


def _check(w, L, **opts):
    X = torch.from_numpy(np.ascontiguousarray(w.X)).cuda()
    dens, counts, plan = kde.kde_eval(X, w.H, w.lo, w.hi, w.M, precision=w.precision, tau=w.tau, **opts)
    assert plan.info.L == (L,)
    f, c_ref, _, _ = O.binned_estimate(w.X, w.H, w.lo, w.hi, w.M, tau=w.tau, **opts)
    assert np.array_equal(counts.cpu().numpy(), c_ref)
    assert np.max(np.abs(dens.cpu().numpy() - f)) <= TOL[w.precision] * np.max(np.abs(f))
