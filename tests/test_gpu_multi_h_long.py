"""Densities of more bandwidths than one parameter upload holds, with odd
column counts and supports from one lag up, on two- and three-factor lines:
each equals the one-bandwidth path bit for bit."""
import numpy as np
import pytest

from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,P_min,nH", [((20, 25), None, 1027), ((33, 20), (0, 449), 65), ((20, 30), (449, 0), 3),
                                        ((40, 41), (81, 99), 130)])
def test_equal_the_one_bandwidth_path(M, P_min, nH):
    rng = np.random.default_rng(nH)
    R = np.zeros((nH, 2, 2))
    R[:, 0, 0], R[:, 1, 1] = np.exp(rng.uniform(-4.5, -1.6, size=(2, nH)))
    R[:, 1, 0] = rng.uniform(-1, 1, size=nH) * R[:, 1, 1]
    H = R @ R.transpose(0, 2, 1)
    lo, hi = [-2.0, -2.0], [2.0, 2.0]
    big = max(H, key=lambda h: np.linalg.eigvalsh(h).max())
    P = kde.kde_plan_info_compute(M, lo, hi, big, P_min=P_min).P
    plan = kde.Plan(M, lo, hi, H[0], P_min=P)
    X = torch.randn(5000, 2, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    c = kde.kde_bin(X, lo, hi, M)
    d = kde.kde_fft_eval_multi(plan, 5000, H, c)
    for h in list(range(min(nH, 5))) + [nH // 2, nH - 1]:
        one = kde.Plan(M, lo, hi, H[h], P_min=P)
        assert one.info.P == plan.info.P
        assert torch.equal(kde.kde_fft_eval(one, c, kde.kde_kernel_grid(one, 5000)), d[h]), h
