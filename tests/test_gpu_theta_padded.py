"""kde_lscv_theta_select on plans padded far beyond any support: the lag sums'
shared memory follows the widest support a candidate can have, not the
padding, so every plan that kde_plan_create accepts takes the call, and the
scores equal the host-built candidates' on the same plan."""
import numpy as np
import pytest

from paper_1508_02766_gb300 import kde
from paper_1508_02766_gb300 import learned as Lm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,P_min", [((64, 64), (128, 4096)), ((40, 256), (80, 4096)),
                                     ((64, 33), (4096, 3800)), ((48, 2048), (96, 4096)),
                                     ((64, 64), (128, 128))])
def test_padding_wider_than_any_support(M, P_min):
    lo, hi = [-6.0, -6.0], [6.0, 6.0]
    plan = kde.Plan(M, lo, hi, 0.01 * np.eye(2), P_min=P_min)
    ns = np.array([1000, 50])
    R = torch.rand(2, *plan.info.P, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    base = np.array([[-0.5, 0.3, -1.0], [-1.5, -0.6, -0.2]])
    offs = 0.5 * Lm.NEIGHBOUR_OFFSETS * Lm.STEP
    refs = Lm.normal_reference_thetas(ns)
    lscv = torch.empty(2, len(offs) + 1, dtype=torch.float64, device="cuda")
    kde.kde_lscv_theta_select(plan, ns, torch.tensor(base, dtype=torch.float32, device="cuda"),
                              [-9.0] * 3, [9.0] * 3, offs, refs, R, lscv=lscv)
    th = np.concatenate([base.astype(np.float32).astype(np.float64)[:, None] + offs, refs[:, None]], axis=1)
    ref = kde.kde_lscv_autocorr_batch(plan, [int(v) for v in ns], Lm.thetas_to_H(th), R).cpu().numpy()
    got = lscv.cpu().numpy()
    # the same FP32 lag sums from FP64 parameters that can differ in the last bit
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-6
