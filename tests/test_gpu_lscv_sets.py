"""A candidate set scored against many datasets as one product: scores and
pair sums equal the one-by-one calls bit for bit, at set counts either side
of the product's line, odd ones and more than one slab, with supports from
one lag to many, a group that is not full, both layouts, FP64 plans (always
one by one) and a support too wide for the product."""
import numpy as np
import pytest

from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cands(rng, count, lo, hi):
    R = np.zeros((count, 2, 2))
    R[:, 0, 0], R[:, 1, 1] = np.exp(rng.uniform(lo, hi, size=(2, count)))
    R[:, 1, 0] = rng.uniform(-1, 1, size=count) * R[:, 0, 0]
    return R @ R.transpose(0, 2, 1)


@pytest.mark.parametrize("nsets,M,count,wide,opts", [
    (7, (40, 33), 37, -0.9, {}), (8, (40, 33), 37, -0.9, {}), (9, (33, 70), 64, -0.4, {}),
    (65, (40, 33), 5, -1.5, {"layout": "wand"}), (300, (33, 40), 21, -1.0, {}),
    (12, (24, 20), 9, -1.0, {"precision": "f64"}), (8, (4, 1000), 3, 2.2, {}),
    (10, (64, 64), 1030, -1.2, {})])
def test_equal_one_by_one(nsets, M, count, wide, opts):
    rng = np.random.default_rng(nsets + count)
    lo, hi = [-4.0, -4.0], [4.0, 4.0 if M[1] < 1000 else 20.0]
    H = _cands(rng, count, -4.0, wide)
    big = max(2.0 * H, key=lambda h: np.linalg.eigvalsh(h).max())
    P = kde.kde_plan_info_compute(M, lo, hi, big, **opts).P
    plan = kde.Plan(M, lo, hi, H[0], P_min=P, **opts)
    cands = kde.LscvCands(plan, H)
    R = torch.rand(nsets, *plan.info.P, dtype=plan.real_dtype(), device="cuda",
                   generator=torch.Generator(device="cuda").manual_seed(1))
    ns = rng.integers(2, 10**6, size=nsets)
    S = torch.empty(nsets, count, 2, dtype=torch.float64, device="cuda")
    got = cands.score_batch(ns, R, pair_sums=S)
    for i in list(range(min(nsets, 10))) + [nsets - 1]:
        S1 = torch.empty(count, 2, dtype=torch.float64, device="cuda")
        one = cands.score(int(ns[i]), R[i], pair_sums=S1)
        assert torch.equal(one, got[i]) and torch.equal(S1, S[i]), i
