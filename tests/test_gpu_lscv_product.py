"""The product kernel of the batched lag sums where its rule takes it (enough
work units times datasets for its few long items): scores equal the one-by-one calls bit for bit, on
either side of the line, with dataset counts that leave its tile of 16 part
empty, more than one launch, supports of one row, beyond one window and of the
widest kind, groups that are not full, and both layouts."""
import numpy as np
import pytest

from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cands(rng, count, lo, hi, M):
    """Bandwidths whose supports spread from lo to hi lags on a grid of unit
    spacing, along axis 1 in six steps (matrices of one width share a warp)."""
    s = np.exp(rng.uniform(np.log(lo), np.log(hi), size=(count, 2))) / 3.7
    s[:, 1] = np.geomspace(lo, hi, 6)[rng.integers(6, size=count)] / 3.7
    r = rng.uniform(-0.7, 0.7, size=count)
    H = np.zeros((count, 2, 2))
    H[:, 0, 0], H[:, 1, 1] = s[:, 0] ** 2, s[:, 1] ** 2
    H[:, 0, 1] = H[:, 1, 0] = r * s[:, 0] * s[:, 1]
    return H


@pytest.mark.parametrize("nsets,M,count,lo,hi,opts,product", [
    (8, (150, 150), 300, 10, 70, {}, True),
    (31, (90, 300), 400, 5, 200, {"range_mode": "wand"}, True),
    (17, (40, 50), 701, 1, 12, {"layout": "wand"}, True),
    (150, (3, 1100), 1000, 2, 400, {"range_mode": "wand"}, True),
    (257, (24, 30), 40, 2, 20, {}, True),
    (7, (150, 150), 400, 10, 70, {}, False),
    (8, (60, 60), 30, 2, 20, {}, False), (12, (256, 256), 32, 20, 190, {}, False)])
def test_equal_one_by_one(nsets, M, count, lo, hi, opts, product):
    rng = np.random.default_rng(nsets * count)
    glo, ghi = [0.0, 0.0], [M[0] - 1.0, M[1] - 1.0]
    H = _cands(rng, count, lo, hi, M)
    infos = [kde.kde_plan_info_compute(M, glo, ghi, a * h, **opts) for h in H for a in (1.0, 2.0)]
    P = np.max([i.P for i in infos], axis=0)
    plan = kde.Plan(M, glo, ghi, H[0], P_min=[int(p) for p in P], **opts)
    cands = kde.LscvCands(plan, H)
    R = torch.rand(nsets, *plan.info.P, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    ns = rng.integers(2, 10**6, size=nsets)
    S = torch.empty(nsets, count, 2, dtype=torch.float64, device="cuda")
    kde.profile_enable(True)
    got = cands.score_batch(ns, R, pair_sums=S)
    names = kde.profile_read()
    kde.profile_enable(False)
    assert ("kde_lscv_ac_sets_kernel" in names) == product
    for i in sorted({0, 1, nsets // 2, nsets - 2, nsets - 1}):
        S1 = torch.empty(count, 2, dtype=torch.float64, device="cuda")
        one = cands.score(int(ns[i]), R[i], pair_sums=S1)
        assert torch.equal(one, got[i]) and torch.equal(S1, S[i]), i
