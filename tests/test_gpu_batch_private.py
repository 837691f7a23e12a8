"""Staged ragged batches whose problems bin into block-private counts: grids of
both shared-memory classes and above them, sample counts either side of the
rule and of a chunk, samples outside; densities equal the persistent form's
(direct adds of the same integers) bit for bit, and the oracle's."""
import numpy as np
import pytest

from oracle import kde_oracle as O
from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_staged_equals_persistent(prec):
    rng = np.random.default_rng(4)
    sizes = [((8, 9), 4096 + 8 * 72 + e) for e in (-1, 0, 5000)]
    sizes += [((64, 96), 70_001), ((64, 97), 90_000), ((128, 128), 200_000), ((128, 192), 210_000),
              ((128, 193), 210_000), ((20, 20), 7)]
    probs, Xs = [], []
    for M, n in sizes:
        X = rng.normal(size=(n, 2))
        X[rng.integers(n, size=n // 50)] = 3.0
        Xs.append(X.astype(np.float32 if prec == "f32" else np.float64))
        probs.append((M, [-3.0, -3.0], [3.0, 3.0], np.array([[0.05, 0.03], [0.03, 0.06]]), n))
    bp = kde.BatchPlan(probs, precision=prec)
    X = torch.from_numpy(np.concatenate(Xs)).cuda()
    bp.set_mode("persistent")
    a = bp.eval(X).clone()
    bp.set_mode("staged")
    b = bp.eval(X)
    assert torch.equal(a, b)
    off = 0
    for (M, lo, hi, H, n), x in zip(probs, Xs):
        got = b[off:off + M[0] * M[1]].reshape(M).cpu().numpy()
        off += M[0] * M[1]
        if n < 10_000:
            f, _, _, _ = O.binned_estimate(x, H, lo, hi, M)
            assert np.max(np.abs(got - f)) <= (1e-12 if prec == "f64" else 1e-5) * np.max(np.abs(f))
