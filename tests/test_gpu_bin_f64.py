"""Binning of FP64 samples at sample counts where a warp's last lanes have
none, with samples outside the grid and on its last nodes: counts and the
number outside equal the oracle's."""
import numpy as np
import pytest

from oracle import kde_oracle as O
from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["direct", "tiled"])
@pytest.mark.parametrize("M", [(41,), (19, 23), (7, 9, 11)])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 127, 129, 4097])
def test_counts_equal_oracle(n, M, method):
    d = len(M)
    rng = np.random.default_rng(n + d)
    lo, hi = np.full(d, -1.0), np.linspace(1.0, 1.5, d)
    X = rng.uniform(-1.1, 1.6, size=(n, d))
    X[rng.integers(n, size=n // 8)] = hi          # last node on every axis
    X[rng.integers(n, size=n // 16)] = np.nan
    X[rng.integers(n, size=n // 16)] = -0.0
    X[0] = lo + 0.1                               # the oracle wants one sample inside
    nout = torch.zeros(1, dtype=torch.int64, device="cuda")
    c = kde.kde_bin(torch.from_numpy(X).cuda(), lo, hi, M, n_outside=nout, method=method)
    ref, out = O.bin_linear(X, lo, hi, M)
    assert np.array_equal(c.cpu().numpy(), ref)
    assert int(nout.item()) == out
