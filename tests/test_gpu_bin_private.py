"""Binning onto few cells (block-private counts in shared memory): sample
counts either side of the rule that takes it, the largest grid it takes and
the first it leaves, blocks that flush twice, samples outside and on the last
nodes, adding into existing counts.  Counts equal the oracle's, or the tiled
method's (the same integers) where there are many samples."""
import numpy as np
import pytest

from oracle import kde_oracle as O
from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _samples(rng, n, d, dtype):
    X = rng.normal(size=(n, d)).astype(dtype)
    X[rng.integers(n, size=n // 64)] = 3.0      # the grid's last nodes
    X[rng.integers(n, size=n // 64)] = -3.0
    X[rng.integers(n, size=n // 256)] = np.nan
    return X


def _line(M):
    return 4096 + {1: 14, 2: 8, 3: 3}[len(M)] * int(np.prod(M))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("extra", [-1, 0, 1023])
@pytest.mark.parametrize("M", [(2,), (101,), (3, 2), (33, 41), (5, 7, 9), (2, 2, 2)])
def test_counts_equal_oracle(M, extra, dtype):
    d, n = len(M), _line(M) + extra
    X = _samples(np.random.default_rng(n), n, d, dtype)
    lo, hi = [-3.0] * d, [3.0] * d
    nout = torch.zeros(1, dtype=torch.int64, device="cuda")
    Xg = torch.from_numpy(X).cuda()
    c = kde.kde_bin(Xg, lo, hi, M, n_outside=nout)
    ref, out = O.bin_linear(X, lo, hi, M)
    assert np.array_equal(c.cpu().numpy(), ref) and int(nout.item()) == out
    kde.kde_bin(Xg, lo, hi, M, counts=c, n_outside=nout, accumulate=True)
    assert np.array_equal(c.cpu().numpy(), 2 * ref) and int(nout.item()) == 2 * out


@pytest.mark.parametrize("M,n", [((24576,), 400_000), ((24577,), 400_000), ((128, 192), 300_000),
                                 ((128, 128), 5_300_000), ((29, 28, 30), 150_001), ((40,), 11_000_000)])
def test_counts_equal_tiled(M, n):
    d = len(M)
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(n, d, device="cuda", generator=g)
    lo, hi = [-3.0] * d, [3.0] * d
    no = torch.zeros(2, dtype=torch.int64, device="cuda")
    a = kde.kde_bin(X, lo, hi, M, n_outside=no[:1])
    b = kde.kde_bin(X, lo, hi, M, n_outside=no[1:], method="tiled")
    assert torch.equal(a, b) and int(no[0]) == int(no[1])
