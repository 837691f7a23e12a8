"""FP64 2-D kernel grids formed by direct sums: supports of one lag, unequal
ones, more frequencies than a block has threads, both column layouts, Wand's
kernel, and either side of the line beyond which the grid is transformed;
every node against the oracle."""
import numpy as np
import pytest

from oracle import kde_oracle as O
from paper_1508_02766_gb300 import kde
from paper_1508_02766_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", ["lines", "simd"])
@pytest.mark.parametrize("M,L0,opts", [((40, 30), 1, {}), ((130, 20), 9, {}), ((20, 300), 5, {}),
                                       ((50, 60), 20, {"layout": "wand"}), ((60, 50), 12, {"range_mode": "per_axis"}),
                                       ((200, 180), 60, {}), ((200, 180), 100, {})])
def test_every_node(M, L0, opts, cols):
    w = W.small_case(M[0] + L0, 2, M, n=1500, precision="f64")
    lam = w.H[0, 0] if opts.get("range_mode") else np.linalg.eigvalsh(w.H).max()
    w.tau = (L0 - 0.5) * (w.hi[0] - w.lo[0]) / (M[0] - 1) / np.sqrt(lam)
    X = torch.from_numpy(np.ascontiguousarray(w.X)).cuda()
    dens, _, plan = kde.kde_eval(X, w.H, w.lo, w.hi, M, precision="f64", tau=w.tau, cols=cols, **opts)
    assert plan.info.L[0] == L0
    f, _, _, _ = O.binned_estimate(w.X, w.H, w.lo, w.hi, M, tau=w.tau, **opts)
    assert np.max(np.abs(dens.cpu().numpy() - f)) <= 1e-12 * np.max(np.abs(f))
