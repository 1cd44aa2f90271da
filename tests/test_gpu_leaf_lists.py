"""Lists of near leaves: by a warp per leaf (few leaves) and a thread per leaf
(more than two per resident warp), one leaf, two leaves, and leaves with more
near leaves or near siblings than a list holds, which walk the tree."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


# (points, dimension, points within eps of a point on average)
@pytest.mark.parametrize("n,d,near", [(1, 3, 4), (20, 2, 4), (40, 3, 4), (3000, 2, 5), (3000, 5, 5), (9000, 3, 2000),
                                      (6000, 2, 2500), (260000, 2, 4), (260000, 3, 5)])
@pytest.mark.parametrize("algo", ["fdbscan", "densebox"])
def test_uniform_points_match_oracle(n, d, near, algo):
    X = np.random.default_rng(n + d).uniform(0.0, 1.0, size=(n, d)).astype(np.float32)
    ball = {2: np.pi, 3: 4.0 * np.pi / 3.0, 5: 8.0 * np.pi ** 2 / 15.0}[d]
    eps = float(np.float32(min(0.5, (near / (n * ball)) ** (1.0 / d))))
    min_pts = 5 if near < 100 else near
    lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), eps, min_pts, algo=algo, want_core=True, sync=True)
    assert_matches_oracle(X, eps, min_pts, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())
