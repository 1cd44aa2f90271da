"""Lists of near leaves made by a thread per leaf: taken when there are more
leaves than two per warp of the launch, which has 1,216 blocks of 8 warps from
311,296 points on. The number of leaves is checked, so that no case changes to
the lists by warps unnoticed. The last case's leaves have more near leaves than
a list holds and walk the tree."""
import numpy as np
import pytest

import oracle
from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu

MOST_BY_WARPS = 2 * 1216 * 8


# (points, dimension, points within eps of a point on average)
@pytest.mark.parametrize("n,d,near", [(600_000, 2, 4), (600_000, 3, 4), (500_000, 5, 3), (500_000, 3, 400)])
def test_uniform_points_match_oracle(n, d, near):
    X = np.random.default_rng(n + d).uniform(0.0, 1.0, size=(n, d)).astype(np.float32)
    ball = {2: np.pi, 3: 4.0 * np.pi / 3.0, 5: 8.0 * np.pi ** 2 / 15.0}[d]
    eps = float(np.float32((near / (n * ball)) ** (1.0 / d)))
    min_pts = 5 if near < 100 else near
    ref = oracle.dbscan(X, eps, min_pts, oracle.MODE_DBSCAN)
    sets = oracle.border_sets(X, eps, ref[1], ref[0])
    pts = torch.from_numpy(X).cuda()
    for algo in ("fdbscan", "densebox"):
        lab, core = gb.dbscan_run(pts, eps, min_pts, algo=algo, want_core=True, sync=True)
        assert gb.last_stats()["leaves"] > MOST_BY_WARPS
        assert_matches_oracle(X, eps, min_pts, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy(), ref=ref,
                              sets=sets)
