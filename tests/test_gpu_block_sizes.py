"""Block sizes of the traversal kernels one after another in a process, in both
directions: those from 672 threads on need more shared memory than a launch
gets by default, a limit that belongs to the kernel and not to the launch."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle
from workloads import blobs

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
def test_large_blocks_in_any_order(dim):
    X = blobs(6000, dim, dim, n_blobs=6, sigma=0.03)
    eps = float(np.float32(0.03))
    pts = torch.from_numpy(np.ascontiguousarray(X, dtype=np.float32)).cuda()
    ref = None
    try:
        for block in (1024, 768, 1024, 672, 64, 768, 1024):
            gb.set_tuning(block, 1.0)
            lab, core = gb.dbscan_run(pts, eps, 5, algo="densebox", want_core=True, sync=True)
            ref = assert_matches_oracle(X, eps, 5, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy(), ref=ref)
    finally:
        gb.set_tuning(0, 0.0)
