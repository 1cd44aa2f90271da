"""Batches at the edges of their row split (instances of no rows, one row, and
around the 32 and 128 rows of a step, many small ones per warp and one large
one), with key and row in one word and, at a tiny eps, too wide for that."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1], [0, 5, 0, 0, 31, 32, 33, 0], [127, 128, 129, 1, 2, 255, 256, 257, 4096, 3],
                                   [7] * 300, [20000, 1, 33]])
@pytest.mark.parametrize("spread", [1.0, 3.0e4])
@pytest.mark.parametrize("algo", ["fdbscan", "densebox"])
def test_batch_matches_oracle(sizes, spread, algo):
    r = np.random.default_rng(len(sizes))
    inst = []
    for k, s in enumerate(sizes):
        x = r.uniform(0.0, 1.0, size=(s, 2 + k % 2))
        x[: s // 2] *= 0.05
        if s > 2:
            x[-1] = spread  # far off: a fine grid over a wide range
        inst.append((x.astype(np.float32), float(np.float32(0.004 + 0.001 * (k % 3))), 2 + k % 4))
    offs = np.cumsum([0] + sizes)
    flat = torch.from_numpy(np.concatenate([x.ravel() for x, _, _ in inst])).cuda()
    core = torch.empty(int(offs[-1]), dtype=torch.uint8, device="cuda")
    lab, core = gb.dbscan_run_batch(flat, offs, [x.shape[1] for x, _, _ in inst], [e for _, e, _ in inst],
                                    [m for _, _, m in inst], core_out=core, algo=algo)
    gb.stream_status()
    for b, (x, e, m) in enumerate(inst):
        if len(x):
            s = slice(int(offs[b]), int(offs[b + 1]))
            assert_matches_oracle(x, e, m, gb.MODE_DBSCAN, lab[s].cpu().numpy(), core[s].cpu().numpy())
