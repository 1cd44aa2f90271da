"""Sorts of one tile, by one block: edges of warps, of the keys per thread and
of the tile, one to eight passes, stable among equal keys; and whole runs of
one tile (keys packed with the index, and key-value pairs)."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 32, 33, 255, 256, 257, 511, 513, 1000, 4095, 4096, 4097])
@pytest.mark.parametrize("bits", [1, 9, 10, 27, 64])
def test_small_sorts_match_stable_argsort(n, bits):
    keys = np.random.default_rng(n + bits).integers(0, 1 << bits, size=n, dtype=np.uint64, endpoint=False) \
        if bits < 64 else np.random.default_rng(n).integers(0, 2**64 - 1, size=n, dtype=np.uint64, endpoint=True)
    keys[:: 3] = keys[0]
    k = torch.from_numpy(keys.view(np.int64).copy()).cuda()
    v = torch.arange(n, dtype=torch.int32, device="cuda")
    gb.sort_pairs_u64(k, v, bits)
    order = np.argsort(keys, kind="stable")
    assert (k.cpu().numpy().view(np.uint64) == keys[order]).all()
    assert (v.cpu().numpy() == order).all()


@pytest.mark.parametrize("n", [2, 100, 4096, 4097])
@pytest.mark.parametrize("algo", ["fdbscan", "densebox"])
@pytest.mark.parametrize("eps", [0.2, 1e-5])
def test_small_runs_match_oracle(n, algo, eps):
    X = np.random.default_rng(n).uniform(0.0, 1.0, size=(n, 3)).astype(np.float32)
    X[: n // 2] *= np.float32(1e-4)
    e = float(np.float32(eps))
    lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), e, 4, algo=algo, want_core=True, sync=True)
    assert_matches_oracle(X, e, 4, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())
