"""The number of BVH leaves against the definition of the tiles: the maximal
subtrees of at most 32 points of the sorted points' radix tree (equal keys
told apart by position), at sizes around the parts that the leaf kernels give
a warp (windows of 32 positions, two at a time) and a block."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


def tiles(keys):
    """Leaves of the radix tree over the sorted keys with position tie-breaks."""
    words = [(int(k) << 32) | i for i, k in enumerate(keys)]
    count, stack = 0, [(0, len(words))]
    while stack:
        a, b = stack.pop()
        if b - a <= 32:
            count += 1
            continue
        bit = (words[a] ^ words[b - 1]).bit_length() - 1
        lo, hi = a, b - 1  # first position of [a, b) with the bit set
        while hi - lo > 1:
            mid = (lo + hi) // 2
            if (words[mid] >> bit) & 1:
                hi = mid
            else:
                lo = mid
        stack += [(a, hi), (hi, b)]
    return count


@pytest.mark.parametrize("dup", [False, True])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 1023, 1024, 1025, 2047, 2049, 20000])
def test_leaf_count(n, dup):
    r = np.random.default_rng(n)
    X = r.uniform(0.0, 1.0, size=(n, 2)).astype(np.float32)
    if dup:  # long runs of equal keys
        X = X[r.integers(0, max(1, n // 50), size=n)]
    pts = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    gb.dbscan_run(pts, 0.01, 3, algo="fdbscan", sync=True)
    m = gb.last_stats()["leaves"]
    lo, hi = X.min(axis=0), X.max(axis=0)
    keys = np.sort(gb.morton_codes(pts, lo, hi, 16).cpu().numpy())
    assert m == tiles(keys)
