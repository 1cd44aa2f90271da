"""Dense cells of every size class of the classification: runs that a thread
walks (up to 64 points), that the block takes (more), that fit a tile (up to
32) or do not, at the end of the sorted order, in 2D to 5D and in batches."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 66, 255, 257, 1025, 3000]


def clumps(sizes, d, seed):
    """One tight clump per size on a lattice of spacing 1 (each inside one
    cell for eps 0.05), plus noise; shuffled."""
    r = np.random.default_rng(seed)
    parts = []
    for i, s in enumerate(sizes):
        centre = np.array([(i >> (2 * k)) & 3 for k in range(d)], dtype=np.float64) + 0.5
        parts.append(centre + r.uniform(-0.002, 0.002, size=(s, d)))
    parts.append(r.uniform(0.0, 4.0, size=(100, d)))
    pts = np.concatenate(parts).astype(np.float32)
    return pts[r.permutation(len(pts))]


@pytest.mark.parametrize("min_pts", [1, 2, 5, 33])
@pytest.mark.parametrize("d", [2, 3, 5])
def test_clumps_match_oracle(d, min_pts):
    X = clumps(SIZES, d, d)
    eps = float(np.float32(0.05))
    pts = torch.from_numpy(X).cuda()
    lab, core = gb.dbscan_run(pts, eps, min_pts, algo="densebox", want_core=True, sync=True)
    assert_matches_oracle(X, eps, min_pts, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())


@pytest.mark.parametrize("n", [64, 65, 257, 4097])
def test_all_points_in_one_cell(n):
    # one run to the end of the sorted order; wide enough for the guard to fail at the larger eps
    X = np.random.default_rng(n).uniform(0.0, 0.01, size=(n, 3)).astype(np.float32)
    for eps in (0.05, 0.011):
        e = float(np.float32(eps))
        lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), e, 4, algo="densebox", want_core=True, sync=True)
        assert_matches_oracle(X, e, 4, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())


def test_clumps_in_a_batch():
    inst = [(clumps(SIZES, 3, 7), 0.05, 5), (clumps([700, 64, 33], 2, 8), 0.05, 3), (clumps([40], 3, 9), 0.06, 2)]
    offs = np.cumsum([0] + [len(x) for x, _, _ in inst])
    flat = np.concatenate([x.ravel() for x, _, _ in inst])
    core = torch.empty(int(offs[-1]), dtype=torch.uint8, device="cuda")
    lab, core = gb.dbscan_run_batch(torch.from_numpy(flat).cuda(), offs, [x.shape[1] for x, _, _ in inst],
                                    [e for _, e, _ in inst], [m for _, _, m in inst], core_out=core)
    gb.stream_status()
    for b, (x, e, m) in enumerate(inst):
        s = slice(int(offs[b]), int(offs[b + 1]))
        assert_matches_oracle(x, float(np.float32(e)), m, gb.MODE_DBSCAN, lab[s].cpu().numpy(), core[s].cpu().numpy())


@pytest.mark.parametrize("d", [2, 3, 5])
def test_cell_near_the_box_of_a_tile_but_near_none_of_its_points(d):
    # two arms of isolated points whose box reaches a dense cell larger than a
    # tile: preprocessing's only candidate leaf, and it drops out for every query
    w = 1.0 / np.sqrt(d)  # cells of eps 1
    X = np.zeros((22 + 40, d))
    X[:11, 0] = X[11:22, 1] = 31.8 * w
    X[:11, 1] = X[11:22, 0] = 1.1 * np.arange(11)
    X[22:, :2] = 32.3 * w + np.random.default_rng(d).uniform(-0.1 * w, 0.1 * w, size=(40, 2))
    X = X.astype(np.float32)
    lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), 1.0, 5, algo="densebox", want_core=True, sync=True)
    assert_matches_oracle(X, 1.0, 5, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())
    assert (lab[:22] == -1).all() and (lab[22:] == 22).all()
