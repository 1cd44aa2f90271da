"""Dense cells at the limits of the classification's classes: runs of equal keys
of up to 8 points are walked by a thread, of up to 1,024 by a warp, longer ones
by the block; at each limit the walk ends with its class full and the next key
another, at the end of the order as well, and a block's list of runs for its
warps is full where nine-point runs follow each other."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu

LIMITS = [7, 8, 9, 10, 1023, 1024, 1025, 1026]


@pytest.fixture(autouse=True)
def cells_of_side_eps_over_root_d():
    gb.set_tuning(128, 1.0)
    yield
    gb.set_tuning(0, 0.0)


def cells(sizes, d, eps, seed):
    """One cell of the grid for each size, filled with so many points, several
    cells apart; a point at the origin fixes the grid. Shuffled."""
    r = np.random.default_rng(seed)
    h = eps / np.sqrt(d)
    parts = [np.zeros((1, d))]
    for i, s in enumerate(sizes):
        cell = np.array([7 * ((i >> (2 * k)) & 3) + 7 for k in range(d)])
        parts.append((cell + 0.5 + r.uniform(-0.1, 0.1, size=(s, d))) * h)
    X = np.concatenate(parts).astype(np.float32)
    return X[r.permutation(len(X))]


@pytest.mark.parametrize("min_pts", [2, 7, 9, 1024])
@pytest.mark.parametrize("d", [2, 3, 5])
def test_one_cell_of_each_size(d, min_pts):
    eps = float(np.float32(0.05))
    X = cells(LIMITS, d, eps, d)
    lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), eps, min_pts, algo="densebox", want_core=True, sync=True)
    assert gb.last_stats()["dense_cells"] == sum(s >= min_pts for s in LIMITS)
    assert_matches_oracle(X, eps, min_pts, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())


@pytest.mark.parametrize("n", LIMITS + [2048, 2049])
def test_all_points_in_one_cell(n):
    X = np.random.default_rng(n).uniform(0.0, 0.01, size=(n, 3)).astype(np.float32)
    for eps in (0.05, 0.011):  # the guard passes, and fails
        e = float(np.float32(eps))
        lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), e, 4, algo="densebox", want_core=True, sync=True)
        assert_matches_oracle(X, e, 4, gb.MODE_DBSCAN, lab.cpu().numpy(), core.cpu().numpy())


def test_rounds_full_of_nine_point_runs():
    # One nine-point clump in every 7th cell of each axis, and a point far off
    # that fixes the grid's origin: after it every run has nine points, so some
    # round of 16 x 256 positions starts with a run and holds 456 of them.
    side, eps = 102, float(np.float32(1e-3))
    h = eps / np.sqrt(3.0)
    count = side ** 3
    assert 1 + 9 * count > 15 * 152 * 16 * 256, "16 steps a round"
    g = torch.Generator(device="cuda").manual_seed(1)
    cell = torch.arange(count, device="cuda")
    at = torch.stack([cell % side, cell // side % side, cell // (side * side)], dim=1).double()
    centre = (at * 7.0 + 0.5) * h
    pts = centre[:, None, :] + (torch.rand(count, 9, 3, device="cuda", generator=g, dtype=torch.float64) - 0.5) * 0.2 * h
    pts = torch.cat([torch.full((1, 3), -10.0 * h, device="cuda", dtype=torch.float64), pts.reshape(-1, 3)]).float()
    owner = torch.cat([torch.full((1,), -1, device="cuda", dtype=torch.int64), cell.repeat_interleave(9)])
    order = torch.randperm(len(pts), device="cuda", generator=g)
    pts, owner = pts[order].contiguous(), owner[order]
    lab, core = gb.dbscan_run(pts, eps, 9, algo="densebox", want_core=True, sync=True)
    assert gb.last_stats()["dense_cells"] == count
    first = torch.full((count,), 1 << 40, device="cuda", dtype=torch.int64)
    index = torch.arange(len(pts), device="cuda")
    first.scatter_reduce_(0, owner.clamp(min=0), torch.where(owner >= 0, index, 1 << 40), "amin")
    want = torch.where(owner >= 0, first[owner.clamp(min=0)], -1)
    assert torch.equal(lab.long(), want) and torch.equal(core.bool(), owner >= 0)
