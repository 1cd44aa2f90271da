"""Runs whose kernels overlap (up to 2^21 points), over and over on inputs in
turn with nothing waiting between them: every sweep's core flags are those of
single runs, and its core points' labels too; likewise slab-wise runs."""
import numpy as np
import pytest

from workloads import halo_eps, halos

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu

MPS = [2, 5, 10, 20]


def inputs(n):
    return [torch.from_numpy(halos(n, seed, n_halos=max(10, n // 340))).cuda() for seed in (n, n + 1)]


@pytest.mark.parametrize("n", [100_000, 524_287, 1_048_576, 2_097_152])
@pytest.mark.parametrize("algo", ["densebox", "fdbscan"])
def test_sweeps_repeat_and_agree_with_single_runs(n, algo):
    eps = halo_eps(n)
    refs = []
    for pts in inputs(n):
        runs = [gb.dbscan_run(pts, eps, m, algo=algo, want_core=True, sync=True) for m in MPS]
        refs.append((pts, torch.stack([r[1] for r in runs]), torch.stack([r[0] for r in runs])))
    wrong = torch.zeros(3, dtype=torch.int64, device="cuda")
    for _ in range(100):
        for pts, core, lab in refs:
            sl, sc = gb.dbscan_run_multi(pts, eps, MPS, algo=algo, want_core=True)
            wrong[0] += (sc != core).sum()
            wrong[1] += ((sl != lab) & (core != 0)).sum()
            wrong[2] += ((sl == -1) != (lab == -1)).sum()
    gb.stream_status()
    assert wrong.tolist() == [0, 0, 0]


def test_slabs_repeat():
    n = 300_000
    X = halos(n, 5, n_halos=900)
    eps = halo_eps(n)
    lab, core = gb.dbscan_run(torch.from_numpy(X).cuda(), eps, 10, want_core=True, sync=True)
    core = core.cpu().numpy().astype(bool)
    lab = lab.cpu().numpy()
    for _ in range(20):
        sl, sc = gb.dbscan_run_slabs(X, eps, 10, slab_points=40_000)
        np.testing.assert_array_equal(sc, core)
        np.testing.assert_array_equal(sl[core], lab[core])
