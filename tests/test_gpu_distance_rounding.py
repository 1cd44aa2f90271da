"""Pairs at eps to the last bit. Adjacency is fl(...fl(fl(d0 d0) + fl(d1 d1))...)
<= fl(eps eps), every product and sum rounded by itself; a fused multiply-add
gives another last bit for about a fifth of all pairs. The pairs here are those
where the two fall on different sides of eps, each on its own except for
companions that only its first point is near: that point is core exactly where
the pair is adjacent."""
import numpy as np
import pytest

from tests.parity import assert_matches_oracle

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu

f32 = np.float32


def defined(d):
    s = d[:, 0] * d[:, 0]
    for k in range(1, d.shape[1]):
        s = s + d[:, k] * d[:, k]
    return s


def fused(d):
    x = d.astype(np.float64)  # a product of two floats is exact in 64 bits
    s = d[:, 0] * d[:, 0]
    for k in range(1, d.shape[1]):
        s = (s.astype(np.float64) + x[:, k] * x[:, k]).astype(f32)
    return s


def border_pairs(dim, eps, seed, want=600):
    """p and q, one pair per cell of a lattice of spacing 6 eps, whose defined
    and fused squared distances lie on different sides of eps squared."""
    r = np.random.default_rng(seed)
    side = int(1.0 / (6.0 * eps))
    p, q, used = [], [], set()
    for _ in range(40):
        m = 400000
        cell = r.integers(0, side, size=(m, dim))
        v = r.normal(size=(m, dim))
        v *= eps * r.uniform(1.0 - 2e-6, 1.0 + 2e-6, size=(m, 1)) / np.linalg.norm(v, axis=1, keepdims=True)
        a = ((cell + 0.5) * (6.0 * eps) + r.uniform(-0.2, 0.2, size=(m, dim)) * eps).astype(f32)
        b = (a + v).astype(f32)
        e2 = f32(eps) * f32(eps)
        for i in np.nonzero((defined(a - b) <= e2) != (fused(a - b) <= e2))[0]:
            c = tuple(cell[i])
            if c not in used:
                used.add(c)
                p.append(a[i])
                q.append(b[i])
        if len(p) >= want:
            break
    assert len(p) >= min(want, side**dim // 4), len(p)
    return np.array(p), np.array(q)


def clouds(dim, eps, min_pts, seed):
    """The pairs with min_pts - 2 companions of p each, opposite to q: within
    0.3 eps of p and farther than eps from q."""
    p, q = border_pairs(dim, eps, seed)
    r = np.random.default_rng(seed + 1)
    u = (q - p) / np.linalg.norm(q - p, axis=1, keepdims=True)
    parts = [p, q]
    for _ in range(min_pts - 2):
        parts.append((p - u * eps * r.uniform(0.1, 0.3, size=(len(p), 1))).astype(f32))
    X = np.concatenate(parts)
    core = np.zeros(len(X), dtype=bool)
    core[: len(p)] = defined(p - q) <= f32(eps) * f32(eps)
    if min_pts == 2:
        core[len(p):] = core[: len(p)]
    order = r.permutation(len(X))
    return X[order], core[order]


EPS = {2: 0.002, 3: 0.01, 5: 0.02, 8: 0.04}


@pytest.mark.parametrize("min_pts", [2, 3, 12, 40])
@pytest.mark.parametrize("algo", ["fdbscan", "densebox"])
@pytest.mark.parametrize("dim", [2, 3, 5, 8])
def test_pairs_at_eps(dim, algo, min_pts):
    eps = float(f32(EPS[dim]))
    X, core = clouds(dim, eps, min_pts, dim)
    lab, got = gb.dbscan_run(torch.from_numpy(X).cuda(), eps, min_pts, algo=algo, want_core=True, sync=True)
    got = got.cpu().numpy().astype(bool)
    assert (got == core).all(), f"{(got != core).sum()} of {len(X)} core flags"
    assert_matches_oracle(X, eps, min_pts, gb.MODE_DBSCAN, lab.cpu().numpy(), got)


@pytest.mark.parametrize("dim", [2, 3])
def test_pairs_at_eps_in_sweeps_and_batches(dim):
    eps = float(f32(EPS[dim]))
    sets = [clouds(dim, eps, m, dim + m) for m in (3, 12)]
    for X, _ in sets:
        pts = torch.from_numpy(X).cuda()
        lab, got = gb.dbscan_run_multi(pts, eps, [3, 12], want_core=True)
        gb.stream_status()
        for k, mp in enumerate((3, 12)):
            assert_matches_oracle(X, eps, mp, gb.MODE_DBSCAN, lab.reshape(2, -1)[k].cpu().numpy(),
                                  got.reshape(2, -1)[k].cpu().numpy())
    flat = torch.from_numpy(np.concatenate([X.ravel() for X, _ in sets])).cuda()
    offs = np.cumsum([0] + [len(X) for X, _ in sets])
    got = torch.empty(int(offs[-1]), dtype=torch.uint8, device="cuda")
    lab, got = gb.dbscan_run_batch(flat, offs, [dim, dim], [eps, eps], [3, 12], core_out=got)
    gb.stream_status()
    for b, (X, core) in enumerate(sets):
        assert (got[int(offs[b]):int(offs[b + 1])].cpu().numpy().astype(bool) == core).all()
