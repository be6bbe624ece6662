"""The proximity query where coordinates are large beside the contact thickness: pairs and
weights bit for bit those of the oracle's FP32 test over every vertex and triangle."""
import numpy as np
import pytest
import torch

from oracle import proximity as px
from paper_2008_00409_gb300 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    from paper_2008_00409_gb300 import build
    build.build()
    from paper_2008_00409_gb300 import pcloth
    return pcloth


def _query(pc, x, tris, delta):
    """Pairs and weights of a mesh of separate triangles at positions x."""
    x = np.ascontiguousarray(x, np.float32)
    rest = np.zeros_like(x)  # any valid rest shape: right-angled triangles side by side
    rest[:, 0] = np.arange(len(x)) // 3 * 2.0 + (np.arange(len(x)) % 3 == 1)
    rest[:, 1] = np.arange(len(x)) % 3 == 2
    wl = wk.Workload("separate", rest, np.ascontiguousarray(tris, np.int32), np.zeros(0, np.int32), x,
                     np.zeros_like(x), 1.0 / 200.0, wk.Material(), [], 1)
    cl = pc.Cloth(wl, max_contacts=100000)
    got_p, got_w = cl.proximity(delta)
    got = got_p.cpu().numpy(), got_w.cpu().numpy()
    cl.close()
    return got


def _brute(x, tris, delta):
    """The oracle's FP32 test on all pairs (its query looks within boxes grown by twice delta,
    which the rounding of large coordinates exceeds)."""
    pairs, weights = [], []
    for p in range(len(x)):
        w, d2 = px.closest_point(x[p][None], *(x[tris[:, k]] for k in range(3)))
        hit = np.nonzero((d2 < np.float32(delta) * np.float32(delta)) & (tris != p).all(1))[0]
        pairs.append(np.concatenate([np.full((len(hit), 1), p), tris[hit]], 1))
        weights.append(w[hit])
    return np.concatenate(pairs).astype(np.int32), np.concatenate(weights)


# (seed, which corner of the long triangles lies at the vertices): with a slack that grows with the
# vertex's own coordinates only, a box test drops a few of these pairs
@pytest.mark.parametrize("seed,corner", [(1, 1), (2, 2)])
def test_long_triangles_with_a_corner_at_a_vertex_near_the_origin(pc, seed, corner):
    rng = np.random.default_rng(seed)
    n, delta, length = 250, 3e-5, 1000.0
    at = np.full((n, 3), 0.5)
    b = at + delta * rng.normal(size=(n, 3))
    d, e = (-np.abs(rng.normal(size=(n, 3))) for _ in range(2))
    a = b + length * d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(0.3, 1.0, (n, 1))
    c = b + length * e / np.linalg.norm(e, axis=1)[:, None]
    long = np.roll(np.stack([b, a, c], 1), corner, axis=1)
    p = at + 2.0 * delta * rng.normal(size=(n, 3))
    small = np.stack([p, p + [40.0, 0.0, 0.0], p + [0.0, 40.0, 0.0]], 1)
    x = np.concatenate([long, small]).reshape(-1, 3).astype(np.float32)
    tris = np.arange(6 * n).reshape(-1, 3)
    want_p, want_w = _brute(x, tris, delta)
    # the case is what it says: pairs whose vertex the grown box and such a slack leave out
    A = x[want_p[:, 1:]]
    lo, hi, q = A.min(1) - 1.01 * delta, A.max(1) + 1.01 * delta, x[want_p[:, 0]]
    slack = (0.05 * delta + 1e-6 * np.abs(q).sum(1))[:, None]
    assert ((q < lo - slack) | (q > hi + slack)).any(1).sum() > 0
    got_p, got_w = _query(pc, x, tris, delta)
    np.testing.assert_array_equal(got_p, want_p)
    np.testing.assert_array_equal(got_w.view(np.uint32), want_w.view(np.uint32))


def test_triangles_at_both_ends_of_the_cell_range(pc):
    """Cells are of one box's size and their coordinates reach from -2^20 to 2^20 - 1: triangles in
    both of these along every axis, and a pair at each end."""
    delta, e = 0.125, 0.75
    tri = np.array([[0.0, 0.0, 0.0], [e, 0.0, 0.0], [0.0, e, 0.0]])
    # at the origin: the largest grown box, whose edge is the cell; there 2 pads are exact
    cell = np.float32((np.float32(e) + 2 * np.float32(delta * np.float32(1.01))) * np.float32(1.001))
    end = (np.floor((2.0 ** 20 - 0.5) * cell * 8) / 8)  # whole eighths: units in the last place there
    x = []
    for base in (np.zeros(3), [end - 1.0, end - 1.0, end - 0.25], np.full(3, -end + 0.25)):
        x += [tri + base, tri + base + [0.25, 0.25, 0.0]]
    x = np.concatenate(x).astype(np.float32)
    pad = np.float32(np.float32(delta) * np.float32(1.01))
    lo, hi = np.floor((x.min(0) - pad) / cell), np.floor((x.max(0) + pad) / cell)
    assert (hi == 2 ** 20 - 1).all() and (lo == -2 ** 20).all()
    tris = np.arange(len(x)).reshape(-1, 3)
    want_p, want_w = _brute(x, tris, delta)
    assert set(want_p[:, 0] // 6) == {0, 1, 2}
    got_p, got_w = _query(pc, x, tris, delta)
    np.testing.assert_array_equal(got_p, want_p)
    np.testing.assert_array_equal(got_w.view(np.uint32), want_w.view(np.uint32))


def test_time_does_not_hang_on_empty_cells(pc):
    """Two sheets with hundreds of thousands of empty cells between them (inside the cell table) take
    no longer than the same sheets half a millimetre apart and half as much again."""
    took = []
    for gap in (5e-4, 0.1):
        wl = wk.stacked_sheets(301, 2, seed=4, gap=gap, contact_frac=0.0)
        cl = pc.Cloth(wl, max_contacts=4 * wl.V)
        times = []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            cl.proximity(5.5e-4)
            e[1].record()
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]))
        took.append(float(np.median(times[2:])))
        cl.close()
    assert took[1] <= 1.5 * took[0], took
