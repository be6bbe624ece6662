"""Patterns and values of steps in which vertices have many contacts: rows ordered by a thread, by a
warp, and the key sort, against the FP64 oracle (pattern exact, values
within the per-block tolerance of _helpers)."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2008_00409_gb300 import workloads as wk
from tests import _helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    from paper_2008_00409_gb300 import build
    build.build()
    from paper_2008_00409_gb300 import pcloth
    return pcloth


def _np(t):
    return t.detach().cpu().numpy()


def _check(pc, wl, pairs, seed):
    """Compares one assembly with the oracle's; returns the launches of the pattern call."""
    pairs = np.ascontiguousarray(pairs[[len(set(q)) == 4 for q in pairs.tolist()]], np.int32)
    w = np.random.default_rng(seed).dirichlet([1.0, 1.0, 1.0], len(pairs)).astype(np.float32)
    cl, om = pc.Cloth(wl, max_contacts=len(pairs)), oracle.Mesh.from_workload(wl)
    tp, tw, s = torch.from_numpy(pairs).cuda(), torch.from_numpy(w).cuda(), cl.alloc_system()
    n0 = pc.pc_launch_count(cl.ctx)
    pc.pc_assemble_pattern(cl.ctx, tp, tw, s["row_ptr"], s["col_idx"])
    launches = pc.pc_launch_count(cl.ctx) - n0
    cl.assemble(tp, tw, sysbuf=s)
    rp, ci, vals, b = om.assemble(wl.x0.astype(np.float64), wl.v0.astype(np.float64), pairs, w, wl.h)
    np.testing.assert_array_equal(_np(s["row_ptr"]), rp)
    np.testing.assert_array_equal(_np(s["col_idx"])[: s["nnzb"]], ci)
    assert H.block_errors(rp, ci, _np(s["vals"])[: 9 * s["nnzb"]], vals).max() <= 0
    assert H.rel_l2(_np(s["b"]), b) <= 1e-5
    cl.close()
    return launches, pairs


# the last row of a thread and the first of a warp (24 where there are few rows), the last of the
# warps and the first that is sorted; a vertex on both sides of its contacts
@pytest.mark.parametrize("star", [8, 24, 25, 65, 128, 129, 300, 1024, 1025])
def test_one_vertex_with_many_contacts(pc, star):
    wl = wk.square_cloth(48, seed=2, contact_frac=0.0)
    rng = np.random.default_rng(star)
    hub = 20 * 48 + 20
    far = rng.permutation(np.nonzero((wl.tris > 30 * 48).all(1))[0])
    own = wl.tris[np.nonzero((wl.tris == hub).any(1))[0][0]]
    n = star // 2
    others = rng.permutation(np.setdiff1d(np.arange(48 * 48), own))[:n]
    pairs = np.concatenate([np.concatenate([np.full((star - n, 1), hub), wl.tris[far[: star - n]]], 1),
                            np.concatenate([others[:, None], np.tile(own, (n, 1))], 1)])
    launches, used = _check(pc, wl, rng.permutation(pairs), star)
    assert (used == hub).sum() == star
    # a sort takes tens of launches
    assert (launches <= 10) == (star <= 1024), launches


# every vertex with a few dozen contacts, rows of unequal length side by side; few rows (4 per warp)
# and many (32, a thread for up to 64)
@pytest.mark.parametrize("n,per", [(20, 12.0), (64, 12.0), (64, 40.0), (281, 3.0)])
def test_every_vertex_with_many_contacts(pc, n, per):
    wl = wk.square_cloth(n, seed=2, contact_frac=0.0)
    rng = np.random.default_rng(n)
    P = int(per * wl.V)
    p = np.minimum((wl.V * rng.random(P) ** 2).astype(np.int64), wl.V - 1)
    pairs = np.concatenate([p[:, None], wl.tris[rng.integers(0, wl.T, P)]], 1)
    launches, used = _check(pc, wl, pairs, n)
    most = np.bincount(used.reshape(-1), minlength=wl.V).max()
    assert (launches <= 10) == (most <= 1024), (launches, most)


# the edges of a tile of eight rows and of two; a tile of 32 (many rows: 281 x 281 above)
@pytest.mark.parametrize("nx,ny", [(4, 2), (3, 3), (5, 3), (4, 4), (17, 1 + 1)])
def test_values_at_edges_of_small_tiles(pc, nx, ny):
    rest, tris, _ = wk.grid_piece(nx, ny, 0.01 * (nx - 1), 0.01 * (ny - 1), jitter=0.2, flip_prob=0.1, seed=nx)
    wl = wk.Workload("tile", rest, tris, np.array([0], np.int32), rest.copy(), np.zeros_like(rest), 1.0 / 200.0,
                     wk.Material(), [], 1)
    p = np.arange(wl.V, dtype=np.int64)[:, None]
    pairs = np.concatenate([np.repeat(p, wl.T, 0), np.tile(wl.tris, (wl.V, 1))], 1)
    _check(pc, wl, pairs, nx)


def test_values_of_few_rows_with_many_contacts_in_time(pc):
    """12,288 rows of 48 contacts beside four times as many of 47: the few rows' contacts are chains
    of loads that nothing else hides (32 rows per CTA and one contact at a time: 0.44 of the many
    rows' time; now 0.34)."""
    took = []
    for n, delta in ((64, 8e-3), (128, 3e-3)):
        wl = wk.proximity_stack(n, 3, delta=delta, per_vertex=40.0)
        cl = pc.Cloth(wl)
        pairs, w = cl.proximity()
        s = cl.assemble(pairs, w)
        times = []
        for _ in range(31):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            pc.pc_assemble_values(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], cl.x, cl.v, pairs, w, cl.h, s["vals"],
                                  s["b"], s["dres"])
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        took.append(float(np.median(times[3:])))
        cl.close()
    assert took[0] <= 0.4 * took[1], took
