"""The routes that the library chooses by size, density or layout, at the sizes where they
change: each against the FP64 oracle or against the general route.

Tolerances. Solutions: the solve's own FP64 residual |b - A dv| / |b|, formed from the
caller's matrix, meets tol (PC_PREC_MIXED's contract, whatever storage the products read);
at 1e-9 dv is within 1e-5 of the oracle (H.DV_RTOL, as the parity tests hold it). Values: the
per-block tolerance of _helpers. Patterns, proximity pairs and weights: exact.
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import mlp as omlp
from oracle import proximity as oprox
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


def _workload(rest, tris, pins, z_jitter=1e-4, seed=3):
    rest = np.ascontiguousarray(rest, np.float32)
    x0 = rest.astype(np.float64).copy()
    x0[:, 2] += z_jitter * wk.normal(seed, 1, rest.shape[0])
    return wk.Workload("custom", rest, np.ascontiguousarray(tris, np.int32), np.asarray(pins, np.int32),
                       x0.astype(np.float32), np.zeros_like(rest), 1.0 / 200.0, wk.Material(), [], seed)


def _grid(nx, ny, seed=21, extra=0):
    """A jittered nx x ny grid, with `extra` vertices that no triangle uses at its end."""
    rest, tris, _ = wk.grid_piece(nx, ny, 0.01 * (nx - 1), 0.01 * (ny - 1), jitter=0.2, flip_prob=0.1, seed=seed)
    if extra:
        rest = np.concatenate([rest, np.full((extra, 3), 0.5, np.float32)])
    return _workload(rest, tris, [0, nx - 1])


def _fan(n):
    """n triangles around one vertex (a cone), a second triangle pair over the same three
    vertices at its side."""
    a = 2.0 * np.pi * np.arange(n) / n
    rest = np.concatenate([[[0.0, 0.0, 0.02]], np.stack([0.1 * np.cos(a), 0.1 * np.sin(a), 0.0 * a], -1),
                           [[0.3, 0.0, 0.0], [0.35, 0.0, 0.0], [0.3, 0.05, 0.0]]])
    tris = [[0, 1 + k, 1 + (k + 1) % n] for k in range(n)]
    tris += [[n + 1, n + 2, n + 3], [n + 1, n + 3, n + 2]]
    return _workload(rest, tris, [1])


def _solve(pc, cl, s, tol=1e-6, **kw):
    dv = torch.zeros(cl.V * 3, device="cuda")
    n0 = pc.pc_launch_count(cl.ctx)
    info, st = pc.pc_pcg_solve(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"], dv,
                               pc.solve_opts(tol=tol, precision=pc.PC_PREC_MIXED, max_iter=50000, **kw))
    assert st == pc.PC_OK and info.rel_res <= tol
    return dv, info, pc.pc_launch_count(cl.ctx) - n0


# one patch; the edges of a 32-row slice; two patch sizes of the resident schedule (32 rows
# per SM, then 64); vertices without elements
@pytest.mark.parametrize("nx,ny,extra", [(2, 2, 0), (31, 1 + 1, 0), (8, 4, 0), (11, 3, 0), (76, 64, 0), (77, 64, 0),
                                         (40, 40, 7)])
@pytest.mark.parametrize("block", [False, True])
def test_resident_solve_matches_oracle(pc, nx, ny, extra, block):
    wl = _grid(nx, ny, extra=extra)
    cl, om = pc.Cloth(wl), oracle.Mesh.from_workload(wl)
    if extra:  # a row without mass has no equation: give those rows one
        s = cl.assemble()
        vals, dres = s["vals"].view(-1, 9), s["dres"].view(-1, 9)
        rp = _np(s["row_ptr"])
        for r in range(cl.V - extra, cl.V):
            vals[rp[r]] = torch.eye(3, device="cuda").reshape(9) * 1e-5
            dres[r] = vals[rp[r]]
        s["b"].view(-1, 3)[cl.V - extra:] = 2e-5
    else:
        s = cl.assemble()
    pre = pc.PC_PRECOND_BLOCK if block else pc.PC_PRECOND_JACOBI
    dv, info, launches = _solve(pc, cl, s, tol=1e-9, schedule=pc.PC_SCHED_GRID, precond=pre)
    assert launches < info.iters + 40  # iterations are not launches of their own
    general, _, _ = _solve(pc, cl, s, tol=1e-9, schedule=pc.PC_SCHED_GRID, precond=pre, storage=pc.PC_STORAGE_FULL)
    assert H.rel_l2(_np(dv), _np(general)) <= H.DV_RTOL
    if extra:
        np.testing.assert_allclose(_np(dv).reshape(-1, 3)[cl.V - extra:], 2.0, rtol=1e-5)
    else:
        rp, ci, vals, b = om.assemble(wl.x0.astype(np.float64), wl.v0.astype(np.float64), None, None, wl.h)
        ref, _, _ = oracle.pcg(rp, ci, vals, b, tol=1e-12)
        assert H.rel_l2(_np(dv), ref) <= H.DV_RTOL
    cl.close()


# the last size whose patches stay on the SMs and the first that streams them (480 rows x 152
# SMs = 72,960), a ragged one beyond, and two sheets with contacts between them
@pytest.mark.parametrize("nx,ny,layers", [(270, 270, 1), (304, 240, 1), (305, 240, 1), (331, 287, 1), (210, 210, 2)])
def test_patch_storage_solves_like_the_full_matrix(pc, nx, ny, layers):
    wl = (wk.stacked_sheets(nx, layers, seed=4, contact_frac=0.05) if layers > 1 else _grid(nx, ny))
    cl = pc.Cloth(wl)
    s = cl.assemble(*cl.contacts_device(0))
    dv, info, _ = _solve(pc, cl, s, tol=1e-9)
    general, ginfo, _ = _solve(pc, cl, s, tol=1e-9, storage=pc.PC_STORAGE_FULL)
    assert abs(info.iters - ginfo.iters) <= 0.12 * ginfo.iters + 5
    # both residuals are below 1e-9; the matrices' condition numbers are a few 1e5
    assert H.rel_l2(_np(dv), _np(general)) <= 1e-5
    again, _, _ = _solve(pc, cl, s, tol=1e-9)
    assert torch.equal(dv, again)  # tickets change who takes a patch, never a sum
    cl.close()


def test_matrix_that_is_not_symmetric_to_the_bit_is_read_as_it_is(pc):
    """One block changed by a unit in the last place: resident records (which keep one block
    for both of its rows) are not used, so the iterations are launches of their own."""
    cl = pc.Cloth(_grid(40, 40))
    s = cl.assemble()
    _, info, launches = _solve(pc, cl, s, schedule=pc.PC_SCHED_GRID)
    assert launches < info.iters
    rp, ci = _np(s["row_ptr"]), _np(s["col_idx"])
    r = cl.V // 2
    k = rp[r] + int(np.nonzero(ci[rp[r]:rp[r + 1]] == r + 1)[0][0])
    v = s["vals"].view(-1, 9)
    v[k, 0] = torch.nextafter(v[k, 0], v[k, 0] * 2)
    dv, info, launches = _solve(pc, cl, s, tol=1e-9, schedule=pc.PC_SCHED_GRID)
    assert launches >= 2 * info.iters
    full, _, _ = _solve(pc, cl, s, tol=1e-9, schedule=pc.PC_SCHED_GRID, storage=pc.PC_STORAGE_FULL)
    assert H.rel_l2(_np(dv), _np(full)) <= H.DV_RTOL
    cl.close()


# V = 16,384 is the largest scan in one CTA; 64 and 65 contacts at one vertex are the last row
# that is ordered in place and the first that sends the step to the sort
@pytest.mark.parametrize("nx,ny,star", [(129, 127, 0), (128, 128, 0), (31, 30, 63), (31, 30, 64), (31, 30, 65), (31, 30, 300)])
def test_pattern_and_values_with_many_contacts_at_a_vertex(pc, nx, ny, star):
    wl = _grid(nx, ny)
    rng = np.random.default_rng(nx + star)
    far = rng.permutation(np.arange(2 * (nx - 1) * (ny - 1) // 2, 2 * (nx - 1) * (ny - 1)))
    tri = wl.tris[far[: max(star, 40)]]
    p = np.zeros(len(tri), np.int32) + (5 if star else 0)
    if not star:
        p = rng.permutation(nx * ny // 3)[: len(tri)].astype(np.int32)
    pairs = np.concatenate([p[:, None], tri], 1).astype(np.int32)[rng.permutation(len(tri))]
    pairs = np.ascontiguousarray(pairs[[len(set(q)) == 4 for q in pairs.tolist()]])
    w = rng.dirichlet([1.0, 1.0, 1.0], len(pairs)).astype(np.float32)
    cl, om = pc.Cloth(wl, max_contacts=len(pairs)), oracle.Mesh.from_workload(wl)
    s = cl.assemble(torch.from_numpy(pairs).cuda(), torch.from_numpy(w).cuda())
    rp, ci, vals, b = om.assemble(wl.x0.astype(np.float64), wl.v0.astype(np.float64), pairs, w, wl.h)
    np.testing.assert_array_equal(_np(s["row_ptr"]), rp)
    np.testing.assert_array_equal(_np(s["col_idx"])[: s["nnzb"]], ci)
    assert H.block_errors(rp, ci, _np(s["vals"])[: 9 * s["nnzb"]], vals).max() <= 0
    cl.close()


# the edges of a tile of 32 rows; a vertex with many elements, and an element that meets a
# vertex twice (a row of hundreds of blocks: the star of 300 above)
@pytest.mark.parametrize("wl", [_grid(5, 3), _grid(16, 1 + 1), _grid(11, 3), _grid(17, 3), _fan(8), _fan(40)],
                         ids=["15", "32", "33", "51", "fan8", "fan40"])
def test_values_at_tile_edges_match_oracle(pc, wl):
    cl, om = pc.Cloth(wl), oracle.Mesh.from_workload(wl)
    rng = np.random.default_rng(1)
    v = torch.from_numpy((0.1 * rng.normal(size=(cl.V, 3))).astype(np.float32)).cuda()
    s = cl.assemble(v=v)
    rp, ci, vals, b = om.assemble(wl.x0.astype(np.float64), _np(v).astype(np.float64), None, None, wl.h)
    np.testing.assert_array_equal(_np(s["col_idx"])[: s["nnzb"]], ci)
    got = _np(s["vals"])[: 9 * s["nnzb"]]
    assert H.block_errors(rp, ci, got, vals).max() <= 0
    # the pair of triangles over the same three vertices is folded flat: the sign of its angle
    # (+pi or -pi), and with it its force, hangs on a rounding
    n = cl.V - (3 if (np.sort(wl.tris[-1]) == np.sort(wl.tris[-2])).all() else 0)
    assert H.rel_l2(_np(s["b"]).reshape(-1, 3)[:n], b.reshape(-1, 3)[:n]) <= 1e-5
    A = {(r, c): got[9 * k: 9 * k + 9].reshape(3, 3) for r in range(cl.V) for k, c in
         zip(range(rp[r], rp[r + 1]), ci[rp[r]:rp[r + 1]])}
    assert all(np.array_equal(B, A[c, r].T) for (r, c), B in A.items())
    cl.close()


# a vertex shared by many separate fans of eight triangles: a row of hundreds of blocks, each
# with few contributions; with contacts between the fans and without
@pytest.mark.parametrize("fans,contacts", [(59, False), (60, False), (60, True), (140, False), (140, True)])
def test_values_of_a_vertex_with_many_blocks(pc, fans, contacts):
    a = 2.0 * np.pi * np.arange(8) / 8
    ring = np.stack([0.1 * np.cos(a), 0.1 * np.sin(a), 0.0 * a], -1)
    rest = np.concatenate([[[0.0, 0.0, 0.02]]] + [ring + [0.0, 0.0, 0.002 * k] for k in range(fans)])
    tris = [[0, 1 + 8 * f + k, 1 + 8 * f + (k + 1) % 8] for f in range(fans) for k in range(8)]
    wl = _workload(rest, tris, [3])
    cl, om = pc.Cloth(wl, max_contacts=fans), oracle.Mesh.from_workload(wl)
    pairs = w = tp = tw = None
    if contacts:
        pairs = np.array([[1 + 8 * f, *tris[8 * (f + 1) + 3]] for f in range(fans // 2)], np.int32)
        w = np.random.default_rng(2).dirichlet([1.0, 1.0, 1.0], len(pairs)).astype(np.float32)
        tp, tw = torch.from_numpy(pairs).cuda(), torch.from_numpy(w).cuda()
    s = cl.assemble(tp, tw)
    rp, ci, vals, b = om.assemble(wl.x0.astype(np.float64), wl.v0.astype(np.float64), pairs, w, wl.h)
    np.testing.assert_array_equal(_np(s["col_idx"])[: s["nnzb"]], ci)
    assert H.block_errors(rp, ci, _np(s["vals"])[: 9 * s["nnzb"]], vals).max() <= 0
    cl.close()


@pytest.mark.parametrize("layers,delta", [(3, 5.5e-4), (5, 1.2e-3), (2, 5e-5)])
def test_proximity_of_many_and_of_far_apart_triangles(pc, layers, delta):
    """More pairs at a vertex than the counting pass remembers (vertices right above each
    other, delta over twice the gap), and a second piece so far away that the cells outnumber the table."""
    wl = wk.stacked_sheets(14, layers, seed=5, contact_frac=0.0, jitter=0.0, flip_prob=0.0)
    if delta < 1e-4:
        wl.rest = wl.rest.copy()
        wl.rest[wl.V // 2:, 0] += 30.0
        wl.x0 = wl.rest.copy()
        wl.x0[wl.V // 2:, 2] += 20.0
        wl.x0[:, 2] += np.where(np.arange(wl.V) % 2, 2e-5, 0.0).astype(np.float32)
    cl = pc.Cloth(wl, max_contacts=400 * wl.V)
    x = torch.from_numpy(wl.x0).cuda()
    pairs = torch.zeros(400 * wl.V, 4, dtype=torch.int32, device="cuda")
    w = torch.zeros(400 * wl.V, 3, device="cuda")
    n = pc.pc_proximity_query(cl.ctx, x, delta, pairs, w)
    ref_pairs, ref_w = oprox.query(wl.x0, wl.tris, delta)
    assert n == len(ref_pairs)
    np.testing.assert_array_equal(_np(pairs)[:n], ref_pairs)
    np.testing.assert_array_equal(_np(w)[:n].view(np.uint32), np.asarray(ref_w, np.float32).view(np.uint32))
    if delta == 1.2e-3:
        assert np.bincount(_np(pairs)[:n, 0]).max() > 16
    cl.close()


# a tile fuller than the 16-block stages in a matrix whose average row is below 15 blocks
@pytest.mark.parametrize("diff", [True, False])
def test_plain_product_with_an_overfull_tile(pc, diff):
    wl = _grid(40, 40)
    rng = np.random.default_rng(2)
    tri = wl.tris[rng.permutation(np.arange(2000, wl.T))[:150]]
    pairs = np.ascontiguousarray(np.concatenate([np.full((150, 1), 40, np.int32), tri], 1))
    w = rng.dirichlet([1.0, 1.0, 1.0], 150).astype(np.float32)
    cl = pc.Cloth(wl, max_contacts=150)
    s = cl.assemble(torch.from_numpy(pairs).cuda(), torch.from_numpy(w).cuda())
    rp, ci = _np(s["row_ptr"]), _np(s["col_idx"])[: s["nnzb"]]
    assert s["nnzb"] <= 15 * cl.V and max(rp[min(r + 32, cl.V)] - rp[r] for r in range(0, cl.V, 32)) > 512
    x = rng.normal(size=3 * cl.V).astype(np.float32)
    y = torch.zeros(3 * cl.V, device="cuda")
    pc.pc_bsr_spmv(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"] if diff else None,
                   torch.from_numpy(x).cuda(), y)
    vals = _np(s["vals"])[: 9 * s["nnzb"]].astype(np.float64).reshape(-1, 3, 3)
    rows = np.repeat(np.arange(cl.V), np.diff(rp))
    X = x.astype(np.float64).reshape(-1, 3)
    u = X[ci] - X[rows] if diff else X[ci]
    terms = np.einsum("kab,kb->ka", vals, u)
    mag = np.einsum("kab,kb->ka", np.abs(vals), np.abs(u))
    ref, bound = np.zeros((cl.V, 3)), np.zeros((cl.V, 3))
    np.add.at(ref, rows, terms)
    np.add.at(bound, rows, mag)
    if diff:
        D = _np(s["dres"]).astype(np.float64).reshape(-1, 3, 3)
        ref += np.einsum("kab,kb->ka", D, X)
        bound += np.einsum("kab,kb->ka", np.abs(D), np.abs(X))
    # a row of n blocks: (3 n + 3) rounded terms in any order, at most 1e-5 of their magnitudes
    assert (np.abs(_np(y).reshape(-1, 3) - ref) <= 1e-5 * bound + 1e-30).all()
    cl.close()


# one row, the edges of a tile, more tiles than CTAs; feature rows that are not 16-byte aligned
@pytest.mark.parametrize("n", [1, 127, 128, 129, 4 * 152 * 128 + 1])
@pytest.mark.parametrize("offset", [0, 1])
def test_inference_tiles_and_alignment(pc, n, offset):
    rng = np.random.default_rng(n)
    params, stats = omlp.init_params(1), np.concatenate([np.zeros(12), np.ones(12), np.zeros(3), np.ones(3)])
    feat = rng.normal(size=(n, 12)).astype(np.float32)
    buf = torch.zeros(12 * n + offset, device="cuda")
    buf[offset:] = torch.from_numpy(feat.reshape(-1)).cuda()
    out = torch.full((n, 3), float("nan"), device="cuda")
    pc.pc_mlp_infer(n, torch.from_numpy(params.astype(np.float32)).cuda(), torch.from_numpy(stats.astype(np.float32)).cuda(),
                    buf[offset:], None, None, out)
    ref = omlp.predict(params.astype(np.float32), stats, feat, np.zeros((n, 3)), bf16=True)
    assert H.rel_l2(_np(out), ref) <= 2e-3  # as tests/test_gpu_mlp.py
