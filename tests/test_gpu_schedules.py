"""Which kernels a grid-schedule solve runs, shown by its launches and by the blocks its products
read, and that the solution is that of the matrix itself (PC_STORAGE_FULL).

Tolerances: solves to a residual of 1e-9 agree within 1e-5 (H.DV_RTOL); a few iterations of the
same recurrence differ by roundings, 1e-5 as well.
"""
import numpy as np
import pytest
import torch

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


def _cloth(pc, nx, ny):
    rest, tris, _ = wk.grid_piece(nx, ny, 0.01 * (nx - 1), 0.01 * (ny - 1), jitter=0.2, flip_prob=0.1, seed=21)
    x0 = rest.astype(np.float64)
    x0[:, 2] += 1e-4 * wk.normal(3, 1, len(rest))
    wl = wk.Workload("grid", rest, tris, np.array([0, nx - 1], np.int32), x0.astype(np.float32), np.zeros_like(rest),
                     1.0 / 200.0, wk.Material(), [], 3)
    cl = pc.Cloth(wl)
    return cl, cl.assemble()


def _solve(pc, cl, s, **kw):
    """dv, iterations, launches and the blocks a product read."""
    kw = {"tol": 1e-9, "precision": pc.PC_PREC_MIXED, "max_iter": 50000, "schedule": pc.PC_SCHED_GRID, **kw}
    dv = torch.zeros(cl.V * 3, device="cuda")
    pc.pc_spmv_stats(cl.ctx)
    pc.pc_set_profiling(cl.ctx, True)
    n0 = pc.pc_launch_count(cl.ctx)
    info, _ = pc.pc_pcg_solve(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"], dv,
                              pc.solve_opts(**kw), allow_not_converged=True)
    launches = pc.pc_launch_count(cl.ctx) - n0
    pc.pc_set_profiling(cl.ctx, False)
    return dv, info.iters, launches, pc.pc_spmv_stats(cl.ctx)[2]


# one patch; the edges of a 32-row slice; the last size whose patches stay on the SMs
@pytest.mark.parametrize("nx,ny", [(2, 2), (31, 2), (8, 4), (11, 3), (76, 64), (77, 64), (304, 240)])
def test_sizes_that_stay_on_the_sms(pc, nx, ny):
    cl, s = _cloth(pc, nx, ny)
    short = _solve(pc, cl, s, precision=pc.PC_PREC_FP32, max_iter=1)
    full = _solve(pc, cl, s, precision=pc.PC_PREC_FP32, tol=1e-5)
    # one launch whatever the iterations
    assert full[2] == short[2] and full[1] > short[1]
    assert full[3] < s["nnzb"] - cl.V or cl.V == 4
    general = _solve(pc, cl, s, storage=pc.PC_STORAGE_FULL)
    assert general[2] >= 2 * general[1]
    assert H.rel_l2(_np(_solve(pc, cl, s)[0]), _np(general[0])) <= H.DV_RTOL
    cl.close()


# the first size that streams its records, a ragged one, and as two kernels per iteration or three
@pytest.mark.parametrize("nx,ny,fuse", [(305, 240, True), (331, 287, True), (331, 287, False)])
def test_sizes_that_stream_their_records(pc, nx, ny, fuse):
    cl, s = _cloth(pc, nx, ny)
    dv, iters, launches, blocks = _solve(pc, cl, s, fuse=fuse)
    assert launches >= (2 if fuse else 3) * iters and blocks < s["nnzb"] - cl.V
    # too short for records: the copy without the diagonal
    short = _solve(pc, cl, s, fuse=fuse, tol=1e-12, precision=pc.PC_PREC_FP32, max_iter=31)
    assert short[1] == 31 and short[3] == s["nnzb"] - cl.V
    general = _solve(pc, cl, s, fuse=fuse, storage=pc.PC_STORAGE_FULL)
    assert general[3] == s["nnzb"]
    assert H.rel_l2(_np(dv), _np(general[0])) <= H.DV_RTOL
    cl.close()


def _in_patch_block(s, row):
    """A block of `row` with its right neighbour (in its patch, on these grids) and its mirror."""
    rp, ci = _np(s["row_ptr"]), _np(s["col_idx"])

    def at(r, c):
        return rp[r] + int(np.nonzero(ci[rp[r]:rp[r + 1]] == c)[0][0])

    return at(row, row + 1), at(row + 1, row)


# resident and streamed records of a matrix that is not symmetric to the bit, in a block that its
# row keeps or in one that another row keeps for it; or that lacks one of the two blocks
@pytest.mark.parametrize("nx,ny", [(40, 40), (305, 240)])
@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("lacking", [False, True])
def test_matrix_that_records_cannot_hold(pc, nx, ny, side, lacking):
    cl, s = _cloth(pc, nx, ny)
    same = _solve(pc, cl, s, tol=1e-12, precision=pc.PC_PREC_FP32, max_iter=40)
    assert same[3] < s["nnzb"] - cl.V
    at = _in_patch_block(s, cl.V // 2)[side]
    vals = s["vals"].view(-1, 9)
    if lacking:
        # positive without the block as well: a diagonal as large as the largest entry on top
        rp, ci = _np(s["row_ptr"]), _np(s["col_idx"])[: s["nnzb"]]
        diag = torch.from_numpy(np.nonzero(ci == np.repeat(np.arange(cl.V), np.diff(rp)))[0]).cuda()
        top = torch.eye(3, device="cuda").reshape(9) * vals.abs().max()
        vals[diag] += top
        s["dres"].view(-1, 9).add_(top)
        n = s["nnzb"]
        keep = torch.arange(n, device="cuda") != at
        t = {k: torch.zeros_like(s[k]) for k in ("col_idx", "vals")}
        t["col_idx"][: n - 1] = s["col_idx"][:n][keep]
        t["vals"].view(-1, 9)[: n - 1] = vals[:n][keep]
        row = cl.V // 2 + side
        rp = s["row_ptr"].clone()
        rp[row + 1:] -= 1
        s = {**s, **t, "row_ptr": rp, "nnzb": n - 1}
    else:
        vals[at, 0] = torch.nextafter(vals[at, 0], vals[at, 0] * 2)
    for iters in (3, 40):
        dv, _, launches, blocks = _solve(pc, cl, s, tol=1e-12, precision=pc.PC_PREC_FP32, max_iter=iters)
        full = _solve(pc, cl, s, tol=1e-12, precision=pc.PC_PREC_FP32, max_iter=iters, storage=pc.PC_STORAGE_FULL)
        if iters == 3 or lacking:
            assert H.rel_l2(_np(dv), _np(full[0])) <= 1e-5
        # (of two blocks one of which is lacking, records can hold the other for its own row)
        if iters == 40 and not lacking:
            assert blocks == s["nnzb"] - cl.V and launches >= 2 * iters
    cl.close()


def test_fused_update_barrier_timeout_and_recovery_on_the_matrix(pc):
    """The fused update meets at a grid barrier once per iteration: with a one-cycle budget the solve
    reports PC_ERR_TIMEOUT, and with the default budget the same context gives the identical solve."""
    cl, s = _cloth(pc, 60, 50)
    ref, iters, launches, blocks = _solve(pc, cl, s, storage=pc.PC_STORAGE_FULL)
    assert launches >= 2 * iters and blocks == s["nnzb"]  # an update is a launch
    pc.pc_set_barrier_wait(cl.ctx, 1)
    with pytest.raises(pc.PcError) as e:
        _solve(pc, cl, s, storage=pc.PC_STORAGE_FULL)
    pc.pc_set_profiling(cl.ctx, False)
    assert e.value.status == pc.PC_ERR_TIMEOUT
    pc.pc_set_barrier_wait(cl.ctx, 0)
    again, n, _, _ = _solve(pc, cl, s, storage=pc.PC_STORAGE_FULL)
    assert n == iters and torch.equal(again, ref)
    cl.close()


# contacts that join the sheets' patches: records hold a few per vertex where they stay on the SMs,
# and half a contact per vertex streamed; the proximity query's several per vertex are the copy's
@pytest.mark.parametrize("n,layers,delta,records", [(64, 3, 5.5e-4, True), (150, 3, 5.5e-4, False),
                                                    (200, 3, 5.5e-4, False)])
def test_contacts_too_dense_for_records(pc, n, layers, delta, records):
    wl = wk.proximity_stack(n, layers, delta=delta)
    cl = pc.Cloth(wl)
    pairs, w = cl.proximity()
    assert pairs.shape[0] > wl.V
    s = cl.assemble(pairs, w)
    dv, iters, launches, blocks = _solve(pc, cl, s)
    assert (launches < iters) == records and (blocks < s["nnzb"] - cl.V) == records
    general = _solve(pc, cl, s, storage=pc.PC_STORAGE_FULL)
    assert H.rel_l2(_np(dv), _np(general[0])) <= H.DV_RTOL
    cl.close()
