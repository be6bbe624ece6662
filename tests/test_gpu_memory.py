"""Device memory that a context holds, as include/pcloth.h states it."""
import numpy as np
import pytest
import torch

from paper_2008_00409_gb300 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    from paper_2008_00409_gb300 import build
    build.build()
    from paper_2008_00409_gb300 import pcloth
    return pcloth


def _held(pc, wl, max_contacts):
    """Bytes that pc_create takes and keeps."""
    t = [torch.from_numpy(np.ascontiguousarray(a, d)).cuda()
         for a, d in ((wl.tris, np.int32), (wl.rest, np.float32), (wl.pins, np.int32))]
    pc.pc_destroy(pc.pc_create(wl.V, wl.T, *t, wl.material, max_contacts))  # modules, the allocator's own pages
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = pc.pc_create(wl.V, wl.T, *t, wl.material, max_contacts)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    pc.pc_destroy(ctx)
    return held


def test_memory_of_a_context_without_contacts(pc):
    """5,500 bytes per vertex of a sheet (two triangles, three hinges, 13 blocks) at most."""
    wl = wk.square_cloth(512, seed=3, contact_frac=0.0)
    assert _held(pc, wl, 0) <= 5500 * wl.V


def test_memory_per_contact(pc):
    """1,500 bytes per contact of max_contacts at most: what a contact can add to the matrix (six
    blocks) in the solver's copies, and its own records."""
    wl = wk.square_cloth(128, seed=3, contact_frac=0.0)
    assert _held(pc, wl, 40 * wl.V) - _held(pc, wl, 0) <= 1500 * 40 * wl.V


def test_context_without_room_for_the_patch_records(pc):
    """All of a context's memory but half of the patch records' free: the context is made, and
    its solves stream the BSR rows."""
    wl = wk.square_cloth(708, seed=3, contact_frac=0.0)
    held = _held(pc, wl, 0)
    store = 560 * wl.V  # of at most 620 bytes per vertex
    torch.cuda.empty_cache()
    block = torch.empty(torch.cuda.mem_get_info()[0] - held + store // 2 - (64 << 20), dtype=torch.uint8, device="cuda")
    cl = pc.Cloth(wl, max_contacts=0)
    del block
    torch.cuda.empty_cache()
    s = cl.assemble()
    dv = torch.zeros(2, cl.V * 3, device="cuda")
    for out, storage in ((dv[0], pc.PC_STORAGE_OFFDIAG), (dv[1], pc.PC_STORAGE_FULL)):
        n0 = pc.pc_launch_count(cl.ctx)
        info, st = pc.pc_pcg_solve(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"], out,
                                   pc.solve_opts(tol=1e-9, precision=pc.PC_PREC_MIXED, max_iter=50000, storage=storage))
        assert st == pc.PC_OK and info.rel_res <= 1e-9
    pc.pc_set_profiling(cl.ctx, True)
    dv[0].zero_()
    pc.pc_pcg_solve(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"], dv[0],
                    pc.solve_opts(tol=1e-9, precision=pc.PC_PREC_MIXED, max_iter=50000))
    assert pc.pc_spmv_stats(cl.ctx)[2] == s["nnzb"] - cl.V  # the copy without the diagonal, no records
    assert ((dv[0] - dv[1]).norm() / dv[1].norm()).item() <= 1e-5
    cl.close()
