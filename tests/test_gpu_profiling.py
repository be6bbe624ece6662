"""pc_spmv_stats of solves whose iterations run inside one launch: every iteration's product is
represented, with a time."""
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


# records of 32, 160 and 480 rows per SM (four, four and two threads per row)
@pytest.mark.parametrize("nx,precision,block", [(64, 1, False), (141, 0, True), (270, 1, False)])
def test_products_of_a_solve_are_counted_and_timed(pc, nx, precision, block):
    cl = pc.Cloth(wk.square_cloth(nx, seed=4, contact_frac=0.0))
    s = cl.assemble()
    dv = [torch.zeros(cl.V * 3, device="cuda") for _ in range(2)]
    opts = pc.solve_opts(tol=1e-5, precision=precision, max_iter=20000, schedule=pc.PC_SCHED_GRID,
                         precond=pc.PC_PRECOND_BLOCK if block else pc.PC_PRECOND_JACOBI)
    args = cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"]
    pc.pc_pcg_solve(*args, dv[0], opts)
    assert pc.pc_spmv_stats(cl.ctx)[0] == 0
    pc.pc_set_profiling(cl.ctx, True)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    n0 = pc.pc_launch_count(cl.ctx)
    e[0].record()
    info, _ = pc.pc_pcg_solve(*args, dv[1], opts)
    e[1].record()
    torch.cuda.synchronize()
    assert pc.pc_launch_count(cl.ctx) - n0 < info.iters
    n, ms, blocks = pc.pc_spmv_stats(cl.ctx)
    assert n == info.iters and 0.0 < ms < e[0].elapsed_time(e[1])
    # a block inside a patch counts once
    assert (s["nnzb"] - cl.V) / 2 <= blocks < s["nnzb"] - cl.V
    assert torch.equal(dv[0], dv[1])
    cl.close()
