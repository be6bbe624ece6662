"""Two host threads, each with a context and a stream of its own, solving at the same time:
every result bit for bit that of the context alone. The kernels' launch limits belong to the
process, so what one solve needs must not take from another's launches.

Only schedules whose kernels never wait for CTAs that may not be resident: the resident one (a
cooperative launch per stretch of iterations) and, for streamed records, the separate update and
direction kernels (fuse = 0).
"""
import threading

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


def _system(pc, n):
    wl = wk.square_cloth(n, seed=11, contact_frac=0.0)
    cl = pc.Cloth(wl)
    return cl, cl.assemble()


def _solve(pc, cl, s, dv, fuse, tol):
    dv.zero_()
    # replacements every 32 iterations: many launches of one solve, with the host in between
    info, st = pc.pc_pcg_solve(cl.ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"], dv,
                               pc.solve_opts(tol=tol, max_iter=20000, precision=pc.PC_PREC_MIXED, refresh_every=32,
                                             schedule=pc.PC_SCHED_GRID, fuse=fuse))
    assert st == pc.PC_OK
    return info.iters


# resident records of 256 and of 32 rows per SM, in the same instantiation of the kernel; streamed
# records, the first system's larger for its contacts
@pytest.mark.parametrize("big,small,fuse,tol", [(190, 48, True, 1e-5), (330, 290, False, 1e-3)])
def test_solves_of_two_threads_do_not_disturb_each_other(pc, big, small, fuse, tol):
    systems = [_system(pc, big), _system(pc, small)]
    if not fuse:  # contacts make the first system's records the larger ones
        cl = systems[0][0]
        wl = wk.square_cloth(big, seed=11, contact_frac=0.05)
        pairs, w = (torch.from_numpy(a).cuda() for a in wl.contacts(0))
        cl.close()
        cl = pc.Cloth(wl)
        systems[0] = (cl, cl.assemble(pairs, w))
    want, bufs = [], []
    for cl, s in systems:
        dv = torch.zeros(cl.V * 3, device="cuda")
        iters = _solve(pc, cl, s, dv, fuse, tol)
        want.append((iters, dv.clone()))
        bufs.append(dv)
    torch.cuda.synchronize()
    failures, stop = [], threading.Event()

    def work(k, rounds):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(rounds):
                    if stop.is_set() and k:
                        return
                    iters = _solve(pc, *systems[k], bufs[k], fuse, tol)
                    torch.cuda.current_stream().synchronize()
                    if iters != want[k][0] or not torch.equal(bufs[k], want[k][1]):
                        failures.append(f"system {k}: another result")
                        return
        except Exception as e:  # reported in the main thread
            failures.append(f"system {k}: {e!r}")
        finally:
            if k == 0:
                stop.set()

    threads = [threading.Thread(target=work, args=(0, 4)), threading.Thread(target=work, args=(1, 400))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
    for cl, _ in systems:
        cl.close()
