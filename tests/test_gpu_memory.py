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
