"""Value assembly with time steps whose square is outside FP32's range: the right-hand side, which
is of first order in h, against the FP64 oracle (relative L2 error 1e-5, as the parity tests)."""
import dataclasses

import numpy as np
import pytest

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


# h^2 kc denormal; h^2 denormal; h^2 zero
@pytest.mark.parametrize("h", [1e-17, 3e-20, 1e-23])
def test_right_hand_side_of_a_tiny_step(pc, h):
    wl = wk.square_cloth(12, seed=5, contact_frac=0.0)
    wl.h = h
    # bending alone: nothing that hides its forces
    wl.material = dataclasses.replace(wl.material, gravity=(0.0, 0.0, 0.0), young=1e-3)
    wl.x0 = wl.x0.copy()
    wl.x0[:, 2] += (0.02 * np.random.default_rng(3).normal(size=wl.V)).astype(np.float32)
    cl, om = pc.Cloth(wl), oracle.Mesh.from_workload(wl)
    s = cl.assemble()
    _, _, _, b = om.assemble(wl.x0.astype(np.float64), wl.v0.astype(np.float64), None, None, np.float64(np.float32(h)))
    got = s["b"].cpu().numpy().astype(np.float64) / h
    assert np.isfinite(got).all()
    assert H.rel_l2(got.reshape(-1, 3), b / h) <= 1e-5
    cl.close()
