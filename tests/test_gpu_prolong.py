"""cgp_prolong: the device form (one launch a level, straight into the caller's array) gives bit
for bit what the host form gives, leaves the same field in the solver, and takes arrays that
share their start or overlap otherwise."""

import ctypes

import numpy as np
import pytest

from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,k", [(square_mesh(3), 1, 1), (square_mesh(5), 3, 2), (square_mesh(7), 2, 0),
                                           (channel_cylinder_mesh(seed=1, h=0.05), 3, 3)])
@pytest.mark.parametrize("layout", ["apart", "same", "overlap"])
def test_device_prolongation_equals_the_host_form(lib, base, levels, k, layout):
    import torch
    from paper_1812_00185_gb300 import binding as cg
    m = cg.Mesh(base.xy, base.tri, base.tag, levels)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=k))
    phi = np.random.default_rng(k).standard_normal(s.nc)
    want = cg.cgp_prolong(s.handle, phi)
    buf = torch.zeros(s.nf + s.nc + 16, dtype=torch.float64, device="cuda")
    at = {"apart": s.nf + 8, "same": 0, "overlap": 3}[layout]
    src, dst = buf[at:at + s.nc], buf[:s.nf]
    src.copy_(torch.from_numpy(phi))
    rc = cg.load().cgp_prolong(s.handle, ctypes.c_void_p(src.data_ptr()), ctypes.c_void_p(dst.data_ptr()),
                               cg.CGP_DEVICE, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == cg.CGP_OK
    assert np.array_equal(dst.cpu().numpy(), want)
    assert np.array_equal(s.vector(cg.CGP_VEC_PHI_F), want)
    s.close()
    m.close()
