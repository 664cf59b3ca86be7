"""GPU check of what a context takes of the device's memory."""

import pytest

from paper_2504_08157_gb300 import xg

pytestmark = pytest.mark.gpu


def test_fp64_context_takes_its_arrays_and_no_more(cuda_device):
    """Five-variable arrays for the state, the stages and the result (4), the
    partial tendency (1), four values a node for the point values and one for
    the heating: 30 a node.  Allocations, a dozen of them, are rounded up to 2 MB,
    and launches may load kernels."""
    import torch
    d = xg.mesh_desc((96, 96, 16), 4, (0.0, 0.0, 0.0), (768.0e3, 768.0e3, 20.0e3), (True, True, False))
    small = xg.xg_mesh_create(xg.mesh_desc((2, 2, 2), 4, (0.0, 0.0, 0.0), (1e3, 1e3, 1e3), (True, True, False)))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    c = xg.xg_mesh_create(d)
    try:
        taken = before - torch.cuda.mem_get_info()[0]
        assert taken <= 30 * 8 * xg.xg_mesh_np(c) + 16 * 2 ** 21
    finally:
        xg.xg_destroy(c)
        xg.xg_destroy(small)
