"""dect_project_noalloc takes every image whose pair textures fit its fixed scratch (16 (nx (ny + 3) + ny (nx + 3)) bytes,
360 x 360), and no larger one."""
import ctypes
import math

import pytest
import torch

from synth import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, ny", [(324, 324), (360, 360), (361, 361), (2048, 62), (2048, 63)])
def test_noalloc_limit_is_the_textures_size(cuda_dev, nx, ny):
    from paper_1905_00934_gb300 import Geometry, dect

    geo = Geometry(G.Geometry(G.PARALLEL, nx, ny, 0.1, 12, 0.1, math.pi, 90, 0.5))
    gen = torch.Generator(device=cuda_dev)
    gen.manual_seed(nx)
    x = torch.rand((2, ny, nx), device=cuda_dev, generator=gen)
    out = torch.zeros((2, 12, 90), device=cuda_dev)
    if 16 * (nx * (ny + 3) + ny * (nx + 3)) <= dect.NOALLOC_SCRATCH_BYTES:
        dect.project_noalloc(geo, x, out)
        assert torch.equal(out, geo.project(x))
    else:
        status = dect.lib().dect_project_noalloc(geo.handle, 2, ctypes.c_void_p(x.data_ptr()),
                                                 ctypes.c_void_p(out.data_ptr()), None)
        assert status == dect.EINVAL and b"scratch" in dect.lib().dect_last_error()
