"""The float64 R and R^T hold the same matrix, entry for entry: R of every single pixel against R^T of every single ray,
bit for bit (a product of one weight and one factor each, so no sum rounds)."""
import math

import numpy as np
import pytest
import torch

from synth import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [G.Geometry(G.PARALLEL, 5, 4, 0.1, 23, 0.05, math.pi, 9, 0.07, 0.01),
                               G.Geometry(G.FAN_FLAT, 4, 6, 0.1, 31, 0.3, 2 * math.pi, 11, 0.13, 0.02, 2.0, 3.4)],
                         ids=["parallel", "fan"])
def test_f64_pair_is_one_matrix_bit_for_bit(cuda_dev, g):
    from paper_1905_00934_gb300 import Geometry

    geo = Geometry(g)
    np_, nr = g.ny * g.nx, g.n_views * g.n_bins
    pixels = torch.eye(np_, dtype=torch.float64, device=cuda_dev).reshape(np_, 1, g.ny, g.nx)
    rays = torch.eye(nr, dtype=torch.float64, device=cuda_dev).reshape(nr, 1, g.n_views, g.n_bins)
    r = torch.stack([geo.project(x).reshape(-1) for x in pixels], 1)
    rt = torch.stack([geo.backproject(y).reshape(-1) for y in rays], 0)
    assert int((r > 0).sum()) > np_ * g.n_views / 2
    assert torch.equal(r, rt)
