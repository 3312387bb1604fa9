"""The float64 projector pair at the edges of its launch shapes: rows of 32 pixels, four lanes per ray, view groups of
eight, single channels, rays almost parallel to an axis far outside the image.

Tolerance 1e-12 (relative L2): positions are float64 (rounding 1e-13 pixel at these sizes) and every sum has at most
a few thousand terms."""
import math

import numpy as np
import pytest
import torch

from conftest import rel_l2
from oracle import projector as oproj
from synth import geometry as G

pytestmark = pytest.mark.gpu

GEOMS = {
    "axis_parallel": G.Geometry(G.PARALLEL, 33, 31, 0.1, 8, 0.0, 2 * math.pi, 90, 0.1, 0.0),
    "one_row": G.Geometry(G.FAN_FLAT, 65, 1, 0.1, 7, 0.2, 2 * math.pi, 33, 0.3, 0.0, 12.0, 20.0),
    "fan_64x32": G.Geometry(G.FAN_FLAT, 64, 32, 0.1, 17, 0.2, 2 * math.pi, 130, 0.11, 0.02, 12.0, 20.0),
    "fine_bins": G.Geometry(G.FAN_FLAT, 9, 40, 0.1, 5, 0.2, 2 * math.pi, 700, 0.01, 0.0, 12.0, 20.0),
}


@pytest.mark.parametrize("nch", [1, 2])
@pytest.mark.parametrize("name", sorted(GEOMS))
def test_f64_pair_matches_oracle(cuda_dev, name, nch):
    from paper_1905_00934_gb300 import Geometry

    g = GEOMS[name]
    rng = np.random.default_rng(4)
    x, y = rng.normal(size=(nch, g.ny, g.nx)), rng.normal(size=(nch, g.n_views, g.n_bins))
    geo = Geometry(g)
    s = geo.project(torch.tensor(x, device=cuda_dev)).cpu().numpy()
    b = geo.backproject(torch.tensor(y, device=cuda_dev)).cpu().numpy()
    assert rel_l2(s, np.stack([oproj.project(g, x[c]) for c in range(nch)])) <= 1e-12
    assert rel_l2(b, np.stack([oproj.backproject(g, y[c]) for c in range(nch)])) <= 1e-12
