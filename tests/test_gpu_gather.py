"""The gathering backprojector at the sizes where it can go wrong: tile edges, detectors much finer (a view's rays
over a tile exceed a staged batch) and much coarser than the pixels, groups of three to five slices, and rays that
are not finite.

Tolerance 1e-5 (relative L2): weights carry 2^-23 pixel, a pixel sums at most a few thousand float32 terms, whose
rounding errors add up to well below 1e-6 of the sum's norm."""
import math

import numpy as np
import pytest
import torch

from conftest import rel_l2, to_dev
from oracle import projector as oproj
from synth import geometry as G
from synth.spectra import SpectralTables

pytestmark = pytest.mark.gpu


def _fan(n, ny, views, bins, pitch_px, offset=0.0):
    """A fan over an n x ny image of 1 mm pixels whose bins are pitch_px pixels apart at the isocentre."""
    return G.Geometry(G.FAN_FLAT, n, ny, 0.1, views, 0.05, 2 * math.pi, bins, 0.1 * pitch_px * 1.7, offset, 30.0, 51.0)


GEOMS = {
    "tile_31x33": _fan(31, 33, 37, 64, 0.8),
    "tile_32x64": _fan(32, 64, 37, 100, 0.8, 0.03),
    "tile_65x1": _fan(65, 1, 21, 80, 0.9),
    "fine_detector": _fan(40, 36, 9, 3000, 0.02),
    "coarse_detector": _fan(70, 67, 50, 21, 5.0),
    "parallel_fine": G.Geometry(G.PARALLEL, 33, 40, 0.1, 17, 0.0, math.pi, 1500, 0.004, 0.0),
}


@pytest.mark.parametrize("name", sorted(GEOMS))
def test_backprojection_matches_oracle_at_edge_sizes(cuda_dev, name):
    from paper_1905_00934_gb300 import Geometry

    g = GEOMS[name]
    y = np.random.default_rng(3).normal(size=(2, g.n_views, g.n_bins))
    geo = Geometry(g)
    ref = np.stack([oproj.backproject(g, np.float32(y[c]).astype(np.float64)) for c in range(2)])
    got = geo.backproject(to_dev(y, cuda_dev)).cpu().numpy()
    assert rel_l2(got, ref) <= 1e-5
    one = geo.backproject(to_dev(y[:1], cuda_dev)).cpu().numpy()
    assert rel_l2(one[0], ref[0]) <= 1e-5


@pytest.mark.parametrize("slices", [3, 5])
def test_groups_of_slices_equal_single_slices(cuda_dev, slices):
    # slices of one geometry share backprojector CTAs two or four at a time; whatever the autotuner picks
    # at a fixed view-group count, every slice has the bits of its own solver
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra, dect

    g = _fan(75, 66, 90, 110, 0.9)
    geo, spec = Geometry(g), Spectra.from_tables(SpectralTables(e_ref_kev=100.0))
    rng = np.random.default_rng(8)
    data = []
    for _ in range(slices):
        m = rng.uniform(0.1, 2.0, size=(2, g.n_views, g.n_bins))
        data.append([to_dev(a, cuda_dev) for a in (m[0], 1.2 * m[1], 1e5 * np.exp(-m[0]), 1e5 * np.exp(-m[1]))])
    outs = []
    for kw in (dict(), dict(bp_slices=2), dict(bp_slices=1)):
        sol = Solver([geo] * slices, spec, bp_view_groups=3, **kw)
        for b, d in enumerate(data):
            sol.set_data(b, *d)
        sol.reconstruct(2)
        outs.append([sol.get(b, dect.X).cpu().numpy() for b in range(slices)])
    for b, d in enumerate(data):
        one = Solver([geo], spec, bp_view_groups=3)
        one.set_data(0, *d)
        one.reconstruct(2)
        x = one.get(0, dect.X).cpu().numpy()
        for o in outs:
            assert np.array_equal(o[b], x), b


@pytest.mark.parametrize("value", [math.inf, math.nan])
def test_a_ray_that_is_not_finite_reaches_its_own_pixels_only(cuda_dev, value):
    from paper_1905_00934_gb300 import Geometry

    g = _fan(70, 50, 12, 90, 0.9)
    y = np.zeros((2, g.n_views, g.n_bins))
    y[0, 5, 40] = 1.0
    w = oproj.backproject(g, y[0])
    y[0, 5, 40] = value
    got = Geometry(g).backproject(to_dev(y, cuda_dev)).cpu().numpy()
    bad = ~np.isfinite(got[0])
    assert bad[w > 1e-5].all() and not bad[w == 0].any()
    assert np.isfinite(got[1]).all()
