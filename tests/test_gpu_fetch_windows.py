"""The backprojector fetches staged rays 64 at a time whatever views they belong to: detectors of few, wide bins, where a
window spans many views, and of one bin; images of one pixel, one tile and ragged ones; both tile sides. One channel of
the single-slice projector is summed by itself: the same bits as beside a second one.

Tolerance 1e-5 (relative L2): weights carry 2^-23 pixel, a pixel sums at most a few thousand float32 terms, whose rounding
errors add up to well below 1e-6 of the sum's norm."""
import math

import numpy as np
import pytest

from conftest import rel_l2, to_dev
from oracle import projector as oproj
from synth import geometry as G
from synth.spectra import SpectralTables

pytestmark = pytest.mark.gpu


def _fan(n, ny, views, bins, pitch_px, offset=0.0):
    r = 0.05 * math.hypot(n, ny)
    return G.Geometry(G.FAN_FLAT, n, ny, 0.1, views, 0.05, 2 * math.pi, bins, 0.17 * pitch_px, offset, 3 * r + 1, 1.7 * (3 * r + 1))


GEOMS = {
    "one_bin": _fan(33, 20, 150, 1, 3.0),
    "one_pixel": _fan(1, 1, 90, 7, 0.5),
    "coarse_16": _fan(130, 64, 300, 12, 16.0, 0.1),
    "coarse_4": _fan(70, 97, 200, 41, 4.0),
    "coarse_parallel": G.Geometry(G.PARALLEL, 64, 65, 0.1, 180, 0.0, math.pi, 9, 1.1, 0.05),
    "many_views": _fan(32, 31, 1100, 30, 1.6),
}


@pytest.mark.parametrize("name", sorted(GEOMS))
def test_backprojection_of_few_bins_matches_oracle(cuda_dev, name):
    from paper_1905_00934_gb300 import Geometry

    g = GEOMS[name]
    y = np.float32(np.random.default_rng(5).uniform(0.5, 1.5, size=(2, g.n_views, g.n_bins))).astype(np.float64)
    geo = Geometry(g)
    ref = np.stack([oproj.backproject(g, y[c]) for c in range(2)])
    assert rel_l2(geo.backproject(to_dev(y, cuda_dev)).cpu().numpy(), ref) <= 1e-5
    assert rel_l2(geo.backproject(to_dev(y[:1], cuda_dev)).cpu().numpy()[0], ref[0]) <= 1e-5


@pytest.mark.parametrize("name", ["coarse_16", "coarse_parallel"])
def test_few_bins_give_the_same_bits_in_every_launch_shape(cuda_dev, name):
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra, dect

    g = GEOMS[name]
    spec, geo = Spectra.from_tables(SpectralTables(e_ref_kev=100.0)), Geometry(g)
    rng = np.random.default_rng(8)
    data = []
    for _ in range(3):
        m = rng.uniform(0.1, 2.0, size=(2, g.n_views, g.n_bins))
        data.append([to_dev(a, cuda_dev) for a in (m[0], 1.2 * m[1], 1e5 * np.exp(-m[0]), 1e5 * np.exp(-m[1]))])
    outs = []
    for kw in (dict(bp_tile=32, bp_slices=1), dict(bp_tile=64, bp_slices=1), dict(bp_tile=64, bp_slices=2),
               dict(bp_slices=4), dict(bp_tile=32, bp_cluster=1)):
        sol = Solver([geo] * 3, spec, bp_view_groups=3, **{"bp_cluster": -1, **kw})
        for b, d in enumerate(data):
            sol.set_data(b, *d)
        sol.reconstruct(2)
        outs.append([sol.get(b, dect.X).cpu().numpy() for b in range(3)])
    for o in outs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(o, outs[0]))


@pytest.mark.parametrize("name", sorted(GEOMS))
def test_one_channel_projection_has_the_bits_of_two(cuda_dev, name):
    import torch

    from paper_1905_00934_gb300 import Geometry

    g = GEOMS[name]
    x = to_dev(np.random.default_rng(2).normal(size=(2, g.ny, g.nx)), cuda_dev)
    geo = Geometry(g)
    both = geo.project(x)
    for c in range(2):
        assert torch.equal(geo.project(x[c:c + 1].contiguous())[0], both[c])


@pytest.mark.parametrize("angle0", [0.0, 1e-17, 1e-9, 1e-4, math.pi / 2, math.pi / 4])
@pytest.mark.parametrize("n, ny", [(1, 1), (2, 31), (64, 5)])
def test_f64_projection_of_rays_along_the_axes_and_the_edges(cuda_dev, n, ny, angle0):
    # a ray's samples are bounded in float32: rays (nearly) along an axis, through, on and beside the image's edges.
    # Tolerance 1e-12 of the largest value: at most 64 float64 terms of one sign
    import torch

    from paper_1905_00934_gb300 import Geometry

    g = G.Geometry(G.PARALLEL, n, ny, 0.1, 2, angle0, math.pi, 4 * max(n, ny) + 9, 0.025, 0.0)
    x = np.random.default_rng(n).uniform(0.1, 1.0, size=(2, ny, n))
    ref = np.stack([oproj.project(g, x[c]) for c in range(2)])
    got = Geometry(g).project(torch.tensor(x, device=cuda_dev)).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
