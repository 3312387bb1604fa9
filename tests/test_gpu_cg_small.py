"""CG steps of small batches form their scalars in the update kernels, those of large ones in kernels of their own: the
same sums in the same order, so a slice alone (small) equals itself in a batch of many (large) bit for bit. Sizes by
the slots per slice: one, a warp's, one more, and the most (256)."""
import math

import numpy as np
import pytest
import torch

from synth import geometry as G
from synth.spectra import SpectralTables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, ny, views, bins, copies", [(9, 11, 12, 20, 500), (64, 128, 40, 96, 24),
                                                         (91, 93, 45, 130, 20), (256, 256, 30, 260, 4)])
@pytest.mark.parametrize("precondition", [1, 0])
def test_small_and_large_batches_give_the_same_bits(cuda_dev, nx, ny, views, bins, copies, precondition):
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra, dect

    spec = Spectra.from_tables(SpectralTables(e_ref_kev=100.0))
    geo = Geometry(G.Geometry(G.PARALLEL, nx, ny, 0.1, views, 0.1, math.pi, bins, 0.1, 0.02))
    rng = np.random.default_rng(nx)
    dev = lambda x: torch.tensor(x, dtype=torch.float32, device=cuda_dev)
    m = rng.uniform(0.1, 3.0, (2, views, bins))
    data = [dev(x) for x in (m[0], m[1], 1e5 * np.exp(-m[0]), 1e5 * np.exp(-m[1]))]
    # the same view groups and sweep for both, so that only the CG's launches differ
    params = dict(bp_view_groups=4, bp_tile=32, bp_cluster=-1, bp_slices=1, precondition=precondition)
    out, launches = [], []
    for n in (1, copies):
        sol = Solver([geo] * n, spec, **params)
        for b in range(n):
            sol.set_data(b, *data)
        sol.reconstruct(2)
        launches.append(sol.stats(0)["count_launches"])
        out.append([sol.get(b, dect.X).cpu().numpy() for b in (0, n - 1)])
    assert launches[0] < launches[1]
    for x in (out[0][1], *out[1]):
        assert np.array_equal(out[0][0], x)
