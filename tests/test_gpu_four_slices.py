"""The backprojector that takes four slices of one geometry per CTA, asked for by itself (bp_slices = 4): full and partial
groups, every storage, both ways of adding the view groups. Each slice has the bits of its own one-slice solver, and the
shape that a solver reports can be asked for again."""
import ctypes
import math

import numpy as np
import pytest

from conftest import to_dev
from synth import geometry as G
from synth.spectra import SpectralTables


def _geometry(n, ny):
    return G.Geometry(G.FAN_FLAT, n, ny, 0.1, 70, 0.05, 2 * math.pi, 110, 0.15, 0.0, 30.0, 51.0)


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["STORE_F32", "STORE_F16", "STORE_BF16"])
@pytest.mark.parametrize("reduce", [-1, 1])
@pytest.mark.parametrize("slices", [2, 3, 4, 5, 7])
def test_four_slices_per_cta_equal_single_slices(cuda_dev, slices, reduce, storage):
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra, dect

    spec = Spectra.from_tables(SpectralTables(e_ref_kev=100.0))
    # the slices of one geometry between two others: groups start and end within the batch
    other, geo = Geometry(_geometry(40, 37)), Geometry(_geometry(75, 66))
    geos = [other] + [geo] * slices + [other]
    rng = np.random.default_rng(slices)
    data = []
    for g in geos:
        m = rng.uniform(0.1, 2.0, size=(2, g.n_views, g.n_bins))
        data.append([to_dev(a, cuda_dev) for a in (m[0], 1.2 * m[1], 1e5 * np.exp(-m[0]), 1e5 * np.exp(-m[1]))])
    shape = dict(bp_view_groups=3, bp_tile=32, bp_cluster=-1, bp_reduce=reduce, storage=getattr(dect, storage))

    def solve(gs, ds, sl):
        sol = Solver(gs, spec, bp_slices=sl, **shape)
        for b, d in enumerate(ds):
            sol.set_data(b, *d)
        sol.reconstruct(2)
        return sol.stats(0)["bp_slices"], [sol.get(b, dect.X).cpu().numpy() for b in range(len(gs))]

    used, out = solve(geos, data, 4)
    assert used == 4
    for b, g in enumerate(geos):
        _, one = solve([g], [data[b]], 1)
        assert np.array_equal(out[b], one[0]), b


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [dict(), dict(bp_slices=4), dict(bp_slices=4, bp_view_groups=-1), dict(bp_slices=2)])
def test_the_reported_shape_can_be_asked_for(cuda_dev, kw):
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra

    spec, geo = Spectra.from_tables(SpectralTables(e_ref_kev=100.0)), Geometry(_geometry(75, 66))
    keys = ("bp_view_groups", "bp_tile", "bp_slices", "bp_cluster")
    first = {k: Solver([geo] * 5, spec, **kw).stats(0)[k] for k in keys}
    assert first["bp_slices"] == kw.get("bp_slices", first["bp_slices"])
    again = Solver([geo] * 5, spec, **{**first, "bp_cluster": 1 if first["bp_cluster"] else -1}).stats(0)
    assert {k: again[k] for k in keys} == first


@pytest.mark.parametrize("kw", [dict(bp_slices=3), dict(bp_slices=5), dict(bp_slices=-1), dict(bp_slices=4, bp_tile=64),
                                dict(bp_slices=4, bp_cluster=1)])
def test_shapes_that_do_not_exist_are_refused(kw):
    # with the other parameter checks, before any handle is used (the handles here are never read)
    from paper_1905_00934_gb300 import dect

    dummy = ctypes.create_string_buffer(4096)
    geoms = (ctypes.c_void_p * 1)(ctypes.addressof(dummy))
    h = ctypes.c_void_p()
    p = dect.params_default(**kw)
    assert dect.lib().dect_admm_create(ctypes.cast(geoms, ctypes.c_void_p), 1, ctypes.addressof(dummy), ctypes.byref(p),
                                       ctypes.byref(h)) == dect.EINVAL
    assert b"bp_slices" in dect.lib().dect_last_error()
