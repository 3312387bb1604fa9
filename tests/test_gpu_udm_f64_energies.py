"""The decomposition in float64 arithmetic (udm_f64 = 1) takes as many energies as spectra may have (512): its tables
outgrow the shared memory that a kernel gets unasked. Bins of zero weight add exact zeros to its sums, so spectra that are
lengthened by such bins give the same images bit for bit."""
import numpy as np
import pytest

from conftest import to_dev
from synth.workloads import small_parallel_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["STORE_F32", "STORE_F16", "STORE_BF16"])
@pytest.mark.parametrize("ne", [496, 497, 501, 505, 512])
def test_udm_f64_with_many_energies(cuda_dev, ne, storage):
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra, dect

    c = small_parallel_case(e_ref_kev=100.0)
    t, geo = c["spectra"], Geometry(c["geom"])
    x0 = np.stack([c["truth_c"], c["truth_p"]]) * 0.9
    out = []
    for extra in (0, ne - len(t.f_kn)):
        more = lambda a, v: np.concatenate([a, np.full(extra, v)])
        spec = Spectra(more(t.s_high, 0.0), more(t.s_low, 0.0), more(t.f_kn, 0.2), more(t.f_p, 0.1))
        sol = Solver([geo], spec, storage=getattr(dect, storage), udm_f64=1, bp_view_groups=4)
        sol.set_data(0, *[to_dev(c[k], cuda_dev) for k in ("m_h", "m_l", "w_h", "w_l")], to_dev(x0, cuda_dev))
        sol.reconstruct(2)
        out.append([sol.get(0, w).cpu().numpy() for w in (dect.X, dect.A, dect.MU)])
    assert np.isfinite(out[1][0]).all()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
