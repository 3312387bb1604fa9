"""The float64 decomposition leaves out the shorter spectrum's sums past its end. With the two spectra and their
measurements exchanged the other one is the longer: the same problem, so the same images to float64 rounding."""
import numpy as np
import pytest

from conftest import rel_l2, to_dev
from synth.workloads import small_parallel_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_pcg, m_udm", [(1, 1), (2, 3)])
def test_f64_exchanged_spectra_give_the_same_images(cuda_dev, n_pcg, m_udm):
    from paper_1905_00934_gb300 import Geometry, Solver, Spectra, dect

    c = small_parallel_case(e_ref_kev=100.0)
    t, geo = c["spectra"], Geometry(c["geom"])
    f = lambda a: to_dev(a, cuda_dev)
    x0 = np.stack([c["truth_c"], c["truth_p"]]) * 0.9
    out = []
    for a, b in (("high", "low"), ("low", "high")):
        s = {"high": t.s_high, "low": t.s_low}
        sol = Solver([geo], Spectra(s[a], s[b], t.f_kn, t.f_p), storage=dect.STORE_F64, n_pcg=n_pcg, m_udm=m_udm)
        sol.set_data(0, f(c["m_" + a[0]]), f(c["m_" + b[0]]), f(c["w_" + a[0]]), f(c["w_" + b[0]]), f(x0))
        sol.reconstruct(5)
        out.append(sol.get(0, dect.X).cpu().numpy().astype(np.float64))
    # 5 iterations of rounding at 1e-16 against steps of order one (float32 images: 6e-8 each)
    assert rel_l2(out[0], out[1]) <= 1e-7
