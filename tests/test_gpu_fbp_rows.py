"""The ramp filter's passes over a detector row: rows of less than one warp, of a whole number of passes, one bin more
and less, and rows split over several CTAs (few views) against the FP64 oracle; non-finite samples."""
import math

import numpy as np
import pytest

from conftest import rel_l2, to_dev
from oracle import fbp as ofbp
from synth import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb, nv", [(1, 5), (2, 160), (15, 5), (511, 160), (513, 20), (1008, 5), (1024, 160),
                                    (1025, 20), (1025, 160), (1537, 160), (4097, 5), (5001, 160)])
def test_fbp_rows_match_oracle(cuda_dev, nb, nv):
    from paper_1905_00934_gb300 import Geometry

    # 40 x 40 pixels over the whole row
    g = G.Geometry(G.PARALLEL, 40, 40, 0.1 * max(nb, 20) / 40, nv, 0.3, math.pi, nb, 0.1, 0.013)
    p = np.random.default_rng(nb).standard_normal((2, nv, nb)).astype(np.float32)
    x = Geometry(g).fbp(to_dev(p, cuda_dev)).cpu().numpy()
    # white noise read at positions of ~4 roundings of nb, sqrt(2) per bin; one wrong bin of the row is > 1e-2
    tol = 1e-5 + 4e-7 * nb
    for c in range(2):
        assert rel_l2(x[c], ofbp.fbp(g, p[c].astype(np.float64))) <= tol


@pytest.mark.parametrize("nb", [64, 1100])
def test_fbp_infinite_sample_counts_once(cuda_dev, nb):
    from paper_1905_00934_gb300 import Geometry

    # one view at angle 0: pixel i reads the row at i * 0.75 + const
    nx = int(nb / 0.75) - 2
    g = G.Geometry(G.PARALLEL, nx, 1, 0.075, 1, 0.0, math.pi, nb, 0.1, 0.0)
    p = np.ones((1, 1, nb), dtype=np.float32)
    hit = nb // 2 + 1
    p[0, 0, hit] = np.inf
    x = Geometry(g).fbp(to_dev(p, cuda_dev)).cpu().numpy().reshape(nx)
    q = np.ones(nb + 1)  # (any finite value: the neighbours in odd steps have -inf, the sample itself +inf)
    q[nb] = 0.0
    q[:nb][(np.arange(nb) - hit) % 2 == 1] = -np.inf
    q[hit] = np.inf
    k = (np.arange(nx) - 0.5 * (nx - 1)) * 0.75 + 0.5 * (nb - 1)
    k0 = np.floor(k).astype(int)
    clear = np.abs(k - np.round(k)) > 1e-3  # away from the bins themselves, where the position's rounding decides
    with np.errstate(invalid="ignore"):
        ref = q[k0] + (k - k0) * (q[k0 + 1] - q[k0])
    for test in (np.isfinite, np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(test(x)[clear], test(ref)[clear])
