"""The decomposition's launch choices give the same bits: one or two rays per thread (by the number of rays, with
ragged last blocks), and the exponential without or with the scaling of small results (by the range of a warp's
rays). Rays are independent, so a long call must equal its rays in short calls exactly."""
import numpy as np
import pytest
import torch

from synth.spectra import SpectralTables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", [0, 1, 4])
@pytest.mark.parametrize("n", [(1 << 17) + 1, (1 << 17) + 129, (1 << 18) - 1])
def test_long_calls_equal_short_calls_bit_for_bit(cuda_dev, n, iters):
    from paper_1905_00934_gb300 import Spectra

    spec = Spectra.from_tables(SpectralTables(e_ref_kev=100.0))
    rng = np.random.default_rng(n + iters)
    a_c = rng.uniform(0.0, 4.0, n)
    a_c[5::997] = rng.uniform(60.0, 300.0, a_c[5::997].size)  # exponentials below float32's normal range
    a_c[7::9973] = np.nan
    a_p = rng.uniform(-0.1, 0.5, n)
    m = np.stack([rng.uniform(0.0, 6.0, n), rng.uniform(0.0, 8.0, n)])
    w = 1e5 * np.exp(-m)

    def dev(x):
        return torch.tensor(x, dtype=torch.float32, device=cuda_dev)

    args = [dev(x) for x in (m[0], m[1], w[0], w[1], a_c, a_p)]
    state = [dev(a_c), dev(a_p), torch.full((n,), 1e-3, device=cuda_dev)]
    status = torch.full((n,), 9, dtype=torch.uint8, device=cuda_dev)
    part, pstatus = [t.clone() for t in state], status.clone()
    spec.decompose(*args, 1e-3, 1e-3, iters, *state, status)
    step = 100_003  # below the size that takes two rays per thread
    for i in range(0, n, step):
        sl = slice(i, min(n, i + step))
        cut = [t[sl].clone() for t in part]
        cs = pstatus[sl].clone()
        spec.decompose(*[t[sl].clone() for t in args], 1e-3, 1e-3, iters, *cut, cs)
        for t, c in zip(part, cut):
            t[sl] = c
        pstatus[sl] = cs
    for t, p in zip(state + [status], part + [pstatus]):
        assert torch.equal(t.view(torch.uint8), p.view(torch.uint8))


@pytest.mark.parametrize("n_both, n_end, ne", [(1, 1, 2), (3, 5, 8), (7, 9, 17), (8, 16, 17), (9, 15, 24), (16, 16, 23),
                                               (20, 22, 30)])
@pytest.mark.parametrize("tail_high", [True, False])
def test_padded_bins_equal_tested_bins_bit_for_bit(cuda_dev, n_both, n_end, ne, tail_high):
    from paper_1905_00934_gb300 import Spectra

    rng = np.random.default_rng(ne)
    s = [rng.uniform(0.1, 1.0, ne) * (np.arange(ne) < (n_end if long else n_both)) for long in (tail_high, not tail_high)]
    f_kn, f_p = rng.uniform(0.1, 0.3, ne), rng.uniform(0.05, 2.0, ne)
    n = 5000
    m = rng.uniform(0.0, 4.0, (2, n))
    a = [rng.uniform(0.0, 4.0, n), rng.uniform(0.0, 0.5, n)]

    def run(f_last):
        # a bin that neither spectrum has: a large coefficient there takes every ray off the padded path
        f_kn[ne - 1] = f_last
        spec = Spectra(s[0], s[1], f_kn, f_p)
        dev = lambda x: torch.tensor(x, dtype=torch.float32, device=cuda_dev)
        state = [dev(a[0]), dev(a[1]), torch.full((n,), 1e-3, device=cuda_dev)]
        status = torch.zeros(n, dtype=torch.uint8, device=cuda_dev)
        spec.decompose(dev(m[0]), dev(m[1]), dev(np.exp(-m[0])), dev(np.exp(-m[1])), dev(a[0]), dev(a[1]), 1e-3, 1e-3,
                       3, *state, status)
        return torch.stack(state).view(torch.int32), status

    for x, y in zip(run(0.2), run(1e6)):
        assert torch.equal(x, y)
