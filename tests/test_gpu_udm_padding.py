"""A block of 8 energies that holds the end of a spectrum runs unrolled with zero weights where no exponential
underflows, and bin by bin otherwise: the same bits. Every block gets a bin that neither spectrum has; a large coefficient
there sends the block, for every ray, down the other way and adds an exact zero to each sum."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_both, n_end, ne", [(1, 1, 2), (3, 5, 8), (7, 9, 17), (8, 16, 17), (9, 15, 24), (16, 16, 23),
                                               (20, 22, 30), (121, 121, 121), (60, 117, 121)])
@pytest.mark.parametrize("tail_high", [True, False])
@pytest.mark.parametrize("last", [False, True])  # the block's first or last bin that does not end a spectrum
def test_unrolled_blocks_equal_tested_bins_bit_for_bit(cuda_dev, n_both, n_end, ne, tail_high, last):
    from paper_1905_00934_gb300 import Spectra, dect

    rng = np.random.default_rng(ne)
    holes = []
    for e0 in range(0, ne, 8):
        free = [e for e in range(e0, min(e0 + 8, ne)) if e not in (n_both - 1, n_end - 1)]
        holes += free[-1:] if last else free[:1]
    s = [rng.uniform(0.1, 1.0, ne) * (np.arange(ne) < (n_end if long else n_both)) for long in (tail_high, not tail_high)]
    for k in s:
        k[holes] = 0.0
    f_kn, f_p = rng.uniform(0.1, 0.3, ne), rng.uniform(0.05, 2.0, ne)
    n = 5000
    a = np.stack([rng.uniform(1.0, 4.0, n), rng.uniform(0.05, 0.5, n)])
    # measurements of a point close by: the steps stay small, so that no exponent turns positive
    t = np.exp(-np.outer(1.02 * a[0], f_kn) - np.outer(0.98 * a[1], f_p))
    m = [-np.log(t @ (k / k.sum())) for k in s]

    def run(f_hole):
        f = f_kn.copy()
        f[holes] = f_hole
        spec = Spectra(s[0], s[1], f, f_p)
        dev = lambda x: torch.tensor(x, dtype=torch.float32, device=cuda_dev)
        state = [dev(a[0]), dev(a[1]), torch.full((n,), 1e-3, device=cuda_dev)]
        status = torch.zeros(n, dtype=torch.uint8, device=cuda_dev)
        spec.decompose(dev(m[0]), dev(m[1]), dev(1e3 * np.exp(-m[0])), dev(1e3 * np.exp(-m[1])), dev(a[0]), dev(a[1]), 1.0,
                       1.0, 3, *state, status)
        model = [torch.zeros(n, device=cuda_dev) for _ in range(4)]
        jac = torch.zeros((n, 4), device=cuda_dev)
        dect.forward_model(spec.handle, dev(a[0]), dev(a[1]), model[0], model[1])
        dect.forward_model(spec.handle, dev(a[0]), dev(a[1]), model[2], model[3], jac)
        return torch.cat([torch.stack(state + model + [status.float()]).T, jac], 1)

    x, y = run(0.2), run(1e6)
    assert bool(torch.isfinite(x).all()) and bool((x[:, 0] > 0.1).all())
    assert bool((x[:, 0] != torch.tensor(a[0], dtype=torch.float32, device=cuda_dev)).any())
    assert torch.equal(x.view(torch.int32), y.view(torch.int32))
