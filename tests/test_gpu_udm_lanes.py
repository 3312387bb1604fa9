"""The lanes of a warp choose the decomposition's exponential together, whatever the rays of the others do: rays that end
early (not finite from the start or after a step) and lanes past the last ray."""
import glob
import os

import numpy as np
import pytest
import torch

from conftest import ROOT
from synth.spectra import SpectralTables


def test_votes_name_every_lane():
    # a mask of the lanes that happen to be active does not promise that they reach the vote together
    for path in glob.glob(os.path.join(ROOT, "paper_1905_00934_gb300", "csrc", "*.cu*")):
        with open(path) as f:
            assert "__activemask" not in f.read(), path


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 31, 33, 70, (1 << 17) + 40])
def test_rays_beside_rays_that_end_early_keep_their_bits(cuda_dev, n):
    from paper_1905_00934_gb300 import Spectra

    spec = Spectra.from_tables(SpectralTables(e_ref_kev=100.0))
    rng = np.random.default_rng(n)
    dev = lambda x: torch.tensor(x, dtype=torch.float32, device=cuda_dev)
    m = rng.uniform(0.1, 5.0, (2, n))
    a = np.stack([rng.uniform(0.0, 4.0, n), rng.uniform(0.0, 0.4, n)])
    w = 1e5 * np.exp(-m)
    clean = [dev(x) for x in (m[0], m[1], w[0], w[1], a[0], a[1])]
    mixed = [t.clone() for t in clean]
    ends = torch.arange(n, device=cuda_dev) % 7 == 3
    mixed[0][ends] = float("nan")                                  # not finite from the start
    mixed[2][torch.arange(n, device=cuda_dev) % 7 == 5] = 1e30      # its first step is not finite
    far = torch.arange(n, device=cuda_dev) % 7 == 6                 # exponentials that underflow

    def run(args, far_start):
        state = [args[4].clone(), args[5].clone(), torch.full((n,), 1e-3, device=cuda_dev)]
        if far_start:
            state[1][far] = 50.0
        status = torch.full((n,), 9, dtype=torch.uint8, device=cuda_dev)
        spec.decompose(*args, 1e-3, 1e-3, 5, *state, status)
        return torch.stack(state + [status.float()])

    same = torch.arange(n, device=cuda_dev) % 7 < 3
    x, y = run(clean, False), run(mixed, True)
    assert torch.equal(x[:, same].view(torch.int32), y[:, same].view(torch.int32))
    assert bool((y[3][ends] == 2).all())


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 31, 33, 255, 257])
def test_forward_model_of_ragged_calls_equals_long_calls(cuda_dev, n):
    from paper_1905_00934_gb300 import Spectra, dect

    spec = Spectra.from_tables(SpectralTables(e_ref_kev=100.0))
    rng = np.random.default_rng(n)
    a = torch.tensor(rng.uniform(0.0, 4.0, 512), dtype=torch.float32, device=cuda_dev)
    p = torch.tensor(rng.uniform(0.0, 0.4, 512), dtype=torch.float32, device=cuda_dev)
    p[::5] = 50.0

    def run(k):
        f = [torch.zeros(512, device=cuda_dev) for _ in range(6)]
        jac = torch.zeros((512, 4), device=cuda_dev)
        dect.forward_model(spec.handle, a[:k], p[:k], f[0][:k], f[1][:k])
        dect.forward_model(spec.handle, a[:k], p[:k], f[2][:k], f[3][:k], jac[:k])
        dect.forward_model_vjp(spec.handle, a[:k], p[:k], a[:k], p[:k], f[4][:k], f[5][:k])
        return torch.cat([torch.stack(f).T, jac], 1)

    x, y = run(512), run(n)
    assert torch.equal(x[:n].view(torch.int32), y[:n].view(torch.int32))
    assert not y[n:].any()  # nothing is written past the last ray
