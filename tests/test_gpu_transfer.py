"""The transfer kernel of the FFT comparator on axes of one and two modes and
at a small relaxation rate, against the closed-form fixed point of the pins
(its other shapes and sets are in test_gpu_fft.py, with the same bar)."""
import numpy as np
import pytest

import oracle
import pins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,order,shape,tau", [
    ("D3Q111", 5, (1, 6, 2), 1.4), ("D3Q111", 5, (12, 1, 1), 1.4), ("D2Q169", 7, (8, 1), 2.0),
    ("D1Q5", 3, (2,), 1.0), ("D3Q19", 1, (2, 2, 2), 1.0), ("D3Q111", 5, (12, 14, 10), 61.8),
    ("D2Q81", 5, (1, 31), 61.8),
])
def test_transfer_at_the_edges(lattice, order, shape, tau):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    rho = np.random.default_rng(17).standard_normal(shape)
    lat = oracle.lattice(lattice, order)
    S, _ = oracle.source(rho, lat, tau, 1.0)
    want = pins.fixed_point(S, lat.vel, lat.phi, lat.chi, 1.0 / tau)
    r = torch.from_numpy(rho).cuda()
    phi = torch.empty_like(r)
    pk.fixed_point_fft(r, phi, pk.problem(lattice, shape, order, tau_lb=tau))
    got = phi.cpu().numpy()
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
