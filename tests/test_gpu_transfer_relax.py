"""The FFT comparator at relaxation times close to 1/2 (omega close to 2), mode
by mode against exact rational arithmetic.

On axes of 1, 2, 3 and 6 sites every cos(k.v) is 1, 1/2, -1/2 or -1, so T(k) is a
rational function of the weights and of omega = 1 / tau_lb, evaluated here with
Python's fractions.  A product of cosines is an eigenvector: Phi = T(k) S.

Bounds, from the operations (eps = 2^-52, d = 2 - omega, kn and kd the sums of
the absolute terms over the absolute sums): a velocity's term is a few products
of table values, one reciprocal and the class sums, under 16 roundings, and the
transforms add a few, so 32 eps (kn + kd) in all; where cos(theta / 2) is not
zero, |1 - (1 - omega) e|^2 = d^2 + 4 (omega - 1) cos^2(theta / 2) carries the
rounding of that cosine, at most 4 eps / d of it."""
import itertools
from fractions import Fraction as Fr

import numpy as np
import pytest

import oracle

COS = {(1, 0): Fr(1), (2, 0): Fr(1), (2, 1): Fr(-1), (3, 0): Fr(1), (3, 1): Fr(-1, 2),
       (3, 2): Fr(-1, 2), (6, 0): Fr(1), (6, 1): Fr(1, 2), (6, 2): Fr(-1, 2), (6, 3): Fr(-1),
       (6, 4): Fr(-1, 2), (6, 5): Fr(1, 2)}


def transfer(lat, omega, n, m):
    """T(k), the conditions of its two sums, and whether every cos(theta) is +-1."""
    w = Fr(omega)
    num = den = an = ad = Fr(0)
    signs = True
    for v, p, c in zip(np.asarray(lat.vel).reshape(-1, 3), lat.phi, lat.chi):
        # k.v in sixths of a turn
        j = sum(int(m[a]) * int(v[a]) * (6 // n[a]) for a in range(3)) % 6
        cos = COS[6, j]
        signs = signs and abs(cos) == 1
        q = 1 - 2 * (1 - w) * cos + (1 - w) ** 2
        a, b = Fr(c) * (cos - (1 - w)) / q, Fr(p) * (2 - w) * (1 - cos) / q
        num, den, an, ad = num + a, den + b, an + abs(a), ad + abs(b)
    T = num / den
    return T, (float(an / abs(num)) if num else np.inf) + float(ad / abs(den)), signs


def mode(n, m):
    """Product of cosines of mode m, exact values, shape (nz, ny, nx)."""
    f = [np.array([float(COS[n[a], int(m[a]) * x % n[a]]) for x in range(n[a])]) for a in range(3)]
    return f[2][:, None, None] * f[1][None, :, None] * f[0][None, None, :]


@pytest.mark.gpu
@pytest.mark.parametrize("lattice,order,n,taus", [
    ("D1Q5", 1, (6, 1, 1), (0.5005, 0.505, 0.52, 0.6, 0.9)),
    ("D2Q25", 3, (6, 2, 1), (0.5005, 0.505, 0.52, 0.6, 0.9)),
    ("D3Q19", 1, (6, 2, 3), (0.5005, 0.505, 0.52, 0.6, 0.9)),
    ("D3Q111", 1, (2, 6, 2), (0.5005, 0.505, 0.52, 0.6, 0.9)),
    ("D3Q111", 3, (3, 2, 6), (0.5005, 0.505, 0.52, 0.6, 0.9)),
    # stable only above these
    ("D1Q9", 5, (6, 1, 1), (0.65, 0.9)), ("D2Q81", 5, (2, 3, 1), (0.65, 0.9)),
    ("D3Q111", 5, (2, 6, 2), (0.7, 0.9)), ("D1Q13", 7, (6, 1, 1), (0.8, 0.99)),
    ("D2Q169", 7, (2, 6, 1), (0.8, 0.99)),
])
def test_transfer_near_omega_two(lattice, order, n, taus):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    lat = oracle.lattice(lattice, order)
    shape = n[::-1][3 - int(lattice[1]):]
    eps = 2.0 ** -52
    for tau in taus:
        omega = 1.0 / tau
        prob = pk.problem(lattice, shape, order, tau_lb=tau)
        checked = 0
        for m in itertools.product(*(range(k // 2 + 1) for k in n)):
            if not any(m):
                continue
            T, cond, signs = transfer(lat, omega, n, m)
            if cond > 1e6:      # T itself cancels at this mode
                continue
            rho = mode(n, m).reshape(shape)
            S = rho * (lat.cs2 * (tau - 0.5))
            r = torch.from_numpy(rho).cuda()
            phi = torch.empty_like(r)
            pk.fixed_point_fft(r, phi, prob)
            got = float((phi.cpu().numpy() * S).sum() / (S * S).sum())
            bound = eps * cond * (32 if signs else 32 + 8 / (2 - omega))
            assert abs(got / float(T) - 1) <= bound, (tau, m, got, float(T), bound)
            checked += 1
        assert checked > 0
