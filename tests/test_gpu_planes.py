"""The plane form of the scalar stencil (tau_lb = 1, 3D) against the stencil
written with torch.roll in binary64."""
import pytest

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12   # the parity bar of every binary64 path


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    return pk


def _rho(shape, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=torch.float64).cuda()


# plane tiles are 32 x 16 sites; the form is taken once tiles and z chunks
# outnumber the SMs.  Ragged in every axis, whole tiles with one
# plane left over, fewer planes than the stencil spans.
@pytest.mark.parametrize("lattice,order", [("D3Q111", 5), ("D3Q19", 1)])
@pytest.mark.parametrize("shape", [(45, 130, 290), (17, 192, 416), (4, 230, 420), (96, 64, 96)])
def test_plane_stencil_matches_rolls(pk, lattice, order, shape):
    import torch
    rho = _rho(shape, 7)
    vel, _, phi, chi, cs2 = pk.lattice_info(lattice, order)
    S = (rho - rho.mean()) * (cs2 * 0.5)

    def apply(w, field):
        out = torch.zeros_like(field)
        for v, c in zip(vel.tolist(), w.tolist()):
            out += c * torch.roll(field, (v[2], v[1], v[0]), (0, 1, 2))
        return out

    St = apply(chi, S)
    old, now = torch.zeros_like(S), St
    for _ in range(3):
        old, now = now, apply(phi, now) + St
    prob = pk.problem(lattice, shape, order, tau_lb=1.0, max_sweeps=100)
    got = torch.empty_like(rho)
    with pk.Plan(prob) as P:
        P.load_source(rho)
        _, st = P.run(4, check_every=4)
        P.phi(got)
    assert float((got - now).norm() / now.norm()) <= FP64_TOL
    want = float((now - old).norm() / now.norm())
    assert st["residual"] == pytest.approx(want, rel=1e-10)


# The finer tiles (32 x 8) and the one-thread-per-site form beyond the resident
# grids: ragged in every axis, whole tiles in one chunk of z, chunks of fewer
# planes than the stencil spans (32 x 16), few tiles.
@pytest.mark.parametrize("lattice,order", [("D3Q111", 5), ("D3Q19", 1)])
@pytest.mark.parametrize("shape", [(53, 163, 62), (47, 152, 160), (5, 640, 640), (29, 30, 31),
                                   (17, 200, 47)])
def test_stencil_forms_match_rolls(pk, lattice, order, shape):
    test_plane_stencil_matches_rolls(pk, lattice, order, shape)
