"""Which kernel a plan's rules choose, and each form of the scalar stencil
against rolls in binary64 on a grid that takes it.

The rules weigh the busiest SM's time, so the shapes below hold for the 152 SMs
of a GB300."""
import pytest

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12   # the parity bar of every binary64 path
SWEEP, SWEEP16, STENCIL, PLANES = range(4)


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the shapes are chosen for 152 SMs")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    return pk


def _rho(shape, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=torch.float64).cuda()


# (kind, planes per chunk or partial sums, rows of a tile).  Planes, for tiles
# of 8 and 16 rows: fewer planes than the stencil spans, one chunk of z, a last
# chunk of fewer planes, more chunks than the largest grid has blocks; then a
# thread per site, in one chain and in the parts of the small grids.
STENCILS = [
    ("D3Q111", 5, (4, 118, 312), (PLANES, 4, 8)),
    ("D3Q111", 5, (7, 446, 64), (PLANES, 7, 8)),
    ("D3Q111", 5, (9, 195, 96), (PLANES, 5, 8)),
    ("D3Q111", 5, (4, 1760, 1440), (PLANES, 4, 16)),
    ("D3Q111", 5, (3, 368, 402), (PLANES, 3, 16)),
    ("D3Q111", 5, (7, 459, 227), (PLANES, 7, 16)),
    ("D3Q111", 5, (17, 59, 621), (PLANES, 6, 16)),
    ("D3Q19", 1, (17, 152, 254), (PLANES, 17, 8)),
    ("D3Q19", 1, (64, 39, 374), (PLANES, 13, 8)),
    ("D3Q19", 1, (30, 39, 639), (PLANES, 10, 8)),
    ("D3Q19", 1, (8, 398, 189), (PLANES, 8, 16)),
    ("D3Q19", 1, (53, 32, 464), (PLANES, 11, 16)),
    ("D3Q111", 5, (4, 230, 420), (STENCIL, 1, 0)),
    ("D3Q111", 5, (2, 200, 201), (STENCIL, 1, 0)),
    ("D3Q19", 1, (45, 130, 290), (STENCIL, 1, 0)),
    ("D2Q81", 5, (301, 203), (STENCIL, 1, 0)),
    ("D3Q111", 5, (20, 21, 22), (STENCIL, 4, 0)),
    ("D2Q169", 7, (61, 90), (STENCIL, 4, 0)),
]


@pytest.mark.parametrize("lattice,order,shape,form", STENCILS)
def test_stencil_form_and_values(pk, lattice, order, shape, form):
    import torch
    rho = _rho(shape, 7)
    vel, _, phi, chi, cs2 = pk.lattice_info(lattice, order)
    S = (rho - rho.mean()) * (cs2 * 0.5)
    axes = tuple(range(len(shape)))

    def apply(w, field):
        out = torch.zeros_like(field)
        for v, c in zip(vel.tolist(), w.tolist()):
            out += c * torch.roll(field, tuple(v[2 - a] for a in range(3))[3 - len(shape):], axes)
        return out

    St = apply(chi, S)
    old, now = torch.zeros_like(S), St
    for _ in range(3):
        old, now = now, apply(phi, now) + St
    prob = pk.problem(lattice, shape, order, tau_lb=1.0, max_sweeps=100)
    got = torch.empty_like(rho)
    with pk.Plan(prob) as P:
        assert P.step_form()[:3] == form
        P.load_source(rho)
        _, st = P.run(4, check_every=4)
        P.phi(got)
    assert st["variant"] == -1
    assert float((got - now).norm() / now.norm()) <= FP64_TOL
    want = float((now - old).norm() / now.norm())
    assert st["residual"] == pytest.approx(want, rel=1e-10)


@pytest.mark.parametrize("lattice,order,shape,tau,variant,resident", [
    ("D1Q13", 7, (64,), 1.0, -1, 1), ("D1Q13", 7, (631,), 1.0, -1, 2),
    ("D2Q169", 7, (64, 64), 1.5, -1, 3), ("D3Q111", 5, (20, 21, 22), 1.0, -1, 2),
    ("D3Q111", 5, (20, 21, 22), 1.5, -1, 3), ("D3Q111", 5, (22, 22, 22), 1.5, -1, 0),
    ("D3Q111", 5, (27, 27, 28), 1.0, -1, 0), ("D2Q25", 3, (64, 64), 1.5, 0, 0),
])
def test_form_of_per_step_checked_runs(pk, lattice, order, shape, tau, variant, resident):
    prob = pk.problem(lattice, shape, order, tau_lb=tau, max_sweeps=100, variant=variant)
    with pk.Plan(prob) as P:
        assert P.step_form()[4] == resident


def test_step_form_refuses_null(pk):
    import ctypes
    assert pk._pkr.pkr_plan_step_form(None, (ctypes.c_int32 * 5)()) == -1
    with pk.Plan(pk.problem("D1Q5", (8,), 1, tau_lb=1.2, max_sweeps=10)) as P:
        assert pk._pkr.pkr_plan_step_form(P._h, None) == -1
