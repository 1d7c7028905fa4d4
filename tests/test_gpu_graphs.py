"""Per-step-checked binary64 runs as captured graphs: pinned geometries and
grids beyond the resident forms (both asserted through the plan's step form).

The graph applies the stopping rule on the device.  Such a run takes the same
steps as the host loop one call at a time, stops at the same step with the same
residual and Phi bit for bit, reports divergence, and goes on correctly."""
import pytest

import oracle

pytestmark = pytest.mark.gpu


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


def _rows(pk, tiles_per_sm):
    """Rows of 64 sites one beyond that many 32-site tiles per SM."""
    import torch
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    return tiles_per_sm * nsm // 2 + 1


# (lattice, order, shape or tiles per SM, tau_lb, variant)
CASES = [
    ("D2Q169", 7, (24, 20), 6.04398, 5), ("D2Q169", 7, (16, 12), 1.0, 2),
    ("D3Q111", 5, (10, 9, 8), 1.3, 0), ("D1Q13", 7, (64,), 1.0, 1),
    ("D3Q111", 5, (3, 5, 64), 1.3, 8),
    ("D2Q25", 3, 4, 1.0, -1),       # scalar stencil beyond 4 tiles per SM
    ("D2Q25", 3, 2, 1.5, -1),       # population sweep beyond 2 tiles per SM
    ("D3Q19", 1, 4, 1.0, -1),
]


@pytest.mark.parametrize("kind", ["rel_l2", "max_abs"])
@pytest.mark.parametrize("lattice,order,shape,tau,variant", CASES)
def test_graph_run_equals_host_steps(pk, lattice, order, shape, tau, variant, kind):
    import torch
    if isinstance(shape, int):
        rows = _rows(pk, shape)
        shape = (rows, 64) if lattice[1] == "2" else (-(-rows // 8), 8, 64)
    rho = _rho(shape, 5)
    prob = pk.problem(lattice, shape, order, tau_lb=tau, max_sweeps=10 ** 6, variant=variant)
    out = [torch.empty_like(rho) for _ in range(2)]
    with pk.Plan(prob) as P, pk.Plan(prob) as H:
        assert P.step_form()[4] == 0
        P.load_source(rho)
        H.load_source(rho)
        # a graph, a second one and a rest of host steps that do not stop, ...
        P.run(150, tol=1e-300, tol_kind=kind, check_every=1)
        for _ in range(150):
            _, h = H.run(1, tol=1e-300, tol_kind=kind, check_every=1)
            if h["residual"] < 1e-300:   # a tiny grid comes to rest exactly
                break
        assert P.steps() == H.steps()
        assert torch.equal(P.phi(out[0]), H.phi(out[1]))
        # ... then on to a tolerance that is passed inside a graph
        tol = max(h["residual"], 1e-13) * 0.5
        _, s = P.run(448, tol=tol, tol_kind=kind, check_every=1)
        for _ in range(448):
            _, h = H.run(1, tol=tol, tol_kind=kind, check_every=1)
            if h["residual"] < tol:
                break
        assert P.steps() == H.steps()
        assert s["residual"] == pytest.approx(h["residual"], rel=1e-9, abs=1e-18)
        assert torch.equal(P.phi(out[0]), H.phi(out[1]))
        # plain steps, and another checked run from an array of the other parity
        P.run(7)
        H.run(7)
        P.run(64, tol=1e-300, tol_kind=kind, check_every=1)
        for _ in range(64):
            _, h = H.run(1, tol=1e-300, tol_kind=kind, check_every=1)
            if h["residual"] < 1e-300:
                break
        assert P.steps() == H.steps()
        assert torch.equal(P.phi(out[0]), H.phi(out[1]))


@pytest.mark.parametrize("lattice,order,shape,tau,variant", CASES[:3])
def test_graph_solve_stops_with_the_oracle(pk, lattice, order, shape, tau, variant):
    import numpy as np
    import torch
    rho = _rho(shape, 21)
    tol = 1e-11
    ref = oracle.solve(rho.cpu().numpy(), lattice, order, tau_lb=tau, tol=tol, tol_kind=0,
                       check_every=1, max_steps=100000)
    phi = torch.empty_like(rho)
    rc, st = pk.solve(rho, phi, pk.problem(lattice, shape, order, tau_lb=tau, tol=tol,
                                           tol_kind="max_abs", check_every=1, max_sweeps=100000,
                                           variant=variant))
    assert rc == 0 and st["sweeps"] == ref.steps and st["variant"] == variant
    got = phi.cpu().numpy()
    assert np.linalg.norm(got - ref.phi) <= 1e-12 * np.linalg.norm(ref.phi)


@pytest.mark.parametrize("shape,tau,variant", [((8, 9, 10), 1.3, 0), (4, 1.0, -1)])
def test_graph_run_reports_divergence(pk, shape, tau, variant):
    """A source that overflows stops the run at its first check."""
    import torch
    if isinstance(shape, int):
        shape = (-(-_rows(pk, shape) // 8), 8, 64)
    rho = _rho(shape, 3)
    prob = pk.problem("D3Q19", shape, 1, tau_lb=tau, epsilon=1e-320, tol=1e-10, check_every=1,
                      max_sweeps=200, variant=variant)
    with pk.Plan(prob) as P:
        assert P.step_form()[4] == 0
        P.load_source(rho)
        rc, _ = P.run(128, tol=1e-10, check_every=1)
        assert rc == -5
    phi = torch.full_like(rho, 7.0)
    with pytest.raises(pk.PkrError) as e:
        pk.solve(rho, phi, prob)
    assert e.value.status == -5
    assert bool((phi == 7.0).all())
