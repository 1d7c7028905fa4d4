"""pkr_stats.variant names what ran: -2 for a population run in cooperative
launches, the geometry for captured graphs and host-stepped runs, -1 for the
scalar stencil."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,tau,variant,steps,want", [
    ((20, 21), 2.0, -1, 64, -2), ((20, 21), 2.0, -1, 63, 5), ((20, 21), 2.0, 3, 64, 3),
    ((20, 21), 1.0, -1, 64, -1), ((130, 140), 2.0, -1, 64, 5),
])
def test_reported_variant_of_per_step_checked_runs(shape, tau, variant, steps, want):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    rho = torch.randn(shape, generator=torch.Generator().manual_seed(3),
                      dtype=torch.float64).cuda()
    phi = torch.empty_like(rho)
    prob = pk.problem("D2Q81", shape, 5, tau_lb=tau, max_sweeps=steps, tol=1e-300, check_every=1,
                      variant=variant)
    with pk.Plan(prob) as P:
        P.load_source(rho)
        _, st = P.run(steps, tol=1e-300, check_every=1)
        assert st["variant"] == want and P.steps() == steps
        _, st = P.run(2)
        assert st["variant"] == (want if want != -2 else 5)   # plain steps again
    if steps >= 64:
        prob.max_sweeps = steps + 1
    _, st = pk.solve(rho, phi, prob)
    assert st["variant"] == want
