"""Runs of per-step-checked binary64 steps that stay on the GPU.

A resident run (steps >= 64, check_every = 1, small grid) must take the same
steps as the host loop does one call at a time: same stopping step, same Phi
bit for bit, and a plan that goes on correctly afterwards."""
import pytest

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


# one block (Q V <= 8192, V <= 512); over blocks, scalar and population form;
# ragged last tiles, edges below the reach, one and several velocity groups
CASES = [
    ("D1Q13", 7, (64,), 1.0), ("D1Q5", 3, (33,), 1.0), ("D1Q5", 1, (512,), 1.0),
    ("D1Q13", 7, (5,), 1.0), ("D2Q25", 3, (17, 19), 1.0), ("D1Q13", 7, (631,), 1.0),
    ("D2Q25", 3, (24, 31), 1.0), ("D2Q169", 7, (33, 32), 1.0), ("D3Q111", 5, (9, 8, 11), 1.0),
    ("D1Q13", 7, (100,), 1.5), ("D1Q5", 1, (1,), 1.5), ("D2Q81", 5, (20, 21), 2.0),
    ("D3Q19", 1, (9, 8, 7), 1.2), ("D2Q169", 7, (5, 40), 6.0), ("D3Q111", 5, (2, 9, 16), 3.0),
]


@pytest.mark.parametrize("kind", ["rel_l2", "max_abs"])
@pytest.mark.parametrize("lattice,order,shape,tau", CASES)
def test_resident_run_equals_host_steps(pk, lattice, order, shape, tau, kind):
    import torch
    rho = _rho(shape, 5)
    prob = pk.problem(lattice, shape, order, tau_lb=tau, max_sweeps=10 ** 6)
    out = [torch.empty_like(rho) for _ in range(2)]
    with pk.Plan(prob) as P, pk.Plan(prob) as H:
        P.load_source(rho)
        H.load_source(rho)
        # 90 steps that do not stop, then on to a tolerance they pass within 400 more
        P.run(90, tol=1e-300, tol_kind=kind, check_every=1)
        for _ in range(90):
            _, h = H.run(1, tol=1e-300, tol_kind=kind, check_every=1)
            if h["residual"] < 1e-300:   # a tiny grid comes to rest exactly
                break
        assert P.steps() == H.steps()
        assert torch.equal(P.phi(out[0]), H.phi(out[1]))
        tol = max(h["residual"], 1e-13) * 0.5
        _, s = P.run(400, tol=tol, tol_kind=kind, check_every=1)
        for _ in range(400):
            _, h = H.run(1, tol=tol, tol_kind=kind, check_every=1)
            if h["residual"] < tol:
                break
        assert P.steps() == H.steps()
        assert s["residual"] == pytest.approx(h["residual"], rel=1e-9, abs=1e-18)
        assert torch.equal(P.phi(out[0]), H.phi(out[1]))
        # plain steps from the state it left
        P.run(7)
        H.run(7)
        assert torch.equal(P.phi(out[0]), H.phi(out[1]))


def test_resident_run_over_several_launches(pk):
    """More steps than one launch takes (8192), and a zero source (stops at once)."""
    import torch
    rho = _rho((160,), 6)
    prob = pk.problem("D1Q5", (160,), 1, tau_lb=1.0, max_sweeps=10 ** 6)
    a, b = torch.empty_like(rho), torch.empty_like(rho)
    with pk.Plan(prob) as P, pk.Plan(prob) as H:
        P.load_source(rho)
        H.load_source(rho)
        P.run(8192 + 8192 + 77, tol=1e-300, check_every=1)
        H.run(8192 + 8192 + 77, check_every=4096)
        assert P.steps() == H.steps()
        assert torch.equal(P.phi(a), H.phi(b))
        P.load_source(torch.zeros_like(rho))
        rc, s = P.run(1000, tol=1e-12, check_every=1)
        assert rc == 0 and s["sweeps"] == 1 and s["residual"] == 0.0
        P.load_source(rho)
        rc, s = P.run(10 ** 6, tol=1e-13, check_every=1)
        assert rc == 0 and s["residual"] < 1e-13
        assert s["sweeps"] > 2 * 8192
