"""Sweeps with several sites per lane against the one-site forms.

binary16 with four sites per lane (x rows of whole 128-site tiles) and binary32
with two (x rows of whole 64-site pairs) do per site what the one-site kernels
do, in the same order: the same Phi bit for bit between residual checks.  A
check's sums run in another order, and binary32 and binary16 steps take the
mass it measures out through the source, so after checks the two agree to
rounding of the storage."""
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


def _run(pk, rho, lattice, order, precision, variant, steps, every):
    import torch
    prob = pk.problem(lattice, rho.shape, order, tau_lb=1.7, max_sweeps=1000, precision=precision,
                      variant=variant)
    phi = torch.empty_like(rho)
    with pk.Plan(prob) as P:
        P.load_source(rho)
        _, st = P.run(steps, check_every=every)
        P.phi(phi)
    return phi, st


def _rho(shape, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=torch.float64).cuda()


# one tile per row (both halos wrap), several, reaches 1 to 6, tile counts that
# leave the last block part full; all with a tile for every resident warp
@pytest.mark.parametrize("lattice,order,shape", [
    ("D3Q111", 5, (31, 30, 128)), ("D3Q111", 5, (7, 67, 256)), ("D3Q111", 5, (3, 103, 384)),
    ("D3Q19", 1, (33, 29, 128)), ("D2Q25", 3, (913, 128)), ("D2Q81", 5, (457, 256)),
    ("D2Q169", 7, (915, 128)), ("D1Q13", 7, (128 * 913,)),
])
def test_binary16_four_sites_per_lane(pk, lattice, order, shape):
    import torch
    rho = _rho(shape, 3)
    for steps, every in ((7, 1000), (8, 4)):
        one, _ = _run(pk, rho, lattice, order, "fp16", 0, steps, every)
        four, st = _run(pk, rho, lattice, order, "fp16", -1, steps, every)
        assert st["variant"] == 1
        if every > steps:
            assert torch.equal(one, four)
        else:
            assert float((one - four).norm() / one.norm()) <= 1e-6


@pytest.mark.parametrize("lattice,order,shape", [
    ("D3Q111", 5, (5, 7, 64)), ("D3Q111", 5, (37, 33, 64)), ("D3Q111", 5, (9, 11, 192)),
    ("D3Q111", 5, (3, 3, 128)), ("D2Q81", 5, (41, 128)), ("D2Q169", 7, (7, 64)),
    ("D2Q169", 7, (13, 320)),
])
def test_binary32_two_sites_per_lane(pk, lattice, order, shape):
    import torch
    last = pk._pkr.pkr_variant_count(pk.LATTICES[lattice]) - 1
    rho = _rho(shape, 4)
    for steps, every in ((7, 1000), (8, 4)):
        pair, _ = _run(pk, rho, lattice, order, "fp32", last - 1, steps, every)
        wide, st = _run(pk, rho, lattice, order, "fp32", last, steps, every)
        assert st["variant"] == last
        if every > steps:
            assert torch.equal(pair, wide)
        else:
            assert float((pair - wide).norm() / pair.norm()) <= 1e-6


@pytest.mark.parametrize("K", [1, 2, 3, 7])
@pytest.mark.parametrize("precision", ["fp64", "fx64", "fp32"])
def test_batch_schedule_at_every_window_length(pk, K, precision):
    """A batch of grids of one tile, a few and many, with windows of K steps:
    each request's Phi is the plan's after the steps it reports."""
    import torch
    shapes = [(3, 4, 2), (9, 8, 11), (20, 30, 25), (3, 3, 3)]
    with pk.Context("D3Q111", 5, precision=precision, check_every=K) as ctx:
        rho = [_rho(s, 10 + j) for j, s in enumerate(shapes)]
        phi = [torch.empty_like(r) for r in rho]
        t = [ctx.submit(r, p, tau_lb=1.7, max_sweeps=5 + 3 * j, tol=0.0)
             for j, (r, p) in enumerate(zip(rho, phi))]
        ctx.run()
        for j, ticket in enumerate(t):
            rc, st = ctx.wait(ticket)
            assert rc == 0 and st["sweeps"] >= 5 + 3 * j and (st["sweeps"] + 1) % K == 0
            # binary32 plans and requests remove the mass at the same steps
            # only from their first check on: compare up to binary32 rounding
            prob = pk.problem("D3Q111", shapes[j], 5, tau_lb=1.7, max_sweeps=1000,
                              precision=precision, variant=2)
            want = torch.empty_like(rho[j])
            with pk.Plan(prob) as P:
                P.load_source(rho[j])
                P.run(st["sweeps"], check_every=1000)
                P.phi(want)
            err = float((phi[j] - want).norm() / want.norm())
            assert err <= (1e-12 if precision != "fp32" else 1e-5), (j, err)
