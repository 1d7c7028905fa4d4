"""The staged binary64 sweep with and without copies ahead of a tile: below and
above the number of rounds of tiles from which a launch takes them (about 1.5
per resident warp group, 4 for D2Q169), on ragged grids, every staged geometry
gives the Phi of the warp-specialised sweep bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,order,shape", [
    ("D3Q111", 5, (30, 31, 33)), ("D3Q111", 5, (40, 41, 37)),
    ("D2Q81", 5, (191, 201)), ("D2Q81", 5, (411, 409)),
    ("D2Q169", 7, (203, 151)), ("D2Q169", 7, (411, 409)),
])
def test_staged_geometries_agree_at_any_number_of_rounds(lattice, order, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    rho = torch.randn(shape, generator=torch.Generator().manual_seed(9),
                      dtype=torch.float64).cuda()
    staged = pk._pkr.pkr_batch_variant_count(pk.LATTICES[lattice])
    out, residual = [], []
    for v in list(range(staged)) + [staged]:      # the last one: warp-specialised
        phi = torch.empty_like(rho)
        prob = pk.problem(lattice, shape, order, tau_lb=1.7, max_sweeps=100, variant=v)
        with pk.Plan(prob) as P:
            P.load_source(rho)
            P.run(4)
            _, st = P.run(4, check_every=4)
            P.phi(phi)
        assert st["variant"] == v
        out.append(phi)
        residual.append(st["residual"])
    for phi, r in zip(out[:-1], residual):
        assert torch.equal(phi, out[-1])
        assert r == pytest.approx(residual[-1], rel=1e-12)
