"""Default geometry of binary32 plans on grids of whole 64-site x pairs: the
x-pairs sweep from 22 pairs per SM on (its six pair slots per SM are then
filled almost four times), never for D2Q169 (three slots); the Phi of the staged
geometry that it replaces bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,order,pairs_per_sm,wide", [
    ("D3Q111", 5, 8, False), ("D3Q111", 5, 21, False), ("D3Q111", 5, 23, True),
    ("D2Q81", 5, 9, False), ("D2Q81", 5, 23, True),
    ("D2Q169", 7, 8, False), ("D2Q169", 7, 30, False),
])
def test_default_geometry_of_binary32(lattice, order, pairs_per_sm, wide):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    rows = -(-pairs_per_sm * nsm // 2)           # rows of two pairs
    shape = (rows, 128) if lattice[1] == "2" else (-(-rows // 8), 8, 128)
    rho = torch.randn(shape, generator=torch.Generator().manual_seed(2),
                      dtype=torch.float64).cuda()
    last = pk._pkr.pkr_variant_count(pk.LATTICES[lattice]) - 1
    out = []
    for v in (-1, last if not wide else 2):
        prob = pk.problem(lattice, shape, order, tau_lb=1.7, max_sweeps=100, precision="fp32",
                          variant=v)
        phi = torch.empty_like(rho)
        with pk.Plan(prob) as P:
            P.load_source(rho)
            _, st = P.run(6, check_every=1000)
            P.phi(phi)
        out.append((phi, st["variant"]))
    assert out[0][1] == (last if wide else 2)
    assert torch.equal(out[0][0], out[1][0])
