"""Forms of the binary16 sweep: which one a grid takes, just below and above the
line of each rule, and the same Phi as one site per lane bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


# tiles of 128 sites per SM, sites of a row, (sites per lane, copies ahead)
@pytest.mark.parametrize("lattice,order,per_sm,nx,form", [
    ("D3Q111", 5, 1, 128, (2, 0)), ("D3Q111", 5, 7.8, 128, (2, 0)), ("D3Q111", 5, 8.1, 128, (4, 1)),
    ("D3Q111", 5, 8.9, 192, (2, 0)), ("D3Q111", 5, 9.2, 192, (2, 1)), ("D3Q111", 5, 9.2, 64, (2, 1)),
    ("D3Q19", 1, 5.8, 128, (2, 0)), ("D3Q19", 1, 6.2, 128, (4, 1)), ("D3Q19", 1, 9.2, 64, (2, 0)),
    ("D2Q25", 3, 9.2, 256, (4, 1)), ("D2Q81", 5, 9.2, 256, (2, 0)), ("D2Q81", 5, 73, 128, (4, 1)),
    ("D2Q169", 7, 6, 128, (2, 0)), ("D2Q169", 7, 73, 128, (2, 0)), ("D2Q169", 7, 73, 256, (4, 1)),
    ("D1Q5", 1, 30, 0, (2, 0)), ("D1Q9", 5, 25, 0, (2, 0)), ("D1Q13", 7, 27, 0, (4, 1)),
])
def test_form_and_values(lattice, order, per_sm, nx, form):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    sites = int(per_sm * nsm) * 128
    if lattice[1] == "1":
        shape = (sites,)
    elif lattice[1] == "2":
        shape = (-(-sites // nx), nx)
    else:
        ny = 7 if sites < 10 ** 6 else 41
        shape = (-(-sites // (nx * ny)), ny, nx)
    rho = torch.randn(shape, generator=torch.Generator().manual_seed(4),
                      dtype=torch.float64).cuda()
    out = []
    for v in (-1, 0):
        prob = pk.problem(lattice, shape, order, tau_lb=1.7, max_sweeps=100, precision="fp16",
                          variant=v)
        phi = torch.empty_like(rho)
        with pk.Plan(prob) as P:
            assert P.step_form()[:3] == ((1,) + form if v < 0 else (1, 1, 0))
            P.load_source(rho)
            P.run(7, check_every=1000)
            P.phi(phi)
        out.append(phi)
    assert torch.equal(out[0], out[1])
