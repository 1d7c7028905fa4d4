"""Status of the FFT comparator when cuFFT gets no work space: PKR_ECUDA for a
finite rho, PKR_EINVAL for a non-finite one (as with work space), phi untouched
both times, and the next call works."""
import pytest

pytestmark = pytest.mark.gpu

V = 4000037      # prime: cuFFT's work area is several times the data


def test_nonfinite_rho_is_refused_before_a_failed_transform():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_05869_gb300 as pk
    prob = pk.problem("D1Q5", (V,), 1, tau_lb=1.0)
    small = pk.problem("D1Q5", (96,), 1, tau_lb=1.0)
    r = torch.randn(V, dtype=torch.float64, generator=torch.Generator().manual_seed(1)).cuda()
    bad = r.clone()
    bad[7] = float("nan")
    phi = torch.full_like(r, 7.0)
    a, b = torch.randn(96, dtype=torch.float64).cuda(), torch.empty(96, dtype=torch.float64).cuda()
    pk.fixed_point_fft(a, b, small)      # loads the kernels that the calls below launch

    def status(rho):
        try:
            pk.fixed_point_fft(rho, phi, prob)
            return 0
        except pk.PkrError as e:
            return e.status

    # the call's own block is 32 V bytes; leave it and a little more free
    for margin in (256, 128, 64, 32):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        held = torch.empty(free - 32 * V - margin * 2 ** 20, dtype=torch.uint8, device="cuda")
        phi.fill_(7.0)
        ok, nan = status(r), status(bad)
        untouched = bool((phi == 7.0).all())
        del held
        torch.cuda.empty_cache()
        if ok != 0:
            break
    assert ok == -6 and untouched, ok
    assert nan == -1
    pk.fixed_point_fft(a, b, small)
    assert bool(torch.isfinite(b).all())
