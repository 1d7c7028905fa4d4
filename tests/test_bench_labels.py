"""The benchmark's kernel labels follow the form that the plan reports
(pkr_plan_step_form), not a guess from the grid's size."""
import pytest

import __graft_entry__  # noqa: F401  (puts the repo root on the path)


@pytest.fixture
def bench(monkeypatch):
    import bench as b
    monkeypatch.setattr(b, "PRECISION", "fp16")
    return b


def test_binary16_labels(bench):
    assert bench.kernel_label(None, 0, (1, 1, 0, 10, 0)) == "sweep_h16_kernel<D3Q111>"
    assert bench.kernel_label(None, 1, (1, 2, 0, 10, 0)) == "sweep_h16p_kernel<D3Q111>"
    assert bench.kernel_label(None, 1, (1, 2, 1, 10, 0)) == \
        "sweep_h16p_kernel<D3Q111> (copies ahead)"
    assert bench.kernel_label(None, 1, (1, 4, 1, 10, 0)) == "sweep_h16w_kernel<D3Q111>"


def test_stencil_labels(bench):
    assert bench.stencil_label((3, 16, 8, 10, 0), 111) == ("stencil_planes_kernel<D3Q111,8>", 47)
    assert bench.stencil_label((3, 16, 16, 10, 0), 19) == ("stencil_planes_kernel<D3Q111,16>", 13)
    assert bench.stencil_label((2, 1, 0, 10, 0), 111) == ("stencil_kernel<D3Q111>", 111)
    assert bench.stencil_label((2, 4, 0, 10, 0), 111) == ("stencil_kernel<D3Q111>", 115)
