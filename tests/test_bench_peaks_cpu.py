"""The benchmark's roofline is the one of the kernels that a workload's sizes select."""
import bench
import pytest
from paper_1905_13298_gb300 import build


@pytest.fixture(scope="module")
def ds():
    build.build_library()
    import paper_1905_13298_gb300 as ds
    return ds


def test_peak_follows_the_route(monkeypatch, ds):
    monkeypatch.setattr(bench, "alu_peak", lambda dev=None: (40.0, 152, 2070.0, "measured"))
    assert bench.route_peak(None, ds.ds_linear_shift_route(64, 784, 512)) == ("alu", 40.0)
    name, tops = bench.route_peak(None, ds.ds_linear_shift_route(8192, 4096, 4096))
    assert name == "tensor" and tops == pytest.approx(40.0 * 2 * 8192 / 17 / 128)
    assert bench.route_peak(None, ds.ds_linear_shift_route(64, 25088, 4096))[0] == "tensor"
    assert bench.route_peak(None, ds.ds_conv2d_shift_route(1, 512, 7, 7, 512, 3, 3, 1, 1, 1, 1))[0] == "alu"
