"""The size rules that choose a call's kernels, at sizes where both choices were timed (GB300, us per call).

Each entry: the sizes, the route, and the times of the CUDA cores, the rows-as-lanes and the columns-as-lanes tensor-core
kernels where they were taken.  The route must be the fastest of them, to 5%, or 1.5 us where all are short."""
import pytest

CC, TC, SWAP = 0, 1, 2
FC = [
    # M, K, N, route, CUDA cores, rows as lanes, columns as lanes
    (8, 25088, 4096, CC, None, None, None),
    (1024, 1028, 128, SWAP, 35.4, 56.4, 31.0),
    (384, 1368, 256, SWAP, 33.5, 58.0, 29.0),
    (256, 4100, 128, SWAP, 49.1, 64.2, 31.9),
    (384, 5464, 64, SWAP, 41.4, 49.6, 33.1),
    (384, 10924, 64, SWAP, 64.8, 61.9, 41.7),
    (1024, 7725, 48, TC, 102.5, 57.8, 98.8),
    (384, 10924, 128, SWAP, 98.0, 81.0, 44.0),
    (1024, 2900, 256, SWAP, 86.0, 60.0, 43.0),
    (129, 1440, 4096, TC, 116.0, 55.0, 60.0),
    (129, 2036, 4096, TC, 155.1, 62.5, 88.8),
    (129, 1021, 4096, TC, 92.8, 51.9, 61.5),
    (1024, 5796, 128, SWAP, 91.0, 69.0, 62.0),
    (1024, 5797, 128, TC, 98.6, 71.8, 80.1),
    (1024, 8196, 128, TC, 124.0, 75.0, 89.0),
    (64, 25088, 4096, SWAP, 565.0, None, 189.0),
    (8192, 4096, 4096, TC, 9930.0, 1460.0, None),
]
CONV = [
    # N, C, H, W, K, R, stride, pad, route, CUDA cores, tensor cores
    (4, 128, 32, 32, 128, 1, 1, 0, TC, 31.2, 32.1),
    (5, 128, 39, 39, 128, 1, 1, 0, TC, 37.2, 33.0),
    (5, 512, 23, 23, 64, 1, 1, 0, TC, 37.4, 31.6),
    (5, 16, 60, 60, 32, 3, 1, 1, TC, 33.9, 30.7),
    (32, 64, 56, 56, 64, 3, 1, 1, TC, 295.0, 109.0),
    (32, 64, 56, 56, 64, 1, 1, 0, CC, None, None),
]


@pytest.fixture(scope="module")
def ds():
    from paper_1905_13298_gb300 import build
    build.build_library()
    import paper_1905_13298_gb300 as ds
    ds.lib()
    return ds


def _fastest(times, route):
    known = {i: t for i, t in enumerate(times) if t is not None}
    assert not known or known[route] <= max(1.05 * min(known.values()), min(known.values()) + 1.5)


@pytest.mark.parametrize("case", FC)
def test_fc_route(ds, case):
    M, K, N, route, *times = case
    assert ds.ds_linear_shift_route(M, K, N) == route
    _fastest(times, route)


# the same without amax_io: M, K, N, route, CUDA cores, rows as lanes, columns as lanes
FC_NO_BOUND = [
    (16, 25088, 4096, CC, 538.9, None, 744.3),
    (9, 25088, 4096, CC, 539.0, None, 744.2),
    (64, 25088, 4096, SWAP, 1162.1, None, 747.6),
    (128, 4096, 4096, SWAP, 417.6, None, 248.6),
    (64, 4096, 1000, SWAP, 96.9, None, 82.1),
    (384, 10924, 128, SWAP, 177.5, 319.8, 100.0),
    (1024, 2052, 512, SWAP, 219.0, 249.0, 140.0),
    (384, 684, 4096, TC, 226.0, 169.0, 181.0),
    (1024, 68, 4096, CC, 82.0, None, 94.0),
    (1024, 4096, 4096, TC, 2955.3, 1594.7, None),
]
CONV_NO_BOUND = [
    # N, C, H, W, K, R, stride, pad, route, CUDA cores, tensor cores in tiles of 64 columns
    (4, 16, 171, 171, 16, 3, 1, 1, CC, 124.9, 164.6),
    (5, 16, 88, 88, 16, 3, 1, 1, TC, 103.0, 60.5),
    (4, 16, 121, 121, 16, 3, 1, 1, CC, 67.9, 100.7),
    (5, 3, 119, 119, 16, 7, 1, 3, TC, 188.8, 103.9),
    (4, 3, 169, 169, 16, 7, 1, 3, CC, 121.2, 147.0),
    (5, 128, 181, 181, 16, 1, 1, 0, TC, 243.0, 191.8),
    (4, 128, 17, 17, 512, 1, 1, 0, TC, 45.6, 37.0),
    (4, 512, 32, 32, 128, 1, 1, 0, TC, 83.0, 50.0),
    (32, 64, 56, 56, 64, 3, 1, 1, TC, 559.0, 388.8),
]


@pytest.mark.parametrize("case", FC_NO_BOUND)
def test_fc_route_without_a_bound(ds, case):
    M, K, N, route, *times = case
    assert ds.ds_linear_shift_route(M, K, N, False) == route
    _fastest(times, route)


@pytest.mark.parametrize("case", CONV)
def test_conv_route(ds, case):
    B, C, H, W, K, R, st, pd, route, *times = case
    assert ds.ds_conv2d_shift_route(B, C, H, W, K, R, R, st, st, pd, pd) == route
    _fastest(times, route)


@pytest.mark.parametrize("case", CONV_NO_BOUND)
def test_conv_route_without_a_bound(ds, case):
    B, C, H, W, K, R, st, pd, route, *times = case
    assert ds.ds_conv2d_shift_route(B, C, H, W, K, R, R, st, st, pd, pd, False) == route
    _fastest(times, route)


def test_refused_sizes_have_no_route(ds):
    assert ds.ds_linear_shift_route(0, 64, 64) == -1
    assert ds.ds_linear_shift_route(64, 0, 64) == -1
    assert ds.ds_linear_shift_route(64, 64, 65535 * 64 + 1) == -1
    assert ds.ds_linear_shift_route(1 << 40, 1 << 40, 1) == -1
    assert ds.ds_conv2d_shift_route(1, 64, 8, 8, 64, 9, 9, 1, 1, 0, 0) == -1  # kernel larger than the image
    assert ds.ds_conv2d_shift_route(1, 64, 8, 8, 64, 3, 3, 0, 1, 0, 0) == -1
    assert ds.ds_conv2d_shift_route(1, 1 << 20, 1 << 10, 1 << 10, 64, 1, 1, 1, 1, 0, 0) == -1
