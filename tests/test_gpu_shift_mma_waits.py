"""The integer tensor-core kernel when its bounded waits run out: nothing is made up, and the next call is right.

With the limit cut to one cycle a launch's waits give up.  The call returns, the fault flag reads 1 and then 0, every
output is either the right one or left as it was, and the reported max|y| is 2^31, which no proof of 32-bit sums
accepts.  With the default limit restored the same call gives every output.  Rows and columns as lanes, a tile a CTA
and the reduction split over a cluster, 32-bit and forced 64-bit sums (two passes of a split tile)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CANARY = 0x5A5A5A5A
FC = [
    (64, 8192, 4096),    # columns as lanes, split
    (64, 512, 19500),    # columns as lanes, a tile a CTA
    (256, 8192, 512),    # rows as lanes, split
    (2560, 2048, 1024),  # rows as lanes, a tile a pair of CTAs
]
CONV = [
    (8, 64, 56, 64, 3),   # 64-column tiles, more of them than pairs
    (8, 512, 12, 512, 3),  # 128-column tiles, split
]


def _codes(g, shape):
    s = torch.randint(-1, 2, shape, device="cuda", generator=g, dtype=torch.int8)
    return s, torch.randint(-12, -7, shape, device="cuda", generator=g, dtype=torch.int8)


def _check(ds, call, shape):
    def run():
        y = torch.full(shape, CANARY, dtype=torch.int32, device="cuda")
        amax_io = torch.zeros(2, dtype=torch.int32, device="cuda")
        call(y, amax_io)
        torch.cuda.synchronize()
        return y, int(amax_io.cpu().numpy().view(np.uint32)[1])

    assert ds.ds_bf16_fault_flag() == 0
    try:
        ds.ds_bf16_set_wait_limit(1)
        y_cut, amax_cut = run()
    finally:
        ds.ds_bf16_set_wait_limit(0)
    assert ds.ds_bf16_fault_flag() == 1
    assert ds.ds_bf16_fault_flag() == 0  # read and cleared
    want, amax = run()
    assert ds.ds_bf16_fault_flag() == 0
    assert not bool((want == CANARY).any())
    assert amax == int(want.long().abs().max())
    assert bool(((y_cut == want) | (y_cut == CANARY)).all())
    assert bool((y_cut == CANARY).any())
    assert amax_cut == 1 << 31


@pytest.mark.parametrize("flags", [0, 16])
@pytest.mark.parametrize("shape", FC)
def test_fc_gives_up_cleanly(dslib, shape, flags):
    ds, (M, K, N) = dslib, shape
    g = torch.Generator("cuda").manual_seed(M + K)
    w = ds.pack_shift_weights(*_codes(g, (N, K)))
    x = torch.randint(-(1 << 20), 1 << 20, (M, K), device="cuda", generator=g, dtype=torch.int32)
    _check(ds, lambda y, a: ds.ds_linear_shift(x, w.desc, None, y, M, K, N, flags | ds.DS_AMAX_OUT, a), (M, N))


@pytest.mark.parametrize("flags", [0, 16])
@pytest.mark.parametrize("geom", CONV)
def test_conv_gives_up_cleanly(dslib, geom, flags):
    ds, (B, C, H, K, R) = dslib, geom
    g = torch.Generator("cuda").manual_seed(B + C)
    w = ds.pack_shift_weights(*_codes(g, (K, C, R, R)))
    x = torch.randint(-(1 << 20), 1 << 20, (B, C, H, H), device="cuda", generator=g, dtype=torch.int32)
    _check(ds, lambda y, a: ds.ds_conv2d_shift(x, w.desc, None, None, y, B, C, H, H, K, R, R, 1, 1, 1, 1,
                                               flags | ds.DS_AMAX_OUT, a), (B, K, H, H))
