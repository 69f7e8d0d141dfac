"""The tensor-core shift sums at the edges of their tiles, runs and digit ranges.

Reference: the operator in float64 on the GPU, one library product per shift value (every sum is below 2^53, so it is
exact), then bias, saturation, residual and ReLU.  The results are integers with one correct value: no tolerance.
The sizes are the smallest ones that the dispatch rules send to the kernel (2^27 terms for FC, 2^26 for convolutions)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _gen(seed):
    return torch.Generator("cuda").manual_seed(seed)


def _codes(g, shape, kind):
    n = int(np.prod(shape))
    t = torch.rand(n, device="cuda", generator=g)
    s = torch.where(t < 0.1, 0, torch.where(t < 0.55, -1, 1))
    if kind == "uniform":
        p = torch.randint(-15, 1, (n,), device="cuda", generator=g)
    elif kind == "plain":  # every weight +1: the largest sums
        s, p = torch.ones_like(s), torch.zeros(n, device="cuda", dtype=torch.int64)
    else:  # around a centre that keeps the columns' weights small
        up, down = (torch.empty(n, device="cuda").geometric_(0.5, generator=g) for _ in range(2))
        p = (-10 + up - down).clamp_(-15, 0)
    return s.to(torch.int8).reshape(shape), p.to(torch.int8).reshape(shape)


def _values(g, shape, top):
    """Signed values up to +-top with the extremes of every digit range among them."""
    x = torch.randint(-top, top, shape, device="cuda", generator=g, dtype=torch.int64)
    edge = torch.tensor([-top, top - 1, top if top < 2 ** 31 else top - 1, 0, -1, 65535, -65536, 32768], device="cuda")
    edge = edge.clamp(-top, top if top < 2 ** 31 else top - 1)
    flat = x.reshape(-1)
    flat[:: max(1, flat.numel() // 97)] = edge[torch.arange(flat[:: max(1, flat.numel() // 97)].numel(), device="cuda") % 8]
    return x.to(torch.int32)


def _sum(x, s, p, product):
    acc = 0
    for k in range(16):
        w = torch.where(p == -k, s, torch.zeros_like(s)).double()
        acc = acc + product((x >> k).double(), w)
    return acc


def _finish(acc, bias, residual=None, relu=False):
    lo, hi = -2.0 ** 31, 2.0 ** 31 - 1
    y = (acc + bias).clamp(lo, hi)
    if residual is not None:
        y = (y + residual).clamp(lo, hi)
    return (y.clamp(min=0) if relu else y).to(torch.int32)


# M, K, N, max |x|, codes.  M <= 128: weights as lanes; else rows as lanes, in pairs of 128
FC = [
    (9, 4096, 4096, 1 << 17, "centred"),
    (17, 4099, 2050, 1 << 20, "uniform"),         # K not a multiple of 4 or 16, two runs, ragged columns
    (64, 2064, 1030, (1 << 20) + 1, "centred"),   # two digits
    (65, 2052, 1025, 1 << 24, "uniform"),         # two row tiles of the swapped roles
    (128, 2048, 520, 1 << 28, "centred"),         # three digits
    (129, 1030, 1100, 1 << 31, "uniform"),        # four digits, a second pair tile of one row
    (300, 7700, 66, 1 << 20, "uniform"),          # three runs, 64-column tiles with a ragged one
    (257, 4100, 129, 1 << 14, "plain"),           # unbounded columns of equal weights
    (1030, 1031, 127, 1 << 20, "plain"),
]


@pytest.mark.parametrize("case", FC)
@pytest.mark.parametrize("flags", [0, 16])  # 32-bit sums where proven / always 64-bit
def test_fc(dslib, case, flags):
    ds, (M, K, N, top, kind) = dslib, case
    g = _gen(M * 31 + K + flags)
    s, p = _codes(g, (N, K), kind)
    x, b = _values(g, (M, K), top), torch.randint(-(1 << 16), 1 << 16, (N,), device="cuda", generator=g, dtype=torch.int32)
    amax_io = torch.zeros(2, dtype=torch.int32, device="cuda")
    y = ds.linear_shift(x, ds.pack_shift_weights(s, p), b, relu=bool(M & 1), amax_io=amax_io, flags=flags | ds.DS_AMAX_OUT)
    want = _finish(_sum(x, s, p, lambda a, w: a @ w.t()), b.double(), relu=bool(M & 1))
    assert torch.equal(y, want)
    assert int(amax_io.cpu().numpy().view(np.uint32)[1]) == int(want.long().abs().max())
    assert ds.ds_bf16_fault_flag() == 0


def test_fc_without_a_bound(dslib):
    """amax_io = NULL: four digits and 64-bit sums whatever the values."""
    g = _gen(5)
    s, p = _codes(g, (1030, 2052), "centred")
    x = _values(g, (64, 2052), 1 << 18)
    y = dslib.linear_shift(x, dslib.pack_shift_weights(s, p))
    assert torch.equal(y, _finish(_sum(x, s, p, lambda a, w: a @ w.t()), 0.0))


# B, C, H, W, K, R, S, stride, pad, max |x|, codes
CONV = [
    (2, 64, 24, 24, 130, 3, 3, 1, 1, 1 << 20, "centred"),
    (4, 65, 17, 16, 64, 3, 3, 1, 1, 1 << 18, "centred"),          # 64-column tiles, a partial last slot
    (1, 15, 40, 33, 160, 5, 5, 1, 2, 1 << 20, "uniform"),         # 25 taps
    (2, 3, 128, 126, 64, 7, 7, 2, 3, 1 << 17, "centred"),         # 49 taps, stride 2
    (3, 130, 20, 20, 500, 1, 1, 1, 0, 1 << 24, "centred"),        # 1x1, two digits
    (6, 200, 31, 29, 256, 1, 1, 2, 0, 1 << 31, "uniform"),        # 1x1 / 2, four digits
    (5, 40, 33, 34, 200, 3, 3, 2, 1, 1 << 20, "plain"),
    (4, 96, 20, 19, 65, 3, 2, 1, 1, 1 << 16, "centred"),          # a kernel that is not square
    (8, 512, 12, 12, 512, 3, 3, 1, 1, 1 << 20, "centred"),        # reduction split over a cluster
]


@pytest.mark.parametrize("case", CONV)
@pytest.mark.parametrize("flags", [0, 16])
def test_conv(dslib, case, flags):
    ds, (B, C, H, W, K, R, S, st, pd, top, kind) = dslib, case
    g = _gen(B * 77 + C + K + flags)
    s, p = _codes(g, (K, C, R, S), kind)
    x, b = _values(g, (B, C, H, W), top), torch.randint(-(1 << 16), 1 << 16, (K,), device="cuda", generator=g, dtype=torch.int32)
    OH, OW = (H + 2 * pd - R) // st + 1, (W + 2 * pd - S) // st + 1
    res = torch.randint(-(1 << 31), (1 << 31) - 1, (B, K, OH, OW), device="cuda", generator=g, dtype=torch.int32) if C & 1 else None
    amax_io = torch.zeros(2, dtype=torch.int32, device="cuda")
    y = ds.conv2d_shift(x, ds.pack_shift_weights(s, p), (R, S), b, (st, st), (pd, pd), relu=bool(K & 1), residual=res,
                        amax_io=amax_io, flags=flags | ds.DS_AMAX_OUT)
    xp = torch.nn.functional.pad(x, (pd,) * 4)

    def product(a, w):
        cols = a.unfold(2, R, st).unfold(3, S, st).permute(0, 2, 3, 1, 4, 5).reshape(B * OH * OW, C * R * S)
        return cols @ w.reshape(K, -1).t()

    acc = _sum(xp, s, p, product).reshape(B, OH, OW, K).permute(0, 3, 1, 2)
    want = _finish(acc, b.double()[None, :, None, None], res, relu=bool(K & 1))
    assert torch.equal(y, want)
    assert int(amax_io.cpu().numpy().view(np.uint32)[1]) == int(want.long().abs().max())


@pytest.mark.parametrize("geom", [(4, 64, 34, 34, 128, 3, 2, 1), (4, 64, 35, 33, 130, 3, 2, 0), (2, 40, 49, 50, 128, 5, 2, 2)])
def test_strided_input_gradient(dslib, geom):
    """The tap phases of a strided layer's gradient, several in one launch, against the implicit GEMM."""
    ds, (B, C, H, W, K, R, st, pd) = dslib, geom
    g = _gen(sum(geom))
    s, p = _codes(g, (K, C, R, R), "centred")
    OH, OW = (H + 2 * pd - R) // st + 1, (W + 2 * pd - R) // st + 1
    dy = _values(g, (B, K, OH, OW), 1 << 18)
    w = ds.pack_shift_weights_backward(s, p, (st, st))
    got = []
    for flags in (0, ds.DS_CONV_IM2COL):
        dx = torch.full((B, C, H, W), 7, dtype=torch.int32, device="cuda")
        ds.ds_conv2d_shift_backward_x(dy, w.desc, dx, B, C, H, W, K, R, R, st, st, pd, pd, flags,
                                      torch.zeros(2, dtype=torch.int32, device="cuda"))
        got.append(dx)
    assert torch.equal(*got)


@pytest.mark.parametrize("n", [1, 3, 4096, 16383, 16384, 16385])
@pytest.mark.parametrize("offset", [0, 1])
def test_absmax_at_the_small_kernels_edge(dslib, n, offset):
    """One-block and many-block maxima, with and without 16-byte alignment, over an older larger word."""
    x = _values(_gen(n), (n + 1,), 1 << 30)[offset:offset + n]
    word = torch.full((1,), 0x7FFFFFFF, dtype=torch.int32, device="cuda")
    dslib.ds_absmax(x, n, word)
    assert int(word.item()) == int(x.long().abs().max())
