"""The tensor-core shift sums where a CTA walks several tiles, runs, digits and column halves, and at the accumulators' limit.

Sizes are chosen by what the launcher does with them, and each test asserts the route: grids that cannot be split (at
least as many tiles as CTAs or pairs of them), more tiles than CTAs, reductions over one run of 3840 indices, and split
ones.  Reference: float64 products on the GPU, exact (every sum is below 2^53); results are integers with one correct
value, so there is no tolerance."""
import numpy as np
import pytest
import torch

from test_gpu_guard import X_CANARY, Y_CANARY, Guarded
from test_gpu_shift_mma import _codes, _finish, _gen, _values

pytestmark = pytest.mark.gpu

TC, SWAP = 1, 2


def _sum(x, s, p, product):
    acc = 0
    for k in (-torch.unique(p.long())).tolist():
        acc = acc + product((x >> k).double(), torch.where(p == -k, s, torch.zeros_like(s)).double())
    return acc


def _fc_want(x, s, p, b, relu=False):
    return _finish(_sum(x, s, p, lambda a, w: a @ w.t()), b.double(), relu=relu)


# M, K, N, max |x|, route
FC = [
    (2600, 4000, 1000, 1 << 20, TC),     # 88 tiles of 256 x 128 on 76 pairs, two runs
    (2600, 3999, 1000, 1 << 20, TC),     # the same with rows that are not 16-byte aligned
    (2500, 4100, 1025, 1 << 26, TC),     # three digits, two runs, a tile of one column
    (19500, 4000, 60, 1 << 20, TC),      # 77 tiles of 256 x 64, two runs, ragged columns
    (19500, 3999, 64, 1 << 24, TC),
    (128, 4000, 9800, 1 << 20, SWAP),    # 154 tiles of 64 rows x 128 columns on 152 CTAs, two runs
    (70, 3999, 20000, 1 << 22, SWAP),    # two digits, a row tile of six
    (512, 8200, 300, 1 << 20, TC),       # split over 8 pairs
    (512, 8201, 300, 1 << 31, TC),       # four digits
    (700, 600, 1000, 1 << 25, SWAP),    # 11 row tiles of the swapped roles
]


@pytest.mark.parametrize("flags", [0, 16])
@pytest.mark.parametrize("case", FC)
def test_fc(dslib, case, flags):
    ds, (M, K, N, top, route) = dslib, case
    assert ds.ds_linear_shift_route(M, K, N) == route
    g = _gen(M + K + flags)
    s, p = _codes(g, (N, K), "uniform")
    x, b = _values(g, (M, K), top), torch.randint(-(1 << 16), 1 << 16, (N,), device="cuda", generator=g, dtype=torch.int32)
    amax_io = torch.zeros(2, dtype=torch.int32, device="cuda")
    y = ds.linear_shift(x, ds.pack_shift_weights(s, p), b, relu=bool(M & 4), amax_io=amax_io, flags=flags | ds.DS_AMAX_OUT)
    want = _fc_want(x, s, p, b, relu=bool(M & 4))
    assert torch.equal(y, want)
    assert int(amax_io.cpu().numpy().view(np.uint32)[1]) == int(want.long().abs().max())
    assert ds.ds_bf16_fault_flag() == 0


# B, C, H, W, K, R, S, stride, pad, max |x|
CONV = [
    (8, 96, 28, 27, 65, 3, 2, 1, 1, 1 << 16),    # a kernel that is not square, 65 columns
    (8, 65, 28, 28, 64, 3, 3, 1, 1, 1 << 18),    # 64-column tiles, a partial last slot
    (8, 63, 56, 56, 60, 3, 3, 1, 1, 1 << 20),    # 98 tiles of 64 columns on 76 pairs, residual
    (8, 63, 56, 56, 130, 3, 3, 1, 1, 1 << 24),   # 196 tiles of 128 columns, two digits, residual
    (8, 450, 40, 40, 60, 3, 3, 2, 1, 1 << 31),   # more indices than a run, four digits
]


@pytest.mark.parametrize("flags", [0, 16])
@pytest.mark.parametrize("case", CONV)
def test_conv(dslib, case, flags):
    ds, (B, C, H, W, K, R, S, st, pd, top) = dslib, case
    assert ds.ds_conv2d_shift_route(B, C, H, W, K, R, S, st, st, pd, pd) == TC
    g = _gen(B * 77 + C + K + flags)
    s, p = _codes(g, (K, C, R, S), "uniform" if C == 450 else "centred")
    x, b = _values(g, (B, C, H, W), top), torch.randint(-(1 << 16), 1 << 16, (K,), device="cuda", generator=g, dtype=torch.int32)
    OH, OW = (H + 2 * pd - R) // st + 1, (W + 2 * pd - S) // st + 1
    res = torch.randint(-(1 << 31), (1 << 31) - 1, (B, K, OH, OW), device="cuda", generator=g, dtype=torch.int32) if C == 63 else None
    amax_io = torch.zeros(2, dtype=torch.int32, device="cuda")
    y = ds.conv2d_shift(x, ds.pack_shift_weights(s, p), (R, S), b, (st, st), (pd, pd), relu=C == 65, residual=res,
                        amax_io=amax_io, flags=flags | ds.DS_AMAX_OUT)
    xp = torch.nn.functional.pad(x, (pd,) * 4)

    def product(a, w):
        cols = a.unfold(2, R, st).unfold(3, S, st).permute(0, 2, 3, 1, 4, 5).reshape(B * OH * OW, C * R * S)
        return cols @ w.reshape(K, -1).t()

    acc = _sum(xp, s, p, product).reshape(B, OH, OW, K).permute(0, 3, 1, 2)
    want = _finish(acc, b.double()[None, :, None, None], res, relu=C == 65)
    assert torch.equal(y, want)
    assert int(amax_io.cpu().numpy().view(np.uint32)[1]) == int(want.long().abs().max())


def _limit_case(kind, g, M, K, N):
    """Inputs and codes whose fp32 accumulators end in [2^23, 2^24), odd sums among them, or get there and come back."""
    s = torch.ones((N, K), device="cuda", dtype=torch.int8)
    p = torch.full((N, K), -4, device="cuda", dtype=torch.int8)
    rnd = lambda lo, hi: torch.randint(lo, hi, (M, K), device="cuda", generator=g, dtype=torch.int32)  # noqa: E731
    if kind == "features":          # x >> 4 up to 4095, 4096 times: the bound 2^16 sum |w| = 2^24 is met
        return rnd(61440, 65536), s, p
    if kind == "negative":          # the same features against digits of -1 that cancel them
        return rnd(-4096, 0), s, p
    if kind == "returning":         # up to 2^23 and back down through every value
        s[:, K // 2:] = -1
        return rnd(61440, 65536), s, p
    if kind == "digits":            # digits up to 16 at sh = 7, odd ones from sh = 15
        p[:] = -7
        p[:, ::64] = -15
        return rnd(15 << 16, (1 << 20) + 1), s, p
    # runs of a tile without a bound: one column of large weights, the others at the most a run's terms can be
    p[:] = -8
    p[::128] = 0
    return rnd(0xFF000, 1 << 20), s, p


@pytest.mark.parametrize("kind", ["features", "negative", "returning", "digits", "runs"])
@pytest.mark.parametrize("shape", [(2600, 1000, TC), (64, 19500, SWAP)])
def test_sums_near_the_accumulators_limit(dslib, kind, shape):
    """Grids that are not split, so that one accumulator takes the whole sum (or a whole run of 3840 terms)."""
    ds, (M, N, route) = dslib, shape
    K = 7680 if kind == "runs" else 4096
    assert ds.ds_linear_shift_route(M, K, N) == route
    g = _gen(len(kind))
    x, s, p = _limit_case(kind, g, M, K, N)
    b = torch.zeros(N, device="cuda", dtype=torch.int32)
    y = ds.linear_shift(x, ds.pack_shift_weights(s, p), b, amax_io=torch.zeros(2, dtype=torch.int32, device="cuda"))
    assert torch.equal(y, _fc_want(x, s, p, b))


def _guarded_weights(ds, s, p):
    n_out = s.shape[0]
    k_red = s.numel() // n_out
    nb = ds.ds_packed_weight_bytes(n_out, k_red)
    blob = Guarded(nb, torch.uint8, 0xFF)
    desc = ds.ds_pack_shift_weights(s.reshape(n_out, k_red), p.reshape(n_out, k_red), n_out, k_red, blob.view, nb)
    return desc, blob


@pytest.mark.parametrize("shape", [(9, 4099, 4099, SWAP), (65, 2052, 1025, SWAP), (2565, 1031, 1001, TC), (19457, 131, 61, TC)])
def test_fc_stays_inside_its_buffers(dslib, shape):
    """Canaries around every buffer: a read past an input would change the results, a write past an output shows."""
    ds, (M, K, N, route) = dslib, shape
    assert ds.ds_linear_shift_route(M, K, N) == route
    g = _gen(M)
    s, p = _codes(g, (N, K), "uniform")
    x, b = _values(g, (M, K), 1 << 20), torch.randint(-(1 << 16), 1 << 16, (N,), device="cuda", generator=g, dtype=torch.int32)
    desc, blob = _guarded_weights(ds, s, p)
    xg = Guarded(x.numel(), torch.int32, X_CANARY, x.cpu().numpy())
    bg = Guarded(N, torch.int32, X_CANARY, b.cpu().numpy())
    yg = Guarded(M * N, torch.int32, Y_CANARY)
    ag = Guarded(2, torch.int32, Y_CANARY, np.zeros(2, np.int32))
    ds.ds_linear_shift(xg.view, desc, bg.view, yg.view, M, K, N, ds.DS_AMAX_OUT, ag.view)
    for buf in (xg, bg, yg, ag, blob):
        assert buf.margins_intact()
    assert torch.equal(yg.view.reshape(M, N), _fc_want(x, s, p, b))


@pytest.mark.parametrize("geom", [(4, 67, 29, 31, 67, 3, 2, 1, 1), (5, 131, 21, 23, 513, 1, 1, 1, 0), (2, 3, 129, 127, 67, 7, 7, 2, 3)])
def test_conv_stays_inside_its_buffers(dslib, geom):
    ds, (B, C, H, W, K, R, S, st, pd) = dslib, geom
    assert ds.ds_conv2d_shift_route(B, C, H, W, K, R, S, st, st, pd, pd) == TC
    g = _gen(sum(geom))
    s, p = _codes(g, (K, C, R, S), "centred")
    x = _values(g, (B, C, H, W), 1 << 20)
    OH, OW = (H + 2 * pd - R) // st + 1, (W + 2 * pd - S) // st + 1
    res = torch.randint(-(1 << 20), 1 << 20, (B, K, OH, OW), device="cuda", generator=g, dtype=torch.int32)
    desc, blob = _guarded_weights(ds, s, p)
    xg = Guarded(x.numel(), torch.int32, X_CANARY, x.cpu().numpy())
    rg = Guarded(res.numel(), torch.int32, X_CANARY, res.cpu().numpy())
    yg = Guarded(res.numel(), torch.int32, Y_CANARY)
    ag = Guarded(2, torch.int32, Y_CANARY, np.zeros(2, np.int32))
    ds.ds_conv2d_shift(xg.view, desc, None, rg.view, yg.view, B, C, H, W, K, R, S, st, st, pd, pd,
                       ds.DS_RESIDUAL | ds.DS_AMAX_OUT, ag.view)
    for buf in (xg, rg, yg, ag, blob):
        assert buf.margins_intact()
    xp = torch.nn.functional.pad(x, (pd,) * 4)

    def product(a, w):
        cols = a.unfold(2, R, st).unfold(3, S, st).permute(0, 2, 3, 1, 4, 5).reshape(B * OH * OW, C * R * S)
        return cols @ w.reshape(K, -1).t()

    want = _finish(_sum(xp, s, p, product).reshape(B, OH, OW, K).permute(0, 3, 1, 2), 0.0, res)
    assert torch.equal(yg.view.reshape(res.shape), want)


@pytest.mark.parametrize("shape", [(33, 4100, 1030, SWAP), (300, 8300, 500, SWAP), (2600, 1030, 1000, TC)])
def test_fc_without_a_bound(dslib, shape):
    """amax_io = NULL: four digits and 64-bit sums, whatever the values."""
    ds, (M, K, N, route) = dslib, shape
    assert ds.ds_linear_shift_route(M, K, N, False) == route
    g = _gen(M)
    s, p = _codes(g, (N, K), "uniform")
    x, b = _values(g, (M, K), 1 << 31), torch.randint(-(1 << 16), 1 << 16, (N,), device="cuda", generator=g, dtype=torch.int32)
    assert torch.equal(ds.linear_shift(x, ds.pack_shift_weights(s, p), b), _fc_want(x, s, p, b))


@pytest.mark.parametrize("geom", [(8, 256, 14, 300, 3, 1), (4, 130, 41, 513, 1, 0), (3, 64, 40, 65, 3, 1)])
def test_conv_without_a_bound(dslib, geom):
    """The same for convolutions (tiles of 64 columns, more of them than 128-column ones) and their gradient."""
    ds, (B, C, H, K, R, pd) = dslib, geom
    assert ds.ds_conv2d_shift_route(B, C, H, H, K, R, R, 1, 1, pd, pd, False) == TC
    g = _gen(sum(geom))
    s, p = _codes(g, (K, C, R, R), "uniform")
    x = _values(g, (B, C, H, H), 1 << 31)
    y = ds.conv2d_shift(x, ds.pack_shift_weights(s, p), (R, R), None, (1, 1), (pd, pd))
    xp = torch.nn.functional.pad(x, (pd,) * 4)

    def product(a, w):
        cols = a.unfold(2, R, 1).unfold(3, R, 1).permute(0, 2, 3, 1, 4, 5).reshape(B * H * H, C * R * R)
        return cols @ w.reshape(K, -1).t()

    assert torch.equal(y, _finish(_sum(xp, s, p, product).reshape(B, H, H, K).permute(0, 3, 1, 2), 0.0))
    w = ds.pack_shift_weights_backward(s, p, (1, 1))
    got = []
    for flags in (0, ds.DS_CONV_IM2COL):
        dx = torch.full((B, C, H, H), 7, dtype=torch.int32, device="cuda")
        ds.ds_conv2d_shift_backward_x(y, w.desc, dx, B, C, H, H, K, R, R, 1, 1, pd, pd, flags, None)
        got.append(dx)
    assert torch.equal(*got)


def _small_calls(ds, seed):
    """One FC call (columns as lanes, split) and one convolution (pairs, split): closures over fresh tensors, and checks."""
    g = _gen(seed)
    s, p = _codes(g, (1030, 2052), "uniform")
    x, b = _values(g, (64, 2052), 1 << 20), torch.randint(-(1 << 16), 1 << 16, (1030,), device="cuda", generator=g, dtype=torch.int32)
    w, a = ds.pack_shift_weights(s, p), torch.zeros(2, dtype=torch.int32, device="cuda")
    sc, pc = _codes(g, (130, 64, 3, 3), "centred")
    xc = _values(g, (2, 64, 24, 24), 1 << 20)
    wc, ac = ds.pack_shift_weights(sc, pc), torch.zeros(2, dtype=torch.int32, device="cuda")
    y = torch.empty((64, 1030), dtype=torch.int32, device="cuda")
    yc = torch.empty((2, 130, 24, 24), dtype=torch.int32, device="cuda")

    def call(stream):
        ds.ds_linear_shift(x, w.desc, b, y, 64, 2052, 1030, 0, a, stream)
        ds.ds_conv2d_shift(xc, wc.desc, None, None, yc, 2, 64, 24, 24, 130, 3, 3, 1, 1, 1, 1, 0, ac, stream)

    def check():
        assert torch.equal(y, _fc_want(x, s, p, b))
        cols = torch.nn.functional.pad(xc, (1,) * 4).unfold(2, 3, 1).unfold(3, 3, 1).permute(0, 2, 3, 1, 4, 5).reshape(1152, 576)
        want = _finish(_sum(cols, sc.reshape(130, -1), pc.reshape(130, -1), lambda v, u: v @ u.t()), 0.0)
        assert torch.equal(yc.permute(0, 2, 3, 1).reshape(1152, 130), want)

    return call, check, (x, xc)


def test_calls_on_two_threads_and_streams(dslib):
    import threading
    work = [_small_calls(dslib, seed) for seed in (3, 4)]
    torch.cuda.synchronize()
    errors = []

    def go(call):
        try:
            stream = torch.cuda.Stream()
            for _ in range(20):
                call(stream.cuda_stream)
            stream.synchronize()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=go, args=(w[0],)) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for _, check, _ in work:
        check()


def test_captured_calls_follow_new_inputs(dslib):
    call, check, inputs = _small_calls(dslib, 5)
    call(torch.cuda.current_stream().cuda_stream)  # kernel attributes are set at the first launch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(torch.cuda.current_stream().cuda_stream)
    for shift in (1, 2):
        for t in inputs:
            t.copy_(torch.roll(t, shift, 0) >> shift)
        graph.replay()
        torch.cuda.synchronize()
        check()
