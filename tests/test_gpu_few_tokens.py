"""Contractions over few tokens: the edges of the tiles, stages and MMA steps that short
examples and small experts reach."""
import numpy as np
import pytest
import torch

import oracle
from few_plan import SMS, plan
from gpu_util import assert_close, f64, hbits, host, setup_linear

pytestmark = pytest.mark.gpu


def _shape(rows, features, contraction):
    """(largest token tile, features of a tile, depth, stages, code slots) of the product's launch."""
    p = plan(rows, features, contraction)
    assert p is not None and torch.cuda.get_device_properties(0).multi_processor_count == SMS
    return (p.largest, p.features, p.depth, p.stages, p.slots) if p.limit else None


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("M", [1, 15, 16, 17, 127, 129, 145])
def test_scale_gradient_of_few_tokens(fmt, M):
    """Part of a stage's MMA steps (16 tokens each), rows and columns that end inside a tile,
    16-byte and narrower gradient stores, and a mask that starts at an odd address."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    for N, K in ((72, 160), (264, 512)):
        wl = synth.custom("few", fmt, M, N, K, seed=300 + M)
        w, X, dY = setup_linear(wl, wl.linears[0])
        G = K // wl.block
        store = torch.zeros(N * G + 1, dtype=torch.uint8, device="cuda")
        mask = store[1:].view(N, G)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(M)
        mask.copy_(torch.rand(N, G, generator=gen, device="cuda") < 0.9)
        g = h.sq_scale_grad(w, X, dY, mask=mask)
        h.sq_sync()
        ref = oracle.scale_grad(fmt, host(w.codes), hbits(X), hbits(dY), mask=host(mask))
        assert_close(f64(g), ref, what=f"g {fmt} {M}x{N}x{K}")
        assert not np.any(f64(g)[host(mask) == 0])


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("N,K", [(264, 512), (136, 96), (40, 288)])
def test_scale_gradient_masks_at_any_address(fmt, N, K):
    """The mask is read in words where its address and its rows allow and in bytes elsewhere:
    at every address the gradient is the unmasked one times the mask, bit for bit."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    wl = synth.custom("few", fmt, 50, N, K, seed=N + K)
    w, X, dY = setup_linear(wl, wl.linears[0])
    G = K // wl.block
    full = h.sq_scale_grad(w, X, dY)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(K)
    bits = torch.rand(N, G, generator=gen, device="cuda") < 0.7
    for start in range(5):
        store = torch.full((N * G + 5,), 7, dtype=torch.uint8, device="cuda")
        mask = store[start:start + N * G].view(N, G)
        mask.copy_(bits)
        g = h.sq_scale_grad(w, X, dY, mask=mask)
        h.sq_sync()
        assert torch.equal(g, full * bits), start


@pytest.mark.parametrize("fmt", [0, 1])
def test_scale_gradient_beyond_the_tables(fmt):
    """More experts than the kernel keeps in shared memory, and a weight of more tiles."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    E, N, K = 1100, 16, 64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(fmt)
    codes = torch.randint(0, 256, (E, N, K // 2), generator=gen, device="cuda", dtype=torch.uint8)
    scales = torch.full((E, N, K // (16 if fmt == 0 else 32)), 0x38, dtype=torch.uint8, device="cuda")
    gw = pkg.GroupedWeight(fmt, E, N, K, codes, scales, [1.0] * E)
    off = [0]
    for e in range(E):
        off.append(off[-1] + e % 4)
    X = torch.randn(off[-1], K, generator=gen, device="cuda").bfloat16()
    dY = torch.randn(off[-1], N, generator=gen, device="cuda").bfloat16()
    g = h.sq_grouped_scale_grad(gw, off, X, dY)
    h.sq_sync()
    for e in (0, 1, 2, 3, 1023, 1024, 1025, 1027, 1098, 1099):
        a, b = off[e], off[e + 1]
        ref = oracle.scale_grad(fmt, host(codes[e]), hbits(X[a:b]), hbits(dY[a:b]))
        assert_close(f64(g[e]), ref, what=f"g of expert {e}")

    wl = synth.custom("few", fmt, 20, 8712, 8224, seed=fmt)   # 35 x 33 tiles
    w, X, dY = setup_linear(wl, wl.linears[0])
    g = h.sq_scale_grad(w, X, dY)
    h.sq_sync()
    rows = np.array([0, 255, 256, 4095, 4096, 7935, 7936, 8191, 8192, 8447, 8448, 8711])
    ref = oracle.scale_grad(fmt, host(w.codes), hbits(X), hbits(dY), rows=rows)
    assert_close(f64(g)[rows], ref, what="g of a large weight")


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("M,N,K", [
    (1, 8, 32),          # one MMA step of everything
    (16, 120, 160), (17, 136, 96),   # a feature tile's edge, half a stage of the contraction
    (129, 264, 544),     # two token tiles
    (250, 4104, 1056),   # 128-token tiles of unequal fill
    (33, 25000, 192),    # more tiles than SMs: 64-deep stages, no more of them than the rings hold
    (150, 25000, 96), (60, 25000, 160)])
def test_few_token_products(fmt, M, N, K):
    """Forward and input gradient of sizes that run on the few-token kernel in one or both
    directions: ragged tiles on every side, both depths of a stage."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    wl = synth.custom("few", fmt, M, N, K, seed=M + N + K, kind="outlier")
    w, X, dY = setup_linear(wl, wl.linears[0])
    Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    dX = torch.full((M, K), float("nan"), dtype=torch.bfloat16, device="cuda")
    h.sq_fwd(w, X, Y)
    h.sq_bwd_dx(w, dY, dX)
    h.sq_sync()
    codes, scales = host(w.codes), host(w.scales)
    assert_close(f64(Y), oracle.fwd(fmt, codes, scales, w.ws2, hbits(X)), what="Y")
    assert_close(f64(dX), oracle.dx(fmt, codes, scales, w.ws2, hbits(dY)), what="dX")


@pytest.mark.parametrize("fmt", [0, 1])
def test_pair_kernel_ragged_edges(fmt):
    """Sizes whose forward and input gradient run on the 512 x 256 tiles, ragged on every side."""
    assert _shape(2085, 2824, 2592) is None and _shape(2085, 2592, 2824) is None
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    wl = synth.custom("pair", fmt, 2085, 2824, 2592, seed=12)
    w, X, dY = setup_linear(wl, wl.linears[0])
    Y, dX = h.sq_fwd(w, X), h.sq_bwd_dx(w, dY)
    h.sq_sync()
    codes, scales = host(w.codes), host(w.scales)
    rng = np.random.default_rng(5)
    m = np.concatenate([[0, 2084, 2084, 0], rng.integers(0, 2085, 3000)])
    n = np.concatenate([[0, 2823, 0, 2823], rng.integers(0, 2824, 3000)])
    k = np.concatenate([[0, 2591, 0, 2591], rng.integers(0, 2592, 3000)])
    assert_close(f64(Y)[m, n], oracle.fwd_at(fmt, codes, scales, w.ws2, hbits(X), m, n), what="Y")
    assert_close(f64(dX)[m, k], oracle.dx_at(fmt, codes, scales, w.ws2, hbits(dY), m, k), what="dX")


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("M", [2136, 2304, 2305, 2559])   # last 512-row tile: 88, 256, 257, 511 rows
def test_pair_kernel_last_tiles(fmt, M):
    """The last row tile of the 512 x 256 tiles: part of a half, one half, a row more, one short."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    N, K = 2568, 2080
    assert _shape(M, N, K) is None and _shape(M, K, N) is None
    h = pkg.Handle()
    wl = synth.custom("pair", fmt, M, N, K, seed=M)
    w, X, dY = setup_linear(wl, wl.linears[0])
    # rows behind the outputs must stay as they are
    Y = torch.full((M + 8, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    dX = torch.full((M + 8, K), float("nan"), dtype=torch.bfloat16, device="cuda")
    h.sq_fwd(w, X, Y[:M])
    h.sq_bwd_dx(w, dY, dX[:M])
    h.sq_sync()
    assert torch.isnan(Y[M:]).all() and torch.isnan(dX[M:]).all()
    last = np.arange(M // 512 * 512, M)
    codes, scales = host(w.codes), host(w.scales)
    rows = np.concatenate([[0], last])
    assert_close(f64(Y[:M])[rows], oracle.fwd(fmt, codes, scales, w.ws2, hbits(X)[rows]), what="Y")
    assert_close(f64(dX[:M])[rows], oracle.dx(fmt, codes, scales, w.ws2, hbits(dY)[rows]), what="dX")


def test_few_token_and_pair_kernels_agree_bit_for_bit():
    """A row of the output does not depend on the batch it is in: 100 tokens alone (few-token
    kernel) and as the head of 4096 (pair kernel), forward and input gradient."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    for fmt in (0, 1):
        wl = synth.custom("bits", fmt, 4096, 4104, 2080, seed=7, kind="outlier")
        w, X, dY = setup_linear(wl, wl.linears[0])
        Y, dX = h.sq_fwd(w, X), h.sq_bwd_dx(w, dY)
        Yf, dXf = h.sq_fwd(w, X[:100]), h.sq_bwd_dx(w, dY[:100])
        h.sq_sync()
        assert torch.equal(Y[:100], Yf) and torch.equal(dX[:100], dXf)


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("M,N,K", [(1, 72, 4128), (96, 4104, 1056), (33, 2056, 544), (190, 4128, 288), (16, 9728, 96)])
def test_few_token_tiles_of_64_features(fmt, M, N, K):
    """Tiles of 64 features: ragged last tiles, one to three 32-token boxes, two token tiles,
    contractions shorter and longer than the code ring; each row as in a large batch, bit for bit."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    h = pkg.Handle()
    wl = synth.custom("few", fmt, 4096, N, K, seed=M + N + K, kind="outlier")
    w, X, dY = setup_linear(wl, wl.linears[0])
    Y, dX = h.sq_fwd(w, X[:M]), h.sq_bwd_dx(w, dY[:M])
    Yb, dXb = h.sq_fwd(w, X), h.sq_bwd_dx(w, dY)
    h.sq_sync()
    codes, scales = host(w.codes), host(w.scales)
    assert_close(f64(Y), oracle.fwd(fmt, codes, scales, w.ws2, hbits(X[:M])), what="Y")
    assert_close(f64(dX), oracle.dx(fmt, codes, scales, w.ws2, hbits(dY[:M])), what="dX")
    assert torch.equal(Y, Yb[:M]) and torch.equal(dX, dXb[:M])


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("M,N,K,fwd,dx", [
    # one direction with two CTAs per SM (64-deep stages), 17 or 19 fills of 6, 4 or 3 code slots;
    # the other with the longest contraction of a CTA alone
    (30, 19592, 2400, (32, 128, 64, 3, 6), (32, 64, 128, 4, 12)),
    (60, 19592, 2080, (64, 128, 64, 3, 4), (64, 64, 128, 4, 11)),
    (190, 19592, 2080, (192, 128, 64, 2, 3), (96, 64, 128, 4, 4)),
    (30, 2400, 19616, (32, 64, 128, 4, 12), (32, 128, 64, 3, 6)),
    (60, 2088, 19616, (64, 64, 128, 4, 11), (64, 128, 64, 3, 4)),
    (190, 2088, 19616, (96, 64, 128, 4, 4), (192, 128, 64, 2, 3)),
    # 256-token tiles, two code slots
    (1000, 4104, 2080, (256, 128, 128, 2, 2), (128, 128, 128, 2, 11)),
    (1000, 2088, 4128, (128, 128, 128, 2, 11), (256, 128, 128, 2, 2)),
])
def test_few_token_rings_wrap(fmt, M, N, K, fwd, dx):
    """Every ring of every shape turns over several times; each row as in a large batch (pair
    kernel), bit for bit, and samples against the oracle."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    big = 4096
    assert _shape(M, N, K) == fwd and _shape(M, K, N) == dx
    assert _shape(big, N, K) is None and _shape(big, K, N) is None
    h = pkg.Handle()
    wl = synth.custom("few", fmt, big, N, K, seed=M + N + K, kind="outlier")
    w, X, dY = setup_linear(wl, wl.linears[0])
    Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    dX = torch.full((M, K), float("nan"), dtype=torch.bfloat16, device="cuda")
    h.sq_fwd(w, X[:M], Y)
    h.sq_bwd_dx(w, dY[:M], dX)
    Yb, dXb = h.sq_fwd(w, X), h.sq_bwd_dx(w, dY)
    h.sq_sync()
    assert torch.equal(Y, Yb[:M]) and torch.equal(dX, dXb[:M])
    codes, scales = host(w.codes), host(w.scales)
    rng = np.random.default_rng(M)
    m, n, k = (np.concatenate([[0, v - 1], rng.integers(0, v, 2000)]) for v in (M, N, K))
    assert_close(f64(Y)[m, n], oracle.fwd_at(fmt, codes, scales, w.ws2, hbits(X[:M]), m, n), what="Y")
    assert_close(f64(dX)[m, k], oracle.dx_at(fmt, codes, scales, w.ws2, hbits(dY[:M]), m, k), what="dX")


def _rows(seed, experts, most):
    """Token counts: an expert without rows, one of a single row, the rest up to `most`."""
    rng = np.random.default_rng(seed)
    return [0, 1, *(int(v) for v in rng.integers(0, most + 1, experts - 2))]


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("rows,N,K,fwd,dx", [
    ([9] * 128, 2624, 1376, (16, 128, 64, 3, 6), (16, 128, 64, 3, 6)),
    (_rows(1, 64, 30), 2080, 1568, (32, 128, 64, 3, 6), (32, 128, 64, 3, 6)),
    (_rows(2, 32, 60), 1160, 2080, (64, 128, 64, 3, 4), (64, 128, 64, 3, 4)),
    (_rows(3, 32, 90), 1160, 2080, (80, 128, 64, 2, 6), (80, 128, 64, 2, 6)),
    (_rows(4, 40, 190), 1032, 1184, (192, 128, 64, 2, 3), (192, 128, 64, 2, 3)),
    (_rows(5, 128, 300), 768, 1056, (192, 128, 64, 2, 3), (192, 128, 64, 2, 3)),
], ids=["9_rows", "to_30", "to_60", "to_90", "to_190", "to_300"])
def test_grouped_few_token_products(fmt, rows, N, K, fwd, dx):
    """Experts with few rows, more tiles than SMs (two CTAs per SM): every expert as the dense call
    on it alone (CTAs alone on their SMs, other rings), bit for bit, some against the oracle."""
    import paper_2609_04526_gb300 as pkg
    from paper_2609_04526_gb300 import synth
    assert _shape(rows, N, K) == fwd and _shape(rows, K, N) == dx
    h = pkg.Handle()
    wl = synth.custom_moe("few", fmt, rows, N, K, seed=sum(rows) + N, kind="outlier")
    ex = synth.gen_experts(wl, wl.linears[0], device="cuda")
    gw = pkg.GroupedWeight(ex.fmt, ex.E, ex.N, ex.K, ex.codes, ex.scales, ex.ws2)
    off = synth.offsets_of(rows)
    X = synth.gen_act(wl, "x", M=off[-1], device="cuda")
    dY = synth.gen_dy(wl, wl.linears[0], M=off[-1], device="cuda")
    Y = torch.full((off[-1], N), float("nan"), dtype=torch.bfloat16, device="cuda")
    dX = torch.full((off[-1], K), float("nan"), dtype=torch.bfloat16, device="cuda")
    h.sq_grouped_fwd(gw, off, X, Y)
    h.sq_grouped_bwd_dx(gw, off, dY, dX)
    h.sq_sync()
    checked = {1, len(rows) // 2, len(rows) - 1, int(np.argmax(rows))}
    for e in range(len(rows)):
        a, b = off[e], off[e + 1]
        if a == b:
            continue
        w = gw.expert(e)
        w.scales = w.scales.clone()   # the dense entry points take 16-byte aligned planes
        Yd, dXd = h.sq_fwd(w, X[a:b].clone()), h.sq_bwd_dx(w, dY[a:b].clone())
        assert torch.equal(Y[a:b], Yd) and torch.equal(dX[a:b], dXd), e
        if e in checked:
            c, s = host(w.codes), host(w.scales)
            assert_close(f64(Y[a:b]), oracle.fwd(fmt, c, s, w.ws2, hbits(X[a:b])), what=f"Y of expert {e}")
            assert_close(f64(dX[a:b]), oracle.dx(fmt, c, s, w.ws2, hbits(dY[a:b])), what=f"dX of expert {e}")
    h.sq_sync()
