"""Contractions over few tokens: the edges of the tiles, stages and MMA steps that short
examples and small experts reach."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_close, f64, hbits, host, setup_linear

pytestmark = pytest.mark.gpu


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
    (250, 4104, 1056),   # 256-token tiles
    (33, 25000, 192),    # more tiles than SMs: 64-deep stages
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
