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
