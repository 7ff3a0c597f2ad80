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
