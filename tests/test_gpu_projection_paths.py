"""The projection's short paths (several blocks at a time, quotients by a reciprocal) and the
adapter projection's larger tiles, bit for bit against the oracle."""
import math
import struct

import numpy as np
import pytest
import torch

import oracle
from gpu_util import hbits, host

pytestmark = pytest.mark.gpu


def _f32(bits):
    return struct.unpack("<f", struct.pack("<I", bits))[0]


# tensor scales: ordinary, a power of two, significands 1 to 3 (and one more) from a multiple
# of 2^20, and both ends of the range the reciprocal is used in
SCALES = [0.0123456, 2.0 ** -7, _f32(0x3C500001), _f32(0x3C4FFFFE), _f32(0x3C500003), _f32(0x3C500004),
          _f32(0x3C4FFFFC), 2.0 ** -90, 2.0 ** -91, 1.5 * 2.0 ** 90, 2.0 ** 112]


def _latents(ws2, rng):
    """Around every rounding point of the grid, its ends, zeros of both signs, subnormals,
    infinities and NaN, in an order that mixes them within groups of four."""
    w = np.float32(ws2)
    mids = [(2 * n + 1) * 2.0 ** -10 for n in range(8)] + [(2 * m + 17) * 2.0 ** (e - 4) for e in range(-6, 9) for m in range(8)]
    vals = []
    with np.errstate(all="ignore"):
        for m in mids:
            v = np.float32(np.float32(m) * w)
            for step in (-2, -1, 0, 1, 2):
                u = (v.view(np.int32) + np.int32(step)).view(np.float32)
                vals += [u, np.float32(-u)]
        cap = np.float32(448.0) * w
        vals += [cap, -cap, np.nextafter(cap, np.float32(np.inf)), -np.nextafter(cap, np.float32(np.inf)), 2 * cap, 0.0, -0.0,
                 np.float32(1e-45), np.float32(-1e-45), np.inf, -np.inf, np.nan]
        vals = np.array(vals, dtype=np.float32)
        vals = np.concatenate([vals, (rng.standard_normal(4000) * 100).astype(np.float32) * w])
    vals = vals[rng.permutation(vals.size)]
    return np.resize(vals, (math.ceil(vals.size / 16), 16))


@pytest.mark.parametrize("ws2", SCALES)
def test_projected_and_merged_bytes(ws2):
    import paper_2609_04526_gb300 as pkg
    h = pkg.Handle()
    L = _latents(ws2, np.random.default_rng(1))
    t = torch.from_numpy(L).cuda()
    z = lambda d: torch.zeros(L.shape, dtype=d, device="cuda")  # noqa: E731
    nf = torch.zeros(1, dtype=torch.int32, device="cuda")
    old = torch.randint(0, 120, L.shape, dtype=torch.uint8, device="cuda")
    p = {"latent": t, "bytes": z(torch.uint8), "mask": z(torch.uint8), "ws2": ws2, "nonfinite": nf}
    m = {"latent": t, "bytes": old.clone(), "ws2": ws2, "ongrid_delta": z(torch.float32),
         "changed": torch.zeros(1, dtype=torch.int64, device="cuda")}
    h.sq_project_planes(pkg.NVFP4, [p])
    h.sq_merge_planes(pkg.NVFP4, [m])
    h.sq_sync()
    rb, rm, rnf = oracle.project(pkg.NVFP4, L, ws2)
    assert np.array_equal(host(p["bytes"]), rb) and np.array_equal(host(p["mask"]), rm) and int(nf.item()) == rnf
    assert np.array_equal(host(m["bytes"]), rb) and int(m["changed"].item()) == int((host(old) != rb).sum())
    scale = torch.arange(256, dtype=torch.uint8).view(torch.float8_e4m3fn).float().numpy() * np.float32(ws2)
    with np.errstate(all="ignore"):
        delta = scale[rb] - scale[host(old)]
    got = host(m["ongrid_delta"])
    ok = ~np.isnan(delta)
    assert np.array_equal(np.isnan(got), ~ok) and np.array_equal(got[ok].view(np.uint32), delta[ok].view(np.uint32))


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("N,G,r", [(7300, 376, 32), (6500, 380, 33), (19999, 100, 64), (19500, 128, 65), (6500, 508, 131)])
def test_adapter_projection_in_large_tiles(fmt, N, G, r):
    """Ragged rows and blocks, odd ranks, and ranks of one, two and three chunks of 64."""
    import paper_2609_04526_gb300 as pkg
    h = pkg.Handle()
    rng = np.random.default_rng(N + G + r)
    ws2 = 0.00371 if fmt == 0 else 1.0
    base = torch.from_numpy(rng.integers(40, 120, (N, G), dtype=np.uint8)).cuda()
    B = torch.from_numpy(rng.standard_normal((N, r)).astype(np.float32) * 2e-3).cuda().to(torch.bfloat16)
    A = torch.from_numpy(rng.standard_normal((r, G)).astype(np.float32)).cuda().to(torch.bfloat16)
    mask = torch.zeros(N, G, dtype=torch.uint8, device="cuda")
    nf = torch.zeros(1, dtype=torch.int32, device="cuda")
    lat = torch.zeros(N, G, dtype=torch.float32, device="cuda")
    b, _, _ = h.sq_project_lowrank(fmt, base, B, A, ws2, 16.0 / r, mask_out=mask, nonfinite=nf, latent_out=lat)
    h.sq_sync()
    rb, rm, rnf, rL = oracle.project_lowrank(fmt, host(base), hbits(B), hbits(A), ws2, 16.0 / r)
    assert np.array_equal(host(lat).view(np.uint32), rL.view(np.uint32))
    assert np.array_equal(host(b), rb) and np.array_equal(host(mask), rm) and int(nf.item()) == rnf
