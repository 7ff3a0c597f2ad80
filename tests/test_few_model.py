"""The host side of the few-token forward and input gradient (no GPU).

few_ring and few_limit in csrc/sq_internal.h size its shared memory and choose between it
and the pair kernel. Checked here by compiling them into a host program: every plan that
can be chosen fits its limits, and the choice follows the estimates it is made from."""
import math
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_04526_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
SMS = 152

PROGRAM = r"""
#include <cstdio>
#include "sq_internal.h"
int main() {
  long long M, F, K;
  while (std::scanf("%lld %lld %lld", &M, &F, &K) == 3) {
    auto tiles_at = [&](int limit) { const int t = sqi::few_tile_tokens(M, limit); return (int64_t)((M + t - 1) / t); };
    const int64_t pair = ((M + 511) / 512) * ((F + 255) / 256);
    const int limit = sqi::few_limit(tiles_at, M, F, K, pair, SMS);
    int tokens = 0, alone = 0, feat = 0;
    sqi::FewRing r{};
    double few = 0;
    if (limit) {
      tokens = sqi::few_tile_tokens(M, limit);
      alone = tiles_at(limit) * ((F + 127) / 128) <= SMS;
      feat = sqi::few_features(tiles_at(limit), tokens, F, SMS);
      r = sqi::few_ring(tokens, alone, feat);
      few = sqi::few_us(tiles_at(limit), (double)M / tiles_at(limit), F, K, SMS);
    }
    std::printf("%d %d %d %d %d %d %d %d %d %.9g %.9g\n", limit, tokens, alone, feat, r.depth, r.stage_bytes, r.stages,
                r.slots, r.bytes, few, sqi::pair_us(pair, K, SMS));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda.h")):
        pytest.skip("no host C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("few_model")
    src, exe = d / "few_model.cpp", d / "few_model"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", f"-DSMS={SMS}", f"-I{CSRC}", f"-I{CUDA_INC}", str(src), "-o", str(exe)], check=True)

    def run(cases):
        out = subprocess.run([str(exe)], input="".join("%d %d %d\n" % c for c in cases), capture_output=True, text=True,
                             check=True).stdout.split("\n")
        return [tuple(float(v) for v in line.split()) for line in out if line]
    return run


def test_every_plan_fits(plan):
    rng = random.Random(3)
    log = lambda hi: int(math.exp(rng.uniform(0, math.log(hi))))  # noqa: E731
    cases = [(log(1 << 31) if i % 4 else log(2000), 8 * log(1 << 21), 32 * log(1 << 19)) for i in range(4000)]
    cases += [(m, f, 4096) for m in range(1, 1100, 7) for f in (8, 128, 136, 1024, 4096, 14336)]
    chosen = 0
    for (M, F, K), (limit, tokens, alone, feat, depth, stage, stages, slots, nbytes, few, pair) in zip(cases, plan(cases)):
        if not limit:
            continue
        chosen += 1
        assert few < 0.97 * pair
        assert tokens % 16 == 0 and 16 <= tokens <= limit <= 256 and (tokens <= 192 or alone)
        assert depth == (128 if alone else 64) and stage == (feat + math.ceil(tokens / 32) * 32) * depth * 2
        assert (stages == 4 if feat == 64 else 2 <= stages <= 3) and 2 <= slots <= 12
        assert nbytes == stages * stage + slots * 8192 + 1024
        # shared memory of a CTA (227 KiB less the static part), or of two on an SM (228 KiB less 1 KiB each)
        assert nbytes + 512 <= 227 * 1024 if alone else 2 * (nbytes + 512 + 1024) <= 228 * 1024
        assert tokens * 256 <= nbytes - 1024  # the epilogue's bf16 tile
        # a set of decode warps can tell its use of a code slot from the use before
        reuse, sets = slots * 128 / depth, 4 if feat == 64 else 2
        assert (reuse % sets == 0 or reuse >= sets + stages) and sets <= max(stages, 2)
        if feat == 64:  # the MMAs' rows past the tile's read no further than the code ring
            assert alone and tokens <= 96 and slots * 8192 > 16384
        # the codes run ahead of the stages in flight
        assert slots >= math.ceil(stages * depth / 128) + (0 if depth == 128 and stages in (2, 4) else 1)
    assert chosen > 500


def test_measured_sides(plan):
    """(tokens, output features, contraction) -> whether the few-token kernel was the faster one."""
    sides = {(16, 4096, 4096): True, (187, 4096, 4096): True, (1024, 4096, 4096): True, (2048, 4096, 4096): False,
             (2048, 1024, 4096): True, (2048, 4096, 1024): False, (512, 14336, 4096): False, (64, 256, 512): True,
             (4096, 4096, 4096): False, (1999, 4096, 14336): False, (32768, 14336, 4096): False}
    for case, r in zip(sides, plan(list(sides))):
        assert bool(r[0]) == sides[case], case


@pytest.mark.parametrize("rows,F,K", [([128, 16, 16, 16], 1024, 4096), ([97, 1, 1], 640, 2080), ([8] * 7 + [256], 512, 2048),
                                      ([96, 5, 60], 1024, 4096), ([192] + [3] * 12, 1024, 1024)])
def test_estimate_is_of_the_launched_shape(rows, F, K):
    """Ragged experts: the tile shape follows the largest tile, and so does the estimate."""
    from few_plan import plan as plan_of
    p = plan_of(rows, F, K)
    if p is None:
        pytest.skip("no host C++ compiler or CUDA headers")
    assert p.limit and p.ctas <= SMS
    stage = 0.43 if p.features == 64 else 0.56 + 0.0015 * max(0, p.largest - 128)
    assert p.features == (64 if p.largest <= 96 and p.tiles * math.ceil(F / 64) <= SMS else 128)
    assert math.isclose(p.few_us, 4.8 + math.ceil(K / 128) * stage, rel_tol=1e-6)
