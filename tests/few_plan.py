"""Which kernel and tile shape a forward or input gradient gets: the host rules of
csrc/sq_internal.h compiled into a small program, for tests that need a certain plan."""
import atexit
import functools
import os
import shutil
import subprocess
import tempfile
from collections import namedtuple

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_04526_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
SMS = 152

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "sq_internal.h"
int main() {
  long long F, K, E;
  while (std::scanf("%lld %lld %lld", &F, &K, &E) == 3) {
    std::vector<long long> rows(E);
    long long M = 0, pair = 0;
    for (auto &r : rows) {
      if (std::scanf("%lld", &r) != 1) return 1;
      M += r;
      pair += (r + sqi::kPairMTile - 1) / sqi::kPairMTile * ((F + sqi::kPairNTile - 1) / sqi::kPairNTile);
    }
    auto tiles_at = [&](int limit) {
      int64_t n = 0;
      for (auto r : rows)
        if (r > 0) n += (r + sqi::few_tile_tokens(r, limit) - 1) / sqi::few_tile_tokens(r, limit);
      return n;
    };
    auto largest_at = [&](int limit) {
      int n = 0;
      for (auto r : rows)
        if (r > 0) n = std::max(n, sqi::few_tile_tokens(r, limit));
      return n;
    };
    const int limit = sqi::few_limit(tiles_at, M, F, K, pair, SMS, largest_at);
    if (!limit) {
      std::printf("0 0 0 0 0 0 0 0 %.9g %.9g\n", 0.0, sqi::pair_us(pair, K, SMS));
      continue;
    }
    const int largest = largest_at(limit);
    const int64_t tiles = tiles_at(limit);
    const int feat = sqi::few_features(tiles, largest, F, SMS);
    const int64_t ctas = tiles * ((F + feat - 1) / feat);
    const sqi::FewRing r = sqi::few_ring(largest, ctas <= SMS, feat);
    std::printf("%d %d %lld %lld %d %d %d %d %.9g %.9g\n", limit, largest, (long long)tiles, (long long)ctas, feat, r.depth,
                r.stages, r.slots, sqi::few_us(tiles, (double)M / tiles, F, K, SMS, largest), sqi::pair_us(pair, K, SMS));
  }
  return 0;
}
"""

# limit, largest, ...: of the few-token launch; all 0 where the pair kernel runs
Plan = namedtuple("Plan", "limit largest tiles ctas features depth stages slots few_us pair_us")


@functools.lru_cache(maxsize=1)
def _program():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda.h")):
        return None
    d = tempfile.mkdtemp(prefix="few_plan")
    atexit.register(shutil.rmtree, d, True)
    src, exe = os.path.join(d, "few_plan.cpp"), os.path.join(d, "few_plan")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", f"-DSMS={SMS}", f"-I{CSRC}", f"-I{CUDA_INC}", src, "-o", exe], check=True)
    return exe


def plan(rows, features, contraction):
    """Plan of a product over these token rows (a number: dense, a list: per expert) with this
    many output features (forward N, input gradient K) and this contraction; None without a
    host compiler."""
    if _program() is None:
        return None
    rows = [rows] if isinstance(rows, int) else list(rows)
    out = subprocess.run([_program()], input=" ".join(map(str, [features, contraction, len(rows), *rows])), capture_output=True,
                         text=True, check=True).stdout.split()
    return Plan(*[int(v) for v in out[:8]], float(out[8]), float(out[9]))
