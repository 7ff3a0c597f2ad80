// Forward and input gradient over few tokens (sm_103a): short examples, one-sequence
// calls of narrow linears, experts with tens to hundreds of rows.
//
//   MODE_FWD  Y[m,n]  = sum_k X[m,k] W[n,k]      MODE_DX  dX[m,k] = sum_n dY[m,n] W[n,k]
//
// The 512 x 256 tiles of sq_gemm_pair_kernel leave most SMs without a tile there, and
// most rows of a tile empty. This kernel turns the product around: the decoded weights
// are the MMA's A operand (128 output features) and up to 256 tokens its N, so the
// tensor work follows the token count. Every output is still the sum of the same K = 16
// steps in the same order, so its bits do not depend on which of the two kernels ran
// (the contraction is not split over CTAs for that reason).
//
// Three rings feed the MMA warp: packed codes (TMA, run far ahead: the first touches of a
// weight take 2,000 to 3,000 cycles), activations (TMA) and the weights that the decode
// warps make of the codes; the last two share stages. Three shapes:
//   128-deep stages, 16 decode warps in two sets, one CTA per SM: launches of at most one
//   CTA per SM.
//   The same with 64 features and four sets: where twice as many tiles still have an SM each.
//   64-deep stages, 8 decode warps, two CTAs per SM, so that one computes while the other
//   starts up, waits for memory or drains: larger launches.
//
// Measured (forward; before: the pair kernel): 4096 x 4096 at 187 tokens 43 -> 18.5 us, 1024 x
// 4096 at 2048 tokens 44 -> 25 us, 128 experts of 768 x 2048 with 128 rows each 131 -> 87 us,
// of 2880 x 2880 with 16 rows each 566 -> 271 us (2.1 TB/s of codes). Bound by latency: with
// two CTAs per SM (128 experts of 768 x 2048, 128 rows each) the schedulers issue in 52 % of
// the cycles forward and 51 % in the input gradient, the tensor pipe is busy for 29 and 24 %,
// DRAM at 31 and 24 % of its rate, and of the warps waiting most (4.1 and 3.9 per issue) wait on
// the long scoreboard; a CTA alone issues in 43 %. clock64 traces of one CTA show what a stage's
// chain consists of (a barrier test ~110 cycles, a commit ~100, a TMA load ~150, beside the
// decode): hence the long stages, and one elected lane per warp.
// Codes and activations have a TMA warp each: with one for both a stage of a CTA alone took
// 0.60 us where it takes 0.54 (4096 x 4096 at 187 tokens 24.7 -> 22.6 us, 4096 x 14336 at 64
// tokens 71.9 -> 61.6 us; the experts' launches, two CTAs per SM, are unchanged); in tiles of
// 64 features 0.43 us (18.5 and 46 us).
// Codes loaded by the decode warps into registers, four units ahead, were 20-50 % slower and
// the experts' forward half as fast; 64-deep stages took 29-33 us for the 25 us launches.
#include <climits>

#include "sq_gemm_kernels.cuh"

namespace sqi {
namespace {

struct FewCfg {
  static constexpr int kF = kFewFeatures;       // output features of a tile (the MMA's M)
  static constexpr int kBoxRows = kFewBoxRows;  // tokens of the smallest TMA box (128 bytes x 32 rows, 4 KiB)
  static constexpr int kBox = kBoxRows * 128;
  static constexpr int kC = kFewSlotBytes;      // 8 KiB: the codes of 128 x 128 weights (64-byte rows, 64-byte swizzle)
  static constexpr int kAhead = 8;              // units whose scale bytes are in registers
  static constexpr int kMaxStages = kFewMaxStages;
  static constexpr int kMaxSlots = kFewMaxSlots;
};

struct FewParams {
  const uint8_t *scales;
  float ws2;
  int64_t M, N, K;
  uint16_t *out;
  int *err;
  const FewTile *tiles;  // grouped: the token tiles; dense: null
  int tile_tokens;       // dense: tokens of a tile
  int ftiles;            // feature tiles
  int box_rows;          // token rows of a stage's activations
  int stages, stage_bytes;
  int slots;             // of the code ring
  int tmem_cols;
};
struct FewMaps {
  CUtensorMap box[3];  // the activations: grouped, in boxes of 32, 64 and 128 tokens; dense, [0] a tile's tokens
  CUtensorMap codes;   // the packed codes in 64-byte x 128-row boxes
};

// Barrier arrivals and TMA loads issued by one elected lane of a converged warp.
__device__ __forceinline__ void expect_tx_elect(uint64_t *bar, uint32_t bytes) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xFFFFFFFF;\n\t"
      "@e mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
      "r"(bytes)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_elect(uint32_t dst, const CUtensorMap *map, uint64_t *bar, int32_t x,
                                                  int32_t y) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xFFFFFFFF;\n\t"
      "@e cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];\n\t}" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// After an abort: waits, with a limit each, for the copies into a ring's slots in flight, of
// `fills` made so far. All of them (the last may land first); a stage that its decode warps gave
// up only ends at the limit.
__device__ __noinline__ void drain_ring(uint64_t *full, int fills, int slots) {
  for (int i = (fills > slots ? fills - slots : 0); i < fills; ++i)
    mbar_drain(&full[i % slots], static_cast<uint32_t>(i / slots) & 1u);
}

// BK: contraction depth of a stage. WARPS: decode warps, which then run the epilogue.
// GROUPS: see the decode warps. FEAT: output features of a tile; of 64 the MMAs' upper 64
// rows multiply whatever the shared memory holds, into accumulator lanes that nothing reads.
template <int MODE, int FMT, int BK, int WARPS, int GROUPS, int FEAT>
__global__ void __launch_bounds__(32 * (WARPS + 3), 16 / WARPS)
    sq_gemm_few_kernel(const __grid_constant__ FewMaps maps, const FewParams p) {
  using C = FewCfg;
  constexpr int kTmaWarp = WARPS, kMmaWarp = WARPS + 1, kCodeWarp = WARPS + 2, kThreads = 32 * (WARPS + 3);
  constexpr int kA = FEAT * BK * 2;                          // decoded weights of a stage
  constexpr int kUnits = FEAT / 32 * BK * GROUPS / (32 * WARPS);  // 32-weight units of a thread per stage
  constexpr int kPer = 128 / BK;                             // stages of a code slot
  static_assert(GROUPS % kPer == 0 && C::kAhead % kUnits == 0, "a group's stages share one half of their slots");
  extern __shared__ uint8_t few_smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(few_smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t bars[2 * C::kMaxStages + 2 * C::kMaxSlots + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  volatile int *abort_flag = &abort_word;
  // One barrier per stage says that it is complete (the activation boxes' bytes and the
  // weights' decode warps): each test costs the MMA warp ~110 cycles.
  uint64_t *full = bars;                    // [stages] 1 arrival + tx, and the arrivals of one group's warps
  uint64_t *empty = full + C::kMaxStages;   // [stages] the MMAs reading the stage are done (commit)
  uint64_t *cfull = empty + C::kMaxStages;  // [slots] the codes landed                     (1 arrival + tx)
  uint64_t *cempty = cfull + C::kMaxSlots;  // [slots] its stages' warps have read them     (their arrivals)
  uint64_t *done = cempty + C::kMaxSlots;   // every MMA of the tile is done                (commit)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.stages;
  const int tt = static_cast<int>(blockIdx.x) / p.ftiles, ft = static_cast<int>(blockIdx.x) - tt * p.ftiles;
  FewTile tile;
  if (p.tiles) {
    tile = p.tiles[tt];
  } else {
    tile.expert = 0;
    tile.row0 = tt * p.tile_tokens;
    tile.rows = static_cast<int>(p.M - tile.row0 < p.tile_tokens ? p.M - tile.row0 : p.tile_tokens);
    tile.ws2 = p.ws2;
  }
  const int64_t F = MODE == MODE_FWD ? p.N : p.K;   // output features
  const int64_t Kc = MODE == MODE_FWD ? p.K : p.N;  // contraction
  const int64_t f0 = static_cast<int64_t>(ft) * FEAT;
  const int cnt = static_cast<int>((Kc + BK - 1) / BK);  // stages
  const int boxes = (tile.rows + C::kBoxRows - 1) / C::kBoxRows;

  uint8_t *code_ring = smem + S * p.stage_bytes;
  // The two TMA warps set up the barriers they wait on and start at once; the others meet
  // them at `start` before they touch one.
  auto start = [] { asm volatile("barrier.sync 1, %0;" ::"n"(kThreads) : "memory"); };

  if (warp == kCodeWarp) {
    // ------------------------------------------------------ packed codes
    // The whole warp walks the slots and an elected lane issues (see the MMA warp). A slot
    // holds 128 rows x 64 bytes: FWD 128 feature rows x 128 k, DX 128 contraction rows x
    // 128 feature columns (a tile of 64 features uses the first half).
    if (lane == 0) {
      for (int c = 0; c < p.slots; ++c) {
        mbar_init(&cfull[c], 1);
        mbar_init(&cempty[c], kPer * (WARPS / GROUPS));
      }
      abort_word = 0;
      fence_barrier_init();
      fence_proxy_async_smem();
    }
    __syncwarp();
    asm volatile("barrier.arrive 1, %0;" ::"n"(kThreads) : "memory");
    const int fills = (cnt + kPer - 1) / kPer;
    const int cx = MODE == MODE_FWD ? 0 : static_cast<int>(f0 / 2);
    const int cy = static_cast<int>(tile.expert * p.N) + (MODE == MODE_FWD ? static_cast<int>(f0) : 0);
    int j = 0, c = 0;  // slots filled, the next one and its use parity
    uint32_t ph = 0;
    for (; j < fills; ++j) {
      if (j >= p.slots && !__all_sync(0xFFFFFFFFu, mbar_wait(&cempty[c], ph ^ 1u, abort_flag, p.err))) break;
      expect_tx_elect(&cfull[c], C::kC);
      tma_load_2d_elect(smem_u32(code_ring) + c * C::kC, &maps.codes, &cfull[c], cx + (MODE == MODE_FWD ? j * 64 : 0),
                        cy + (MODE == MODE_FWD ? 0 : j * 128));
      if (++c == p.slots) {
        c = 0;
        ph ^= 1u;
      }
    }
    if (*abort_flag) drain_ring(cfull, j, p.slots);
    __syncwarp();
  } else if (warp == kTmaWarp) {
    // ------------------------------------------------------ activations
    if (lane == 0) {
      for (int s = 0; s < S; ++s) {
        mbar_init(&full[s], 1 + WARPS / GROUPS);
        mbar_init(&empty[s], 1);
      }
      mbar_init(done, 1);
      abort_word = 0;
      fence_barrier_init();
      fence_proxy_async_smem();
    }
    __syncwarp();
    asm volatile("barrier.arrive 1, %0;" ::"n"(kThreads) : "memory");
    int it = 0, s = 0;
    uint32_t ph = 0, dst = smem_u32(smem) + kA;
    // Rows past the tile's last token (the next expert's, or zeros past M) only fill
    // accumulator columns that nothing stores.
    for (; it < cnt; ++it) {
      if (it >= S && !__all_sync(0xFFFFFFFFu, mbar_wait(&empty[s], ph ^ 1u, abort_flag, p.err))) break;
      expect_tx_elect(&full[s], static_cast<uint32_t>((p.tiles ? boxes * C::kBoxRows : p.box_rows) * (BK * 2)));
#pragma unroll
      for (int h = 0; h < BK / 64; ++h) {  // 64-wide chunks of the contraction
        const int x = it * BK + 64 * h;
        const uint32_t d = dst + h * p.box_rows * 128;
        if (!p.tiles) {  // dense: one box holds a tile's tokens
          tma_load_2d_elect(d, &maps.box[0], &full[s], x, tile.row0);
        } else {  // the largest boxes that the tile's 32-token units fill
          int b = 0;
          for (; b + 4 <= boxes; b += 4)
            tma_load_2d_elect(d + b * C::kBox, &maps.box[2], &full[s], x, tile.row0 + b * C::kBoxRows);
          if (boxes & 2) {
            tma_load_2d_elect(d + b * C::kBox, &maps.box[1], &full[s], x, tile.row0 + b * C::kBoxRows);
            b += 2;
          }
          if (boxes & 1) tma_load_2d_elect(d + b * C::kBox, &maps.box[0], &full[s], x, tile.row0 + b * C::kBoxRows);
        }
      }
      dst += p.stage_bytes;
      if (++s == S) {
        s = 0;
        dst = smem_u32(smem) + kA;
        ph ^= 1u;
      }
    }
    if (*abort_flag) drain_ring(full, it, S);
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------ MMA issuer
    tmem_alloc(&tmem_slot, p.tmem_cols);
    tc_fence_before();
    __syncwarp();
    start();
    tc_fence_after();
    // The whole warp walks the stages and one elected lane issues: warp-uniform
    // descriptors stay in uniform registers, where a single lane's would be moved there
    // for every MMA (65 to 110 cycles per MMA against 30).
    const uint32_t tmem = tmem_slot;
    const int n16 = (tile.rows + 15) & ~15;
    const uint32_t idesc = idesc_bf16(C::kF, n16, MODE == MODE_FWD ? 0 : 1, 0);
    // weights: FWD K-major (64-wide chunks of FEAT rows, 32 bytes per K step), DX MN-major
    // (64-feature atoms of BK contraction rows, 16 rows = 2 KiB per K step); activations
    // K-major in 64-wide chunks. Rows 64-127 of a 64-feature tile are what follows in the
    // shared memory: at most 16 KiB past the weights, less than the code ring behind the
    // last stage.
    const uint32_t base = smem_u32(smem);
    const uint64_t ad0 = MODE == MODE_FWD ? smem_desc_sw128(base, 16, 1024) : smem_desc_sw128(base, BK * 128, 1024);
    const uint64_t bd0 = smem_desc_sw128(base + kA, 16, 1024);
    const uint32_t chunk = static_cast<uint32_t>(p.box_rows) * 128 >> 4;  // of the activations, in descriptor units
    const uint32_t step = static_cast<uint32_t>(p.stage_bytes) >> 4;
    uint32_t so = 0;  // the slot's offset in descriptor units
    int s = 0;
    uint32_t ph = 0;
    for (int it = 0; it < cnt; ++it) {
      if (!__all_sync(0xFFFFFFFFu, mbar_wait(&full[s], ph, abort_flag, p.err))) break;
      tc_fence_after();
      const uint64_t ad = ad0 + so, bd = bd0 + so;
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk)
        umma_bf16_elect(tmem, ad + ((MODE == MODE_FWD ? (kk >> 2) * (FEAT * 128) + (kk & 3) * 32 : kk * 2048) >> 4),
                        bd + (kk >> 2) * chunk + ((kk & 3) * 32 >> 4), idesc, (it > 0 || kk > 0) ? 1u : 0u);
      umma_commit_elect(&empty[s]);
      so += step;
      if (++s == S) {
        s = 0;
        so = 0;
        ph ^= 1u;
      }
    }
    umma_commit_elect(done);
    mbar_drain(done, 0);
  } else {
    // ------------------------------------------------------ decode
    // The warps form GROUPS groups; group g decodes stages g, g + GROUPS, ..., kUnits
    // 32-weight units per thread and stage, so one proxy fence and one barrier arrival
    // serve kUnits units and GROUPS stages are being decoded at a time. FWD: a stage is
    // FEAT feature rows x BK k; DX: BK contraction rows x FEAT feature columns. The 8 lanes
    // that share a shared-memory wavefront hold 8 different rows.
    constexpr int kGroupThreads = 32 * WARPS / GROUPS;
    constexpr int kAcross = MODE == MODE_FWD ? BK / 32 : FEAT / 32;  // units of a row
    constexpr int kRowStep = kGroupThreads / kAcross;         // rows between a thread's units
    const int grp = threadIdx.x / kGroupThreads;
    const int u = threadIdx.x % kGroupThreads;
    const int row = (u & 7) + 8 * (u / (8 * kAcross));
    const int q = (u >> 3) % kAcross;  // which 32 of the row
    constexpr int B = FMT == 0 ? 16 : 32;
    const int64_t G = p.K / B;
    // position of the thread's first unit in the weight
    const int64_t n0 = MODE == MODE_FWD ? f0 + row : row;
    const int64_t k0 = MODE == MODE_FWD ? 32 * q : f0 + 32 * q;
    const uint8_t *sp = p.scales + (static_cast<int64_t>(tile.expert) * p.N + n0) * G + k0 / B;
    // Scale bytes run kAhead units ahead in registers, so their pointer and the rows left
    // move on every kUnits loads.
    const int srow = static_cast<int>(G);
    const int64_t sstep = static_cast<int64_t>(GROUPS) * (MODE == MODE_FWD ? BK / B : BK * static_cast<int64_t>(srow));
    sp += grp * (sstep / GROUPS);
    // rows of the weight from the thread's first one on, at the loads' stage, and stages
    // whose 32 weights lie inside it
    int rows_left = static_cast<int>(p.N - n0 < INT_MAX ? p.N - n0 : INT_MAX) - (MODE == MODE_FWD ? 0 : grp * BK);
    int stages_left = cnt - grp;
    if (MODE == MODE_FWD) {
      const int64_t in = k0 < p.K ? (p.K - k0 + BK - 1) / BK - grp : 0;
      if (in < stages_left) stages_left = static_cast<int>(in);
    } else if (k0 >= p.K) {
      stages_left = 0;
    }
    uint32_t sw[C::kAhead];
    auto load = [&](int r) -> uint32_t {  // scale bytes of unit r of the loads' stage
      // Outside the weight byte 0, for NVFP4 a scale of zero. For MXFP4 it is 2^-127, and the
      // other operand or the store makes up for it: TMA fills the activations with zeros past
      // the contraction's end, and features past the last are not stored.
      uint32_t sc = 0;
      if (stages_left > 0 && r * kRowStep < rows_left) {
        const uint8_t *s = sp + static_cast<int64_t>(r * kRowStep) * srow;
        sc = FMT == 0 ? __ldg(reinterpret_cast<const unsigned short *>(s)) : __ldg(s);
      }
      if (r == kUnits - 1) {
        sp += sstep;
        stages_left -= GROUPS;
        if (MODE != MODE_FWD) rows_left -= GROUPS * BK;
      }
      return sc;
    };
#pragma unroll
    for (int d = 0; d < C::kAhead; ++d) sw[d] = load(d % kUnits);
    // the first unit's codes in the slot (of 64-deep stages, the thread's are all the first
    // or all the second half of their slots), and its 16-byte chunks in the stage's
    // 128-byte-swizzled tile
    const int half = grp % kPer;
    const uint32_t c_off = MODE == MODE_FWD ? row * 64 + (((half * kAcross + q) ^ ((row >> 1) & 3)) << 4)
                                            : (half * BK + row) * 64 + ((q ^ ((row >> 1) & 3)) << 4);
    uint32_t off[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      off[c] = (q >> 1) * (MODE == MODE_FWD ? FEAT * 128 : BK * 128) + row * 128 + (((4 * (q & 1) + c) ^ (row & 7)) << 4);
    __syncwarp();
    start();
    bool ok = true;
    int s = grp;  // ring slot and use parity of the group's stage (GROUPS <= stages)
    uint32_t ph = 0;
    int cs = grp / kPer;  // code slot and its use parity (few_ring: which slot counts this can follow)
    uint32_t cph = 0;
    while (cs >= p.slots) {
      cs -= p.slots;
      cph ^= 1u;
    }
    for (int it0 = grp; it0 < cnt && ok; it0 += C::kAhead / kUnits * GROUPS) {
#pragma unroll
      for (int d = 0; d < C::kAhead; ++d) {
        const int it = it0 + d / kUnits * GROUPS;
        if (it >= cnt) break;
        if (d % kUnits == 0 && !(ok = mbar_wait(&cfull[cs], cph, abort_flag, p.err))) break;
        uint32_t sc_lo, sc_hi;
        if (FMT == 0) {
          sc_lo = scale_bf16x2<0>(sw[d] & 0xFFu);
          sc_hi = scale_bf16x2<0>(sw[d] >> 8);
        } else {
          sc_lo = sc_hi = scale_bf16x2<1>(sw[d]);
        }
        const uint4 cw = lds128(smem_u32(code_ring) + cs * C::kC + c_off + (d % kUnits) * kRowStep * 64);
        const uint32_t words[4] = {cw.x, cw.y, cw.z, cw.w};
        uint32_t o[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          e2m1x8_to_bf16(words[c], o[c]);
#pragma unroll
          for (int i = 0; i < 4; ++i) o[c][i] = bf16x2_mul(o[c][i], c < 2 ? sc_lo : sc_hi);
        }
        sw[d] = load(d % kUnits);
        if (d % kUnits == 0 && it >= S && !(ok = mbar_wait(&empty[s], ph ^ 1u, abort_flag, p.err))) break;
        const uint32_t base = smem_u32(smem) + s * p.stage_bytes + (d % kUnits) * kRowStep * 128;
#pragma unroll
        for (int c = 0; c < 4; ++c) st_shared_v4(base + off[c], o[c][0], o[c][1], o[c][2], o[c][3]);
        if (d % kUnits == kUnits - 1) {
          fence_proxy_async_smem();  // this thread's shared-memory writes -> async proxy
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(&full[s]);
            mbar_arrive(&cempty[cs]);  // the warp's code reads are done
          }
          if ((s += GROUPS) >= S) {
            s -= S;
            ph ^= 1u;
          }
          cs += GROUPS / kPer;
          while (cs >= p.slots) {
            cs -= p.slots;
            cph ^= 1u;
          }
        }
      }
    }
  }

  // ------------------------------------------------------ epilogue
  // The decode warps scale the accumulator (lane = feature, column = token), round it to
  // bf16 and put it into shared memory as [token][128 features], over the stages (their
  // MMAs are done), then store whole row segments, 16 bytes per lane.
  __syncwarp();
  if (warp < WARPS) {
    mbar_wait(done, 0, abort_flag, p.err);
    __syncwarp();
    tc_fence_after();
    const float scale = FMT == 0 ? tile.ws2 : 1.0f;
    const uint32_t t_row = tmem_slot + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint32_t tokens_smem = smem_u32(smem);
#pragma unroll 1
    for (int c = 32 * (warp >> 2); c < tile.rows && (warp & 3) < FEAT / 32; c += 8 * WARPS) {
      uint32_t v[32];
      tmem_ld32(t_row + c, v);
      tmem_ld_wait();
      const uint32_t dst = tokens_smem + (c * C::kF + (warp & 3) * 32 + lane) * 2;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const unsigned short h = __bfloat16_as_ushort(__float2bfloat16_rn(__uint_as_float(v[i]) * scale));
        asm volatile("st.shared.b16 [%0], %1;" ::"r"(dst + i * C::kF * 2), "h"(h) : "memory");
      }
    }
    asm volatile("barrier.sync 2, %0;" ::"n"(32 * WARPS) : "memory");
    uint16_t *out = p.out + static_cast<int64_t>(tile.row0) * F + f0;
    const int f = 8 * (threadIdx.x & 15);
    if (f < FEAT && f0 + f < F) {
      for (int t = threadIdx.x >> 4; t < tile.rows; t += 2 * WARPS) {
        const uint4 v = lds128(tokens_smem + (t * C::kF + f) * 2);
        *reinterpret_cast<uint4 *>(out + static_cast<int64_t>(t) * F + f) = v;
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_slot, p.tmem_cols);
  }
}

template <int MODE, int FMT, int BK, int WARPS, int GROUPS, int FEAT>
cudaError_t launch_one(const FewParams &p, const FewMaps &maps, int64_t units, int smem, cudaStream_t stream) {
  static int done_mask = 0;  // per device ordinal (first 31)
  int dev = 0;
  cudaGetDevice(&dev);
  const auto kernel = sq_gemm_few_kernel<MODE, FMT, BK, WARPS, GROUPS, FEAT>;
  if (!(done_mask & (1 << (dev & 31)))) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  WARPS == 16 ? kFewSmemAlone : kFewSmemBytes)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  cudaSharedmemCarveoutMaxShared)) != cudaSuccess)
      return e;
    done_mask |= 1 << (dev & 31);
  }
  kernel<<<static_cast<unsigned>(units), 32 * (WARPS + 3), smem, stream>>>(maps, p);
  return cudaGetLastError();
}

template <int BK, int WARPS, int GROUPS, int FEAT>
cudaError_t launch_shape(const FewArgs &a, const FewParams &p, const FewMaps &maps, int smem, cudaStream_t stream) {
  if (a.mode == MODE_FWD)
    return a.fmt == 0 ? launch_one<MODE_FWD, 0, BK, WARPS, GROUPS, FEAT>(p, maps, a.units, smem, stream)
                      : launch_one<MODE_FWD, 1, BK, WARPS, GROUPS, FEAT>(p, maps, a.units, smem, stream);
  return a.fmt == 0 ? launch_one<MODE_DX, 0, BK, WARPS, GROUPS, FEAT>(p, maps, a.units, smem, stream)
                    : launch_one<MODE_DX, 1, BK, WARPS, GROUPS, FEAT>(p, maps, a.units, smem, stream);
}

}  // namespace

cudaError_t launch_few(const FewArgs &a, const CUtensorMap (&tmX)[3], const CUtensorMap &tmCodes, int sm_count,
                       cudaStream_t stream) {
  const FewMaps maps = {{tmX[0], tmX[1], tmX[2]}, tmCodes};
  const FewRing ring = few_ring(a.tile_tokens, a.units <= sm_count, a.features);
  if (ring.slots < 2) return cudaErrorInvalidValue;
  FewParams p;
  p.scales = a.scales;
  p.ws2 = a.ws2;
  p.M = a.M;
  p.N = a.N;
  p.K = a.K;
  p.out = a.out;
  p.err = a.err;
  p.tiles = a.tiles;
  p.tile_tokens = a.tile_tokens;
  p.ftiles = static_cast<int>(((a.mode == MODE_FWD ? a.N : a.K) + a.features - 1) / a.features);
  p.box_rows = few_box_rows(a.tile_tokens);
  p.stage_bytes = ring.stage_bytes;
  p.stages = ring.stages;
  p.slots = ring.slots;
  for (p.tmem_cols = 32; p.tmem_cols < a.tile_tokens; p.tmem_cols *= 2) {
  }
  if (a.features == kFewNarrow)
    return ring.depth == 128 ? launch_shape<128, 16, kFewGroupsNarrow, kFewNarrow>(a, p, maps, ring.bytes, stream)
                             : cudaErrorInvalidValue;
  return ring.depth == 128 ? launch_shape<128, 16, kFewGroups, kFewFeatures>(a, p, maps, ring.bytes, stream)
                           : launch_shape<64, 8, kFewGroups, kFewFeatures>(a, p, maps, ring.bytes, stream);
}

}  // namespace sqi
