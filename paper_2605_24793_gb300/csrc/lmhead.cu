// LM head fused with argmax and log-prob statistics (Sec. 3.1 Eq. 2: the
// target prediction y_tilde is the argmax of each block row's logits;
// Eq. 23: l_i = x[y_hat_i] - lse).  The M x V logits never reach memory.
//
// tcgen05 swap-AB GEMM: the vocabulary is the MMA M dimension and the verify
// rows are N (padded to a multiple of 32, <= 256 per slice), so a handful of rows
// still fills the tensor core and W -- the only large operand -- is streamed from
// HBM exactly once.  Two CTAs of a cluster share every MMA (cta_group::2, M = 256
// vocabulary rows, 128 of them in each CTA's TMEM): each loads its 128 W rows and
// half of the hidden rows, so an SM takes in 32 KB per 64-wide k-block at 256 rows
// instead of 48.  Persistent pairs (76 on 152 SMs) walk the vocabulary tiles; with
// more than 256 rows, pairs side by side take the row slices of the same tile, so
// W still comes from HBM once.  In each CTA warp 0 issues the TMA loads of W (128B
// swizzle, evict-first) and warp 10 those of the hidden rows (evict-last) into a
// ring of stages (one warp's bulk copies are processed one after another); in the
// pair's leader warp 1 issues the MMAs into one of two TMEM accumulators; warps
// 2-9 fold the finished accumulator into statistics while the next tile is
// multiplied.  A warp may only read the TMEM lane quarter (warp id mod 4), so two
// epilogue warps share each quarter and take alternate 32-column chunks: a chunk
// is transposed through the warp's own shared buffer, after which a lane owns one
// hidden row and folds 32 logits into registers that last over all tiles -- about
// 12 instructions a logit, no shuffles, no barriers.  (A butterfly over the lanes
// with an exponential per merge took 20 us per 256-row tile, exposed after the last
// tile and the bound at d <= 2048; this takes about 3.)  A second small kernel
// merges the per-CTA partials.
//
// Bound: HBM up to about 200 rows, then the operands' way into the SMs (about 13.5
// TB/s over the chip) and the tensor pipe.  The MMAs of a k-block are issued by a
// converged warp, four to a statement: from one diverged thread an MMA took 100 cycles
// and several times that beside the epilogue's warps on its scheduler, which held up the
// mainloop for as long as an epilogue ran (all modes: 128 rows 188 -> 181 us, sampling
// 207 -> 187.5; 384 rows 346 -> 281).  Measured on GB300, us per call, one CTA per MMA
// with the butterfly -> this kernel:
//   Qwen3-8B (d 4096, V 151936)   6 rows 187.3 -> 181 to 184 (the copy peak),
//     128 rows 200.7 -> 180.1, 256 rows 238.9 -> 196.2
//   Qwen3-32B (d 5120)            256 rows 289.5 -> 243.4 (0.95 of the copy peak)
//   Llama-3-8B (V 128256)         384 rows 375.1 -> 244.9, 512 rows 421.5 -> 297.9
//     (1.81 PFLOP/s)
//   d 1024, V 32003               256 rows 55.7 -> 22.2, 512 rows 110.7 -> 30.6
//
// Statistics are kept as a tuple (m, i, sec, s, t): max logit, its lowest
// id, second largest logit, s = sum e^(x-m), t = sum e^(x-m) (x-m); then
// lse = m + log s and entropy = log s - t/s.
//
// Stochastic decoding (Sec. 3.1, App. C.3: candidates drawn at temperature
// T = 1) uses the same kernel with KEYED = true: the target candidate is a
// sample of softmax(x / T) taken by the Gumbel-max rule, argmax_v of
// k_v = x_v / T + g_v with g_v = -log(-log u_v).  u comes from Philox4x32-10
// (Salmon et al., SC 2011) keyed by a 64-bit seed read from device memory, at
// counter (v, m / 4, 0, 0), output m % 4, so a thread that owns vocab id v and
// four consecutive rows makes one generator call.  The tuple then carries the
// best key k and i becomes its id; m, sec, s, t stay statistics of the logits.
//
// Speculative sampling (the distribution-preserving baseline at temperature
// T, Sec. 3.1) needs the target's whole distribution at the row where a draft
// token is rejected, so a third mode (MODE_LOGITS) scales the logits by 1 / T,
// writes them out ([M, V] fp32) and keeps the statistics of the scaled logits.
#include <cuda.h>
#include <math.h>

#include <atomic>

#include "../../include/cospec.h"
#include "cospec_device.cuh"
#include "cospec_internal.h"

namespace cospec {

namespace {

constexpr int BM = 128;                 // vocab rows of a tile per CTA
constexpr int BMP = 2 * BM;             // vocab rows of a tile: MMA M of a CTA pair
constexpr int BK = 64;                  // K elements per stage (one 128-byte swizzle row)
constexpr int A_BYTES = BM * BK * 2;    // 16 KB
constexpr int EPI_WARPS = 8;            // two per TMEM lane quarter
constexpr int EPI_THREADS = 32 * EPI_WARPS;
constexpr int H_WARP = 2 + EPI_WARPS;   // producer of the hidden-row boxes
constexpr int NUM_THREADS = 64 + EPI_THREADS + 32;   // W producer, MMA, epilogue, hidden producer
constexpr int MAX_ROWS = 256;           // rows per slice
constexpr int MAX_CHUNKS = MAX_ROWS / 64;   // 32-column chunks of a tile per epilogue warp
constexpr uint64_t WAIT_NS = 2000000000ull;

struct Stat {
  float m;
  int i;
  float sec;
  float s;
  float t;
  float k;    // KEYED only: largest perturbed key, whose id is i
};

CS_DEV Stat stat_identity() { return Stat{-INFINITY, 0x7fffffff, -INFINITY, 0.f, 0.f, -INFINITY}; }

// max that passes NaN on, so that a NaN logit reaches the log-sum-exp
CS_DEV float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

template <bool KEYED>
CS_DEV Stat stat_merge(const Stat& a, const Stat& b) {
  Stat r;
  bool a_hi;
  if (KEYED) {
    const bool a_key = (a.k > b.k) || (a.k == b.k && a.i < b.i);
    r.k = a_key ? a.k : b.k;
    r.i = a_key ? a.i : b.i;
    a_hi = a.m >= b.m;
  } else {
    a_hi = (a.m > b.m) || (a.m == b.m && a.i < b.i);
    r.i = a_hi ? a.i : b.i;
    r.k = 0.f;
  }
  const Stat& hi = a_hi ? a : b;
  const Stat& lo = a_hi ? b : a;
  r.m = hi.m;
  r.sec = fmaxf(fmaxf(hi.sec, lo.sec), lo.m);
  if (!(lo.s <= 0.f)) {                  // NaN too
    const float dm = max_nan(lo.m - hi.m, -126.f);   // e^-126 is 0 in float
    const float e = __expf(dm);
    r.s = hi.s + lo.s * e;
    r.t = hi.t + e * (lo.t + lo.s * dm);
  } else {
    r.s = hi.s;
    r.t = hi.t;
  }
  return r;
}

template <bool KEYED>
CS_DEV Stat stat_shfl_xor(const Stat& a, int off) {
  Stat r;
  r.m = __shfl_xor_sync(0xffffffffu, a.m, off);
  r.i = __shfl_xor_sync(0xffffffffu, a.i, off);
  r.sec = __shfl_xor_sync(0xffffffffu, a.sec, off);
  r.s = __shfl_xor_sync(0xffffffffu, a.s, off);
  r.t = __shfl_xor_sync(0xffffffffu, a.t, off);
  r.k = KEYED ? __shfl_xor_sync(0xffffffffu, a.k, off) : 0.f;
  return r;
}

// The warps' transposition buffers: 32 columns x 32 vocabulary ids of floats each, column by column,
// the 16-byte chunks of a column exchanged by its number, so that both a store of one column by the 32
// lanes and a 16-byte load of one chunk of 32 columns touch every bank once.
constexpr int XP_BYTES = 32 * 32 * 4;
CS_DEV uint32_t xp_off(int col, int v) {     // in floats
  return (uint32_t)(col * 32 + (((v >> 2) ^ (col & 7)) << 2) + (v & 3));
}

// Running statistics of one column (a hidden row) over the vocabulary ids of one lane: s and t are
// relative to m.
struct RowStat {
  float m;
  int i;
  float sec;
  float s;
  float t;
  float k;
};

// Fold 32 logits of ids v0 .. v0 + 31 (ascending, so a tie keeps the lowest id) into a column's
// statistics.  KEYED: the id is that of the best key instead (row_keys).
template <bool KEYED>
CS_DEV void row_fold(RowStat& r, const float (&x)[32], int v0) {
  constexpr float LOG2E = 1.4426950408889634f;
  const float m_old = r.m;
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const bool up = x[j] > r.m;
    r.sec = fmaxf(r.sec, fminf(x[j], r.m));
    if (!KEYED) r.i = up ? v0 + j : r.i;
    r.m = fmaxf(r.m, x[j]);
  }
  // finite, so that a logit of +infinity gives an infinite (not undefined) sum
  const float base = r.m == -INFINITY ? 0.f : fminf(r.m, 3.4028235e38f);
  // e^-126 is 0 in float: the bound keeps 0 * infinity out of t
  const float dm = fmaxf(m_old - base, -126.f);
  const float f = r.s > 0.f ? exp2_approx(dm * LOG2E) : 1.f;
  float s4[4] = {r.s * f, 0.f, 0.f, 0.f}, t4[4] = {f * fmaf(r.s, dm, r.t), 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const float d = max_nan(x[j] - base, -126.f);
    const float e = exp2_approx(d * LOG2E);
    s4[j & 3] += e;
    t4[j & 3] = fmaf(e, d, t4[j & 3]);
  }
  r.s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
  r.t = (t4[0] + t4[1]) + (t4[2] + t4[3]);
}

struct LmParams {
  const int32_t* draft_for_row;  // [M]
  float* stats;                  // [M][5]
  float4* part;                  // [rows of the launch][parts]: (m, sec, s, t)
  int* part_idx;                 // [rows][parts]
  float* part_k;                 // [rows][parts], KEYED only
  int parts;                     // CTAs that hold partials of a row
  const unsigned long long* seed;  // KEYED only: Philox key (low word, high word)
  float inv_temp;                // KEYED and LOGITS: 1 / T
  float* logits;                 // LOGITS only: [M][V] x / T
  int n_mma;
  int passes;                    // row slices of n_mma rows; pair i takes slice row_slice0 + i % passes
  int row_slice0, M;
  int d, V, num_tiles, stages;
  uint32_t tmem_cols;
  int* err;
};

struct SmemLayout {
  uint32_t a_off, b_off, xp_off, bar_off, total;
};

// The transposition buffers hold the per-quarter statistics ([4][n_mma] tuples) at the end.
__host__ __device__ inline SmemLayout lm_layout(int stages, int n_mma) {
  SmemLayout L;
  L.a_off = 0;
  L.b_off = (uint32_t)stages * A_BYTES;
  L.xp_off = L.b_off + (uint32_t)stages * (n_mma / 2) * 128;
  L.bar_off = L.xp_off + (uint32_t)EPI_WARPS * XP_BYTES;
  L.total = L.bar_off + (uint32_t)(2 * stages + 5) * 8 + 16;
  return L;
}
static_assert(4 * MAX_ROWS * 24 <= EPI_WARPS * XP_BYTES, "the quarters' tuples fit the buffers");

enum : int { MODE_GREEDY = 0, MODE_KEYED = 1, MODE_LOGITS = 2 };

template <int MODE>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    lmhead_kernel(const __grid_constant__ CUtensorMap tmap_w,
                  const __grid_constant__ CUtensorMap tmap_h, const LmParams p) {
  constexpr bool KEYED = MODE == MODE_KEYED;
  constexpr bool LOGITS = MODE == MODE_LOGITS;
  extern __shared__ uint8_t smem_raw[];
  // TMA with 128B swizzle and the UMMA descriptors need 1024-byte alignment.
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const SmemLayout L = lm_layout(p.stages, p.n_mma);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.bar_off);
  uint64_t* empty = full + p.stages;
  uint64_t* tfull = empty + p.stages;    // [2]
  uint64_t* tempty = tfull + 2;          // [2]
  uint64_t* mma_done = tempty + 2;       // [1]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_ctarank();      // 0: the pair's leader
  const int pair = (int)blockIdx.x >> 1;
  const int row0 = (p.row_slice0 + pair % p.passes) * p.n_mma;   // this pair's hidden rows
  const int n_rows = min(p.n_mma, p.M - row0);
  const int tile0 = pair / p.passes, tile_step = ((int)gridDim.x >> 1) / p.passes;
  const int kblocks = p.d / BK;
  const uint32_t b_bytes = (uint32_t)(p.n_mma / 2) * 128u;       // hidden rows held by each CTA

  if (tid == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 2);               // (leader) its W and its hidden-row producer
      mbar_init(&empty[s], 1);
    }
    mbar_init(&tfull[0], 1);
    mbar_init(&tfull[1], 1);
    mbar_init(&tempty[0], 2 * EPI_WARPS);   // (leader) the epilogue warps of both CTAs
    mbar_init(&tempty[1], 2 * EPI_WARPS);
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_h);
  }
  if (warp == 1) tmem_alloc_pair(tmem_holder, p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  cluster_arrive();                         // both CTAs' barriers are initialised
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  // The hidden rows may come from the previous kernel; the W producer
  // (warp 0) reads nothing that does and starts streaming at once.
  if (warp != 0) griddep_wait();
  const uint32_t idesc = idesc_bf16_f32(BMP, p.n_mma);

  if (warp == 0 || warp == H_WARP) {
    // ------------------------------------------------------------ producers
    // A warp's bulk copies are processed one after another, so the W boxes
    // (warp 0) and the hidden-row boxes (warp H_WARP) come from two warps of
    // each CTA.  Each CTA loads its own half of both operands; all bytes of a
    // stage are counted on the leader's barrier, which the leader's two
    // producers arm for both CTAs.  The first ring's worth of W stages streams
    // before the wait for the previous kernel (W does not depend on it).
    if (lane == 0) {
      const bool is_w = warp == 0;
      const uint64_t pol = is_w ? l2_policy_evict_first() : l2_policy_evict_last();
      const void* map = is_w ? (const void*)&tmap_w : (const void*)&tmap_h;
      const uint32_t bytes = is_w ? (uint32_t)A_BYTES : b_bytes;
      const uint32_t buf = smem_u32(smem + (is_w ? L.a_off : L.b_off));
      const int y0 = is_w ? rank * BM : row0 + rank * (p.n_mma / 2);
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued_mask = 0, issued_parity = 0;   // last load per stage (stages <= 16)
      bool ok = true;
      int li = 0;                        // loads so far, in (tile, k-block) order
      for (int tile = tile0; tile < p.num_tiles && ok; tile += tile_step) {
        const int y = is_w ? y0 + tile * BMP : y0;
        for (int kb = 0; kb < kblocks; ++kb, ++li) {
          if (li >= p.stages && (!mbar_wait(&empty[stage], phase ^ 1u, WAIT_NS) || *abort_flag)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * bytes);
          tma_load_2d_pair(buf + (uint32_t)stage * bytes, map, dsmem_map(smem_u32(&full[stage]), 0),
                           kb * BK, y, pol);
          issued_mask |= 1u << stage;
          issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
          if (++stage == p.stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) {
        set_err(p.err, ERR_TIMEOUT);
        *abort_flag = 1;
        // let every issued copy land before shared memory is released (the
        // peer's are counted on the leader's barriers; both CTAs stay until
        // the leader is through)
        if (rank == 0)
          for (int s = 0; s < p.stages; ++s)
            if (issued_mask & (1u << s)) mbar_wait(&full[s], (issued_parity >> s) & 1u, WAIT_NS);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader)
    // (the whole warp walks along; one elected thread acts)
    if (rank == 0) {
      const uint32_t on = elect_one();
      const uint64_t a_desc = smem_desc_sw128(smem_u32(smem + L.a_off));
      const uint64_t b_desc = smem_desc_sw128(smem_u32(smem + L.b_off));
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int it = 0;
      for (int tile = tile0; tile < p.num_tiles && ok; tile += tile_step, ++it) {
        const int acc = it & 1;
        const uint32_t aph = (uint32_t)(it >> 1) & 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(&tempty[acc], aph ^ 1u, WAIT_NS)) && !*abort_flag;
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * p.n_mma);
        for (int kb = 0; kb < kblocks; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(&full[stage], phase, WAIT_NS));
          if (!ok) break;
          tc_fence_after();
          umma_bf16_pair_k64_on(on, d_tmem, a_desc + (uint64_t)(stage * (A_BYTES >> 4)),
                                b_desc + (uint64_t)((uint32_t)stage * (b_bytes >> 4)), idesc, kb != 0 ? 1u : 0u);
          umma_commit_pair_on(on, &empty[stage], 3);
          if (++stage == p.stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        umma_commit_pair_on(on, &tfull[acc], 3);
      }
      if (!ok && on) {
        set_err(p.err, ERR_TIMEOUT);
        *abort_flag = 1;
      }
      // (both CTAs wait for it below)
      umma_commit_pair_on(on, mma_done, 3);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // A warp reads 32 columns (hidden rows) of its 32 TMEM lanes (vocabulary
    // ids) at a time, transposes the block through its own shared buffer, and
    // then every lane folds the 32 logits of one column into statistics that
    // stay in its registers over all tiles: no shuffles and no barriers.
    const int q = warp & 3;               // TMEM lane quarter this warp may access
    const int ew = warp - 2;              // epilogue warp index
    const int half = ew >> 2;             // which alternate 32-column chunks it takes
    const int etid = tid - 64;
    const int nchunks = (n_rows + 31) / 32;
    const uint32_t tempty_leader = dsmem_map(smem_u32(tempty), 0);
    float* xp = reinterpret_cast<float*>(smem + L.xp_off + (uint32_t)ew * XP_BYTES);
    uint32_t seed_lo = 0, seed_hi = 0;
    if (KEYED) {
      const unsigned long long sd = *p.seed;
      seed_lo = (uint32_t)sd;
      seed_hi = (uint32_t)(sd >> 32);
    }
    RowStat run[MAX_CHUNKS];
    int draft[MAX_CHUNKS];
#pragma unroll
    for (int c = 0; c < MAX_CHUNKS; ++c) {
      run[c] = RowStat{-INFINITY, 0x7fffffff, -INFINITY, 0.f, 0.f, -INFINITY};
      const int col = (half + 2 * c) * 32 + lane;
      draft[c] = col < n_rows ? p.draft_for_row[row0 + col] : -2;
    }
    // x: the lane's 32 columns (of one id) -> the 32 ids of one column; ids past the vocabulary -inf
    auto transpose = [&](float (&x)[32], bool valid) {
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 32; ++c) xp[xp_off(c, lane)] = valid ? x[c] : -INFINITY;
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(xp + xp_off(lane, j));
        x[j] = v.x;
        x[j + 1] = v.y;
        x[j + 2] = v.z;
        x[j + 3] = v.w;
      }
    };
    int it = 0;
    for (int tile = tile0; tile < p.num_tiles; tile += tile_step, ++it) {
      const int acc = it & 1;
      const uint32_t aph = (uint32_t)(it >> 1) & 1u;
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull[acc], aph, WAIT_NS))) {
        if (lane == 0) {
          set_err(p.err, ERR_TIMEOUT);
          *abort_flag = 1;
        }
        break;
      }
      tc_fence_after();
      const int v0 = tile * BMP + rank * BM + q * 32;
      const bool valid = v0 + lane < p.V;
      const uint32_t tbase = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * p.n_mma);
#pragma unroll
      for (int c = 0; c < MAX_CHUNKS; ++c) {
        const int ch = half + 2 * c;
        if (ch >= nchunks) break;          // warp-uniform
        float x[32];
        tmem_ld32(tbase + (uint32_t)(ch * 32), x);
        if (LOGITS) {
          // x / T, written row by row: the warp's 32 lanes hold 32 consecutive
          // vocabulary ids of one row, so each store is one 128-byte line
          float* dst = p.logits + (size_t)(row0 + ch * 32) * p.V + v0 + lane;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            x[j] *= p.inv_temp;
            if (valid && ch * 32 + j < n_rows) *dst = x[j];
            dst += p.V;
          }
        }
        transpose(x, valid);
        row_fold<KEYED>(run[c], x, v0);
        const int at = draft[c] - v0;      // the drafted id's logit, if it is one of these
        if ((unsigned)at < 32u && draft[c] < p.V)
          p.stats[(size_t)(row0 + ch * 32 + lane) * 5 + 4] = xp[xp_off(lane, at)];
        if (KEYED) {
          // 16 columns at a time, not unrolled: eight generators' code for each of four chunks was
          // fetched more slowly than it ran (us, d 64, V 128: 8 rows 11.3 -> 8.6, 200 rows 35.2 -> 19.5; d 1024,
          // V 32003: 256 rows 53.6 -> 40.0); columns past the last 16 with a row draw nothing
          __syncwarp();
#pragma unroll 1
          for (int j0 = 0; j0 < 32 && ch * 32 + j0 < n_rows; j0 += 16) {
            float k16[16];
            tq_ld16(tbase + (uint32_t)(ch * 32 + j0), k16);
            tq_wait_ld16(k16);
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
              const uint4 u = philox4x32_10(
                  make_uint4((uint32_t)(v0 + lane), (uint32_t)((row0 + ch * 32 + j0 + j) >> 2), 0u, 0u), seed_lo, seed_hi);
              k16[j + 0] = fmaf(k16[j + 0], p.inv_temp, gumbel_of(u.x));
              k16[j + 1] = fmaf(k16[j + 1], p.inv_temp, gumbel_of(u.y));
              k16[j + 2] = fmaf(k16[j + 2], p.inv_temp, gumbel_of(u.z));
              k16[j + 3] = fmaf(k16[j + 3], p.inv_temp, gumbel_of(u.w));
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) xp[xp_off(j0 + j, lane)] = valid ? k16[j] : -INFINITY;
          }
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const float4 v = *reinterpret_cast<const float4*>(xp + xp_off(lane, j));
            x[j] = v.x;
            x[j + 1] = v.y;
            x[j + 2] = v.z;
            x[j + 3] = v.w;
          }
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const bool up = x[j] > run[c].k;
            run[c].i = up ? v0 + j : run[c].i;
            run[c].k = up ? x[j] : run[c].k;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      // (TMEM reads only, which the tcgen05 fences order: a release to the cluster waits for every
      // store under way; 1024 x 32003, 256 rows: 24.3 -> 23.7 us, 5120 x 151936 264 -> 263)
      if (lane == 0) mbar_arrive_cluster_relaxed(tempty_leader + (uint32_t)acc * 8u);
    }
    griddep_launch_dependents();
    // the four quarters' statistics of every column merge through the buffers
    named_bar_sync(1, EPI_THREADS);        // every warp is through with its own
    float4* s_wt = reinterpret_cast<float4*>(smem + L.xp_off);       // [4][n_mma]
    int* s_wti = reinterpret_cast<int*>(s_wt + 4 * p.n_mma);         // [4][n_mma]
    float* s_wk = reinterpret_cast<float*>(s_wti + 4 * p.n_mma);     // [4][n_mma]
#pragma unroll
    for (int c = 0; c < MAX_CHUNKS; ++c) {
      const int col = (half + 2 * c) * 32 + lane;
      if (col < n_rows) {
        s_wt[q * p.n_mma + col] = make_float4(run[c].m, run[c].sec, run[c].s, run[c].t);
        s_wti[q * p.n_mma + col] = run[c].i;
        if (KEYED) s_wk[q * p.n_mma + col] = run[c].k;
      }
    }
    named_bar_sync(1, EPI_THREADS);
    for (int col = etid; col < n_rows; col += EPI_THREADS) {
      Stat a = stat_identity();
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const float4 v = s_wt[w * p.n_mma + col];
        a = stat_merge<KEYED>(a, Stat{v.x, s_wti[w * p.n_mma + col], v.y, v.z, v.w,
                                      KEYED ? s_wk[w * p.n_mma + col] : 0.f});
      }
      // row by row, so that the merge kernel reads a row's partials side by side
      const size_t at = (size_t)(row0 - p.row_slice0 * p.n_mma + col) * p.parts +
                        (size_t)(2 * (pair / p.passes) + rank);
      p.part[at] = make_float4(a.m, a.sec, a.s, a.t);
      p.part_idx[at] = a.i;
      if (KEYED) p.part_k[at] = a.k;
    }
  }

  tc_fence_before();
  __syncthreads();
  // Neither CTA leaves (or frees its TMEM) while the other may still signal its barriers or the
  // pair's MMAs may write its TMEM: the last signal of the leader's MMAs has arrived in both, and
  // the barrier says so to each.
  if (warp == 1) mbar_wait(mma_done, 0, WAIT_NS);
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc_pair(tmem_base, p.tmem_cols);
  }
}

// Merge the per-CTA partial statistics of every row (one warp per row).
// argmax receives the sampled id when KEYED.
template <bool KEYED>
__global__ void __launch_bounds__(128) lmhead_reduce_kernel(const float4* part, const int* part_idx,
                                                            const float* part_k, int parts,
                                                            int row0, int n_rows, int V,
                                                            const int32_t* draft_for_row,
                                                            int32_t* argmax, float* stats, int* err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 4 + warp;
  griddep_wait();
  griddep_launch_dependents();
  if (row >= n_rows) return;
  Stat a = stat_identity();
  for (int c = lane; c < parts; c += 32) {
    const size_t at = (size_t)row * parts + c;
    const float4 v = part[at];
    a = stat_merge<KEYED>(a, Stat{v.x, part_idx[at], v.y, v.z, v.w, KEYED ? part_k[at] : 0.f});
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) a = stat_merge<KEYED>(a, stat_shfl_xor<KEYED>(a, off));
  if (lane == 0) {
    const int m = row0 + row;
    float* st = stats + (size_t)m * 5;
    if (a.m == INFINITY && a.sec < INFINITY && a.s == INFINITY) {   // one logit is infinite: all the weight
      a.s = 1.f;
      a.t = 0.f;
    }
    const float ls = logf(a.s);
    argmax[m] = a.i < V ? a.i : 0;         // no logit above -inf: the lowest id
    st[0] = a.m;
    st[1] = a.sec;
    st[2] = a.m + ls;
    st[3] = ls - a.t / a.s;
    const int dft = draft_for_row[m];
    if (dft == -1) {
      st[4] = __int_as_float(0x7fc00000);
    } else if (dft < -1 || dft >= V) {
      st[4] = __int_as_float(0x7fc00000);
      set_err(err, ERR_TOKEN);
    }
  }
}

// 2-D bf16 row-major [rows, cols] map with a {64, box_rows} box and 128B swizzle.
bool make_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  const uint64_t dims[2] = {cols, rows};
  const uint64_t strides[1] = {cols * 2};
  const uint32_t box[2] = {(uint32_t)BK, box_rows};
  return encode_tensor_map_bf16(map, base, 2, dims, strides, box);
}

}  // namespace

// Limits already set on each variant of the kernel.
template <int MODE>
KernelLimits& lm_limits() {
  static KernelLimits lim;
  return lim;
}

// CTA pairs of the kernel (one CTA per SM) resident at once on the current device.
int resident_pairs(int num_sms) {
  static std::atomic<int> cache[KL_MAX_DEV];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= KL_MAX_DEV) return num_sms / 2;
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    auto kern = lmhead_kernel<MODE_GREEDY>;
    if (ensure_kernel_limits((const void*)kern, lm_limits<MODE_GREEDY>(), 227 * 1024, false) != cudaSuccess) {
      cudaGetLastError();
      return num_sms / 2;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (num_sms / 2));
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = 227 * 1024;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return num_sms / 2;
    }
    cache[dev].store(n, std::memory_order_relaxed);
  }
  return n < num_sms / 2 ? n : num_sms / 2;
}

LmheadPlan plan_lmhead(int M, int d, int V, int num_sms) {
  LmheadPlan pl{};
  // Rows beyond 256 are cut into slices of equal size (384 rows as 2 x 192:
  // a slice of 256 rows is tensor-bound while a short one is bound by
  // streaming W).  Slice i covers rows [i * n_mma, min(M, (i + 1) * n_mma)).
  // Up to four slices share a launch: pair i takes slice i mod passes, and the
  // pairs of one vocabulary tile run side by side, so W comes from HBM once and
  // from L2 for the other slices.
  const int slices = (M + MAX_ROWS - 1) / MAX_ROWS;
  const int rows = (M + slices - 1) / slices;
  pl.n_mma = (rows + 31) / 32 * 32;      // a pair MMA takes N in steps of 32
  pl.slices = (M + pl.n_mma - 1) / pl.n_mma;
  pl.launches = (pl.slices + 3) / 4;
  pl.passes = (pl.slices + pl.launches - 1) / pl.launches;
  pl.launches = (pl.slices + pl.passes - 1) / pl.passes;
  pl.num_tiles = (V + BMP - 1) / BMP;
  pl.pairs = num_sms / 2 > 0 ? num_sms / 2 : 1;
  const uint32_t budget = 227u * 1024u - 1024u;
  const uint32_t per_stage = A_BYTES + (uint32_t)(pl.n_mma / 2) * 128u;
  int st = (int)((budget - lm_layout(0, pl.n_mma).total) / per_stage);
  if (st > 12) st = 12;
  while (st > 2 && lm_layout(st, pl.n_mma).total > budget) --st;
  pl.stages = st;
  pl.smem_bytes = lm_layout(st, pl.n_mma).total + 1024;
  const size_t per_part = LM_WS_ENTRIES;
  pl.ws_bytes = per_part * (sizeof(float4) + sizeof(int) + sizeof(float));
  return pl;
}

namespace {

template <int MODE>
cudaError_t launch_pass(const CUtensorMap& map_w, const CUtensorMap& map_h, LmParams p, const LmheadPlan& pl,
                        const int32_t* draft_for_row, int32_t* argmax, float* stats, cudaStream_t stream) {
  constexpr bool KEYED = MODE == MODE_KEYED;
  const cudaError_t le = ensure_kernel_limits((const void*)lmhead_kernel<MODE>, lm_limits<MODE>(), 227 * 1024, false);
  if (le != cudaSuccess) return le;
  p.tmem_cols = 32;
  while (p.tmem_cols < (uint32_t)(2 * pl.n_mma)) p.tmem_cols <<= 1;
  p.n_mma = pl.n_mma;
  p.num_tiles = pl.num_tiles;
  p.stages = pl.stages;
  const int pairs = resident_pairs(2 * pl.pairs);
  // Each launch overwrites every partial its merge kernel reads.
  for (int l = 0; l < pl.launches; ++l) {
    p.row_slice0 = l * pl.passes;
    p.passes = pl.slices - p.row_slice0 < pl.passes ? pl.slices - p.row_slice0 : pl.passes;
    int groups = pairs / p.passes;
    if (groups < 1) groups = 1;
    if (groups > pl.num_tiles) groups = pl.num_tiles;
    p.parts = 2 * groups;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * groups * p.passes);
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = pl.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, lmhead_kernel<MODE>, map_w, map_h, p);
    if (e != cudaSuccess) return e;
    const int row0 = p.row_slice0 * pl.n_mma;
    const int n_rows = p.M - row0 < p.passes * pl.n_mma ? p.M - row0 : p.passes * pl.n_mma;
    e = launch_pdl(lmhead_reduce_kernel<KEYED>, dim3((n_rows + 3) / 4), dim3(128), 0, stream,
                   (const float4*)p.part, (const int*)p.part_idx, (const float*)p.part_k, p.parts,
                   row0, n_rows, p.V, draft_for_row, argmax, stats, p.err);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_lmhead(int M, int d, int V, const __nv_bfloat16* hidden,
                          const __nv_bfloat16* w, const int32_t* draft_for_row, int32_t* argmax,
                          float* stats, void* ws, size_t ws_entries, const LmheadPlan& pl, int* err,
                          cudaStream_t stream, const unsigned long long* seed, float inv_temp,
                          float* logits) {
  CUtensorMap map_w, map_h;
  if (!make_map(&map_w, w, (uint64_t)V, (uint64_t)d, BM)) return cudaErrorInvalidValue;
  if (!make_map(&map_h, hidden, (uint64_t)M, (uint64_t)d, (uint32_t)(pl.n_mma / 2)))
    return cudaErrorInvalidValue;
  LmParams p{};
  p.draft_for_row = draft_for_row;
  p.stats = stats;
  p.part = static_cast<float4*>(ws);
  p.part_idx = reinterpret_cast<int*>(p.part + ws_entries);
  p.part_k = reinterpret_cast<float*>(p.part_idx + ws_entries);   // KEYED only
  p.seed = seed;
  p.inv_temp = inv_temp;
  p.logits = logits;
  p.M = M;
  p.d = d;
  p.V = V;
  p.err = err;
  if (seed) return launch_pass<MODE_KEYED>(map_w, map_h, p, pl, draft_for_row, argmax, stats, stream);
  if (logits) return launch_pass<MODE_LOGITS>(map_w, map_h, p, pl, draft_for_row, argmax, stats, stream);
  return launch_pass<MODE_GREEDY>(map_w, map_h, p, pl, draft_for_row, argmax, stats, stream);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the LM-head call.
//
// Some callers cannot give this library device memory: a serving engine that
// reserves almost all of HBM for its KV cache up front and forbids any other
// allocation during decoding, or a plug-in running inside a host framework
// that owns the device's memory and exposes no workspace.  For them the
// per-CTA partial statistics live in one fixed scratch array compiled into
// the library (resident on every GPU that loads it, until the process exits)
// instead of a caller-provided workspace.
//
// The array below is a device symbol: in host code its name is only a
// stand-in, never a device address.  Its address is looked up with
// cudaGetSymbolAddress once per device, on that device's first call.
namespace {

constexpr int NOALLOC_MAX_CTAS = 256;                 // persistent CTAs (one per SM)
constexpr int NOALLOC_MAX_M = 512;                    // rows per call (two 256-row passes)
constexpr size_t NOALLOC_ENTRIES = (size_t)NOALLOC_MAX_CTAS * MAX_ROWS;
// [NOALLOC_ENTRIES] float4 (m, second, s, t) then [NOALLOC_ENTRIES] int (argmax)
static __device__ __align__(256) unsigned char g_lmhead_scratch[NOALLOC_ENTRIES * (sizeof(float4) + sizeof(int))];

std::atomic<void*> g_scratch_addr[64];   // per device; a race only repeats the lookup

// The scratch's device address on the current device, looked up on the
// device's first call; the CUDA error of a failed lookup otherwise.
cudaError_t scratch_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  void* addr = g_scratch_addr[dev].load(std::memory_order_acquire);
  if (!addr) {
    e = cudaGetSymbolAddress(&addr, g_lmhead_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_addr[dev].store(addr, std::memory_order_release);
  }
  *out = addr;
  return cudaSuccess;
}

}  // namespace

}  // namespace cospec

extern "C" COSPEC_API int cospec_lmhead_argmax_features_noalloc(
    int M, int d, int V, const uint16_t* hidden, const uint16_t* w, const int32_t* draft_for_row,
    int32_t* argmax, float* stats, void* stream) {
  using namespace cospec;
  if (M < 0 || d <= 0 || V <= 0) return COSPEC_ERR_INVALID_ARG;
  if (M == 0) return COSPEC_OK;
  if (!hidden || !w || !draft_for_row || !argmax || !stats) return COSPEC_ERR_INVALID_ARG;
  if (d % 64 != 0 || (long long)V > 0x7fffff00LL) return COSPEC_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(hidden) & 15u) || (reinterpret_cast<uintptr_t>(w) & 15u))
    return COSPEC_ERR_INVALID_ARG;
  if (M > NOALLOC_MAX_M) return COSPEC_ERR_UNSUPPORTED;          // beyond the fixed scratch
  const int sms = device_num_sms();
  if (sms <= 0) return cuda_lookup_failed();
  const LmheadPlan pl = plan_lmhead(M, d, V, sms);
  if (2 * pl.pairs > NOALLOC_MAX_CTAS) return COSPEC_ERR_UNSUPPORTED;  // beyond the fixed scratch
  void* scratch = nullptr;
  const cudaError_t se = scratch_address(&scratch);
  if (se != cudaSuccess) return cuda_status(se);
  int* err = device_error_word();
  if (!err) return cuda_lookup_failed();
  return cuda_status(launch_lmhead(M, d, V, reinterpret_cast<const __nv_bfloat16*>(hidden),
                                   reinterpret_cast<const __nv_bfloat16*>(w), draft_for_row, argmax, stats,
                                   scratch, NOALLOC_ENTRIES, pl, err, static_cast<cudaStream_t>(stream)));
}
