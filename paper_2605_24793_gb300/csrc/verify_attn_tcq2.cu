// Verify attention on the tcgen05 tensor cores for more than 128 query rows of
// a KV head (teacher-forced verification pass, Sec. 3.1 Eq. 2 of the paper; the
// arbitrator's regions and causal prefill, Sec. 3.3): one CTA takes up to 256
// query rows as two MMA row tiles (A and B, 128 rows each) that share every
// K/V tile, so the head's cache passes through the SM once, and whose softmax and
// tensor work alternate: while tile A's scores are exponentiated the tensor core
// does B's P.V and next scores, and the other way round.
//
// One CTA owns (sequence b, KV head, row group); the KV range is not split (the planner takes
// the one-tile kernel where a split pays).  The softmax advances in steps of 64 keys.
// Roles by warp:
//   warps 0-2   TMA producers of 128-key K and V tiles (one 2-D box per page and
//               128-byte half, the boxes of a tile split over the warps) into a
//               ring of five slots, K and V in turn; the block's own K/V last;
//   warp 3, 12  MMA issuers of row tile A and B (one elected thread each):
//                 S_g  = Q_g K^T  (M = 128, N = 64 keys, K = D) into one of two
//                                 score buffers of the tile,
//                 O_g += P_g V    (M = 128, N = D, K = 64 keys), P_g read from TMEM
//               in the order P.V(u), S(u + 2): while the softmax works on one of its
//               buffers the tensor core empties and refills the other;
//   warps 4-7   softmax of tile A, warps 8-11 of tile B (one warp per TMEM lane
//               quarter): a thread owns a query row and the 64 scores of a step, and
//               writes P as bf16 over them.
// The maximum is lazy as in the one-tile kernel: m_ref moves (and O and l are
// rescaled) only when a score exceeds it by more than 2^8 in the exp2 domain.
//
// Bound: the tensor pipe's operands.  An MMA of 64 score columns reads 6 KB of shared
// memory and takes about as long as one of 128 (whose 8 KB fill its 64 cycles), so a
// 256 x 128 tile needs about 3100 cycles of MMAs beside the 64 KB that TMA writes: 3900
// measured.  Score tiles of 128 columns leave no room for a second buffer in TMEM and
// make one chain of scores, softmax and P.V (4300-4500 measured, in step or staggered);
// one row tile per CTA is held to about 1900 cycles per 128 rows by the K/V boxes (2 KB
// each, about 58 cycles apart in an SM however many warps issue them).
// Measured (GB300): 212 rows, batch 16 at 512 keys, 22.9 us per layer with one row tile per
// CTA, 16.2 with two, 20.4 with CTA pairs (which take head dimension 128 at more keys or
// units); at 128 keys 10.3 against 16.4 with pairs.
#include <cuda.h>
#include <math.h>

#include "cospec_device.cuh"
#include "cospec_internal.h"

namespace cospec {

namespace {

constexpr int T2_KT = 128;         // keys per cache tile (8 pages) = MMA N of S
constexpr int T2_PPT = T2_KT / 16;
constexpr int T2_PAGE = 16;
constexpr int T2_ROWB = 128;       // bytes of one swizzled smem row
constexpr int T2_M = 128;          // query rows per row tile
constexpr int T2_PROD = 3;
constexpr int T2_MMA_WARP = 3;     // MMA issuer of row tile A
constexpr int T2_SOFT0 = 4;        // softmax warps: tile A 4-7, tile B 8-11
constexpr int T2_MMA_WARP_B = 12;  // MMA issuer of row tile B
constexpr int T2_THREADS = 416;
constexpr int T2_KS = 64;          // keys per softmax step
constexpr int T2_SLOTS = 5;
constexpr float T2_LAZY = 8.f;
constexpr uint64_t T2_WAIT_NS = 2000000000ull;

struct Tcq2Params {
  const int32_t* page_table;
  const int32_t* ctx_len;
  const __nv_bfloat16* q;   // only for the L2 warm-up of the query rows
  __nv_bfloat16* out;
  int B, R, Hq, Hkv, G;
  int JB;           // block rows (j) of a row tile
  int JBQ;          // block rows of the query box: min(R, JB)
  int RG, JG;       // row groups, block rows per group (at most 2 JB)
  int max_pages, num_pages;
  float scale_log2;
  int kv_stable;
  int block_full;
  int* err;
};

template <int D>
struct Tcq2Layout {
  static constexpr int H = D / 64;
  static constexpr int KVB = H * T2_KT * T2_ROWB;       // one slot: [half][128 keys][128 B]
  static constexpr int QH = T2_M * T2_ROWB;             // one half of a row tile's queries
  static constexpr int QOFF = T2_SLOTS * KVB;
  static constexpr int DATA = QOFF + 2 * H * QH;        // ring and query rows
  // barriers: full[5], empty[5], q_full, s_full[2][2], p_full[2][2], pv_done[2], mma_done[2]
  static constexpr int NBAR = 2 * T2_SLOTS + 13;
  static constexpr int HOLDER = DATA + NBAR * 8;
  static constexpr int FLAGS = HOLDER + 8;              // abort, items issued [3], sequence slot
  static constexpr int TOTAL = FLAGS + 24;
  static constexpr uint32_t OCOL = 2 * T2_KT;           // TMEM: S_A[2], S_B[2], O_A, O_B
  static constexpr uint32_t TCOLS = 512u;
};

template <int D>
__global__ void __launch_bounds__(T2_THREADS, 1)
    verify_attn_tcq2_kernel(const __grid_constant__ CUtensorMap map_kp,
                            const __grid_constant__ CUtensorMap map_vp,
                            const __grid_constant__ CUtensorMap map_kb,
                            const __grid_constant__ CUtensorMap map_vb,
                            const __grid_constant__ CUtensorMap map_q, const Tcq2Params p) {
  using LY = Tcq2Layout<D>;
  constexpr int H = LY::H;

  extern __shared__ __align__(16) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + LY::DATA);
  uint64_t* empty = full + T2_SLOTS;
  uint64_t* q_full = empty + T2_SLOTS;
  uint64_t* s_full = q_full + 1;       // [2 tiles][2 buffers]
  uint64_t* p_full = s_full + 4;       // [2][2]
  uint64_t* pv_done = p_full + 4;      // [2]
  uint64_t* mma_done = pv_done + 2;    // [2]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + LY::HOLDER);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + LY::FLAGS);
  volatile int* n_issued = abort_flag + 1;     // [3]: items each producer warp issued (abort tail)
  volatile int* seq_slot = abort_flag + 4;
  uint8_t* qs = smem + LY::QOFF;

  const int kvh = blockIdx.y / p.RG, rg = blockIdx.y % p.RG;
  const int j0 = rg * p.JG;                          // first block row of this group
  const int nj = min(p.JG, p.R - j0);
  const int NT = nj > p.JB ? 2 : 1;                  // row tiles in use
  const int rows_t = p.JB * p.G;                     // query rows of a full tile
  const int NR = nj * p.G;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < T2_SLOTS; ++s) {
      mbar_init(&full[s], T2_PROD);
      mbar_init(&empty[s], (uint32_t)NT);      // both tiles' issuers
    }
    mbar_init(q_full, 1);
    for (int g = 0; g < 2; ++g) {
      const int rows = g < NT ? min(rows_t, NR - g * rows_t) : 32;
      for (int i = 0; i < 2; ++i) {
        mbar_init(&s_full[2 * g + i], 1);
        mbar_init(&p_full[2 * g + i], (uint32_t)((rows + 31) >> 5));   // the tile's warps that own rows
      }
      mbar_init(&pv_done[g], 1);
      mbar_init(&mma_done[g], 1);
    }
    abort_flag[0] = 0;
    n_issued[0] = n_issued[1] = n_issued[2] = 0;
    fence_barrier_init();
  }
  if (warp == T2_MMA_WARP) {
    tmem_alloc(tmem_holder, LY::TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  // (in this order: a dependent under the stable-cache promise reads the cache at once)
  if (!p.kv_stable) griddep_wait();
  griddep_launch_dependents();

  const int b = p.B > RANK_MAX_B ? sequence_in_order(p.ctx_len, p.B, (int)blockIdx.z)
                : p.B > 1        ? sequence_by_rank(p.ctx_len, p.B, (int)blockIdx.z, seq_slot)
                                 : (int)blockIdx.z;
  const int C = p.ctx_len[b];
  const bool bad = (C < 0) || (C > p.max_pages * T2_PAGE);
  if (bad && kvh == 0 && rg == 0 && tid == 0) set_err(p.err, ERR_CTX);
  const int n = bad ? 0 : (C + T2_KT - 1) / T2_KT;   // cache tiles
  const bool do_blk = !bad;                          // then the block's keys
  const int T = n + (do_blk ? 1 : 0);
  const int U = 2 * n + (do_blk ? 1 : 0);            // softmax steps
  const int npages = (C + T2_PAGE - 1) / T2_PAGE;
  const int KBR = (p.R + 15) & ~15;                  // block keys padded to 16
  float mref = -INFINITY, l = 0.f;                   // softmax threads: this row's m_ref and sum

  if (warp < T2_PROD) {
    // ------------------------------------------------------------ producers
    // Items in order K(0), V(0), K(1), V(1), ...; item i goes to slot i % 5.  A
    // warp's bulk copies are processed one after another, so the three warps
    // split the boxes (page x half) of every item.
    constexpr int NKB = H * T2_PPT;
    const int kb0 = warp * NKB / T2_PROD, nkb = (warp + 1) * NKB / T2_PROD - kb0;
    const int e = kb0 + lane;
    if (warp == 0 && lane == 0) {
      tma_prefetch_desc(&map_kp);
      tma_prefetch_desc(&map_vp);
      tma_prefetch_desc(&map_q);
    }
    const uint64_t pol = p.RG > 1 ? l2_policy_evict_normal() : l2_policy_evict_first();
    const int* ptab = p.page_table + (size_t)b * p.max_pages;
    int pid = 0;
    bool ok = true;
    int issued = 0;
    auto issue_cache = [&](int i) {
      const int t = i >> 1, tensor = i & 1, st = i % T2_SLOTS;
      if ((i & 7) == 0) {                // 32 page ids = the next 4 tiles, one per lane
        const int e2 = t * T2_PPT + lane;
        pid = (e2 < npages) ? __ldg(ptab + e2) : 0;
      }
      const int np = min(T2_PPT, npages - t * T2_PPT);
      const int pg = e / H;              // box e: page e / H, half e % H
      int pgid = __shfl_sync(0xffffffffu, pid, (t & 3) * T2_PPT + (pg & 7));
      if (lane == 0) {
        const int hi = min(kb0 + nkb, np * H);
        mbar_arrive_expect_tx(&full[st], (uint32_t)(max(0, hi - kb0) * T2_PAGE * T2_ROWB));
      }
      __syncwarp();
      if (lane < nkb && pg < np) {
        if ((unsigned)pgid >= (unsigned)p.num_pages) {
          set_err(p.err, ERR_PAGE);
          pgid = 0;
        }
        const int h = e % H;
        tma_load_3d(smem_u32(smem + st * LY::KVB + h * (T2_KT * T2_ROWB) + pg * (T2_PAGE * T2_ROWB)),
                    tensor ? (const void*)&map_vp : (const void*)&map_kp, &full[st], 0,
                    (pgid * p.Hkv + kvh) * T2_PAGE, h, pol);
      }
      __syncwarp();
    };
    auto wait_slot = [&](int i) -> bool {
      if (i < T2_SLOTS) return true;
      const bool w = mbar_wait(&empty[i % T2_SLOTS], (uint32_t)((i / T2_SLOTS) - 1) & 1u, T2_WAIT_NS);
      return __all_sync(0xffffffffu, w) && !*abort_flag;
    };
    const int pre = min(2 * n, T2_SLOTS);
    for (int i = 0; i < pre; ++i) {      // with the stable-cache promise: before the wait
      issue_cache(i);
      ++issued;
    }
    // the block K/V comes from the previous kernel (warp 0 loads it)
    if (p.kv_stable && warp == 0) griddep_wait();
    for (int i = pre; i < 2 * n && ok; ++i) {
      if (!wait_slot(i)) {
        ok = false;
        break;
      }
      issue_cache(i);
      ++issued;
    }
    for (int i = 2 * n; i < 2 * T && ok; ++i) {
      if (!wait_slot(i)) {
        ok = false;
        break;
      }
      // one box per tensor: KBR rows from block row 0 of this head, all
      // halves, landing as [half][KBR rows][128 B]
      const int st = i % T2_SLOTS;
      if (lane == 0) {
        if (warp == 0) {
          mbar_arrive_expect_tx(&full[st], (uint32_t)(H * KBR * T2_ROWB));
          tma_load_4d(smem_u32(smem + st * LY::KVB), (i & 1) ? (const void*)&map_vb : (const void*)&map_kb,
                      &full[st], 0, b * p.R, 0, kvh, pol);
        } else {
          mbar_arrive(&full[st]);
        }
      }
      __syncwarp();
      ++issued;
    }
    if (lane == 0) {
      n_issued[warp] = issued;
      if (!ok) {
        set_err(p.err, ERR_TIMEOUT);
        *abort_flag = 1;
      }
    }
  } else if (warp == T2_MMA_WARP || warp == T2_MMA_WARP_B) {
    // ------------------------------------------------------------ MMA issuers
    // (the whole warp walks along; one elected thread acts)
    const int g = warp == T2_MMA_WARP ? 0 : 1;
    if (U > 0 && g < NT) {
      const uint32_t on = elect_one();
      if (g == 0) {
        if (p.kv_stable) griddep_wait();   // the query rows come from the previous kernel
        if (on) {
          const uint64_t qpol = l2_policy_evict_first();
          const int qrows = p.G * p.JBQ;   // rows a query box writes
          mbar_arrive_expect_tx(q_full, (uint32_t)(NT * H * qrows * T2_ROWB));
          for (int i = 0; i < NT; ++i)
            for (int h = 0; h < H; ++h)
              tma_load_4d(smem_u32(qs + (i * H + h) * LY::QH), &map_q, q_full, 0, kvh * p.G,
                          b * p.R + j0 + i * p.JB, h, qpol);
        }
        __syncwarp();
      }
      const uint32_t sbase = smem_u32(smem);
      const uint64_t qd = smem_desc_sw128(sbase + LY::QOFF + g * H * LY::QH);
      const uint64_t k_desc = smem_desc_sw128(sbase);
      const uint32_t idesc_pv = idesc_bf16_f32(T2_M, D) | (1u << 16);   // B (V) MN-major
      const uint32_t s_tmem = tmem_base + (uint32_t)(g * T2_KT);
      const uint32_t o_tmem = tmem_base + LY::OCOL + (uint32_t)(g * D);
      auto wait_full = [&](int i) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(&full[i % T2_SLOTS], (uint32_t)(i / T2_SLOTS) & 1u, T2_WAIT_NS)) &&
               !*abort_flag;
      };
      // Step u: keys 64 (u & 1) .. of cache tile u / 2, or the block's (u == 2n).
      // Descriptor addresses count 16-byte units.
      auto issue_s = [&](int u) {
        const bool blk = u == 2 * n;
        const int nk = blk ? KBR : T2_KS;
        const int slot = (u & ~1) % T2_SLOTS;              // item 2 t of the ring
        const uint64_t khalf = (uint64_t)((blk ? KBR : T2_KT) * (T2_ROWB >> 4));
        const uint64_t kd = k_desc + (uint64_t)(slot * (LY::KVB >> 4) + (u & 1) * (T2_KS * T2_ROWB >> 4));
        const uint32_t dst = s_tmem + (uint32_t)((u & 1) * T2_KS);
        const uint32_t idesc_qk = idesc_bf16_f32(T2_M, nk);
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            umma_bf16_on(on, dst, qd + (uint64_t)(h * (LY::QH >> 4) + ks * 2), kd + h * khalf + (uint64_t)(ks * 2),
                         idesc_qk, (h | ks) != 0 ? 1u : 0u);
        umma_commit_on(on, &s_full[2 * g + (u & 1)]);
        if (blk || (u & 1)) umma_commit_on(on, &empty[slot]);
      };
      auto issue_pv = [&](int u) {
        const bool blk = u == 2 * n;
        const int slot = (u | 1) % T2_SLOTS;               // item 2 t + 1
        const uint32_t src = s_tmem + (uint32_t)((u & 1) * T2_KS);
        const uint32_t vb = sbase + (uint32_t)(slot * LY::KVB + (u & 1) * (T2_KS * T2_ROWB));
        // 16 keys = 8 TMEM columns of P and 16 rows of V (2 KB) per MMA
        if (blk) {
          const uint64_t vd = tq_desc_mn_sw128(vb, (uint32_t)(KBR * T2_ROWB));
          for (int ks = 0; ks < KBR / 16; ++ks)
            umma_bf16_tmem_a_on(on, o_tmem, src + (uint32_t)(ks * 8), vd + (uint64_t)(ks * 128), idesc_pv,
                                (u > 0 || ks > 0) ? 1u : 0u);
        } else {
          const uint64_t vd = tq_desc_mn_sw128(vb, (uint32_t)(T2_KT * T2_ROWB));
          const uint32_t acc0 = u > 0 ? 1u : 0u;
#pragma unroll
          for (int ks = 0; ks < T2_KS / 16; ++ks)
            umma_bf16_tmem_a_on(on, o_tmem, src + (uint32_t)(ks * 8), vd + (uint64_t)(ks * 128), idesc_pv,
                                ks > 0 ? 1u : acc0);
        }
        umma_commit_on(on, &pv_done[g]);
        if (blk || (u & 1)) umma_commit_on(on, &empty[slot]);
      };
      // tcgen05 MMAs of one thread run in issue order, so S(u + 2) may be issued over P(u) once its
      // P.V is.
      bool ok = __all_sync(0xffffffffu, mbar_wait(q_full, 0, T2_WAIT_NS));
      for (int u = 0; u < min(2, U) && ok; ++u) {
        if ((u & 1) == 0) ok = wait_full(u);
        if (!ok) break;
        tc_fence_after();
        issue_s(u);
      }
      for (int u = 0; u < U && ok; ++u) {
        ok = __all_sync(0xffffffffu, mbar_wait(&p_full[2 * g + (u & 1)], (uint32_t)(u >> 1) & 1u, T2_WAIT_NS)) &&
             !*abort_flag;
        if (ok && (u & 1) == 0) ok = wait_full(u + 1);
        if (!ok) break;
        tc_fence_after();
        issue_pv(u);
        if (u + 2 < U) {
          if ((u & 1) == 0) ok = wait_full(u + 2);
          if (!ok) break;
          tc_fence_after();
          issue_s(u + 2);
        }
      }
      if (!ok && on) {
        set_err(p.err, ERR_TIMEOUT);
        *abort_flag = 1;
      }
      // every MMA issued by this thread completes before TMEM is released
      umma_commit_on(on, &mma_done[g]);
      mbar_wait(&mma_done[g], 0, T2_WAIT_NS);
    }
  } else {
    // ------------------------------------------------------------ softmax
    const int sw = warp - T2_SOFT0;
    const int g = sw >> 2, q = sw & 3;   // row tile, TMEM lane quarter
    const int r = q * 32 + lane;         // this thread's row of the tile
    if (p.kv_stable) {
      // warm L2 with the group's query rows before the MMA thread's loads
      for (int e = sw * 32 + lane; e < NR * (D * 2 / 128); e += 256) {
        const int rr = e / (D * 2 / 128), part_ = e % (D * 2 / 128);
        const int j = j0 + rr / p.G, gg = rr % p.G;
        prefetch_l2(p.q + (((size_t)b * p.R + j) * p.Hq + (size_t)kvh * p.G + gg) * D + part_ * 64);
      }
    }
    const int rows_g = g < NT ? min(rows_t, NR - g * rows_t) : 0;
    const bool rvalid = r < rows_g;
    const int jr = j0 + g * p.JB + (rvalid ? r / p.G : 0);       // block row of this query row
    // the last block key this row sees: its own row (causal) or the whole block
    const int blim = p.block_full ? p.R - 1 : min(jr, p.R - 1);
    const float sc = p.scale_log2;
    const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t orow = lane_base + LY::OCOL + (uint32_t)(g * D);
    if (q * 32 < rows_g) {
      for (int u = 0; u < U; ++u) {
        const int bi = 2 * g + (u & 1);
        const bool blk = u == 2 * n;
        const int nk = blk ? KBR : T2_KS;        // score columns of this step
        if (!__all_sync(0xffffffffu, mbar_wait(&s_full[bi], (uint32_t)(u >> 1) & 1u, T2_WAIT_NS)) || *abort_flag) {
          if (lane == 0) {
            set_err(p.err, ERR_TIMEOUT);
            *abort_flag = 1;
          }
          break;
        }
        tc_fence_after();
        const uint32_t srow = lane_base + (uint32_t)(g * T2_KT + (u & 1) * T2_KS);
        // keys 0..lim of this step are visible to this row; padding rows give
        // rows of P and O that nothing reads and decide nothing.  A block step
        // has 16 to 64 score columns; the rest holds an older step's.
        const int left = C - u * T2_KS;          // context keys from here on
        const int lim = blk ? blim : min(T2_KS, left) - 1;
        float x0[32], x1[32];
        tq_ld32(srow, x0);
        tq_ld32(srow + 32, x1);
        tq_wait_ld32(x0);
        tq_wait_ld32(x1);
        if (__any_sync(0xffffffffu, rvalid && lim < T2_KS - 1) || blk) {
#pragma unroll
          for (int k = 0; k < 32; ++k) {
            x0[k] = k <= lim ? x0[k] : -INFINITY;
            x1[k] = 32 + k <= lim ? x1[k] : -INFINITY;
          }
        }
        float m4[4] = {x0[0], x0[1], x0[2], x0[3]};
#pragma unroll
        for (int k = 4; k < 32; ++k) m4[k & 3] = fmaxf(m4[k & 3], x0[k]);
#pragma unroll
        for (int k = 0; k < 32; ++k) m4[k & 3] = fmaxf(m4[k & 3], x1[k]);
        const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * sc;
        // move the reference only when a score exceeds it by 2^8 (the first
        // step always sets it: m_ref starts at -inf)
        const bool up = rvalid && mx > mref + T2_LAZY;
        float alpha = 1.f;
        if (up) {
          alpha = (mref == -INFINITY) ? 0.f : exp2_approx(mref - mx);
          mref = mx;
          l *= alpha;
        }
        if (__any_sync(0xffffffffu, up && u > 0)) {
          // O holds steps 0..u-1: wait for the last of them, then scale the row
          const bool okp = __all_sync(0xffffffffu, mbar_wait(&pv_done[g], (uint32_t)(u - 1) & 1u, T2_WAIT_NS));
          tc_fence_after();
          if (okp) {
#pragma unroll 1
            for (int c = 0; c < D / 16; ++c) {
              float o[16];
              tq_ld16(orow + c * 16, o);
              tq_wait_ld();
              uint32_t w[16];
#pragma unroll
              for (int k = 0; k < 16; ++k) w[k] = __float_as_uint(o[k] * alpha);
              tq_st16(orow + c * 16, w);
            }
          } else if (lane == 0) {
            set_err(p.err, ERR_TIMEOUT);
          }
        }
        // P = 2^(score * scale - m_ref) in bf16, two keys per TMEM column, over
        // this buffer's scores (masked keys give exactly 0)
        const float nb = (mref == -INFINITY) ? 0.f : -mref;
        float l4[4] = {0.f, 0.f, 0.f, 0.f};
        auto exp_store = [&](float (&x)[32], int k0) {
          uint32_t pk[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float p0 = exp2_approx(fmaf(x[2 * k], sc, nb));
            const float p1 = exp2_approx(fmaf(x[2 * k + 1], sc, nb));
            l4[k & 3] += p0 + p1;
            pk[k] = pack_bf16(p0, p1);
          }
          tq_st16(srow + k0 / 2, pk);
        };
        exp_store(x0, 0);
        exp_store(x1, 32);
        l += (l4[0] + l4[1]) + (l4[2] + l4[3]);
        // V rows of keys outside the context (or past the block) may hold
        // stale bytes: each tile's warps zero them before their own P.V reads
        // them, so that their zero weights contribute 0.
        const int vr = blk ? p.R : min(T2_KS, max(0, left));
        if (vr < nk) {
          const int i = u | 1, st = i % T2_SLOTS;
          if (__all_sync(0xffffffffu, mbar_wait(&full[st], (uint32_t)(i / T2_SLOTS) & 1u, T2_WAIT_NS))) {
            uint8_t* vb = smem + st * LY::KVB + (u & 1) * (T2_KS * T2_ROWB);
            const int vhalf = (blk ? KBR : T2_KT) * T2_ROWB, nthr = ((rows_g + 31) & ~31);
            for (int e = r; e < (nk - vr) * H * 8; e += nthr) {
              const int row = vr + e / (H * 8), rem = e % (H * 8);
              *reinterpret_cast<uint4*>(vb + (rem / 8) * vhalf + row * T2_ROWB + (rem % 8) * 16) =
                  make_uint4(0u, 0u, 0u, 0u);
            }
            fence_proxy_async_smem();
          }
        }
        tq_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[bi]);
      }
      if (U > 0 && !*abort_flag) {
        const bool okp = __all_sync(0xffffffffu, mbar_wait(&pv_done[g], (uint32_t)(U - 1) & 1u, T2_WAIT_NS));
        if (!okp && lane == 0) {
          set_err(p.err, ERR_TIMEOUT);
          *abort_flag = 1;
        }
      }
      tc_fence_after();
    }
  }
  __syncthreads();
  tc_fence_after();

  // ---------------------------------------------------------------- output
  // Every softmax thread writes its normalised row.
  const bool have = T > 0 && !*abort_flag;
  const bool soft = warp >= T2_SOFT0 && warp < T2_MMA_WARP_B;
  const int sg = (warp - T2_SOFT0) >> 2, sq = (warp - T2_SOFT0) & 3;
  const int sr = sq * 32 + lane;
  const int srows = soft && sg < NT ? min(rows_t, NR - sg * rows_t) : 0;
  const bool owner = sr < srows;           // this thread holds a query row
  if (sq * 32 < srows) {
    const uint32_t orow = tmem_base + ((uint32_t)(sq * 32) << 16) + LY::OCOL + (uint32_t)(sg * D);
    const int rr = owner ? sg * rows_t + sr : 0;
    const int j = j0 + rr / p.G, hq = rr % p.G;
    __nv_bfloat16* dst = p.out + (((size_t)b * p.R + j) * p.Hq + (size_t)kvh * p.G + hq) * D;
    const float inv = (have && l > 0.f) ? 1.f / l : 0.f;
#pragma unroll 1
    for (int c = 0; c < D / 16; ++c) {
      float o[16];
      if (have) {
        tq_ld16(orow + c * 16, o);
        tq_wait_ld();
      }
      if (owner) {
        uint4 w0, w1;
        auto pk = [&](int i) { return have ? pack_bf16(o[i] * inv, o[i + 1] * inv) : 0u; };
        w0.x = pk(0);
        w0.y = pk(2);
        w0.z = pk(4);
        w0.w = pk(6);
        w1.x = pk(8);
        w1.y = pk(10);
        w1.z = pk(12);
        w1.w = pk(14);
        *reinterpret_cast<uint4*>(dst + c * 16) = w0;
        *reinterpret_cast<uint4*>(dst + c * 16 + 8) = w1;
      }
    }
  }

  // After an abort a copy may still be in flight: wait (bounded) for the last
  // fill of every slot a producer used before shared memory goes.
  if (*abort_flag && tid == 0) {
    const int ni = max(n_issued[0], max(n_issued[1], n_issued[2]));
    for (int st = 0; st < T2_SLOTS && st < ni; ++st) {
      const int last = st + ((ni - 1 - st) / T2_SLOTS) * T2_SLOTS;
      mbar_wait(&full[st], (uint32_t)(last / T2_SLOTS) & 1u, T2_WAIT_NS);
    }
    if (T > 0) mbar_wait(q_full, 0, T2_WAIT_NS);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == T2_MMA_WARP) {
    __syncwarp();
    tmem_dealloc(tmem_base, LY::TCOLS);
  }
}

// At least 118 KB, so that two CTAs (each wants all of TMEM) never share an SM.
template <int D>
size_t tcq2_smem_bytes() {
  const size_t need = (size_t)Tcq2Layout<D>::TOTAL + 1024;
  return need > 118 * 1024 ? need : 118 * 1024;
}

template <int D>
KernelLimits& tcq2_limits() {
  static KernelLimits lim;
  return lim;
}

template <int D>
cudaError_t launch_tcq2_t(const CUtensorMap* maps, const Tcq2Params& p, cudaStream_t stream) {
  const size_t smem = tcq2_smem_bytes<D>();
  auto kern = verify_attn_tcq2_kernel<D>;
  const cudaError_t e = ensure_kernel_limits((const void*)kern, tcq2_limits<D>(), smem, false);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(1, p.Hkv * p.RG, p.B), dim3(T2_THREADS), smem, stream, maps[0], maps[1], maps[2],
                    maps[3], maps[4], p);
}

}  // namespace

cudaError_t launch_verify_attn_tcq2(const AttnArgs& a, const AttnPlan& pl, int* err, cudaStream_t stream) {
  const int H = a.D / 64;
  const int G = a.Hq / a.Hkv;
  if (pl.jb * G > T2_M || pl.jg > 2 * pl.jb || pl.cluster != 1) return cudaErrorInvalidValue;
  CUtensorMap maps[5];
  // Pool as {64 columns, rows, half}: a {64, 16, 1} box is one 128-byte half
  // of one page of one head.
  const uint64_t pool_rows = (uint64_t)a.num_pages * a.Hkv * T2_PAGE;
  const uint64_t dp[3] = {64, pool_rows, (uint64_t)H};
  const uint64_t sp[2] = {(uint64_t)a.D * 2, 128};
  const uint32_t bp[3] = {64, T2_PAGE, 1};
  // Block K/V as {64 columns, batch*rows, half, head}: one box per (b, head).
  const int KBR = (a.R + 15) & ~15;
  const uint64_t db[4] = {64, (uint64_t)a.B * a.R, (uint64_t)H, (uint64_t)a.Hkv};
  const uint64_t sb[3] = {(uint64_t)a.Hkv * a.D * 2, 128, (uint64_t)a.D * 2};
  const uint32_t bb[4] = {64, (uint32_t)KBR, (uint32_t)H, 1};
  // Query rows as {64 columns, head, batch*rows, half}: a {64, G, JBQ, 1}
  // box is one half of the rows (j, g) of a row tile, in order j*G + g.
  const uint64_t dq[4] = {64, (uint64_t)a.Hq, (uint64_t)a.B * a.R, (uint64_t)H};
  const uint64_t sq[3] = {(uint64_t)a.D * 2, (uint64_t)a.Hq * a.D * 2, 128};
  const uint32_t bq[4] = {64, (uint32_t)G, (uint32_t)pl.jbq, 1};
  if (!encode_tensor_map_bf16(&maps[0], a.k_pages, 3, dp, sp, bp) ||
      !encode_tensor_map_bf16(&maps[1], a.v_pages, 3, dp, sp, bp) ||
      !encode_tensor_map_bf16(&maps[2], a.k_blk, 4, db, sb, bb) ||
      !encode_tensor_map_bf16(&maps[3], a.v_blk, 4, db, sb, bb) ||
      !encode_tensor_map_bf16(&maps[4], a.q, 4, dq, sq, bq))
    return cudaErrorInvalidValue;
  Tcq2Params p{};
  p.page_table = a.page_table;
  p.ctx_len = a.ctx_len;
  p.q = a.q;
  p.out = a.out;
  p.B = a.B;
  p.R = a.R;
  p.Hq = a.Hq;
  p.Hkv = a.Hkv;
  p.G = G;
  p.JB = pl.jb;
  p.JBQ = pl.jbq;
  p.RG = pl.rg;
  p.JG = pl.jg;
  p.max_pages = a.max_pages;
  p.num_pages = a.num_pages;
  p.scale_log2 = a.scale * 1.4426950408889634f;
  p.kv_stable = a.kv_stable;
  p.block_full = a.block_full;
  p.err = err;
  if (a.D == 128) return launch_tcq2_t<128>(maps, p, stream);
  if (a.D == 64) return launch_tcq2_t<64>(maps, p, stream);
  return cudaErrorInvalidValue;
}

}  // namespace cospec
