// Verify attention on the tcgen05 tensor cores for more than 128 query rows of
// a KV head with D = 128 (teacher-forced verification pass, Sec. 3.1 Eq. 2 of the
// paper; the arbitrator's regions and causal prefill, Sec. 3.3): a cluster of two CTAs
// takes up to 256 query rows, 128 in each, and one MMA works for both
// (cta_group::2, M = 256): each CTA loads half of every K/V tile and the tensor
// cores read the other half from its peer, so a tile's boxes, shared-memory
// writes and B operands are halved per SM.
//
// The clusters are persistent: each takes its share of the units (sequence b, KV head, row
// group of at most 256 rows; the KV range is not split, the planner takes the one-tile
// kernel where a split pays), longest contexts first and back and forth over the clusters, and
// its loads and scores run on into the next unit while the last one is written out.
// Roles by warp, in both CTAs unless said otherwise:
//   warp 0      TMA producer of K: its CTA's 64 keys of each 128-key tile, one 2-D box per
//               page and 128-byte half ([half][64 keys][128 B]);
//   warp 1      TMA producer of V: the 128 keys of the tile, its CTA's 64 columns ([128 keys][128 B]);
//               rings of four stages, a unit's own block K/V as its last tile.  The bytes of
//               both CTAs count on the leader's barriers, except a V tile that may hold rows
//               to be zeroed (the last cache tile, the block), which counts in its CTA;
//   warp 2      query rows, into one of two buffers; zeroes what such a V tile holds beyond
//               its keys and tells the leader, tiles ahead of their use (telling it with P would
//               put a release to the cluster, thousands of cycles, in each unit's last tiles);
//   warp 3      in the leader (cluster rank 0) the MMA issuer:
//                 S   = Q K^T   (M = 256, N = 128 keys, K = D) into one of two
//                               score buffers of each CTA's TMEM,
//                 O_h += P_h V  (M = 256, N = D, K = 64 keys) for each key half h, P_h
//                               read from TMEM (written over its scores);
//   warps 4-11  softmax of the CTA's 128 rows, two groups of four warps (one per TMEM
//               lane quarter), group h key columns 64 h .. 64 h + 63 of every tile with a
//               reference maximum, a sum and an accumulator O_h of its own, put
//               together at the end of the unit; they write its rows.
// The maximum is lazy as in the one-tile kernel: m_ref moves (and O_h and l are
// rescaled) only when a score exceeds it by more than 2^8 in the exp2 domain.
//
// Bound: the instruction issue of one scheduler.  The MMA issuer shares it with a quarter of the
// softmax, which takes about 1100 cycles of a 128-key tile by itself and 1450 beside the issuer;
// the tile's 16 MMAs take 1024 cycles of the tensor pipe, its loads about 930 (16 boxes
// of 2 KB per SM).  So the issuer runs over plain tiles in a loop of its own, four MMAs per
// statement, and every wait but the issuer's and the softmax's sleeps between polls (one loop for
// all tiles, with the units' ends in it: 1800 cycles per tile).  P is made against the reference as
// it stands while the tile's maximum is found (1450 -> 1435 cycles).
// Measured (GB300, us per layer back to back, against two row tiles per CTA): 212-row regions at
// 4096 keys, batch 8 39.2 -> 32.0, batch 16 77.5 -> 60.9; batch 32 at 2048..8192 keys 155 -> 133;
// four layers of a 4096-token causal prefill (32 / 8 heads) 570 -> 485.  One unit per cluster
// and a launch of as many clusters as units instead of persistent ones: the prefill took 638 (8 us
// per cluster of start, first loads and output, which now overlap).
#include <cuda.h>
#include <math.h>

#include "cospec_device.cuh"
#include "cospec_internal.h"

namespace cospec {

namespace {

constexpr int TP_D = 128;          // head dimension: two 128-byte halves of a key row
constexpr int TP_KT = 128;         // keys per cache tile (8 pages) = MMA N of S
constexpr int TP_PPT = TP_KT / 16;
constexpr int TP_PAGE = 16;
constexpr int TP_ROWB = 128;       // bytes of one swizzled smem row
constexpr int TP_M = 128;          // query rows per CTA
constexpr int TP_NS = 4;           // ring stages
constexpr int TP_MMA_WARP = 3;
constexpr int TP_SOFT0 = 4;
constexpr int TP_THREADS = 384;
constexpr float TP_LAZY = 8.f;
constexpr uint64_t TP_WAIT_NS = 2000000000ull;
// shared memory, the same offsets in both CTAs
constexpr int TP_KV = TP_KT * TP_ROWB;                 // a CTA's half of a K (or V) tile: 16 KB
constexpr int TP_STAGE = 2 * TP_KV;
constexpr int TP_QH = TP_M * TP_ROWB;                  // one half of the query rows
constexpr int TP_QOFF = TP_NS * TP_STAGE;              // two buffers of [half][128 rows][128 B]
constexpr int TP_OUT = TP_QOFF + 2 * 2 * TP_QH;        // 4 KB per softmax warp: its output rows
constexpr int TP_BARS = TP_OUT + 8 * 32 * TP_ROWB;
// full_k[NS], full_v[NS], tail_v[NS], tail_ok[NS], empty_k[NS], empty_v[NS], q_full[2], q_empty[2], s_full[2],
// p_full[2], pv_done[2 halves], o_full, mma_done
constexpr int TP_NBAR = 6 * TP_NS + 12;
constexpr int TP_HOLDER = TP_BARS + TP_NBAR * 8;
constexpr int TP_FLAGS = TP_HOLDER + 8;                // abort, then fills (below)
constexpr int TP_UNITS = (TP_FLAGS + 32 + 15) & ~15;   // the cluster's units: b, C, KV head, first block row
constexpr int TP_MAXU = 32;
constexpr int TP_TOTAL = TP_UNITS + TP_MAXU * 16;
constexpr uint32_t TP_OCOL = 2 * TP_KT;                // TMEM columns: S[2], O_0, O_1
constexpr uint32_t TP_TCOLS = 512u;

template <bool B>
struct TpTag {
  static constexpr bool value = B;
};

struct TcpParams {
  const int32_t* page_table;
  const int32_t* ctx_len;
  __nv_bfloat16* out;
  int B, R, Hq, Hkv, G;
  int JB;           // block rows (j) of a CTA
  int JBQ;          // block rows of the query box: min(R, JB)
  int RG, JG;       // row groups, block rows per group (at most 2 JB)
  int max_pages, num_pages;
  float scale_log2;
  int kv_stable;
  int block_full;
  int* err;
};

__global__ void __launch_bounds__(TP_THREADS, 1)
    verify_attn_tcp_kernel(const __grid_constant__ CUtensorMap map_kp,
                           const __grid_constant__ CUtensorMap map_vp,
                           const __grid_constant__ CUtensorMap map_kb,
                           const __grid_constant__ CUtensorMap map_vb,
                           const __grid_constant__ CUtensorMap map_q, const TcpParams p) {
  constexpr int D = TP_D, NS = TP_NS;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full_k = reinterpret_cast<uint64_t*>(smem + TP_BARS);   // leader's: both CTAs' bytes
  uint64_t* full_v = full_k + NS;
  uint64_t* tail_v = full_v + NS;      // this CTA's V of a unit's last cache tile, of its block
  uint64_t* tail_ok = tail_v + NS;     // leader's: zeroed in both CTAs
  uint64_t* empty_k = tail_ok + NS;
  uint64_t* empty_v = empty_k + NS;
  uint64_t* q_full = empty_v + NS;     // leader's: [2]
  uint64_t* q_empty = q_full + 2;      // [2]
  uint64_t* s_full = q_empty + 2;      // [2]
  uint64_t* p_full = s_full + 2;       // leader's: [2], every softmax warp of both CTAs
  uint64_t* pv_done = p_full + 2;      // [2 halves]
  uint64_t* o_full = pv_done + 2;      // a unit's last products
  uint64_t* mma_done = o_full + 1;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + TP_HOLDER);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + TP_FLAGS);
  // for an abort: K fills, stages filled with V and their next phases (leader's barriers, this
  // CTA's), query fills
  volatile int* fills = abort_flag + 1;
  int4* list = reinterpret_cast<int4*>(smem + TP_UNITS);
  uint8_t* qs = smem + TP_QOFF;

  const int rank = (int)cluster_ctarank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int Y = p.Hkv * p.RG, units = Y * p.B;
  const int ncl = (int)gridDim.x >> 1, cl = (int)blockIdx.x >> 1;
  const int KBR = (p.R + 31) & ~31;          // block keys padded to 32: 16 or 32 in a CTA's K

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full_k[s], 1);
      mbar_init(&full_v[s], 1);
      mbar_init(&tail_v[s], 1);
      mbar_init(&tail_ok[s], 2);
      mbar_init(&empty_k[s], 1);
      mbar_init(&empty_v[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1);
      mbar_init(&q_empty[i], 1);
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], 16);
      mbar_init(&pv_done[i], 1);
    }
    mbar_init(o_full, 1);
    mbar_init(mma_done, 1);
    for (int i = 0; i < 7; ++i) abort_flag[i] = 0;
    fence_barrier_init();
  }
  if (warp == TP_MMA_WARP) tmem_alloc_pair(tmem_holder, TP_TCOLS);
  // (in this order: a dependent under the stable-cache promise reads the cache at once)
  if (!p.kv_stable) griddep_wait();
  griddep_launch_dependents();
  // Sequences longest context first (ties to the lower index); a larger batch in index
  // order, from the longer end.
  const bool ranked = p.B <= TP_THREADS;
  int* c_all = reinterpret_cast<int*>(smem + TP_OUT);
  int* order = c_all + TP_THREADS;
  if (ranked) {
    if (tid < p.B) c_all[tid] = p.ctx_len[tid];
    __syncthreads();
    if (tid < p.B) {
      const int ci = c_all[tid];
      int r = 0;
#pragma unroll 4
      for (int j = 0; j < p.B; ++j) r += (c_all[j] > ci) | ((c_all[j] == ci) & (j < tid));
      order[r] = tid;
    }
    __syncthreads();
  }
  // The cluster's units (C < 0: not processed, its rows are zero): the k-th goes up or down the
  // clusters as k is even or odd.
  const int rounds = (units + ncl - 1) / ncl, last = (rounds - 1) * ncl + ((rounds & 1) ? cl : ncl - 1 - cl);
  const int nunits = rounds - (last >= units ? 1 : 0);
  if (tid < nunits) {
    const int u = tid * ncl + ((tid & 1) ? ncl - 1 - cl : cl);
    const int z = u / Y, y = u - z * Y, kvh = y / p.RG;
    const int b = ranked ? order[z] : sequence_in_order(p.ctx_len, p.B, z);
    const int C = p.ctx_len[b];
    const bool bad = (C < 0) || (C > p.max_pages * TP_PAGE);
    if (bad && rank == 0) set_err(p.err, ERR_CTX);
    list[tid] = make_int4(b, bad ? -1 : C, kvh, (y - kvh * p.RG) * p.JG);
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();                      // both CTAs' barriers are initialised
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  struct Unit {
    int b, C, kvh, jg0, n, T;            // T = n cache tiles and the block's, 0: not processed
  };
  auto fetch = [&](int k, Unit& w) -> bool {
    if (k >= nunits) return false;
    const int4 bc = list[k];
    w.b = bc.x;
    w.C = bc.y;
    w.kvh = bc.z;
    w.jg0 = bc.w;
    w.n = bc.y < 0 ? 0 : (bc.y + TP_KT - 1) / TP_KT;
    w.T = bc.y < 0 ? 0 : w.n + 1;
    return true;
  };

  if (warp < 2) {
    // ------------------------------------------------------------ producers
    // Lane e issues box e of this CTA's eight: K page 4 rank + e / 2, half e % 2; V
    // page e, half `rank`.
    const int tensor = warp;
    uint64_t* my_full = tensor ? full_v : full_k;
    uint64_t* my_empty = tensor ? empty_v : empty_k;
    const uint32_t lead_full = dsmem_map(smem_u32(my_full), 0);
    const int pg = tensor ? lane : 4 * rank + (lane >> 1);
    const int h = tensor ? rank : (lane & 1);
    const uint32_t off = (uint32_t)(tensor ? TP_KV + lane * (TP_PAGE * TP_ROWB)
                                           : (lane & 1) * (64 * TP_ROWB) + (lane >> 1) * (TP_PAGE * TP_ROWB));
    if (lane == 0) tma_prefetch_desc(tensor ? &map_vp : &map_kp);
    const uint64_t pol = p.RG > 1 ? l2_policy_evict_normal() : l2_policy_evict_first();
    const uint32_t sbase = smem_u32(smem);
    int i = 0;                           // tiles so far: ring position
    bool ok = true, waited = !p.kv_stable;
    uint32_t used0 = 0u, phase0 = 0u, used1 = 0u, phase1 = 0u;   // V fills by stage: leader's, this CTA's
    auto wait_slot = [&]() -> bool {
      if (i < NS) return true;
      const bool w = mbar_wait_idle(&my_empty[i % NS], (uint32_t)((i / NS) - 1) & 1u, TP_WAIT_NS, 100u);
      return __all_sync(0xffffffffu, w) && !*abort_flag;
    };
    auto fill = [&](bool tail) {
      const uint32_t bit = 1u << (i % NS);
      used0 |= tail ? 0u : bit;
      phase0 ^= tail ? 0u : bit;
      used1 |= tail ? bit : 0u;
      phase1 ^= tail ? bit : 0u;
      if (lane == 0) {
        if (!tensor) {
          fills[0] = i + 1;
        } else {
          fills[1] = (int)used0;
          fills[2] = (int)phase0;
          fills[3] = (int)used1;
          fills[4] = (int)phase1;
        }
      }
    };
    Unit w;
    for (int k = 0; ok && fetch(k, w); ++k) {
      if (w.T == 0) continue;
      const int* ptab = p.page_table + (size_t)w.b * p.max_pages;
      const int npages = (w.C + TP_PAGE - 1) / TP_PAGE;
      int pid = 0;
      for (int t = 0; t < w.n; ++t) {
        if ((t & 3) == 0) {              // 32 page ids = the next 4 tiles, one per lane
          const int e2 = t * TP_PPT + lane;
          pid = (e2 < npages) ? __ldg(ptab + e2) : 0;
        }
        ok = wait_slot();
        if (!ok) break;
        const int st = i % NS;
        const int np = min(TP_PPT, npages - t * TP_PPT);
        int pgid = __shfl_sync(0xffffffffu, pid, (t & 3) * TP_PPT + (pg & 7));
        const bool tail = tensor && t == w.n - 1;      // counts on this CTA's own barrier
        fill(tail);
        if (lane == 0) {
          if (tail)
            mbar_arrive_expect_tx(&tail_v[st], (uint32_t)(np * TP_PAGE * TP_ROWB));
          else if (rank == 0)
            mbar_arrive_expect_tx(&my_full[st], (uint32_t)(np * TP_PAGE * 2 * TP_ROWB));
        }
        __syncwarp();
        if (lane < TP_PPT && pg < np) {
          if ((unsigned)pgid >= (unsigned)p.num_pages) {
            set_err(p.err, ERR_PAGE);
            pgid = 0;
          }
          const uint32_t dst = sbase + (uint32_t)(st * TP_STAGE) + off;
          const int y = (pgid * p.Hkv + w.kvh) * TP_PAGE;
          if (tail)
            tma_load_3d(dst, &map_vp, &tail_v[st], 0, y, h, pol);
          else
            tma_load_3d_pair(dst, tensor ? (const void*)&map_vp : (const void*)&map_kp, lead_full + st * 8, 0, y, h,
                             pol);
        }
        __syncwarp();
        ++i;
      }
      if (!ok) break;
      if (!waited) {                     // the block K/V comes from the previous kernel
        griddep_wait();
        waited = true;
      }
      ok = wait_slot();
      if (!ok) break;
      // K: KBR / 2 block rows from row rank * KBR / 2, both halves ([half][KBR / 2 rows][128 B]);
      // V: KBR block rows, half `rank`
      const int st = i % NS;
      fill(tensor != 0);
      if (lane == 0) {
        const uint32_t dst = sbase + (uint32_t)(st * TP_STAGE + tensor * TP_KV);
        if (tensor) {
          mbar_arrive_expect_tx(&tail_v[st], (uint32_t)(KBR * TP_ROWB));
          tma_load_4d(dst, &map_vb, &tail_v[st], 0, w.b * p.R, rank, w.kvh, pol);
        } else {
          if (rank == 0) mbar_arrive_expect_tx(&full_k[st], (uint32_t)(2 * KBR * TP_ROWB));
          tma_load_4d_pair(dst, &map_kb, lead_full + st * 8, 0, w.b * p.R + rank * (KBR / 2), 0, w.kvh, pol);
        }
      }
      __syncwarp();
      ++i;
    }
    if (!waited) griddep_wait();
    if (lane == 0 && !ok) {
      set_err(p.err, ERR_TIMEOUT);
      *abort_flag = 1;
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ query rows, ends of V
    if (p.kv_stable) griddep_wait();     // the query rows come from the previous kernel
    const uint64_t qpol = l2_policy_evict_first();
    const uint32_t qbytes = (uint32_t)(2 * p.G * p.JBQ * TP_ROWB);   // two boxes
    const uint32_t lead_ok = dsmem_map(smem_u32(tail_ok), 0);
    bool ok = true;
    int iq = 0, kq = 0;                  // units whose rows were asked for
    auto load_q = [&]() {
      Unit w;
      w.T = 0;
      while (w.T == 0 && fetch(kq, w)) ++kq;
      if (w.T == 0) return;
      if (iq >= 2)
        ok = __all_sync(0xffffffffu, mbar_wait_idle(&q_empty[iq & 1], (uint32_t)((iq >> 1) - 1) & 1u, TP_WAIT_NS, 100u)) &&
             !*abort_flag;
      if (!ok) return;
      if (lane == 0) {
        if (rank == 0) mbar_arrive_expect_tx(&q_full[iq & 1], 2 * qbytes);
        const uint32_t bar = dsmem_map(smem_u32(&q_full[iq & 1]), 0);
        for (int h = 0; h < 2; ++h)
          tma_load_4d_pair(smem_u32(qs + ((iq & 1) * 2 + h) * TP_QH), &map_q, bar, 0, w.kvh * p.G,
                           w.b * p.R + w.jg0 + rank * p.JB, h, qpol);
        fills[5] = iq + 1;
      }
      __syncwarp();
      ++iq;
    };
    load_q();
    int i = 0;                           // tiles before this unit
    uint32_t phase = 0u;                 // parity of the next fill of tail_v, by stage
    Unit w;
    for (int k = 0; ok && fetch(k, w); ++k) {
      if (w.T == 0) continue;
      load_q();                          // the next unit's
      for (int t = w.n > 0 ? w.n - 1 : 0; t < w.T && ok; ++t) {
        const int st = (i + t) % NS;
        const bool blk = t == w.n;
        ok = __all_sync(0xffffffffu, mbar_wait_idle(&tail_v[st], (phase >> st) & 1u, TP_WAIT_NS, 100u)) && !*abort_flag;
        if (!ok) break;
        phase ^= 1u << st;
        // stale bytes may be NaN: the zero weights of these keys must contribute 0
        const int vr = blk ? p.R : w.C - t * TP_KT, nk = blk ? KBR : TP_KT;
        uint8_t* vb = smem + st * TP_STAGE + TP_KV;
        for (int e = lane; e < (nk - vr) * 8; e += 32)
          *reinterpret_cast<uint4*>(vb + vr * TP_ROWB + e * 16) = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_ok + (uint32_t)(st * 8));
      }
      i += w.T;
    }
    if (lane == 0 && !ok) {
      set_err(p.err, ERR_TIMEOUT);
      *abort_flag = 1;
    }
  } else if (warp == TP_MMA_WARP) {
    // ------------------------------------------------------------ MMA issuer
    // (the whole warp walks along; one elected thread acts)
    if (rank == 0) {
      const uint32_t on = elect_one();
      const uint32_t sbase = smem_u32(smem);
      const uint64_t q_desc = smem_desc_sw128(sbase + TP_QOFF);
      const uint64_t k_desc = smem_desc_sw128(sbase);
      const uint32_t idesc_pv = idesc_bf16_f32(2 * TP_M, D) | (1u << 16);   // B (V) MN-major
      bool ok = true;
      auto wait_all = [&](uint64_t* bar, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(bar, parity & 1u, TP_WAIT_NS));
      };
      // Two cursors over the tiles of the cluster's units: scores (two ahead), products.
      struct Cursor {
        int k, T, t, i, units;           // unit, its tiles (0: no more), tile of it, tiles and units so far
      };
      auto enter = [&](Cursor& c) {      // the next unit that is processed
        int T = 0;
        while (T == 0 && ++c.k < nunits) {
          const int C = list[c.k].y;
          T = C < 0 ? 0 : (C + TP_KT - 1) / TP_KT + 1;
        }
        c.T = T;
        c.t = 0;
      };
      auto advance = [&](Cursor& c) {
        ++c.i;
        if (++c.t == c.T) {
          ++c.units;
          enter(c);
        }
      };
      Cursor cs{-1, 0, 0, 0, 0}, cp;
      enter(cs);
      cp = cs;
      // (descriptor addresses count 16-byte units)
      auto ready_s = [&]() -> bool {
        return (cs.t > 0 || wait_all(&q_full[cs.units & 1], (uint32_t)(cs.units >> 1))) &&
               wait_all(&full_k[cs.i % NS], (uint32_t)(cs.i / NS));
      };
      auto issue_s = [&]() {
        const int st = cs.i % NS;
        const int nk = cs.t == cs.T - 1 ? KBR : TP_KT;
        const uint64_t qd = q_desc + (uint64_t)((cs.units & 1) * (2 * TP_QH >> 4));
        const uint64_t kd = k_desc + (uint64_t)(st * (TP_STAGE >> 4));
        const uint64_t khalf = (uint64_t)((nk / 2) * (TP_ROWB >> 4));
        const uint32_t idesc_qk = idesc_bf16_f32(2 * TP_M, nk);
        const uint32_t dst = tmem_base + (uint32_t)((cs.i & 1) * TP_KT);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          umma_bf16_pair_k64_on(on, dst, qd + (uint64_t)(h * (TP_QH >> 4)), kd + h * khalf, idesc_qk, h);
        umma_commit_pair_on(on, &s_full[cs.i & 1], 3);
        umma_commit_pair_on(on, &empty_k[st], 3);      // K of this stage is free once S is done
        if (cs.t == cs.T - 1) umma_commit_pair_on(on, &q_empty[cs.units & 1], 3);
        advance(cs);
      };
      // O_h += P_h V over keys 64 h .. of the tile (the block tile is all in half 0)
      auto issue_pv = [&](int h) {
        const uint32_t vb = sbase + (uint32_t)((cp.i % NS) * TP_STAGE + TP_KV + h * (64 * TP_ROWB));
        const uint32_t src = tmem_base + (uint32_t)((cp.i & 1) * TP_KT + h * 64);
        const uint32_t dst = tmem_base + TP_OCOL + (uint32_t)(h * D);
        // 16 keys = 8 TMEM columns and 16 rows of V (2 KB) per MMA
        const uint64_t vd = tq_desc_mn_sw128(vb, (uint32_t)TP_KV);
        const uint32_t acc0 = cp.t > 0 ? 1u : 0u;
        if (cp.t == cp.T - 1) {
          for (int ks = 0; ks < KBR / 16; ++ks)
            umma_bf16_tmem_a_pair_on(on, dst, src + (uint32_t)(ks * 8), vd + (uint64_t)(ks * 128), idesc_pv,
                                     ks > 0 ? 1u : acc0);
        } else {
          umma_bf16_tmem_a_pair_k64_on(on, dst, src, vd, idesc_pv, acc0);
        }
        umma_commit_pair_on(on, &pv_done[h], 3);
      };
      // S of tile i + 2 goes to buffer i & 1, last read (as P) by the P.V products of tile
      // i: tcgen05 MMAs of one thread run in issue order, so S may be issued once
      // those are.
      for (int j = 0; j < 2 && cs.T > 0 && ok; ++j) {
        ok = ready_s();
        if (!ok) break;
        tc_fence_after();
        issue_s();
      }
      uint32_t vphase = 0u, zphase = 0u; // parities of the next fills, by stage
      while (ok && cp.T > 0) {
        // plain tiles whose S two ahead is a plain tile of the same unit
        const int plain = cp.T - 3 - cp.t;
        if (plain > 0) {
          int i = cp.i;
          const int i_end = i + plain;
          const uint64_t qd = q_desc + (uint64_t)((cp.units & 1) * (2 * TP_QH >> 4));
          const uint32_t idesc_qk = idesc_bf16_f32(2 * TP_M, TP_KT);
          uint32_t acc = cp.t > 0 ? 1u : 0u;
          for (; i < i_end; ++i) {
            const int sv = i % NS, sk = (i + 2) % NS;
            const uint32_t buf = tmem_base + (uint32_t)((i & 1) * TP_KT);
            const uint64_t vd = tq_desc_mn_sw128(sbase + (uint32_t)(sv * TP_STAGE + TP_KV), (uint32_t)TP_KV);
            const uint64_t kd = k_desc + (uint64_t)(sk * (TP_STAGE >> 4));
            ok = wait_all(&full_v[sv], vphase >> sv) && wait_all(&full_k[sk], (uint32_t)((i + 2) / NS)) &&
                 wait_all(&p_full[i & 1], (uint32_t)(i >> 1));
            if (!ok) break;
            vphase ^= 1u << sv;
            tc_fence_after();
            umma_bf16_tmem_a_pair_k64_on(on, tmem_base + TP_OCOL, buf, vd, idesc_pv, acc);
            umma_commit_pair_on(on, &pv_done[0], 3);
            umma_bf16_tmem_a_pair_k64_on(on, tmem_base + TP_OCOL + D, buf + 64, vd + (64 * TP_ROWB >> 4), idesc_pv, acc);
            umma_commit_pair_on(on, &pv_done[1], 3);
            umma_commit_pair_on(on, &empty_v[sv], 3);
            umma_bf16_pair_k64_on(on, buf, qd, kd, idesc_qk, 0u);
            umma_bf16_pair_k64_on(on, buf, qd + (TP_QH >> 4), kd + (64 * TP_ROWB >> 4), idesc_qk, 1u);
            umma_commit_pair_on(on, &s_full[i & 1], 3);
            umma_commit_pair_on(on, &empty_k[sk], 3);
            acc = 1u;
          }
          cp.t += plain;
          cp.i += plain;
          cs.t += plain;
          cs.i += plain;
          if (!ok) break;
        }
        // everything else before P, so that the products are issued in one go
        const int st = cp.i % NS;
        if (cp.t < cp.T - 2) {
          ok = wait_all(&full_v[st], vphase >> st);
          vphase ^= 1u << st;
        } else {
          ok = wait_all(&tail_ok[st], zphase >> st);
          zphase ^= 1u << st;
        }
        const bool next = cs.T > 0;
        if (ok && next) ok = ready_s();
        if (ok) ok = wait_all(&p_full[cp.i & 1], (uint32_t)(cp.i >> 1));
        if (!ok) break;
        tc_fence_after();
        issue_pv(0);
        if (cp.t < cp.T - 1) issue_pv(1);
        umma_commit_pair_on(on, &empty_v[st], 3);
        if (cp.t == cp.T - 1) umma_commit_pair_on(on, o_full, 3);
        if (next) issue_s();
        advance(cp);
      }
      if (!ok && on) {
        set_err(p.err, ERR_TIMEOUT);
        *abort_flag = 1;
      }
      // (both CTAs wait for it below: every MMA completes before TMEM is released)
      umma_commit_pair_on(on, mma_done, 3);
    }
  } else if (warp >= TP_SOFT0) {
    // ------------------------------------------------------------ softmax
    const int sw = warp - TP_SOFT0;
    const int grp = sw >> 2;             // key-column half of every tile
    const int q = sw & 3;                // TMEM lane quarter of this warp
    const int r = q * 32 + lane;         // this thread's query row of the CTA
    const int kc0 = grp * (TP_KT / 2);   // first key column of this half
    const float sc = p.scale_log2;
    const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t ocol = TP_OCOL + (uint32_t)(grp * D);   // this half's O
    const uint32_t lead_p = dsmem_map(smem_u32(p_full), 0);
    uint8_t* stage = smem + TP_OUT + sw * (32 * TP_ROWB);  // this warp's output rows
    int i0 = 0;                          // tiles before this unit
    int pv0 = 0, pv1 = 0;                // P.V products before it, by half
    int nu = 0;                          // units before it
    for (int k = 0;; ++k) {
      int n, T, C, NR, blim;
      bool rvalid;
      {
        Unit w;
        if (!fetch(k, w)) break;
        n = w.n;
        T = w.T;
        C = w.C;
        NR = max(0, min(min(p.JG, p.R - w.jg0) - rank * p.JB, p.JB)) * p.G;   // this CTA's query rows
        rvalid = r < NR;
        const int jr = w.jg0 + rank * p.JB + (rvalid ? r / p.G : 0);          // block row of this query row
        // the last block key this row sees: its own row (causal) or the whole block
        blim = p.block_full ? p.R - 1 : min(jr, p.R - 1);
      }
      float mref = -INFINITY, l = 0.f;                     // this row half's m_ref and sum
      // ---- tiles
      if (*abort_flag) T = n = 0;
      auto tile = [&](int t, auto plain_tag) -> bool {
        constexpr bool PLAIN = decltype(plain_tag)::value;   // not the last cache tile, not the block
        const int i = i0 + t;
        const bool blk = !PLAIN && t == n;
        const int nk = blk ? KBR : TP_KT / 2;      // score columns of this half
        if (!__all_sync(0xffffffffu, mbar_wait(&s_full[i & 1], (uint32_t)(i >> 1) & 1u, TP_WAIT_NS))) {
          if (lane == 0) {
            set_err(p.err, ERR_TIMEOUT);
            *abort_flag = 1;
          }
          return false;
        }
        const int left = C - t * TP_KT - kc0;      // context keys from here on
        // (the tcgen05 fences order P; an arrival with a release to the cluster takes thousands
        // of cycles)
        auto answer = [&]() {
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster_relaxed(lead_p + (uint32_t)((i & 1) * 8));
        };
        if (q * 32 >= NR || (blk && grp)) {        // nothing to exponentiate
          answer();
          return true;
        }
        tc_fence_after();
        const uint32_t srow = lane_base + (uint32_t)((i & 1) * TP_KT + kc0);
        // keys 0..lim of this half are visible to this row (raw scores; the
        // scale is positive, so it is applied with the exponent).  Padding
        // rows (r >= NR) give rows of P and O that nothing reads, so they
        // decide neither the masking nor a rescale.  A block tile has 16 to 64
        // score columns; the rest of the half holds an earlier tile's.
        const int lim = blk ? blim : min(TP_KT / 2, left) - 1;
        float x0[32], x1[32];
        tq_ld32(srow, x0);
        tq_ld32(srow + 32, x1);
        tq_wait_ld32(x0);
        tq_wait_ld32(x1);
        if (!PLAIN && (__any_sync(0xffffffffu, rvalid && lim < TP_KT / 2 - 1) || blk)) {
#pragma unroll
          for (int k = 0; k < 32; ++k) {
            x0[k] = k <= lim ? x0[k] : -INFINITY;
            x1[k] = 32 + k <= lim ? x1[k] : -INFINITY;
          }
        }
        // P = 2^(score * scale - m_ref) in bf16, two keys per TMEM column, over
        // this half's scores (masked keys give exactly 0)
        float2 l2[2];
        auto exponentiate = [&]() {
          const float nb = (mref == -INFINITY) ? 0.f : -mref;
          const float2 sc2 = make_float2(sc, sc), nb2 = make_float2(nb, nb);
          l2[0] = l2[1] = make_float2(0.f, 0.f);
          auto half = [&](float (&x)[32], int k0) {
            uint32_t pk[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float2 e = fma2(make_float2(x[2 * k], x[2 * k + 1]), sc2, nb2);
              const float2 pp = make_float2(exp2_approx(e.x), exp2_approx(e.y));
              l2[k & 1] = add2(l2[k & 1], pp);
              pk[k] = pack_bf16(pp.x, pp.y);
            }
            tq_st16(srow + k0 / 2, pk);
          };
          half(x0, 0);
          half(x1, 32);
        };
        // With the reference as it stands, beside the tile's maximum: it moves only when a
        // score exceeds it by 2^8 (the first tile always sets it: m_ref starts at
        // -inf), and P is made once more then.
        exponentiate();
        float m4[4] = {x0[0], x0[1], x0[2], x0[3]};
#pragma unroll
        for (int k = 4; k < 32; ++k) m4[k & 3] = fmaxf(m4[k & 3], x0[k]);
#pragma unroll
        for (int k = 0; k < 32; ++k) m4[k & 3] = fmaxf(m4[k & 3], x1[k]);
        const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * sc;
        const bool up = rvalid && mx > mref + TP_LAZY;
        if (__any_sync(0xffffffffu, up)) {
          float alpha = 1.f;
          if (up) {
            alpha = (mref == -INFINITY) ? 0.f : exp2_approx(mref - mx);
            mref = mx;
            l *= alpha;
          }
          if (t > 0) {
            // O_h holds tiles 0..t-1: wait for the last of them, then scale the row
            const bool okp =
                __all_sync(0xffffffffu, mbar_wait_idle(&pv_done[grp], (uint32_t)((grp ? pv1 : pv0) + t - 1) & 1u, TP_WAIT_NS));
            tc_fence_after();
            if (okp) {
#pragma unroll 1
              for (int c = 0; c < D / 16; ++c) {
                float o[16];
                tq_ld16(lane_base + ocol + c * 16, o);
                tq_wait_ld();
                uint32_t w[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) w[k] = __float_as_uint(o[k] * alpha);
                tq_st16(lane_base + ocol + c * 16, w);
              }
            } else if (lane == 0) {
              set_err(p.err, ERR_TIMEOUT);
            }
          }
          exponentiate();
        }
        l += (l2[0].x + l2[0].y) + (l2[1].x + l2[1].y);
        tq_wait_st();
        tc_fence_before();
        answer();
        return true;
      };
      bool ok = true;
      int t = 0;
      for (; t < n - 1 && ok; ++t) ok = tile(t, TpTag<true>{});
      for (; t < T && ok; ++t) ok = tile(t, TpTag<false>{});
      // ---- output
      // The two halves of a row are put together: common maximum, weighted sums.  Each group
      // writes half of the row's columns, through shared memory so that a store covers
      // whole 128-byte rows.
      if (T > 0) {
        const bool done = !*abort_flag && mbar_wait_idle(o_full, (uint32_t)nu & 1u, TP_WAIT_NS);
        ++nu;
        if (!__all_sync(0xffffffffu, done) && lane == 0) {
          set_err(p.err, ERR_TIMEOUT);
          *abort_flag = 1;
        }
        tc_fence_after();
      }
      i0 += T;
      pv0 += T;
      pv1 += n;
      float2* xch = reinterpret_cast<float2*>(stage);
      const float2* xch_o = reinterpret_cast<const float2*>(smem + TP_OUT + (sw ^ 4) * (32 * TP_ROWB));
      xch[lane] = make_float2(mref, l);
      named_bar_sync(1 + q, 64);
      const float2 o_ml = xch_o[lane];
      named_bar_sync(1 + q, 64);
      const bool have = T > 0 && !*abort_flag;
      if (q * 32 < NR) {
        Unit w;
        fetch(k, w);
        const int j0 = w.jg0 + rank * p.JB;  // first block row of this CTA
        const float mm = fmaxf(mref, o_ml.x);
        const float wm = (mref == -INFINITY) ? 0.f : exp2_approx(mref - mm);   // this half's weight
        const float wo = (o_ml.x == -INFINITY) ? 0.f : exp2_approx(o_ml.x - mm);
        const float ls = grp ? o_ml.y * wo + l * wm : l * wm + o_ml.y * wo;
        const float inv = (have && ls > 0.f) ? 1.f / ls : 0.f;
        const float w0_ = (grp ? wo : wm) * inv, w1_ = (grp ? wm : wo) * inv;
        const bool have1 = have && n > 0;    // half 1 holds cache tiles only
#pragma unroll
        for (int c = 0; c < 2; ++c) {        // 32 columns at a time, from both accumulators
          float o[32], o1[32];
          if (have) {
            tq_ld32(lane_base + TP_OCOL + (grp * 2 + c) * 32, o);
            if (have1) tq_ld32(lane_base + TP_OCOL + D + (grp * 2 + c) * 32, o1);
            tq_wait_ld32(o);
            if (have1) tq_wait_ld32(o1);
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = !have ? 0.f : have1 ? o[i] * w0_ + o1[i] * w1_ : o[i] * w0_;
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
            uint4 v;
            v.x = pack_bf16(o[i], o[i + 1]);
            v.y = pack_bf16(o[i + 2], o[i + 3]);
            v.z = pack_bf16(o[i + 4], o[i + 5]);
            v.w = pack_bf16(o[i + 6], o[i + 7]);
            *reinterpret_cast<uint4*>(stage + lane * TP_ROWB + (((c * 4 + i / 8) ^ (lane & 7)) * 16)) = v;
          }
        }
        tc_fence_before();                   // (the next unit's products wait for this warp's P)
        __syncwarp();
        const int chunk = lane & 7;
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          const int row = it * 4 + (lane >> 3), rr = q * 32 + row;
          if (rr < NR) {
            const int j = j0 + rr / p.G, g = rr % p.G;
            *reinterpret_cast<uint4*>(p.out + (((size_t)w.b * p.R + j) * p.Hq + (size_t)w.kvh * p.G + g) * D +
                                      grp * 64 + chunk * 8) =
                *reinterpret_cast<const uint4*>(stage + row * TP_ROWB + ((chunk ^ (row & 7)) * 16));
          }
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  if (warp == TP_MMA_WARP) mbar_wait_idle(mma_done, 0, TP_WAIT_NS);
  // Neither CTA leaves, or gives its TMEM back, while the other's copies or products may still
  // touch it.  An abort in one is known to both after the barrier.
  if (*abort_flag && tid == 0)
    dsmem_store_u32(dsmem_map(smem_u32(const_cast<int*>(abort_flag)), (uint32_t)(rank ^ 1)), 1u);
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  if (*abort_flag) {
    // A copy may still be in flight: wait (bounded) for the last fill of every stage
    // that was used (the leader's barriers count both CTAs' bytes), then meet again.
    if (tid == 0) {
      for (int st = 0; st < NS; ++st) {
        const int nk_ = fills[0];
        if (rank == 0 && st < nk_)
          mbar_wait_idle(&full_k[st], (uint32_t)((st + ((nk_ - 1 - st) / NS) * NS) / NS) & 1u, TP_WAIT_NS);
        if (rank == 0 && ((fills[1] >> st) & 1)) mbar_wait_idle(&full_v[st], (uint32_t)((fills[2] >> st) & 1) ^ 1u, TP_WAIT_NS);
        if (rank == 0 && st < 2 && st < fills[5])
          mbar_wait_idle(&q_full[st], (uint32_t)((fills[5] - 1 - st) >> 1) & 1u, TP_WAIT_NS);
        if ((fills[3] >> st) & 1) mbar_wait_idle(&tail_v[st], (uint32_t)((fills[4] >> st) & 1) ^ 1u, TP_WAIT_NS);
      }
    }
    __syncthreads();
    cluster_arrive();
    cluster_wait();
  }
  if (warp == TP_MMA_WARP) {
    __syncwarp();
    tmem_dealloc_pair(tmem_base, TP_TCOLS);
  }
}

KernelLimits& tcp_limits() {
  static KernelLimits lim;
  return lim;
}

constexpr size_t TP_SMEM = (size_t)TP_TOTAL + 1024;
static_assert(TP_SMEM <= 232448, "227 KB of shared memory");

cudaLaunchConfig_t tcp_config(cudaLaunchAttribute* attr, int clusters, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * clusters);
  cfg.blockDim = dim3(TP_THREADS, 1, 1);
  cfg.dynamicSmemBytes = TP_SMEM;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

}  // namespace

cudaError_t launch_verify_attn_tcp(const AttnArgs& a, const AttnPlan& pl, int* err, cudaStream_t stream) {
  const int G = a.Hq / a.Hkv;
  if (a.D != TP_D || pl.jb * G > TP_M || pl.jg > 2 * pl.jb || pl.cluster != 1 || pl.resident < 1)
    return cudaErrorInvalidValue;
  CUtensorMap maps[5];
  // Pool as {64 columns, rows, half}: a {64, 16, 1} box is one 128-byte half
  // of one page of one head.
  const uint64_t pool_rows = (uint64_t)a.num_pages * a.Hkv * TP_PAGE;
  const uint64_t dp[3] = {64, pool_rows, 2};
  const uint64_t sp[2] = {(uint64_t)a.D * 2, 128};
  const uint32_t bp[3] = {64, TP_PAGE, 1};
  // Block K/V as {64 columns, batch*rows, half, head}.
  const uint32_t KBR = (uint32_t)((a.R + 31) & ~31);
  const uint64_t db[4] = {64, (uint64_t)a.B * a.R, 2, (uint64_t)a.Hkv};
  const uint64_t sb[3] = {(uint64_t)a.Hkv * a.D * 2, 128, (uint64_t)a.D * 2};
  const uint32_t bk[4] = {64, KBR / 2, 2, 1};
  const uint32_t bv[4] = {64, KBR, 1, 1};
  // Query rows as {64 columns, head, batch*rows, half}: a {64, G, JBQ, 1}
  // box is one half of the rows (j, g) of a CTA, in order j*G + g.
  const uint64_t dq[4] = {64, (uint64_t)a.Hq, (uint64_t)a.B * a.R, 2};
  const uint64_t sq[3] = {(uint64_t)a.D * 2, (uint64_t)a.Hq * a.D * 2, 128};
  const uint32_t bq[4] = {64, (uint32_t)G, (uint32_t)pl.jbq, 1};
  if (!encode_tensor_map_bf16(&maps[0], a.k_pages, 3, dp, sp, bp) ||
      !encode_tensor_map_bf16(&maps[1], a.v_pages, 3, dp, sp, bp) ||
      !encode_tensor_map_bf16(&maps[2], a.k_blk, 4, db, sb, bk) ||
      !encode_tensor_map_bf16(&maps[3], a.v_blk, 4, db, sb, bv) ||
      !encode_tensor_map_bf16(&maps[4], a.q, 4, dq, sq, bq))
    return cudaErrorInvalidValue;
  TcpParams p{};
  p.page_table = a.page_table;
  p.ctx_len = a.ctx_len;
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
  const cudaError_t e = ensure_kernel_limits((const void*)verify_attn_tcp_kernel, tcp_limits(), TP_SMEM, true);
  if (e != cudaSuccess) return e;
  // one cluster per pair of SMs, or as many more as keep a cluster's list of units short enough
  const long long units = (long long)a.B * a.Hkv * pl.rg, least = (units + TP_MAXU - 1) / TP_MAXU;
  const long long fit = units < pl.resident ? units : pl.resident;
  const long long clusters = fit > least ? fit : least;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = tcp_config(attr, (int)clusters, stream);
  return cudaLaunchKernelEx(&cfg, verify_attn_tcp_kernel, maps[0], maps[1], maps[2], maps[3], maps[4], p);
}

}  // namespace cospec
