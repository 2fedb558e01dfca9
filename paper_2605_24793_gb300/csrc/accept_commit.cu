// Accepted length, emitted tokens (Sec. 3.3 Eq. 15; App. F, Inference
// Procedure) and the commit of the accepted rows' K/V into the paged cache.
//
// One kernel, a thread-block cluster of up to eight CTAs per sequence.  A rejected
// mismatch is Delta_i = 0 and a_i = 0; s = position of the first one (ballot +
// ffs), else K+1.  The cluster's CTAs take the layers in turn and copy block
// rows 0..s-1 of the staging K and V into cache positions C..C+s-1 (C = ctx_len
// before the round) with 16-byte loads and stores, four of each tensor in
// flight per thread; CTA 0 emits y_hat_1..y_hat_{s-1}, y_tilde_s and advances
// ctx_len by s once every CTA of the cluster has read it.
//
// Bound: latency at small batches (one launch, two dependent loads, the copy), HBM
// at large ones.
// Measured (GB300, cold, batch 16, 32 layers): a commit kernel of one CTA per (layer,
// sequence) and a scan kernel after it 10.5 + 3.6 us; this one launch 10.1 us.
#include "cospec_device.cuh"
#include "cospec_internal.h"

namespace cospec {

namespace {

constexpr int CT = 512;              // threads
constexpr int MAX_CLUSTER = 8;       // CTAs per sequence
constexpr int UNROLL = 4;
constexpr int MAX_SPAN = 3;          // pages that 32 rows can touch

__global__ void __launch_bounds__(CT)
    accept_commit_kernel(const CommitArgs a, int capacity, int* err) {
  __shared__ int s_len, s_ctx;
  __shared__ int s_page[MAX_SPAN];
  const int b = blockIdx.y, rank = blockIdx.x, nrank = gridDim.x;
  const int K = a.K, R = K + 1;
  const int tid = threadIdx.x, lane = tid & 31;
  griddep_wait();
  griddep_launch_dependents();
  int dft = 0, tgt = 0, s = 0;
  if (tid < 32) {
    const int C = a.ctx_len[b];
    const bool act = lane < K;
    dft = act ? a.draft[(size_t)b * K + lane] : 0;
    tgt = lane < R ? a.argmax[(size_t)b * R + lane] : 0;
    const bool rejected = act && dft != tgt && a.accept[(size_t)b * K + lane] == 0;
    const unsigned rej = __ballot_sync(0xffffffffu, rejected);
    s = rej ? __ffs(rej) : R;                // 1-based position of the first rejection
    const bool fits = C >= 0 && C + s <= capacity;
    if (lane == 0) {
      s_len = s;
      s_ctx = fits ? C : -1;                 // -1: nothing is committed (flagged by CTA 0)
      if (rank == 0 && !fits) set_err(err, ERR_CTX);
    }
    if (fits && a.L > 0 && lane < MAX_SPAN) {
      const int pg = C / a.P + lane;
      s_page[lane] = pg * a.P < C + s ? a.page_table[(size_t)b * a.max_pages + pg] : 0;
    }
  }
  __syncthreads();
  if (nrank > 1) cluster_arrive();           // this CTA has read ctx_len
  if (rank == 0 && tid < 32) {
    if (lane < R) a.emitted[(size_t)b * R + lane] = lane < s - 1 ? dft : lane == s - 1 ? tgt : -1;
    if (lane == 0) a.accept_len[b] = s;
  }
  const int C = s_ctx, n_rows = s_len;
  if (C >= 0) {
    const unsigned chunks = (unsigned)a.D / 8;                   // 16-byte chunks per (row, head)
    const unsigned per_row = (unsigned)a.Hkv * chunks, per_layer = (unsigned)n_rows * per_row;
    const unsigned layers = rank < a.L ? (unsigned)((a.L - rank + nrank - 1) / nrank) : 0u;
    const int off0 = C % a.P;
    // (the layers in blocks whose chunks count in 32 bits)
    const unsigned lblk = max(1u, (1u << 24) / per_layer);
    for (unsigned l0 = 0; l0 < layers; l0 += lblk) {
      const unsigned total = min(lblk, layers - l0) * per_layer;
      for (unsigned e0 = tid; e0 < total; e0 += CT * UNROLL) {
        uint4 kv[UNROLL], vv[UNROLL];
        size_t dst[UNROLL];
        bool ok[UNROLL];
#pragma unroll
        for (int i = 0; i < UNROLL; ++i) {
          const unsigned e = e0 + i * CT;
          ok[i] = e < total;
          if (!ok[i]) continue;
          const unsigned li = l0 + e / per_layer, rem = e % per_layer;
          const unsigned t = rem / per_row, x = rem % per_row, h = x / chunks, c = x % chunks;
          const int l = rank + (int)li * nrank;
          const int slot = off0 + (int)t;
          const int page = s_page[slot / a.P];
          if ((unsigned)page >= (unsigned)a.num_pages) {
            if (c == 0) set_err(err, ERR_PAGE);
            ok[i] = false;
            continue;
          }
          const size_t src = ((((size_t)l * a.B + b) * R + t) * a.Hkv + h) * a.D + (size_t)c * 8;
          dst[i] = (size_t)l * a.pool_layer_stride +
                   (((size_t)page * a.Hkv + h) * a.P + (slot % a.P)) * a.D + (size_t)c * 8;
          kv[i] = __ldg(reinterpret_cast<const uint4*>(a.k_blk + src));
          vv[i] = __ldg(reinterpret_cast<const uint4*>(a.v_blk + src));
        }
#pragma unroll
        for (int i = 0; i < UNROLL; ++i)
          if (ok[i]) {
            *reinterpret_cast<uint4*>(a.k_pages + dst[i]) = kv[i];
            *reinterpret_cast<uint4*>(a.v_pages + dst[i]) = vv[i];
          }
      }
    }
  }
  __syncwarp();
  if (nrank > 1) cluster_wait();
  if (rank == 0 && tid == 0 && C >= 0) a.ctx_len[b] = C + n_rows;
}

}  // namespace

cudaError_t launch_accept_commit(const CommitArgs& a, int* err, cudaStream_t stream) {
  if (a.B == 0) return cudaSuccess;
  const int capacity = a.max_pages * a.P;
  const int nrank = a.L < 1 ? 1 : a.L < MAX_CLUSTER ? a.L : MAX_CLUSTER;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nrank, a.B);
  cfg.blockDim = dim3(CT);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = nrank;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = nrank > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, accept_commit_kernel, a, capacity, err);
}

}  // namespace cospec
