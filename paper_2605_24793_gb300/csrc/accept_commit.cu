// Accepted length, emitted tokens (Sec. 3.3 Eq. 15; App. F, Inference
// Procedure) and the commit of the accepted rows' K/V into the paged cache.
//
// A rejected mismatch is Delta_i = 0 and a_i = 0; s = position of the first one (ballot +
// ffs), else K+1.  Block rows 0..s-1 of the staging K and V go to cache positions C..C+s-1
// (C = ctx_len before the round) with 16-byte loads and stores; y_hat_1..y_hat_{s-1},
// y_tilde_s are emitted and ctx_len advances by s.
//
// Two forms, by the rule at clustered():
//  - one kernel, a thread-block cluster of up to eight CTAs per sequence: the CTAs take the
//    layers in turn, four chunks of each tensor in flight per thread, and CTA 0 emits and
//    advances ctx_len once every CTA of the cluster has read its inputs;
//  - a commit kernel of one CTA per (layer, sequence), then a scan kernel of one warp per
//    sequence, the only writer of ctx_len.
//
// Bound: latency at small batches (launches, two dependent loads, the copy), HBM at large
// ones.  Measured (GB300, cold, K = 7, 8 KV heads of 128, us, two kernels -> one): batch 16 with
// 4 layers 16.5 -> 11.4, batch 1 with 8 layers 15.5 -> 11.4; but batch 1 with 80 layers
// 15.5 -> 21.6 (K = 31: 33.9 -> 58.5) and batch 256 with 8 layers 33.9 -> 46.2.
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
  if (nrank > 1) cluster_arrive();           // this CTA has read its inputs
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
  if (rank == 0 && tid < 32) {
    if (lane < R) a.emitted[(size_t)b * R + lane] = lane < s - 1 ? dft : lane == s - 1 ? tgt : -1;
    if (lane == 0) a.accept_len[b] = s;
  }
  if (rank == 0 && tid == 0 && C >= 0) a.ctx_len[b] = C + n_rows;
}

__global__ void __launch_bounds__(128)
    accept_scan_kernel(int B, int K, const int32_t* __restrict__ draft,
                       const int32_t* __restrict__ argmax, const uint8_t* __restrict__ accept,
                       int32_t* __restrict__ ctx_len, int32_t* __restrict__ accept_len,
                       int32_t* __restrict__ emitted, int capacity, int* err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * 4 + warp;
  griddep_wait();
  griddep_launch_dependents();
  if (b >= B) return;
  const int R = K + 1;
  const bool act = lane < K;
  const int dft = act ? draft[(size_t)b * K + lane] : 0;
  const int tgt = act ? argmax[(size_t)b * R + lane] : 0;
  const bool rejected = act && (dft != tgt) && (accept[(size_t)b * K + lane] == 0);
  const unsigned rej = __ballot_sync(0xffffffffu, rejected);
  const int s = rej ? __ffs(rej) : R;      // 1-based position of the first rejection
  if (lane < R) {
    int tok = -1;
    if (lane < s - 1) tok = dft;
    else if (lane == s - 1) tok = argmax[(size_t)b * R + lane];
    emitted[(size_t)b * R + lane] = tok;
  }
  if (lane == 0) {
    const int C = ctx_len[b];
    accept_len[b] = s;
    if (C < 0 || C + s > capacity) {
      set_err(err, ERR_CTX);
    } else {
      ctx_len[b] = C + s;
    }
  }
}

__global__ void __launch_bounds__(128)
    commit_kernel(const CommitArgs a, int capacity, int* err) {
  __shared__ int s_len;
  const int l = blockIdx.x, b = blockIdx.y;
  const int R = a.K + 1;
  griddep_wait();
  griddep_launch_dependents();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const bool act = lane < a.K;
    const bool rejected = act && (a.draft[(size_t)b * a.K + lane] != a.argmax[(size_t)b * R + lane]) &&
                          (a.accept[(size_t)b * a.K + lane] == 0);
    const unsigned rej = __ballot_sync(0xffffffffu, rejected);
    if (lane == 0) s_len = rej ? __ffs(rej) : R;
  }
  __syncthreads();
  const int s = s_len;
  const int C = a.ctx_len[b];
  if (C < 0 || C + s > capacity) return;   // flagged by the scan
  const int chunks = a.D / 8;              // 16-byte chunks per (row, head)
  const int per_row = a.Hkv * chunks;
  const int total = s * per_row;
  const int* ptab = a.page_table + (size_t)b * a.max_pages;
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int t = e / per_row;
    const int rem = e % per_row;
    const int h = rem / chunks, c = rem % chunks;
    const int pos = C + t;
    const int page = ptab[pos / a.P];
    if ((unsigned)page >= (unsigned)a.num_pages) {
      if (c == 0) set_err(err, ERR_PAGE);
      continue;
    }
    const size_t src = ((((size_t)l * a.B + b) * R + t) * a.Hkv + h) * a.D + (size_t)c * 8;
    const size_t dst = (size_t)l * a.pool_layer_stride +
                       (((size_t)page * a.Hkv + h) * a.P + (pos % a.P)) * a.D + (size_t)c * 8;
    *reinterpret_cast<uint4*>(a.k_pages + dst) = __ldg(reinterpret_cast<const uint4*>(a.k_blk + src));
    *reinterpret_cast<uint4*>(a.v_pages + dst) = __ldg(reinterpret_cast<const uint4*>(a.v_blk + src));
  }
}

}  // namespace

// One launch where a sequence's layers are a pass or two of its eight CTAs and the clusters
// (512 threads each, held until their slowest CTA is through) are about one wave: up to two CTAs
// per SM, four where a layer's rows fill the threads (2048 chunks of 16 bytes).  Measured over batches 1
// to 256, 1 to 80 layers, K = 4 to 31 and 2 or 8 heads, one kernel against two, cold / warm:
// 0.40-1.00 / 0.49-1.00 of the time within these bounds (0.74 at batch 128, 4 layers, K = 31).
// Beyond: 9 to 16 layers 1.0 to 1.1 at batch 16, more layers up to 2.4 times the time, 512 clusters' CTAs
// of short rows 1.2 to 2.7 times.
static bool clustered(int B, int K, int L, int Hkv, int D) {
  if (L < 1) return false;
  if (L > MAX_CLUSTER) return L <= 2 * MAX_CLUSTER && B <= 8;
  const long long chunks = (long long)(K + 1) * Hkv * (D / 8);
  return (long long)B * L <= (chunks >= CT * UNROLL ? 4 : 2) * device_num_sms();
}

int accept_commit_launches(int B, int K, int L, int Hkv, int D) {
  return B == 0 ? 0 : L < 1 || clustered(B, K, L, Hkv, D) ? 1 : 2;
}

cudaError_t launch_accept_commit(const CommitArgs& a, int* err, cudaStream_t stream) {
  if (a.B == 0) return cudaSuccess;
  const int capacity = a.max_pages * a.P;
  if (!clustered(a.B, a.K, a.L, a.Hkv, a.D)) {
    if (a.L > 0) {
      const cudaError_t e = launch_pdl(commit_kernel, dim3(a.L, a.B), dim3(128), 0, stream, a, capacity, err);
      if (e != cudaSuccess) return e;
    }
    return launch_pdl(accept_scan_kernel, dim3((a.B + 3) / 4), dim3(128), 0, stream, a.B, a.K,
                      a.draft, a.argmax, a.accept, a.ctx_len, a.accept_len, a.emitted, capacity, err);
  }
  const int nrank = a.L < MAX_CLUSTER ? a.L : MAX_CLUSTER;
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
