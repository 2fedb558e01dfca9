// RL stage of CoSpec (Sec. 3.4): per-decision shaped rewards, rollout
// returns, rebalanced group-normalised advantages, per-decision advantages
// and the clipped objective with its entropy and KL terms.
//
// One CTA of 16 warps (4 for many small groups) per prompt group.  The call is bound by memory (27
// bytes per decision with the objective) as long as two things stay off its
// path: uncoalesced access and 64-bit arithmetic, of which an SM issues only
// about two multiply-adds per clock.  So
//  - a CTA works on tiles of a round per thread.  A thread takes its round to find s,
//    i* and the effective set (its K flags become bit masks, four flags per
//    instruction), and the tile's decisions are then walked in memory order, so
//    every large access is a run of consecutive addresses;
//  - per-position values stay in 32 bits where that is exact (g, rho) and in
//    pairs of 32-bit floats (about 2^-46 relative) where the result needs more:
//    the decision advantages, and the logarithms, products and sums of the entropy
//    and the KL divergence; a round's share of the return and the sums of these are
//    in 64 bits (a few operations per round: returns that differ in their last bits alone
//    decide a standardisation whose sigma is as small);
//  - the effective decisions (a fifth of all positions) are compacted through
//    a per-warp queue, so that the objective's arithmetic runs on full warps;
//  - inputs outside the range where the pairs hold (infinities, NaN, huge or
//    tiny values, a probability of exactly 0 or 1 in the reference policy)
//    take the same formulas in 64 bits.
// Warp 0 forms the group statistics in 64 bits between the two passes (so
// that the standardisation of nearly equal returns is not decided by 32-bit
// rounding).  Every sum has a fixed order: repeated calls agree bit for bit.
// Per-group partial sums of the objective go to the workspace and a one-CTA
// kernel adds them in a fixed order.
// Measured (GB300, 256 prompts x 8 rollouts of up to 64 rounds at K = 25, 1.66 M
// decisions with the objective; time of the call's kernels): a lane per round
// walking its K bytes, everything in 64 bits, 790 us; a warp per round with
// ballots and pairs 95-107 us; this split 49.5 us (0.9 TB/s, instruction-bound:
// about 330 warp instructions a round).  The call's host side takes 47 us.
#include <math.h>

#include "../../include/cospec.h"
#include "cospec_device.cuh"
#include "cospec_internal.h"

namespace cospec {

namespace {

constexpr int RL_LOSS_THREADS = 256;

struct RLArgs {
  int num_groups, num_rollouts, num_rounds, K;
  const int32_t* group_off;
  const uint8_t* correct;
  const int32_t* round_off;
  const uint8_t* match;
  const uint8_t* accept;
  const float* ell;
  cospec_rl_params prm;
  const float* ratio;
  const float* p_new;
  const float* p_ref;
  float* g;
  uint8_t* eff;
  float* rho;
  float* J;
  float* Jbar;
  float* adv;
  float* adv_dec;
  double* ws_j;      // [num_rollouts] returns
  double* ws_abs;    // [num_rollouts] sum |g| of each rollout, then the factor of its decisions' advantages
  float2* ws_c;      // [num_rollouts] ws_abs once it holds the decisions' factor, as a pair
  double* part;      // [num_groups][3] objective partial sums
  int* err;
};


CS_DEV double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------- pairs of floats
// An unevaluated sum h + l with |l| <= ulp(h) / 2 (Dekker 1971; Knuth's
// two-sum): about 2^-46 relative, in 32-bit instructions.
struct F2 {
  float h, l;
};

CS_DEV F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return F2{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
CS_DEV F2 quick_two_sum(float a, float b) {          // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return F2{s, __fsub_rn(b, __fsub_rn(s, a))};
}
CS_DEV F2 two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return F2{p, __fmaf_rn(a, b, -p)};
}
CS_DEV F2 add(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h), t = two_sum(a.l, b.l);
  const F2 u = quick_two_sum(s.h, __fadd_rn(s.l, t.h));
  return quick_two_sum(u.h, __fadd_rn(u.l, t.l));
}
CS_DEV F2 neg(F2 a) { return F2{-a.h, -a.l}; }
CS_DEV F2 mul(F2 a, F2 b) {
  const F2 p = two_prod(a.h, b.h);
  return quick_two_sum(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}
CS_DEV F2 mul(float a, F2 b) {
  const F2 p = two_prod(a, b.h);
  return quick_two_sum(p.h, __fmaf_rn(a, b.l, p.l));
}
// (a.h + a.l) / (b.h + b.l) by two quotient digits
CS_DEV F2 div(F2 a, F2 b) {
  const float q1 = __fdividef(a.h, b.h);
  const F2 r = add(a, neg(mul(q1, b)));
  const float q2 = __fdividef(r.h, b.h);
  const F2 r2 = add(r, neg(mul(q2, b)));
  const F2 q = quick_two_sum(q1, q2);
  return quick_two_sum(q.h, __fadd_rn(q.l, __fdividef(r2.h, b.h)));
}
CS_DEV double to_double(F2 a) { return (double)a.h + (double)a.l; }
CS_DEV F2 warp_sum(F2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = add(v, F2{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
  return v;
}

// log of a normal positive float as a pair, by table (Tang, ACM TOMS 1990): x = 2^e m with m in
// [0.707, 1.414), inv ~ 1 / m a multiple of 2^-8, r = m inv - 1 with |r| <= 2^-7 (25 bits: a pair),
//   log x = e log 2 - log inv + log(1 + r),   log(1 + r) = r - r^2/2 + r^3 (1/3 - r/4 + ...).
// Around m = 1 inv is 1, so log(1 + r) keeps its relative accuracy there.
// Entry j - 90 (j = floor(128 m)): inv, -log inv in two parts.
__device__ const float RL_LOG_TAB[91][3] = {
    {1.4140625f, -0x1.62c830p-2f, 0x1.a8c70ep-27f}, {1.3984375f, -0x1.576772p-2f, 0x1.1754b2p-27f},
    {1.3828125f, -0x1.4be5fap-2f, 0x1.5110ecp-27f}, {1.3671875f, -0x1.404308p-2f, -0x1.a1a9f8p-28f},
    {1.35546875f, -0x1.377266p-2f, -0x1.5fec2ep-29f}, {1.33984375f, -0x1.2b9304p-2f, 0x1.51d8b6p-28f},
    {1.328125f, -0x1.229420p-2f, 0x1.0c21a6p-28f}, {1.3125f, -0x1.1675cap-2f, -0x1.7574c2p-27f},
    {1.30078125f, -0x1.0d46b6p-2f, 0x1.0ca916p-27f}, {1.28515625f, -0x1.00e6c4p-2f, -0x1.6b5408p-28f},
    {1.2734375f, -0x1.ef0adcp-3f, -0x1.7b8b26p-28f}, {1.26171875f, -0x1.dc1bcap-3f, -0x1.57d8fap-32f},
    {1.25f, -0x1.c8ff7cp-3f, -0x1.e6a688p-29f}, {1.23828125f, -0x1.b5b51ap-3f, 0x1.704a5cp-31f},
    {1.2265625f, -0x1.a23bc2p-3f, 0x1.d4a9cep-35f}, {1.21484375f, -0x1.8e928ep-3f, 0x1.7792c0p-31f},
    {1.203125f, -0x1.7ab890p-3f, -0x1.086c84p-30f}, {1.19140625f, -0x1.66acd4p-3f, -0x1.3956a8p-30f},
    {1.1796875f, -0x1.526e5ep-3f, -0x1.d0da1cp-30f}, {1.16796875f, -0x1.3dfc2cp-3f, 0x1.e2673ap-28f},
    {1.16015625f, -0x1.303d72p-3f, 0x1.c6e00cp-29f}, {1.1484375f, -0x1.1b72aep-3f, 0x1.5a130cp-28f},
    {1.13671875f, -0x1.067152p-3f, 0x1.a6b4d2p-28f}, {1.12890625f, -0x1.f0a30cp-4f, -0x1.162a66p-36f},
    {1.1171875f, -0x1.c5e548p-4f, -0x1.eb78e8p-29f}, {1.109375f, -0x1.a926d4p-4f, 0x1.6d4aa8p-30f},
    {1.09765625f, -0x1.7da766p-4f, -0x1.af625ap-29f}, {1.08984375f, -0x1.60658ap-4f, -0x1.26ea18p-29f},
    {1.08203125f, -0x1.42edccp-4f, 0x1.59b910p-32f}, {1.0703125f, -0x1.16536ep-4f, -0x1.d46f5cp-29f},
    {1.0625f, -0x1.f0a30cp-5f, -0x1.162a66p-37f}, {1.0546875f, -0x1.b42dd8p-5f, 0x1.dcd1c8p-30f},
    {1.04296875f, -0x1.58a5bap-5f, -0x1.f91c9ap-30f}, {1.03515625f, -0x1.1b0d98p-5f, -0x1.247b30p-30f},
    {1.02734375f, -0x1.b9fc02p-6f, -0x1.ebe466p-32f}, {1.01953125f, -0x1.3cea44p-6f, -0x1.a352bap-33f},
    {1.01171875f, -0x1.7dc476p-7f, 0x1.fbd624p-37f}, {1.0f, 0x0.0p+0f, 0x0.0p+0f},
    {1.0f, 0x0.0p+0f, 0x0.0p+0f}, {0.98828125f, 0x1.82448ap-7f, 0x1.c45156p-34f},
    {0.98046875f, 0x1.432a92p-6f, 0x1.660330p-32f}, {0.97265625f, 0x1.c63d2ep-6f, 0x1.82955ep-31f},
    {0.96484375f, 0x1.252f32p-5f, 0x1.f1a308p-30f}, {0.95703125f, 0x1.67c950p-5f, -0x1.a56894p-30f},
    {0.953125f, 0x1.894aa2p-5f, -0x1.6c0998p-30f}, {0.9453125f, 0x1.ccb73cp-5f, 0x1.bbb65ap-30f},
    {0.9375f, 0x1.08598cp-4f, -0x1.4c38c0p-29f}, {0.9296875f, 0x1.2aa04ap-4f, 0x1.11c5eap-30f},
    {0.92578125f, 0x1.3bdf5ap-4f, 0x1.f47b9ap-30f}, {0.91796875f, 0x1.5e95a4p-4f, 0x1.b2f23ap-29f},
    {0.91015625f, 0x1.8197e2p-4f, 0x1.e81c7ep-29f}, {0.90625f, 0x1.9335e6p-4f, -0x1.535b3cp-31f},
    {0.8984375f, 0x1.b6ac88p-4f, 0x1.b5ab64p-29f}, {0.890625f, 0x1.da7276p-4f, 0x1.c22352p-31f},
    {0.88671875f, 0x1.ec7398p-4f, 0x1.850890p-31f}, {0.87890625f, 0x1.08598cp-3f, -0x1.4c38c0p-28f},
    {0.875f, 0x1.1178e8p-3f, 0x1.13f23ep-30f}, {0.8671875f, 0x1.23d712p-3f, 0x1.493840p-28f},
    {0.86328125f, 0x1.2d1610p-3f, 0x1.90d028p-28f}, {0.85546875f, 0x1.3fb45ap-3f, 0x1.664a32p-29f},
    {0.8515625f, 0x1.4913d8p-3f, 0x1.99dab0p-30f}, {0.84375f, 0x1.5bf406p-3f, 0x1.6a87b6p-28f},
    {0.83984375f, 0x1.6574ecp-3f, -0x1.73ecc6p-31f}, {0.83203125f, 0x1.7898d8p-3f, 0x1.51131cp-29f},
    {0.828125f, 0x1.823c16p-3f, 0x1.5468f0p-29f}, {0.82421875f, 0x1.8beafep-3f, 0x1.671fd2p-28f},
    {0.81640625f, 0x1.9f6c40p-3f, 0x1.c2259ap-29f}, {0.8125f, 0x1.a93ed4p-3f, -0x1.ba930ep-30f},
    {0.80859375f, 0x1.b31d86p-3f, -0x1.148638p-28f}, {0.80078125f, 0x1.c6ffbcp-3f, 0x1.bc03dcp-29f},
    {0.796875f, 0x1.d10380p-3f, -0x1.b35430p-28f}, {0.79296875f, 0x1.db13dcp-3f, -0x1.e56ed8p-28f},
    {0.7890625f, 0x1.e530f0p-3f, -0x1.8efedep-35f}, {0.78125f, 0x1.f991c6p-3f, 0x1.967670p-28f},
    {0.77734375f, 0x1.01eae6p-2f, -0x1.3b272ep-27f}, {0.7734375f, 0x1.071386p-2f, 0x1.35618ap-32f},
    {0.76953125f, 0x1.0c42d6p-2f, 0x1.d858b8p-28f}, {0.765625f, 0x1.1178e8p-2f, 0x1.13f23ep-29f},
    {0.7578125f, 0x1.1bf996p-2f, 0x1.ad35cap-29f}, {0.75390625f, 0x1.214456p-2f, 0x1.a1d71ap-27f},
    {0.75f, 0x1.269622p-2f, -0x1.d9648ep-27f}, {0.74609375f, 0x1.2bef08p-2f, -0x1.91b656p-29f},
    {0.7421875f, 0x1.314f1ep-2f, 0x1.d35ce4p-30f}, {0.73828125f, 0x1.36b678p-2f, -0x1.283ddep-27f},
    {0.734375f, 0x1.3c2528p-2f, -0x1.1999d0p-27f}, {0.73046875f, 0x1.419b42p-2f, 0x1.eaf464p-29f},
    {0.7265625f, 0x1.4718dcp-2f, 0x1.38e20ep-29f}, {0.72265625f, 0x1.4c9e0ap-2f, -0x1.e8d3c4p-30f},
    {0.71875f, 0x1.522ae0p-2f, 0x1.ce28f6p-28f}, {0.71484375f, 0x1.57bf76p-2f, -0x1.86e5c0p-27f},
    {0.7109375f, 0x1.5d5bdep-2f, -0x1.4d41a0p-31f},};

CS_DEV F2 log1p_small(F2 r) {            // |r| <= 2^-6: the series to r^9
  const F2 q = two_prod(r.h, r.h);
  float c = 0.11111111f;
  c = fmaf(c, r.h, -0.125f);
  c = fmaf(c, r.h, 0.14285714f);
  c = fmaf(c, r.h, -0.16666667f);
  c = fmaf(c, r.h, 0.2f);
  c = fmaf(c, r.h, -0.25f);
  c = fmaf(c, r.h, 0.33333333f);
  const F2 s = two_sum(r.h, -0.5f * q.h);
  // the parts below: r.l (1 - r), the square's rounding, the cubic and up
  float lo = fmaf(-r.h, r.l, r.l);
  lo = fmaf(-0.5f, q.l, lo);
  const F2 t = two_sum(s.l, __fmul_rn(__fmul_rn(r.h, q.h), c));
  const F2 u = quick_two_sum(s.h, t.h);
  return quick_two_sum(u.h, __fadd_rn(u.l, __fadd_rn(t.l, lo)));
}

CS_DEV F2 log_pair(float x, const float (*tab)[3]) {
  const int bits = __float_as_int(x);
  int e = (bits >> 23) - 127;
  float m = __int_as_float((bits & 0x7fffff) | 0x3f800000);
  if (m >= 1.4140625f) {
    m *= 0.5f;
    ++e;
  }
  const float* t = tab[(int)(m * 128.f) - 90];
  const F2 mi = two_prod(m, t[0]);
  const F2 lr = log1p_small(two_sum(__fsub_rn(mi.h, 1.f), mi.l));
  // log 2 in three parts, the first of 16 bits (e times it is exact)
  const float fe = (float)e;
  const F2 b = two_prod(fe, 0x1.7f7d1cp-20f);
  F2 s = add(F2{__fmul_rn(fe, 0x1.62e4p-1f), 0.f}, F2{b.h, fmaf(fe, 0x1.ef357ap-45f, b.l)});
  s = add(s, F2{t[1], t[2]});
  return add(s, lr);
}

struct RLReciprocals {
  double v[65];
  constexpr RLReciprocals() : v{} {
    for (int i = 1; i <= 64; ++i) v[i] = 1.0 / i;
  }
};
__device__ const RLReciprocals RL_RCP;   // 1 / i

CS_DEV double bern_entropy(double p) {
  double h = 0.0;
  if (p > 0.0) h -= p * log(p);
  if (p < 1.0) h -= (1.0 - p) * log(1.0 - p);
  return h;
}

CS_DEV double bern_kl(double p, double q) {
  double k = 0.0;
  if (p > 0.0) k += p * log(p / q);
  if (p < 1.0) k += (1.0 - p) * log((1.0 - p) / (1.0 - q));
  return k;
}

// ---------------------------------------------------------------- one round
struct RoundMasks {
  unsigned long long eff;    // effective decisions
  unsigned long long acc;    // of these, accepted ones before the first rejection
  int s, istar, n;           // stop position, first mismatch (0: none), number of effective ones
};

CS_DEV RoundMasks rl_masks(unsigned long long mism, unsigned long long zero, unsigned long long one, int K) {
  const unsigned long long rej = mism & zero;
  RoundMasks r;
  r.istar = mism ? __ffsll((long long)mism) : 0;
  r.s = rej ? __ffsll((long long)rej) : K + 1;
  const int last = r.s < K ? r.s : K;                   // 1 .. 64
  r.eff = mism & (~0ull >> (64 - last));
  r.acc = r.eff & one & ~rej;                           // a rejection is the last of eff, if any
  r.n = __popcll(r.eff);
  return r;
}

// Four flag bytes at byte `at` of an array of `total` bytes whose first byte is `skew` bytes past a
// word boundary: from the two words around them, byte by byte at the array's ends.
CS_DEV uint32_t load_flags4(const uint8_t* base, long long at, long long total, uint32_t skew) {
  const uint32_t sh = (uint32_t)(at + skew) & 3u;
  const long long w = at - sh;                          // first byte of the word that holds `at`
  if (w >= 0 && w + 8 <= total) {
    const uint32_t* q = reinterpret_cast<const uint32_t*>(base + w);
    return __funnelshift_r(__ldg(q), __ldg(q + 1), 8 * sh);
  }
  uint32_t v = 0;
  for (int b = 0; b < 4; ++b)
    if (at + b < total) v |= (uint32_t)base[at + b] << (8 * b);
  return v;
}
// Bit j of the result: byte j of v equals b (v's bytes all compared at once).
CS_DEV uint32_t bytes_equal(uint32_t v, uint32_t b) {
  return ((__vcmpeq4(v, b) & 0x08040201u) * 0x01010101u) >> 24;
}

// The objective's terms of one effective decision in 64 bits, for the inputs the pairs do not hold.
__device__ __noinline__ double3 rl_terms64(double A, float rt_, float p_, float q_, double ce) {
  const double rt = (double)rt_;
  const double rc = fmin(fmax(rt, 1.0 - ce), 1.0 + ce);
  return make_double3(fmin(rt * A, rc * A), bern_entropy((double)p_), bern_kl((double)p_, (double)q_));
}

struct RLQueue {             // per warp: effective decisions waiting for the objective
  long long e[64];
  F2 a[64];
};

struct RLSums {              // per lane: pair sums, and the 64-bit sums of the general path
  F2 surr, ent, kl;
  double surr64, ent64, kl64;
  bool wide;
};

CS_DEV void rl_objective64(const RLArgs& a, long long e, double A, RLSums& s) {
  const double3 t = rl_terms64(A, a.ratio[e], a.p_new[e], a.p_ref[e], (double)a.prm.clip_eps);
  s.wide = true;
  s.surr64 += t.x;
  s.ent64 += t.y;
  s.kl64 += t.z;
}

CS_DEV void rl_objective(const RLArgs& a, const float (*tab)[3], long long e, F2 A, RLSums& s) {
  const float rt = a.ratio[e], p = a.p_new[e], q = a.p_ref[e];
  const float ce = a.prm.clip_eps;
  // p_new may be exactly 0 or 1 (a saturated sigmoid): its 0 log 0 terms are 0
  const bool fast = fabsf(rt) < 1e10f && ce < 1e10f && (p == 0.f || p >= 1e-30f) && p <= 1.f &&
                    q >= 1e-30f && q < 1.f;
  if (!fast) {
    rl_objective64(a, e, to_double(A), s);
    return;
  }
  // min(rt A, rc A): A times the smaller of rt and rc, or the larger for A < 0.  The clip bounds
  // 1 -+ ce have more bits than a float: pairs again.
  {
    const F2 lo = two_sum(1.f, -ce), hi = two_sum(1.f, ce);
    const bool below = rt < lo.h || (rt == lo.h && 0.f < lo.l);
    const bool above = rt > hi.h || (rt == hi.h && 0.f > hi.l);
    F2 w{rt, 0.f};
    if (A.h >= 0.f ? above : below) w = above ? hi : lo;
    s.surr = add(s.surr, mul(w, A));
  }
  const F2 p1 = two_sum(1.f, -p), q1 = two_sum(1.f, -q);
  const F2 lp = p > 0.f ? log_pair(p, tab) : F2{0.f, 0.f};
  F2 lp1{0.f, 0.f};
  if (p1.h > 0.f) {
    lp1 = log_pair(p1.h, tab);
    lp1 = add(lp1, F2{__fdividef(p1.l, p1.h), 0.f});
  }
  const F2 pp{p, 0.f};
  s.ent = add(s.ent, neg(add(mul(p, lp), mul(p1, lp1))));
  // KL: log(p / q) from the difference when the two are close, so that the two terms, nearly equal
  // and opposite, cancel without losing the result
  const F2 dp = two_sum(p, -q), q2{q, 0.f};
  const F2 r1 = div(dp, q2), r2 = neg(div(dp, q1));
  F2 l1 = log1p_small(r1), l2 = log1p_small(r2);
  if (fabsf(r1.h) > 0.015625f) l1 = add(lp, neg(log_pair(q, tab)));
  if (fabsf(r2.h) > 0.015625f) {
    l2 = log_pair(q1.h, tab);
    l2 = add(lp1, neg(add(l2, F2{__fdividef(q1.l, q1.h), 0.f})));
  }
  F2 k{0.f, 0.f};
  if (p > 0.f) k = mul(pp, l1);
  if (p1.h > 0.f) k = add(k, mul(p1, l2));
  s.kl = add(s.kl, k);
}

// The rollout that round r belongs to: the last of [ma, mb) that starts at or before it.
CS_DEV int rollout_of(const int32_t* round_off, int ma, int mb, int r) {
  int lo = ma, hi = mb;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(round_off + mid) <= r) lo = mid;
    else hi = mid;
  }
  return lo;
}

template <int RL_THREADS>
__global__ void __launch_bounds__(RL_THREADS, 1024 / RL_THREADS) rl_group_kernel(const RLArgs a) {
  constexpr int RL_WARPS = RL_THREADS / 32;
  constexpr int RL_TILE = RL_THREADS;    // rounds per tile, one per thread
  const int x = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int K = a.K;
  __shared__ unsigned long long s_eff[RL_TILE], s_acc[RL_TILE];
  __shared__ double s_ret[RL_TILE];      // a round's share of the return
  __shared__ F2 s_val[RL_TILE];          // its decisions' factor
  __shared__ float s_rho[RL_TILE];
  __shared__ uint8_t s_stop[RL_TILE];    // s, with bit 7: the rollout is correct
  __shared__ uint8_t s_big[RL_TILE];     // the round's return takes the general path
  __shared__ F2 red[3][RL_WARPS];
  __shared__ double red64[3][RL_WARPS];
  __shared__ float s_tab[91][3];
  __shared__ RLQueue s_queue[RL_WARPS];
  griddep_wait();
  griddep_launch_dependents();
  const int m0 = a.group_off[x], m1 = a.group_off[x + 1];
  if (m0 < 0 || m1 < m0 || m1 > a.num_rollouts) {
    if (tid == 0) {
      set_err(a.err, ERR_OFFSETS);
      if (a.part) a.part[3 * x] = a.part[3 * x + 1] = a.part[3 * x + 2] = 0.0;
    }
    return;
  }
  const int nm = m1 - m0;
  auto bad_rollout = [&](int m) {
    const int r0 = a.round_off[m], r1 = a.round_off[m + 1];
    return r0 < 0 || r1 < r0 || r1 > a.num_rounds;
  };
  bool some_bad = false;
  for (int m = m0 + tid; m < m1; m += RL_THREADS) {
    some_bad |= bad_rollout(m);
    a.ws_j[m] = 0.0;
    a.ws_abs[m] = 0.0;
  }
  if (a.part)
    for (int i = tid; i < 91 * 3; i += RL_THREADS) (&s_tab[0][0])[i] = (&RL_LOG_TAB[0][0])[i];
  some_bad = __syncthreads_or(some_bad) != 0;
  if (some_bad && tid == 0) set_err(a.err, ERR_OFFSETS);
  // The rounds of a group are one run of rounds; with bad offsets among its rollouts, those that are
  // good are taken one by one.
  const int spans = some_bad ? nm : 1;

  const double alpha = (double)a.prm.alpha, beta = (double)a.prm.beta;
  const bool alpha_ok = fabsf(a.prm.alpha) < 1e6f;
  const uint32_t inv_k = K > 1 ? 0xffffffffu / (uint32_t)K + 1u : 0u;      // x / K = hi(x inv_k) for x < 2^16
  const long long total = (long long)a.num_rounds * K;
  const uint32_t skew_m = (uint32_t)reinterpret_cast<uintptr_t>(a.match) & 3u;
  const uint32_t skew_a = (uint32_t)reinterpret_cast<uintptr_t>(a.accept) & 3u;

  // ---- g, eff and rho of every round; returns
  for (int sp = 0; sp < spans && nm > 0; ++sp) {
    const int ma = some_bad ? m0 + sp : m0, mb = some_bad ? ma + 1 : m1;
    if (some_bad && bad_rollout(ma)) continue;
    const int ra = a.round_off[ma], rz = a.round_off[mb];
    for (int t0 = ra; t0 < rz; t0 += RL_TILE) {
      const int nr = min(RL_TILE, rz - t0);
      if (tid < nr) {                    // one round per thread
        const int r = t0 + tid;
        const int m = rollout_of(a.round_off, ma, mb, r);
        const bool corr = a.correct[m] != 0;
        const long long e0 = (long long)r * K;
        unsigned long long mism = 0, zero = 0, one = 0;
#pragma unroll 4
        for (int i = 0; i < K; i += 4) {
          const uint32_t vm = load_flags4(a.match, e0 + i, total, skew_m);
          const uint32_t va = load_flags4(a.accept, e0 + i, total, skew_a);
          mism |= (unsigned long long)bytes_equal(vm, 0u) << i;
          zero |= (unsigned long long)bytes_equal(va, 0u) << i;
          one |= (unsigned long long)bytes_equal(va, 0x01010101u) << i;
        }
        mism &= ~0ull >> (64 - K);
        const RoundMasks k = rl_masks(mism, zero, one, K);
        const int num = k.s - k.istar, den = K + 1 - k.istar;
        // num / den of small whole numbers: the 32-bit quotient is the 64-bit one rounded
        const float rho = k.istar ? __fdiv_rn((float)num, (float)den) : 0.f;
        a.rho[r] = k.istar ? rho : __int_as_float(0x7fc00000);
        // this round's share of the return, to 64 bits: n rho from a table of reciprocals, or the
        // accepted |ell| in three floats (each two-sum's rounding goes into the next)
        double v = 0.0;
        bool big = false;
        if (corr) {
          if (k.istar) v = (double)(k.n * num) * RL_RCP.v[den];
        } else {
          float v0 = 0.f, v1 = 0.f, v2 = 0.f;
          for (unsigned long long left = k.eff; left; left &= left - 1) {
            const int i = __ffsll((long long)left) - 1;
            const float l = fabsf(a.ell[e0 + i]);
            big |= !(alpha_ok && l < 1e20f);
            const F2 t = two_sum(v0, ((k.acc >> i) & 1) ? l : 0.f);
            const F2 u = two_sum(v1, t.l);
            v0 = t.h;
            v1 = u.h;
            v2 += u.l;
          }
          v = (double)v0 + ((double)v1 + (double)v2);
        }
        s_eff[tid] = k.eff;
        s_acc[tid] = k.acc;
        s_rho[tid] = rho;
        s_ret[tid] = v;
        s_stop[tid] = (uint8_t)(k.s | (corr ? 128 : 0));
        s_big[tid] = big;
      }
      __syncthreads();
      // the tile's decisions in memory order
      const int ne = nr * K;
      const long long e0 = (long long)t0 * K;
#pragma unroll 4
      for (int q = tid; q < ne; q += RL_THREADS) {
        const int r = K > 1 ? (int)__umulhi((uint32_t)q, inv_k) : q;
        const int i = q - r * K;
        const bool eff = (s_eff[r] >> i) & 1;
        const int stop = s_stop[r];
        float g = 0.f;
        if (eff) {
          if (stop & 128) {
            g = s_rho[r];
          } else {
            const bool acc = (s_acc[r] >> i) & 1, rj = i + 1 == stop;
            const float l = fabsf(a.ell[e0 + q]);
            if (alpha_ok && l < 1e20f)
              g = __fmul_rn(-a.prm.alpha, l) * (acc ? 1.f : 0.f) - (rj ? a.prm.beta : 0.f);
            else
              g = (float)(-alpha * (double)l * (acc ? 1.0 : 0.0) - beta * (rj ? 1.0 : 0.0));
          }
        }
        a.g[e0 + q] = g;
        a.eff[e0 + q] = eff ? 1 : 0;
      }
      // returns of the rollouts that the tile touches: a warp each, its lanes the rounds
      const int mf = rollout_of(a.round_off, ma, mb, t0), ml = rollout_of(a.round_off, ma, mb, t0 + nr - 1);
      for (int m = mf + warp; m <= ml; m += RL_WARPS) {
        const int b0 = max(a.round_off[m], t0) - t0, b1 = min(a.round_off[m + 1], t0 + nr) - t0;
        const bool corr = a.correct[m] != 0;
        double v = 0.0;
        int rejected = 0;
        bool wide = false;
        double dg = 0.0, da = 0.0;
        for (int r = b0 + lane; r < b1; r += 32) {
          const int stop = s_stop[r] & 127;
          if (!s_big[r]) {
            v += s_ret[r];
            rejected += stop <= K ? 1 : 0;
            continue;
          }
          wide = true;                   // the general path: this round's decisions in 64 bits
          for (unsigned long long left = s_eff[r]; left; left &= left - 1) {
            const int i = __ffsll((long long)left) - 1;
            const double l = fabs((double)a.ell[e0 + (long long)r * K + i]);
            const double gv = -alpha * l * (((s_acc[r] >> i) & 1) ? 1.0 : 0.0) - beta * (i + 1 == stop ? 1.0 : 0.0);
            dg += gv;
            da += fabs(gv);
          }
        }
        v = warp_sum(v);
        rejected = __reduce_add_sync(0xffffffffu, rejected);
        if (__any_sync(0xffffffffu, wide)) {
          dg = warp_sum(dg);
          da = warp_sum(da);
        }
        if (lane == 0) {
          const double s = v, rj = (double)rejected;
          a.ws_j[m] += corr ? s : dg - (alpha * s + beta * rj);
          a.ws_abs[m] += corr ? s : da + (fabs(alpha) * s + fabs(beta) * rj);
        }
      }
      __syncthreads();                   // the next tile rewrites the shared arrays
    }
  }
  __syncthreads();
  // ---- group statistics (warp 0): gamma, Jbar, mean, population sigma, Adv
  if (warp == 0) {
    const double eps = (double)a.prm.eps;
    double pos = 0.0, negabs = 0.0;
    int npos = 0;
    for (int m = m0 + lane; m < m1; m += 32) {
      const double j = a.ws_j[m];
      if (a.correct[m]) {
        pos += j;
        ++npos;
      } else {
        negabs += fabs(j);
      }
    }
    pos = warp_sum(pos);
    negabs = warp_sum(negabs);
    npos = __reduce_add_sync(0xffffffffu, npos);
    const double n = (double)nm;
    const double gamma = (npos > 0 && npos < nm) ? negabs / (pos + eps) : 1.0;
    const double eta = (npos == 0) ? (double)a.prm.eta_fail : 1.0;
    double sum = 0.0;
    for (int m = m0 + lane; m < m1; m += 32) sum += a.correct[m] ? gamma * a.ws_j[m] : a.ws_j[m];
    sum = warp_sum(sum);
    const double mu = nm > 0 ? sum / n : 0.0;
    double var = 0.0;
    for (int m = m0 + lane; m < m1; m += 32) {
      const double jb = a.correct[m] ? gamma * a.ws_j[m] : a.ws_j[m];
      var += (jb - mu) * (jb - mu);
    }
    var = warp_sum(var);
    const double sigma = nm > 0 ? sqrt(var / n) : 0.0;
    for (int m = m0 + lane; m < m1; m += 32) {
      const bool corr = a.correct[m] != 0;
      const double j = a.ws_j[m];
      const double jb = corr ? gamma * j : j;
      const double ad = eta * (jb - mu) / (sigma + eps);
      a.J[m] = (float)j;
      a.Jbar[m] = (float)jb;
      a.adv[m] = (float)ad;
      // a decision's advantage is rho Adv, or |g| (Adv / sum |g|): the factor, in 64 bits and as a
      // pair (NaN where a pair does not hold it)
      const double sabs = a.ws_abs[m];
      const double c = corr ? ad : (sabs > 0.0 ? ad / sabs : 0.0);
      const float ch = (float)c;
      const bool holds = c == 0.0 || (fabsf(ch) > 1e-12f && fabsf(ch) < 1e12f);
      a.ws_abs[m] = c;
      a.ws_c[m] = holds ? make_float2(ch, (float)(c - (double)ch)) : make_float2(__int_as_float(0x7fc00000), 0.f);
    }
  }
  __syncthreads();
  // ---- decision advantages and the objective terms
  RLSums sums{};
  RLQueue& qu = s_queue[warp];
  int queued = 0;
  for (int sp = 0; sp < spans && nm > 0; ++sp) {
    const int ma = some_bad ? m0 + sp : m0, mb = some_bad ? ma + 1 : m1;
    if (some_bad && bad_rollout(ma)) continue;
    const int ra = a.round_off[ma], rz = a.round_off[mb];
    for (int t0 = ra; t0 < rz; t0 += RL_TILE) {
      const int nr = min(RL_TILE, rz - t0);
      if (tid < nr) {
        const int m = rollout_of(a.round_off, ma, mb, t0 + tid);
        const float2 c = a.ws_c[m];
        s_val[tid] = F2{c.x, c.y};
        s_stop[tid] = a.correct[m] != 0 ? 128 : 0;
      }
      __syncthreads();
      const int ne = nr * K;
      const long long e0 = (long long)t0 * K;
      const int nq = (ne + 31) & ~31;    // whole warps walk together (ballots below)
#pragma unroll 2
      for (int q = tid; q < nq; q += RL_THREADS) {
        const bool in = q < ne;
        const int r = K > 1 ? (int)__umulhi((uint32_t)q, inv_k) : q;
        const bool eff = in && a.eff[e0 + q] != 0;
        F2 A{0.f, 0.f};
        bool put = false;
        if (eff) {
          const F2 c = s_val[r];
          const float g = a.g[e0 + q];                      // a correct rollout's g is its rho
          const float w = (s_stop[r] & 128) ? g : fabsf(g);
          put = c.h == c.h && (w == 0.f || (w > 1e-12f && w < 1e12f));
          if (put) {
            A = mul(w, c);
          } else {               // the general path: in 64 bits, its objective terms at once
            const double c64 = a.ws_abs[rollout_of(a.round_off, ma, mb, t0 + r)];
            const double A64 = c64 == 0.0 ? 0.0 : (double)w * c64;
            A.h = (float)A64;
            if (a.ratio) rl_objective64(a, e0 + q, A64, sums);
          }
        }
        if (in) a.adv_dec[e0 + q] = A.h;
        if (a.ratio) {
          const unsigned b = __ballot_sync(0xffffffffu, put);
          if (put) {
            const int at = queued + __popc(b & ((1u << lane) - 1u));
            qu.e[at] = e0 + q;
            qu.a[at] = A;
          }
          queued += __popc(b);
          __syncwarp();
          if (queued >= 32) {            // a full warp of effective decisions
            rl_objective(a, s_tab, qu.e[lane], qu.a[lane], sums);
            const int rest = queued - 32;
            long long e2 = 0;
            F2 a2{0.f, 0.f};
            if (lane < rest) {
              e2 = qu.e[32 + lane];
              a2 = qu.a[32 + lane];
            }
            __syncwarp();
            if (lane < rest) {
              qu.e[lane] = e2;
              qu.a[lane] = a2;
            }
            __syncwarp();
            queued = rest;
          }
        }
      }
      __syncthreads();
    }
  }
  if (a.part) {
    if (lane < queued) rl_objective(a, s_tab, qu.e[lane], qu.a[lane], sums);
    const F2 surr = warp_sum(sums.surr), ent = warp_sum(sums.ent), kl = warp_sum(sums.kl);
    const bool wide = __any_sync(0xffffffffu, sums.wide);
    if (wide) {
      sums.surr64 = warp_sum(sums.surr64);
      sums.ent64 = warp_sum(sums.ent64);
      sums.kl64 = warp_sum(sums.kl64);
    }
    if (lane == 0) {
      red[0][warp] = surr;
      red[1][warp] = ent;
      red[2][warp] = kl;
      red64[0][warp] = sums.surr64;
      red64[1][warp] = sums.ent64;
      red64[2][warp] = sums.kl64;
    }
    const bool any_wide = __syncthreads_or(wide) != 0;
    if (tid < 3) {
      F2 t{0.f, 0.f};
      double t64 = 0.0;
      for (int w = 0; w < RL_WARPS; ++w) t = add(t, red[tid][w]);
      if (any_wide)
        for (int w = 0; w < RL_WARPS; ++w) t64 += red64[tid][w];
      a.part[3 * x + tid] = t64 + to_double(t);
    }
  }
}

// Sum of the per-group partials in a fixed order; loss[3] is the objective.
__global__ void __launch_bounds__(RL_LOSS_THREADS) rl_loss_kernel(const double* part, int num_groups,
                                                             cospec_rl_params prm, float* loss) {
  __shared__ double acc[3][RL_LOSS_THREADS];
  griddep_wait();
  griddep_launch_dependents();
  double t[3] = {0.0, 0.0, 0.0};
  for (int x = threadIdx.x; x < num_groups; x += RL_LOSS_THREADS)
    for (int c = 0; c < 3; ++c) t[c] += part[3 * x + c];
  for (int c = 0; c < 3; ++c) acc[c][threadIdx.x] = t[c];
  __syncthreads();
  for (int s = RL_LOSS_THREADS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int c = 0; c < 3; ++c) acc[c][threadIdx.x] += acc[c][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    loss[0] = (float)acc[0][0];
    loss[1] = (float)acc[1][0];
    loss[2] = (float)acc[2][0];
    loss[3] = (float)(-acc[0][0] - (double)prm.beta_h * acc[1][0] + (double)prm.beta_kl * acc[2][0]);
  }
}

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

}  // namespace

}  // namespace cospec

extern "C" COSPEC_API size_t cospec_rl_workspace(int num_groups, int num_rollouts) {
  using namespace cospec;
  if (num_groups < 0 || num_rollouts < 0) return 0;
  return 3 * align256((size_t)num_rollouts * sizeof(double)) +
         align256((size_t)num_groups * 3 * sizeof(double)) + 256;
}

extern "C" COSPEC_API int cospec_rl_advantages(
    int num_groups, int num_rollouts, int num_rounds, int K, const int32_t* group_off,
    const uint8_t* correct, const int32_t* round_off, const uint8_t* match, const uint8_t* accept,
    const float* ell, const cospec_rl_params* params, const float* ratio, const float* p_new,
    const float* p_ref, float* g, uint8_t* eff, float* rho, float* J, float* Jbar, float* adv,
    float* adv_dec, float* loss, void* ws, size_t ws_bytes, void* stream) {
  using namespace cospec;
  if (num_groups < 0 || num_rollouts < 0 || num_rounds < 0 || K < 1 || K > 64 || !params)
    return COSPEC_ERR_INVALID_ARG;
  const cospec_rl_params& pr = *params;
  const float vals[7] = {pr.alpha, pr.beta, pr.eta_fail, pr.eps, pr.clip_eps, pr.beta_h, pr.beta_kl};
  for (float v : vals)
    if (!isfinite(v)) return COSPEC_ERR_INVALID_ARG;
  if (!(pr.eps > 0.f) || pr.clip_eps < 0.f) return COSPEC_ERR_INVALID_ARG;
  const int have_obj = (ratio != nullptr) + (p_new != nullptr) + (p_ref != nullptr);
  if (have_obj != 0 && have_obj != 3) return COSPEC_ERR_INVALID_ARG;
  if (have_obj == 3 && !loss) return COSPEC_ERR_INVALID_ARG;
  if (!group_off || !round_off) return COSPEC_ERR_INVALID_ARG;
  if (num_rollouts > 0 && (!correct || !J || !Jbar || !adv)) return COSPEC_ERR_INVALID_ARG;
  if (num_rounds > 0 && (!match || !accept || !ell || !g || !eff || !rho || !adv_dec))
    return COSPEC_ERR_INVALID_ARG;
  const size_t need = cospec_rl_workspace(num_groups, num_rollouts);
  if (!ws || ws_bytes < need) return COSPEC_ERR_WORKSPACE;
  int* err = device_error_word();
  if (!err) return cuda_lookup_failed();
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255));
  const size_t mb = align256((size_t)num_rollouts * sizeof(double));
  RLArgs a{};
  a.num_groups = num_groups;
  a.num_rollouts = num_rollouts;
  a.num_rounds = num_rounds;
  a.K = K;
  a.group_off = group_off;
  a.correct = correct;
  a.round_off = round_off;
  a.match = match;
  a.accept = accept;
  a.ell = ell;
  a.prm = pr;
  a.ratio = ratio;
  a.p_new = p_new;
  a.p_ref = p_ref;
  a.g = g;
  a.eff = eff;
  a.rho = rho;
  a.J = J;
  a.Jbar = Jbar;
  a.adv = adv;
  a.adv_dec = adv_dec;
  a.ws_j = reinterpret_cast<double*>(base);
  a.ws_abs = reinterpret_cast<double*>(base + mb);
  a.ws_c = reinterpret_cast<float2*>(base + 2 * mb);
  a.part = have_obj ? reinterpret_cast<double*>(base + 3 * mb) : nullptr;
  a.err = err;
  if (num_groups > 0) {
    // Many small groups (more than a wave of 512-thread CTAs, at most 2048 decisions each) in CTAs of 128
    // threads, eight to an SM: a CTA then waits on its own chain of loads and sums more than it
    // works.  us, 512 -> 128 threads: 512 groups of 1.5 rounds, K = 3 24.3 -> 14.0; 2048 of 10, K = 5,
    // with the objective 109 -> 49.5; 512 of 34, K = 31 49.5 -> 35.2.  Beyond: 512 of 132, K = 31
    // (4092 decisions) 69 -> 84; 152 of 34, K = 25 24.3 -> 31.1.
    const bool small = num_groups > 2 * device_num_sms() && (long long)num_rounds * K <= 2048LL * num_groups;
    const cudaError_t e = small ? launch_pdl(rl_group_kernel<128>, dim3(num_groups), dim3(128), 0, st, a)
                                : launch_pdl(rl_group_kernel<512>, dim3(num_groups), dim3(512), 0, st, a);
    if (e != cudaSuccess) return cuda_status(e);
  }
  if (have_obj) {
    const cudaError_t e = launch_pdl(rl_loss_kernel, dim3(1), dim3(RL_LOSS_THREADS), 0, st,
                                     (const double*)a.part, num_groups, pr, loss);
    if (e != cudaSuccess) return cuda_status(e);
  }
  return COSPEC_OK;
}
