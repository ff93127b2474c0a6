// crmc_phase.cu -- the colour-phase kernel of the CR-MC stage (sm_103a).
//
// k_cr_phase: one CTA, or a seat of one, per active domain of one colour of the
// 8-colour checkerboard, for one or several replicas (blockIdx.x) in one launch; the
// domains of a colour are launched densest first (blockIdx.y is the rank in
// the order k_domain_cost and k_domain_rank compute at the start of every sweep), so that the
// long CTAs do not form the tail of the launch.
// The CTA
//   1. stages the domain's particles into a list -- in shared memory, or in a
//      global scratch region when the domain is unusually dense -- with its
//      canonical order (in-domain cell rank, then id) as a list of slots, and
//      the halo particles around it into shared memory (they do not change in
//      the phase);
//   2. draws the phase's random numbers for a chunk of trials at once
//      (Philox4x32-10, counter (trial, domain, phase, purpose));
//   3. runs the m trials of the domain one after another: warp 0 selects the
//      participants (ballot scans of the order); every thread sums its share of
//      the pair changes -- FP32 Coulomb, FP64 WCA of inserted/deleted ions --
//      into 64-bit fixed point, exact and therefore independent of the thread
//      count; warp 0 takes the Metropolis decision and commits the move (or
//      several groups of threads evaluate consecutive trials side by side);
//   4. writes the domain's cells back (id-sorted), if a trial was accepted, and
//      adds its count changes.
// The move rules are those of Sec. II.C of the paper applied to the domain
// (the domain's volume and counts).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <iterator>
#include <cstdint>

#include "crmc_device.cuh"
#include "crmc_kernels.h"

namespace crmc {

namespace {

struct TrialPre {
  uint32_t w0, w1, w2, w3;  // move, site choice, first ion, second ion
  float ax, ay, az, bx, by, bz;
  int rankA, rankB;  // in-domain cell rank of the insertion points, -1 = outside
  uint32_t uhi, ulo; // the two words of the Metropolis uniform
  float lnu_f;       // FP32 ln u (decides unless within LNU_BAND of lnA)
  int pad;
  double lnu;        // FP64 ln u (trial records only)
  // delayed acceptance: the stage-2 uniform (Philox purpose 3)
  uint32_t u2hi, u2lo;
  float lnu2_f;
  int pad2;
  double lnu2;
};

struct Desc {
  float x, y, z, dqlB;  // position, lB * (q_new - q_old)
  int dp, cls, skip;    // WCA presence change, class, list slot (-1 inserted)
};

// a trial's selection; pres: presence of a before / after, b before / after
enum Presence { PA_O = 1, PA_N = 2, PB_O = 4, PB_N = 8 };
struct TrialCtl {
  Desc c[2];
  int nch;    // changed particles needing the energy sweep (0 = decided)
  int flags;  // CR_TRIAL_* bits known before the sweep
  int move;
  int placeA, placeB;  // places in the canonical order (-1 none): the site or first ion, the second ion
  int pres;
  long long ln_ratio_fx, dself_fx;  // 2^-48 fixed point
  float qa_o, qa_n, qb_o, qb_n;  // effective charges of the two changed particles
  unsigned long long id_a, id_b;  // trial records only
  // delayed acceptance: in-domain cell ranks of a and b, stage-1 outcome
  int rka, rkb, go;
  int ewacc;             // Ewald: the trial was accepted (S(k) follows)
  float sur;             // surrogate dE~ (DA)
  long long sur_fx;      // dE~ clamped, 2^-48 fixed point (DA)
};
// the charge (0 when absent) of changed particle x (0: a, 1: b) before / after, its presence, and the
// surrogate's integer changes
__device__ __forceinline__ bool had(const TrialCtl &C, int x) { return C.pres & (x ? PB_O : PA_O); }
__device__ __forceinline__ bool has(const TrialCtl &C, int x) { return C.pres & (x ? PB_N : PA_N); }
__device__ __forceinline__ int q_old(const TrialCtl &C, int x) { return had(C, x) ? __float2int_rn(x ? C.qb_o : C.qa_o) : 0; }
__device__ __forceinline__ int q_new(const TrialCtl &C, int x) { return has(C, x) ? __float2int_rn(x ? C.qb_n : C.qa_n) : 0; }
__device__ __forceinline__ int d_charge(const TrialCtl &C, int x) { return q_new(C, x) - q_old(C, x); }
__device__ __forceinline__ int d_presence(const TrialCtl &C, int x) { return (has(C, x) ? 1 : 0) - (had(C, x) ? 1 : 0); }

// The domain's particles.  A particle keeps its slot of the payload arrays
// while it lives; `ord` holds the canonical order (in-domain cell rank, then
// id) as (slot | kind << ORD_KIND_SHIFT, cell rank), so an insertion or
// deletion moves 8 bytes per entry instead of the 56 of the payload: under the
// global schedule (a list of about 1,250, five trials in six accepted) moving
// the payload by one warp was a third of a trial, and finding the k-th of a
// kind 32 entries at a time another fifth (500 trials in each of 128 boxes:
// 5.96 ms before, 3.21 ms with the order list and 256 entries per scan round).
// pos is in the region's flat frame (frame_x).  A deleted particle's slot goes to a
// free list threaded through its info word; its charge is 0 and its class
// CR_CLS_NONE, so the pair sweep passes over it without a test.
struct DomList {
  float4 *pos, *vel;
  unsigned long long *id;
  long long *lnk;  // site constant ln10 (pH - pK - pI_X) at 2^-48, 0 for non-sites
  int *info;
  uint2 *ord;
};
constexpr int ORD_KIND_SHIFT = 28;
constexpr unsigned ORD_SLOT_MASK = (1u << ORD_KIND_SHIFT) - 1u;
// info word of a free slot: no type, class CR_CLS_NONE, the next free slot + 1
constexpr int INFO_FREE = 15 | (CR_CLS_NONE << INFO_CLS_SHIFT);
// a phase's counters beyond the kind counts (misc)
constexpr int MISC_HW = MISC_N, MISC_FREE = MISC_N + 1, MISC_DIRTY = MISC_N + 2, MISC_RES = MISC_N + 4;
// and the groups' outcomes of a round, for two rounds in turn
constexpr int MISC_TOTAL = MISC_RES + 2 * 8;

// FP32 constants of the pair sweep, kept in registers
struct PairK {
  float Lf, halfL, rc2, alpha, c1, c2, rcf;
};
__device__ __forceinline__ PairK pair_k(const SysParams &P) {
  return PairK{P.Lf, P.halfL, P.rc2, P.alpha, P.c1, P.c2, P.rcf};
}

// box cell of region coordinate i < nr <= nc along an axis (the domain's k
// cells from org first, then the h after them, then the h before)
__device__ __forceinline__ int region_coord(int i, int org, int k, int h, int nr, int nc) {
  int c = (i < k + h) ? org + i : org + i - nr;
  c += c < 0 ? nc : 0;
  return c >= nc ? c - nc : c;
}
// i / n for 0 <= i < 2^20 with r = 1 / n in FP32 (the half keeps the product
// away from whole numbers by far more than its rounding)
__device__ __forceinline__ int div_by(int i, float r) { return (int)(((float)i + 0.5f) * r); }

// Exclusive scan of n ints (shared memory) into pre[0..n] by one warp, each
// lane a run of consecutive entries.  SWAP: what pre held goes into vals.
template <bool SWAP>
__device__ __forceinline__ void warp_scan(int *vals, int n, int *pre) {
  const int lane = threadIdx.x & 31;
  const int per = (n + 31) >> 5;
  const int lo = min(n, lane * per), hi = min(n, lo + per);
  int s = 0;
  for (int i = lo; i < hi; ++i) s += vals[i];
  int x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  int run = x - s;
  for (int i = lo; i < hi; ++i) {
    const int v = vals[i];
    if (SWAP) vals[i] = pre[i];
    pre[i] = run;
    run += v;
  }
  if (lane == 31) pre[n] = x;
}

// largest i with pre[i] <= j (pre ascending, pre[0] = 0, j < pre[n])
__device__ __forceinline__ int upper_idx(const int *pre, int n, int j) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pre[mid] <= j) lo = mid; else hi = mid;
  }
  return lo;
}

// warp: place of the kth (0-based) entry of a kind in the canonical order, -1
// if none.  Long lists are first passed over 256 entries at a time (eight
// loads in flight, one warp sum); the entry is then found by ballots.  Out of
// line: one copy of this code serves every selection (the trial loop is bound
// by instruction fetch).
__device__ __noinline__ int warp_kth(const uint2 *ord, int n, int kind, int kth) {
  const int lane = threadIdx.x & 31;
  int base = 0;
#pragma unroll 1
  while (n - base > 64) {
    int c = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = base + 32 * u + lane;
      const unsigned e = ord[min(j, n - 1)].x >> ORD_KIND_SHIFT;
      c += j < n && e == (unsigned)kind ? 1 : 0;
    }
    c = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
    if (kth < c) break;
    kth -= c;
    base += 256;
  }
#pragma unroll 1
  for (; base < n; base += 32) {
    const int j = base + lane;
    const unsigned m = __ballot_sync(0xffffffffu, j < n && (ord[j].x >> ORD_KIND_SHIFT) == (unsigned)kind);
    const int c = __popc(m);
    if (kth < c) {
      const unsigned hit = __ballot_sync(0xffffffffu, ((m >> lane) & 1u) && __popc(m & ((1u << lane) - 1u)) == kth);
      return base + __ffs(hit) - 1;
    }
    kth -= c;
  }
  return -1;
}

// warp: number of entries with cell rank < r (the ranks ascend); long lists
// are narrowed 32-fold per round
__device__ __noinline__ int warp_lower(const uint2 *ord, int n, int r) {
  const int lane = threadIdx.x & 31;
  int base = 0, len = n;
#pragma unroll 1
  while (len > 32) {
    const int st = (len + 31) >> 5, o = lane * st;
    const int b = __popc(__ballot_sync(0xffffffffu, o < len && (int)ord[base + o].y < r));
    if (b == 0) return base;
    const int skip = (b - 1) * st;
    base += skip;
    len = min(st, len - skip);
  }
  return base + __popc(__ballot_sync(0xffffffffu, lane < len && (int)ord[base + lane].y < r));
}

// warp: open a hole at p (entries [p, n) move up by one), 128 entries per
// round from the top down: every load of a round before its stores
__device__ __forceinline__ void ord_open(uint2 *ord, int n, int p) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int hi = n; hi > p; hi -= 128) {
    const int lo = max(p, hi - 128);
    uint2 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lo + 32 * u + lane < hi) x[u] = ord[lo + 32 * u + lane];
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lo + 32 * u + lane < hi) ord[lo + 32 * u + lane + 1] = x[u];
    __syncwarp();
  }
}

// warp: close place p (entries (p, n) move down by one), 128 per round from
// the bottom up
__device__ __forceinline__ void ord_close(uint2 *ord, int n, int p) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int lo = p + 1; lo < n; lo += 128) {
    uint2 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lo + 32 * u + lane < n) x[u] = ord[lo + 32 * u + lane];
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lo + 32 * u + lane < n) ord[lo + 32 * u + lane - 1] = x[u];
    __syncwarp();
  }
}

// The rounding of a pair's terms, the same in every copy of the code that
// evaluates one (the compiler otherwise picks the products it fuses anew for
// each place a function is inlined at): a pair counts the same whether its
// candidate comes from shared or global memory, in whichever form of the launch
// and in logged sweeps.  Left to the compiler, the two differed in the last bit
// of a distance, and about one trial in 10^8 was decided by where its domain's
// list lay.  The flat frame and the general one add the squares in another
// order; a box has regions of one of them only, and each order is the one that
// chains saved with earlier versions were run with.
template <bool FLAT>
__device__ __forceinline__ float pair_r2(float dx, float dy, float dz) {
  return __fmaf_rn(dz, dz, FLAT ? __fmaf_rn(dy, dy, __fmul_rn(dx, dx)) : __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
}
// shifted Coulomb energy of unit charges at lB = 1: ef = erfc(alpha r), r = r2 rinv
struct PairPhi {
  float ef, r, rinv;
};
__device__ __forceinline__ PairPhi pair_phi(float r2, float alpha) {
  const float rinv = rsqrtf(r2);
  const float r = __fmul_rn(r2, rinv);
  return PairPhi{erfcf(__fmul_rn(alpha, r)), r, rinv};
}
__device__ __forceinline__ float phi_value(const PairPhi &p, float c1, float c2, float rcf) {
  return __fmaf_rn(c2, __fsub_rn(p.r, rcf), __fmaf_rn(p.ef, p.rinv, -c1));
}
__device__ __forceinline__ float phi_gross(const PairPhi &p, float c1, float c2, float rcf) {  // sum of the terms' magnitudes
  return __fmaf_rn(c2, fabsf(__fsub_rn(p.r, rcf)), __fmaf_rn(p.ef, p.rinv, c1));
}

// pair change between the two changed particles: u_new - u_old, Coulomb in
// FP32 and WCA in FP64, into fixed point (without a WCA term the FP64 sum
// reduces to the FP32 change, taken directly)
template <bool WITH_S, bool FLAT>
__device__ __forceinline__ void cc_change_impl(const SysParams &K, const WcaEntry *wca, const TrialCtl &t, long long &acc,
                                               unsigned long long &sacc, int &ov) {
  const Desc &A = t.c[0], &B = t.c[1];
  const float dx = wrap_diff(B.x, A.x, K.Lf, K.halfL);
  const float dy = wrap_diff(B.y, A.y, K.Lf, K.halfL);
  const float dz = wrap_diff(B.z, A.z, K.Lf, K.halfL);
  const float r2 = pair_r2<FLAT>(dx, dy, dz);
  const WcaEntry &w = wca[A.cls * 4 + B.cls];
  float uc[2] = {0.0f, 0.0f};
  double uw[2] = {0.0, 0.0};
  double gs = 0.0;
  bool hit = false;
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const int both = s ? PA_N | PB_N : PA_O | PB_O;
    if ((t.pres & both) != both) continue;
    const float qa = s ? t.qa_n : t.qa_o, qb = s ? t.qb_n : t.qb_o;
    if (r2 < K.rc2 && qa != 0.0f && qb != 0.0f) {
      const PairPhi p = pair_phi(r2, K.alpha);
      const float qq = __fmul_rn(K.lBf, __fmul_rn(qa, qb));
      uc[s] = __fmul_rn(qq, phi_value(p, K.c1, K.c2, K.rcf));
      if (WITH_S) gs += (double)__fmul_rn(fabsf(qq), phi_gross(p, K.c1, K.c2, K.rcf));
    }
    if (w.on && r2 < 1.0001f * w.wcut2) {
      const double ddx = wrap_diff_d(B.x, A.x, K.Ld, K.halfLd), ddy = wrap_diff_d(B.y, A.y, K.Ld, K.halfLd),
                   ddz = wrap_diff_d(B.z, A.z, K.Ld, K.halfLd);
      const double r = sqrt(dist2_d(ddx, ddy, ddz));
      if (r < w.wcut_d) {
        const double sv = r - w.del_d;
        const bool inserted = s == 1 && (!(t.pres & PA_O) || !(t.pres & PB_O));  // both are present after
        if (inserted && sv < 0.5 * w.sig_d) {
          ov = 1;
        } else {
          double g = 0.0;
          uw[s] = wca_energy_d(w, sv, g);
          if (WITH_S) gs += g;
          hit = true;
        }
      }
    }
  }
  const float dc = __fsub_rn(uc[1], uc[0]);
  if (!hit) {  // dw = 0: |dc| < 2^20 decides, fix32(dc) is the sum
    if (dc != 0.0f) {
      if (!(fabsf(dc) < BIG_TERM)) {
        ov = 1;
      } else {
        acc += fix32(dc);
        if (WITH_S) sacc += (unsigned long long)__double2ll_rn(fmin(gs, (double)BIG_TERM) * (double)FIX_SCALE);
      }
    }
    return;
  }
  const double dw = uw[1] - uw[0];
  if (dc != 0.0f || dw != 0.0) {
    if (!(fabs((double)dc + dw) < (double)BIG_TERM)) {
      ov = 1;
    } else {
      acc += fix32(dc) + __double2ll_rn(__dmul_rn(dw, (double)FIX_SCALE));
      if (WITH_S) sacc += (unsigned long long)__double2ll_rn(fmin(gs, (double)BIG_TERM) * (double)FIX_SCALE);
    }
  }
}

// Sums of pair terms returned by value from the out-of-line helpers, so that
// the callers' accumulators stay in registers.
struct PairSum {
  long long acc;
  unsigned long long sacc;
  int ov;
};

constexpr unsigned FULL = 0xffffffffu;
constexpr int QCAP = 96;  // per-warp queue of Coulomb pair terms (up to 31 waiting + 64 new)

// Metropolis comparison ln u < lnA with lnA in 2^-48 fixed point: the FP32
// ln u decides outside LNU_BAND, the FP64 ln u inside it
// (the FP64 logarithm of the band is out of line: rare, and large)
__device__ __noinline__ bool accept_band(long long lnA_fx, uint32_t uhi, uint32_t ulo) {
  return __double2ll_rn(log(unif53(uhi, ulo)) * LNFIX) < lnA_fx;
}
__device__ __forceinline__ bool accept_fx(long long lnA_fx, float lnu_f, uint32_t uhi, uint32_t ulo) {
  const long long lnu_apx = (long long)__float2int_rn(lnu_f * 16777216.0f) << 24;
  const long long diff = lnA_fx - lnu_apx;
  if (diff > LNU_BAND) return true;
  if (diff < -LNU_BAND) return false;
  return accept_band(lnA_fx, uhi, ulo);
}

// Maxwell-Boltzmann velocity of an inserted ion (unit mass, kT = 1): Box-Muller
// on the four 24-bit uniforms of Philox block (trial, domain, phase, purpose),
// purpose 6 for the first inserted ion of a trial and 7 for the second
__device__ __noinline__ float4 ion_velocity(uint32_t k, uint32_t d, uint32_t phi, uint32_t purpose, uint32_t key0,
                                           uint32_t key1) {
  const uint4 w = philox10(k, d, phi, purpose, key0, key1);
  const float u0 = ((float)(w.x >> 8) + 0.5f) * (1.0f / 16777216.0f);
  const float u1 = ((float)(w.y >> 8) + 0.5f) * (1.0f / 16777216.0f);
  const float u2 = ((float)(w.z >> 8) + 0.5f) * (1.0f / 16777216.0f);
  const float u3 = ((float)(w.w >> 8) + 0.5f) * (1.0f / 16777216.0f);
  const float r1 = sqrtf(-2.0f * logf(u0)), r2 = sqrtf(-2.0f * logf(u2));
  float s1, c1, s3, c3;
  sincospif(2.0f * u1, &s1, &c1);
  sincospif(2.0f * u3, &s3, &c3);
  return make_float4(r1 * c1, r1 * s1, r2 * c3, 0.0f);
}

__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// ---- delayed-acceptance surrogate

// shell of a squared integer cell offset inside the 5^3 stencil:
// {0},{1},{2},{3},{4},{5},{6},{8,9,12}
__device__ __forceinline__ int shell_of_n2(int n2) { return n2 <= 6 ? n2 : 7; }

// shell of in-domain cell rank rb relative to rank ra (-1 outside the stencil)
__device__ __forceinline__ int shell_ranks(int ra, int rb, int k) {
  const int dx = rb % k - ra % k, dy = (rb / k) % k - (ra / k) % k, dz = rb / (k * k) - ra / (k * k);
  if (abs(dx) > 2 || abs(dy) > 2 || abs(dz) > 2) return -1;
  return shell_of_n2(dx * dx + dy * dy + dz * dz);
}

// region cell of in-domain rank r shifted by (dx, dy, dz) in [-2, 2]^3
__device__ __forceinline__ int region_of(int r, int dx, int dy, int dz, int k, int nr) {
  int x = r % k + dx, y = (r / k) % k + dy, z = r / (k * k) + dz;
  x += x < 0 ? nr : 0;
  y += y < 0 ? nr : 0;
  z += z < 0 ? nr : 0;
  return x + nr * (y + nr * z);
}

// the eight weights of one 16-byte block times eight inputs, onto a, in input order
__device__ __forceinline__ float mlp_block(const uint4 w, const float4 x0, const float4 x1, float a) {
  a = __fmaf_rn(__uint_as_float(w.x << 16), x0.x, a);
  a = __fmaf_rn(__uint_as_float(w.x & 0xffff0000u), x0.y, a);
  a = __fmaf_rn(__uint_as_float(w.y << 16), x0.z, a);
  a = __fmaf_rn(__uint_as_float(w.y & 0xffff0000u), x0.w, a);
  a = __fmaf_rn(__uint_as_float(w.z << 16), x1.x, a);
  a = __fmaf_rn(__uint_as_float(w.z & 0xffff0000u), x1.y, a);
  a = __fmaf_rn(__uint_as_float(w.w << 16), x1.z, a);
  return __fmaf_rn(__uint_as_float(w.w & 0xffff0000u), x1.w, a);
}

// One dense layer with ReLU for the two input vectors x[2][n_in] -> y[2][128]
// by n threads: each output is its bias plus one FP32 fused multiply-add per
// weight, in input order.  The weights come in 16-byte blocks of eight inputs
// of one output (block kb of output o at kb * 128 + o), so that a warp's loads
// are 512 consecutive bytes and a layer takes 16 of them instead of 128 of 2
// bytes per lane; four blocks are loaded ahead of their use.  Below 256
// threads a thread takes an output of both vectors, so each block is loaded
// once for the two.  (13 polyelectrolyte boxes, delayed-acceptance
// cycles of 3.53 ms with 2-byte loads, 2.94 ms.)
__device__ __noinline__ void mlp_layer(const uint4 *__restrict__ W, const float *__restrict__ b, const float *x,
                                       int n_in, float *y, int tid, int n) {
  const int nb = n_in >> 3;
  const bool both = n < 2 * MLP_H;
#pragma unroll 1
  for (int o = tid; o < (both ? MLP_H : 2 * MLP_H); o += n) {
    const int i = o & (MLP_H - 1);
    const float4 *xa = (const float4 *)(x + (both ? 0 : (o >> 7) * n_in)), *xb = (const float4 *)(x + n_in);
    const uint4 *w = W + i;
    float a0 = __ldg(&b[i]), a1 = a0;
    uint4 nx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) nx[u] = __ldg(&w[min(u, nb - 1) * MLP_H]);
#pragma unroll 1
    for (int k0 = 0; k0 < nb; k0 += 4) {
      uint4 c[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) c[u] = nx[u];
#pragma unroll
      for (int u = 0; u < 4; ++u) nx[u] = __ldg(&w[min(k0 + 4 + u, nb - 1) * MLP_H]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k0 + u >= nb) break;
        a0 = mlp_block(c[u], xa[2 * (k0 + u)], xa[2 * (k0 + u) + 1], a0);
        if (both) a1 = mlp_block(c[u], xb[2 * (k0 + u)], xb[2 * (k0 + u) + 1], a1);
      }
    }
    y[o] = a0 > 0.0f ? a0 : 0.0f;
    if (both) y[MLP_H + o] = a1 > 0.0f ? a1 : 0.0f;
  }
}

// DSF Coulomb change of one queued pair: qp * phi(r), qp = lB dq_c q_j
template <bool WITH_S>
__device__ __forceinline__ void coul_eval(const PairK &K, float r2, float qp, long long &acc,
                                          unsigned long long &sacc, int &ov) {
  const PairPhi p = pair_phi(r2, K.alpha);
  const float du = __fmul_rn(qp, phi_value(p, K.c1, K.c2, K.rcf));
  if (!(fabsf(du) < BIG_TERM)) {
    ov = 1;
  } else {
    acc += fix32(du);
    if (WITH_S) sacc += (unsigned long long)fix32(fminf(__fmul_rn(fabsf(qp), phi_gross(p, K.c1, K.c2, K.rcf)), BIG_TERM));
  }
}

// WCA pre-check radius of a changed particle of class ci against class cj
// (1.0001 x squared cutoff, or -1 when the classes do not interact), and the
// largest over cj: the sweep compares with the latter and looks the former up
// for the few candidates inside it
__device__ __forceinline__ float wca_radius(const WcaEntry &w) { return w.on ? 1.0001f * w.wcut2 : -1.0f; }

// A pair within the WCA range of an inserted / deleted changed particle:
// Coulomb in FP32 and WCA in FP64, evaluated at once (rare).  Not inlined, to
// keep the sweep's loop small; everything it needs comes by value or from
// shared memory (P, w), and its sums come back by value.
template <bool WITH_S>
__device__ __noinline__ PairSum near_pair(const SysParams &P, const WcaEntry &w, float cx, float cy, float cz,
                                          float cdq, int cdp, float xj, float yj, float zj, float qj, float r2) {
  PairSum out{0, 0ull, 0};
  float du = 0.0f, gs = 0.0f;
  const bool any = r2 < P.rc2 && cdq != 0.0f && qj != 0.0f;
  if (any) {
    const PairPhi p = pair_phi(r2, P.alpha);
    const float qq = __fmul_rn(cdq, qj);
    du = __fmul_rn(qq, phi_value(p, P.c1, P.c2, P.rcf));
    if (WITH_S) gs = __fmul_rn(fabsf(qq), phi_gross(p, P.c1, P.c2, P.rcf));
  }
  double du_w = 0.0, gs_w = 0.0;
  int ovw = 0;
  const bool hit = wca_change_d(w, cdp, cx, cy, cz, xj, yj, zj, P.Ld, P.halfLd, du_w, gs_w, ovw);
  if (ovw) {
    out.ov = 1;
  } else if (hit) {
    if (!(fabs((double)du + du_w) < (double)BIG_TERM)) {
      out.ov = 1;
    } else {
      if (any) out.acc += fix32(du);
      out.acc += __double2ll_rn(__dmul_rn(du_w, (double)FIX_SCALE));
      if (WITH_S) out.sacc += (unsigned long long)__double2ll_rn(fmin((double)gs + gs_w, (double)BIG_TERM) * (double)FIX_SCALE);
    }
  } else if (any) {  // beyond the WCA cutoff after all: Coulomb only
    if (!(fabsf(du) < BIG_TERM)) out.ov = 1;
    else {
      out.acc += fix32(du);
      if (WITH_S) out.sacc += (unsigned long long)fix32(fminf(gs, BIG_TERM));
    }
  }
  return out;
}

// the pair between the two changed particles when they lie within WCA range
// of each other (rare; one thread; out of line, with its FP64 branch)
template <bool WITH_S, bool FLAT>
__device__ __noinline__ PairSum cc_change(const SysParams &P, const TrialCtl &t) {
  PairSum out{0, 0ull, 0};
  cc_change_impl<WITH_S, FLAT>(P, P.wca, t, out.acc, out.sacc, out.ov);
  return out;
}

// Flat frame of a region that spans less than half the box: along an axis
// whose region wraps around the periodic boundary (bit i of strad), a
// coordinate x >= L/2 becomes x - L (exact: L/2 <= x < L).  Between two points
// of the region the plain difference in this frame then equals the
// minimum-image difference bit for bit, whichever of the two had been shifted.
__device__ __forceinline__ float frame_x(float x, int strad, int axis, float halfL, float L) {
  return ((strad >> axis) & 1) && x >= halfL ? x - L : x;
}

// a coordinate of the flat frame (frame_x) back in [0, L), exactly
__device__ __forceinline__ float unframe_x(float x, float L) { return x < 0.0f ? x + L : x; }

// every full 32 queued Coulomb pairs of the warp are evaluated with all lanes
// busy; the rest (fewer than 32) stays queued
template <bool WITH_S>
__device__ __forceinline__ void queue_flush(const PairK &K, float2 *q, int &qn, long long &acc,
                                            unsigned long long &sacc, int &ov) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  while (qn >= 32) {  // from the end, so that the rest stays where it is
    __syncwarp();
    const float2 e = q[qn - 32 + lane];
    qn -= 32;
    coul_eval<WITH_S>(K, e.x, e.y, acc, sacc, ov);
  }
  __syncwarp();
}

// A candidate within the largest WCA range of an inserted / deleted changed
// particle c (rare): the pair is evaluated here when it lies within its own
// classes' range (returned true), Coulomb included
template <bool WITH_S>
__device__ __forceinline__ bool near_check(const SysParams &P, const float *wr, const Desc &c, float r2, float xj,
                                           float yj, float zj, float qj, int jcls, long long &acc,
                                           unsigned long long &sacc, int &ov) {
  const int e = c.cls * 4 + jcls;
  if (!(r2 < wr[e])) return false;
  const PairSum p = near_pair<WITH_S>(P, P.wca[e], c.x, c.y, c.z, c.dqlB, c.dp, unframe_x(xj, P.Lf),
                                      unframe_x(yj, P.Lf), unframe_x(zj, P.Lf), qj, r2);
  acc += p.acc;
  sacc += p.sacc;
  ov |= p.ov;
  return true;
}

// One trial's changed particles as the sweep needs them: coordinates in the
// sweep's frame, Coulomb ranges (-1 without a charge change) and the largest
// WCA ranges (-1 when the particle is neither inserted nor deleted)
struct SweepPair {
  float ax, ay, az, bx, by, bz, qA, qB, rcA, rcB, wmA, wmB;
  int skA, skB;
};
__device__ __forceinline__ SweepPair sweep_pair(const PairK &K, const float *wmax, const Desc &A, const Desc &B,
                                                int strad) {
  SweepPair p;
  p.ax = frame_x(A.x, strad, 0, K.halfL, K.Lf);
  p.ay = frame_x(A.y, strad, 1, K.halfL, K.Lf);
  p.az = frame_x(A.z, strad, 2, K.halfL, K.Lf);
  p.bx = frame_x(B.x, strad, 0, K.halfL, K.Lf);
  p.by = frame_x(B.y, strad, 1, K.halfL, K.Lf);
  p.bz = frame_x(B.z, strad, 2, K.halfL, K.Lf);
  p.qA = A.dqlB;
  p.qB = B.dqlB;
  p.rcA = A.dqlB != 0.0f ? K.rc2 : -1.0f;
  p.rcB = B.dqlB != 0.0f ? K.rc2 : -1.0f;
  p.wmA = A.dp != 0 ? wmax[A.cls] : -1.0f;
  p.wmB = B.dp != 0 ? wmax[B.cls] : -1.0f;
  p.skA = A.skip;
  p.skB = B.skip;
  return p;
}

// The pair between the two changed particles, as one more queued Coulomb pair:
// a and b are both present either before the trial or after it, so its change
// is plus or minus one pair energy, in the same form and rounding as a queued
// pair's.  Evaluated by one thread of its own it kept the other warps waiting
// at the trial's barrier.  True when lane 0 of the calling warp queued it;
// within WCA range it is evaluated here.
template <bool WITH_S, bool FLAT>
__device__ __forceinline__ bool queue_changed_pair(const SysParams &P, const PairK &K, const float *wr,
                                                   const TrialCtl &t, float2 *q, long long &acc,
                                                   unsigned long long &sacc, int &ov) {
  const Desc &A = t.c[0], &B = t.c[1];
  const float dx = wrap_diff(B.x, A.x, K.Lf, K.halfL);
  const float dy = wrap_diff(B.y, A.y, K.Lf, K.halfL);
  const float dz = wrap_diff(B.z, A.z, K.Lf, K.halfL);
  const float r2 = pair_r2<FLAT>(dx, dy, dz);
  const bool after = (t.pres & (PA_N | PB_N)) == (PA_N | PB_N);
  const float qq = after ? __fmul_rn(t.qa_n, t.qb_n) : -__fmul_rn(t.qa_o, t.qb_o);
  if (r2 < wr[A.cls * 4 + B.cls]) {
    if ((threadIdx.x & 31) == 0) {
      const PairSum cc = cc_change<WITH_S, FLAT>(P, t);
      acc += cc.acc;
      sacc += cc.sacc;
      ov |= cc.ov;
    }
    return false;
  }
  if (!(r2 < K.rc2) || qq == 0.0f) return false;
  if ((threadIdx.x & 31) == 0) q[0] = make_float2(r2, __fmul_rn(P.lBf, qq));
  return true;
}

// Both changed particles against one candidate (lane-parallel): two distance
// tests; the in-range Coulomb pairs of A and B join the warp's queue with one
// compaction step, and every full 32 queued pairs are evaluated with all
// lanes busy.  cls(): the candidate's class, read only for near candidates.
// FLAT: plain differences in the region's flat frame are the minimum-image
// ones.
template <bool WITH_S, bool FLAT, typename Cls>
__device__ __forceinline__ void offer2(const SysParams &P, const PairK &K, const float *wr, const TrialCtl &ctl,
                                       const SweepPair &p, bool valid, float xj, float yj, float zj, float qj,
                                       Cls cls, float2 *q, int &qn, long long &acc, unsigned long long &sacc,
                                       int &ov) {
  float ax, ay, az, bx, by, bz;
  if (FLAT) {
    ax = xj - p.ax; ay = yj - p.ay; az = zj - p.az;
    bx = xj - p.bx; by = yj - p.by; bz = zj - p.bz;
  } else {
    ax = wrap_diff(xj, p.ax, K.Lf, K.halfL); ay = wrap_diff(yj, p.ay, K.Lf, K.halfL); az = wrap_diff(zj, p.az, K.Lf, K.halfL);
    bx = wrap_diff(xj, p.bx, K.Lf, K.halfL); by = wrap_diff(yj, p.by, K.Lf, K.halfL); bz = wrap_diff(zj, p.bz, K.Lf, K.halfL);
  }
  const float rA = pair_r2<FLAT>(ax, ay, az), rB = pair_r2<FLAT>(bx, by, bz);
  const bool charged = valid && qj != 0.0f;
  bool inA = charged && rA < p.rcA, inB = charged && rB < p.rcB;
  if (valid && (rA < p.wmA || rB < p.wmB)) {
    const int jc = cls();
    if (rA < p.wmA && near_check<WITH_S>(P, wr, ctl.c[0], rA, xj, yj, zj, qj, jc, acc, sacc, ov)) inA = false;
    if (rB < p.wmB && near_check<WITH_S>(P, wr, ctl.c[1], rB, xj, yj, zj, qj, jc, acc, sacc, ov)) inB = false;
  }
  const unsigned mA = __ballot_sync(FULL, inA), mB = __ballot_sync(FULL, inB);
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int nA = __popc(mA);
  if (inA) q[qn + __popc(mA & lt)] = make_float2(rA, __fmul_rn(p.qA, qj));
  if (inB) q[qn + nA + __popc(mB & lt)] = make_float2(rB, __fmul_rn(p.qB, qj));
  qn += nA + __popc(mB);
  if (qn >= 32) queue_flush<WITH_S>(K, q, qn, acc, sacc, ov);
}


// The threads that work on one domain: a whole CTA, or one of its seats.  tid
// of n; `groups` groups of gn threads each evaluate a trial (several groups
// only where a domain has the whole CTA; each is then one warp).  Without
// seats (SEATS false) a domain's barrier is the CTA's.  With seats, seat s has
// barrier s; a kernel with run-time barrier numbers holds all 16 barriers per
// CTA, which limits an SM to four CTAs -- no loss for the 256 threads and more
// of those CTAs, but it halved the residency of 64-thread ones.
constexpr int MAX_GROUPS = 8;
template <bool SEATS>
struct Seat {
  int tid, n, groups, gn, bar;
  __device__ __forceinline__ void sync() const {
    if (SEATS) asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory");
    else __syncthreads();
  }
  __device__ __forceinline__ void group_sync() const {
    if (gn == 32) __syncwarp();
    else sync();
  }
};

// A CTA's domain, in shared memory (so that the trial loop holds none of it
// in registers): where it lies, its random-number counters, its list, and the
// region around it.  The sweep reads the halo on chip (cpos[0 .. nhc), classes
// hcls), the list's payload behind it (cpos[hcs + slot]) when that is in shared
// memory too (in_smem), and what does not fit there from global memory.
struct Dom {
  DomList L;
  const long long *lnt;  // log table
  const int *hpre, *hcell;
  long long log_dom;     // first record of a logged call
  int nhc, hcs;   // halo entries on chip, and their capacity
  int cpos_at, hcls_at, queue_at;  // byte offsets of cpos, hcls and the queues in the seat's shared memory
  int NH, NR;     // halo entries in all; region cells
  int in_smem, strad, flat, list_cap;
  int org[3], off[3], dd[3], d;
  uint32_t phi, key0, key1;
  float wr[20];   // [16] WCA pre-check radii by class pair, [4] their maxima per class
};

// Random numbers of a chunk of trials (Philox purposes 0-3 and 6-7; thread i0
// of a group of `stride` threads takes every stride-th task): the move and
// its choices, both insertion points with their in-domain cell ranks, the
// Metropolis uniform, for delayed acceptance the stage-2 uniform, and the
// velocities of the ions an insertion would add.
template <bool LOG, bool DA>
__device__ __noinline__ void draw_chunk(const SysParams &P, const Dom &D, TrialPre *tp, float4 *tvel, int k0,
                                        int nchunk, int i0, int stride) {
  const int d = D.d, k = P.k, nc = P.nc;
  const uint32_t phi = D.phi, key0 = D.key0, key1 = D.key1;
  const float af = P.af, Lf = P.Lf, scf = P.scf;
  const int *org = D.org, *off = D.off, *dd = D.dd;
  // the Maxwell-Boltzmann velocities an accepted insertion gives its ions
  // (purposes 6, 7), counted from the last thread so that other warps than
  // those of the trials' own numbers draw them
  for (int u = stride - 1 - i0; u < 2 * nchunk; u += stride)
    tvel[u] = ion_velocity((uint32_t)(k0 + (u >> 1)), (uint32_t)d, phi, 6u + (uint32_t)(u & 1), key0, key1);
  for (int t = i0; t < nchunk; t += stride) {
    const uint32_t kk = (uint32_t)(k0 + t);
    const uint4 a = philox10(kk, (uint32_t)d, phi, 0u, key0, key1);
    const uint4 b = philox10(kk, (uint32_t)d, phi, 1u, key0, key1);
    const uint4 c = philox10(kk, (uint32_t)d, phi, 2u, key0, key1);
    TrialPre q;
    q.w0 = a.x; q.w1 = a.y; q.w2 = a.z; q.w3 = a.w;
    q.ax = insert_coord(org[0], b.x, k, nc, af, Lf);
    q.ay = insert_coord(org[1], b.y, k, nc, af, Lf);
    q.az = insert_coord(org[2], b.z, k, nc, af, Lf);
    q.bx = insert_coord(org[0], b.w, k, nc, af, Lf);
    q.by = insert_coord(org[1], c.x, k, nc, af, Lf);
    q.bz = insert_coord(org[2], c.y, k, nc, af, Lf);
    const float xs[2][3] = {{q.ax, q.ay, q.az}, {q.bx, q.by, q.bz}};
    int rk[2];
    for (int s = 0; s < 2; ++s) {
      int l[3];
      bool in = true;
      for (int i = 0; i < 3; ++i) {
        const int cc = cell_of(xs[s][i], scf, nc);
        const int sh = ((cc - off[i]) % nc + nc) % nc;
        in = in && (sh / k == dd[i]);
        l[i] = sh % k;
      }
      rk[s] = in ? l[0] + k * (l[1] + k * l[2]) : -1;
    }
    q.rankA = rk[0];
    q.rankB = rk[1];
    q.uhi = c.z;
    q.ulo = c.w;
    q.lnu_f = logf((float)(c.z >> 5) * 7.450580596923828e-09f + ((float)(c.w >> 6) + 0.5f) * 1.1102230246251565e-16f);
    q.pad = 0;
    q.lnu = LOG ? log(unif53(c.z, c.w)) : 0.0;
    q.u2hi = q.u2lo = 0u;
    q.lnu2_f = 0.0f;
    q.pad2 = 0;
    q.lnu2 = 0.0;
    if (DA) {
      const uint4 e = philox10(kk, (uint32_t)d, phi, 3u, key0, key1);
      q.u2hi = e.x;
      q.u2lo = e.y;
      q.lnu2_f = logf((float)(e.x >> 5) * 7.450580596923828e-09f + ((float)(e.y >> 6) + 0.5f) * 1.1102230246251565e-16f);
      q.lnu2 = LOG ? log(unif53(e.x, e.y)) : 0.0;
    }
    tp[t] = q;
  }
}

// id of the (first) ion a trial inserts
__device__ __forceinline__ unsigned long long new_id(uint32_t phi, int d, int m, int kk) {
  return ((unsigned long long)(phi + 1u) << 32) | (unsigned long long)(2u * ((uint32_t)d * (uint32_t)m + (uint32_t)kk));
}

// slot of the particle at place i of the canonical order, and a slot's
// position in [0, L) (w: charge)
__device__ __forceinline__ int slot_at(const DomList &L, int i) { return (int)(L.ord[i].x & ORD_SLOT_MASK); }
__device__ __forceinline__ float4 raw_pos(const DomList &L, int s, float Lf) {
  const float4 p = L.pos[s];
  return make_float4(unframe_x(p.x, Lf), unframe_x(p.y, Lf), unframe_x(p.z, Lf), p.w);
}

// Proposal of trial kk on the current list (Sec. II.C applied to the domain):
// the move, its participants, the log of the acceptance ratio without the
// energy, the self-energy change and the two changed particles.  Every lane
// of the calling warp computes the same values (the list scans are ballots).
// One path serves the four forms: a is the site, or the first ion of a salt
// move; b the ion paired with it; a listed particle is the kth of its kind,
// an inserted one lies at the trial's point.
template <bool LOG, bool DA>
__device__ __forceinline__ void select_trial(const SysParams &P, const Dom &D, const int *misc, const TrialPre &q,
                                             int kk, TrialCtl &C) {
  const int lane = threadIdx.x & 31;
  const int n = misc[0];
  const int mv = pick32(q.w0, 2 * P.n_react);
  const int r = P.react[mv >> 1];
  const bool fwd = (mv & 1) == 0, salt = r == R_SALT;
  const int kn = r == R_ACID ? K_A0 : K_B0;      // the site's neutral kind; the ionised one follows it
  const float qs = r == R_ACID ? -1.0f : 1.0f;   // its charge when ionised
  const bool listA = !salt || !fwd, listB = !fwd;
  const int kA = salt ? P.kxp : (fwd ? kn : kn + 1), kB = salt || r == R_BASE ? P.kxm : P.kxp;
  const int nA = misc[1 + kA], nB = misc[1 + kB];
  int flags = 0, sA = -1, sB = -1, placeA = -1, placeB = -1;
  if ((listA && nA == 0) || (listB && nB == 0)) {
    flags = CR_TRIAL_NO_ELIGIBLE;
  } else {
    if (fwd && (q.rankA < 0 || (salt && q.rankB < 0))) flags = CR_TRIAL_EDGE;
    if (listA) placeA = warp_kth(D.L.ord, n, kA, pick32(salt ? q.w2 : q.w1, nA));
    if (listB) placeB = warp_kth(D.L.ord, n, kB, pick32(salt ? q.w3 : q.w2, nB));
    // a failed selection would mean the kind counts and the list disagree:
    // record it and reject instead of touching memory outside the list
    if ((listA && placeA < 0) || (listB && placeB < 0)) {
      flags |= CR_TRIAL_NO_ELIGIBLE;
      placeA = placeB = -1;
      if (lane == 0) atomicOr(P.err, ERRB_ARG);
    }
  }
  Desc c0 = {q.ax, q.ay, q.az, 0.0f, 1, P.ion_cls, -1};
  Desc c1 = salt ? Desc{q.bx, q.by, q.bz, 0.0f, 1, P.ion_cls, -1} : c0;
  float qa_o = 0.0f, qa_n = 0.0f, qb_o = 0.0f, qb_n = 0.0f;
  long long lnk = 0;
  int rka = q.rankA, rkb = salt ? q.rankB : q.rankA;
  unsigned long long id_a = ~0ull, id_b = ~0ull;
  if (placeA >= 0) {
    sA = slot_at(D.L, placeA);
    const float4 p = raw_pos(D.L, sA, P.Lf);
    c0 = Desc{p.x, p.y, p.z, 0.0f, salt ? -1 : 0, (D.L.info[sA] >> INFO_CLS_SHIFT) & 3, sA};
    qa_o = p.w;
    lnk = D.L.lnk[sA];
    if (DA) rka = (int)D.L.ord[placeA].y;
    if (LOG) id_a = D.L.id[sA];
  }
  if (placeB >= 0) {
    sB = slot_at(D.L, placeB);
    const float4 p = raw_pos(D.L, sB, P.Lf);
    c1 = Desc{p.x, p.y, p.z, 0.0f, -1, (D.L.info[sB] >> INFO_CLS_SHIFT) & 3, sB};
    qb_o = p.w;
    if (DA) rkb = (int)D.L.ord[placeB].y;
    if (LOG) id_b = D.L.id[sB];
  }
  if (fwd) {
    qa_n = salt ? P.ion_q : qs;
    qb_n = (salt ? -1.0f : -qs) * P.ion_q;
  }
  c0.dqlB = P.lBf * (qa_n - qa_o);
  c1.dqlB = P.lBf * (qb_n - qb_o);
  const int pres = salt ? (fwd ? PA_N | PB_N : PA_O | PB_O) : (fwd ? PA_O | PA_N | PB_N : PA_O | PA_N | PB_O);
  // the combinatorial and chemical factor; the counts after a forward move
  // are one higher, and a reverse move has the inverse form
  const long long *lnt = D.lnt;
  const int up = fwd ? 1 : 0;
  long long ln = P.lnz1_fx - lnt[nB + up];
  if (salt) ln += P.lnz1_fx + P.lnsalt_fx - lnt[nA + up];
  else ln += lnk;
  ln = fwd ? ln : -ln;
  if (!salt) ln += lnt[nA] - lnt[misc[1 + (fwd ? kn + 1 : kn)] + 1];
  // self-energy change: lB s_self (sum of q_new^2 - q_old^2), an integer multiple
  const int sq = (int)(qa_n * qa_n) - (int)(qa_o * qa_o) + (int)(qb_n * qb_n) - (int)(qb_o * qb_o);
  // lane 0 publishes the selection (C lives in shared memory; every lane
  // holds the same values), once every lane has read the previous trial's: a
  // forward salt move scans no list, so nothing else lets the warp meet here
  __syncwarp();
  if (lane == 0) {
    C.c[0] = c0;
    C.c[1] = c1;
    C.nch = flags & (CR_TRIAL_NO_ELIGIBLE | CR_TRIAL_EDGE) ? 0 : 2;
    C.move = 2 * r + (fwd ? 0 : 1);
    C.flags = flags;
    C.placeA = placeA;
    C.placeB = placeB;
    C.pres = pres;
    C.ln_ratio_fx = ln;
    C.dself_fx = P.lBself_fx * (long long)sq;
    C.qa_o = qa_o; C.qa_n = qa_n; C.qb_o = qb_o; C.qb_n = qb_n;
    if (LOG) {  // the ids of a trial without eligible particles stay unused
      const unsigned long long nid = new_id(D.phi, D.d, P.m, kk);
      const bool none = flags & CR_TRIAL_NO_ELIGIBLE;
      C.id_a = listA ? id_a : nid;
      C.id_b = none || listB ? id_b : (salt ? nid + 1u : nid);
    }
    if (DA) {
      C.rka = rka;
      C.rkb = rkb;
      C.go = 1;
      C.sur = 0.0f;
      C.sur_fx = 0;
    }
  }
}

// The part of a region that is not on chip: the halo beyond its capacity
// (dense regions; straight from global memory) and a list in global memory.
// Out of line, as it is rare; the queue (qn entries) is continued and emptied.
template <bool LOG, bool FLAT>
__device__ __noinline__ PairSum sweep_rest(const SysParams &P, const TrialCtl &C, const Dom &Rg, int nlist, int i0,
                                           int stride, float2 *q, int qn) {
  const PairK K = pair_k(P);
  const SweepPair sp = sweep_pair(K, Rg.wr + 16, C.c[0], C.c[1], Rg.strad);
  const int lane = threadIdx.x & 31;
  PairSum out{0, 0ull, 0};
  const float4 *lpos = Rg.L.pos;
  const int *linfo = Rg.L.info;
  const int nover = Rg.NH - Rg.nhc, total = nover + (Rg.in_smem ? 0 : nlist);
#pragma unroll 1
  for (int base = 0; base < total; base += stride) {
    const int u = base + i0;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    bool v = false;
    int cls = 0;
    if (u < nover) {
      const int h = Rg.nhc + u;
      const int i = upper_idx(Rg.hpre, Rg.NR, h);
      const int g = Rg.hcell[i] * P.cap + (h - Rg.hpre[i]);
      p = P.pos[g];
      p.x = frame_x(p.x, Rg.strad, 0, P.halfL, P.Lf);
      p.y = frame_x(p.y, Rg.strad, 1, P.halfL, P.Lf);
      p.z = frame_x(p.z, Rg.strad, 2, P.halfL, P.Lf);
      cls = (P.info[g] >> INFO_CLS_SHIFT) & 3;
      v = true;
    } else if (u < total) {
      const int j = u - nover;
      p = lpos[j];
      cls = (linfo[j] >> INFO_CLS_SHIFT) & 3;
      v = j != sp.skA && j != sp.skB;
    }
    offer2<LOG, FLAT>(P, K, Rg.wr, C, sp, v, p.x, p.y, p.z, p.w, [&] { return cls; }, q, qn, out.acc, out.sacc, out.ov);
  }
  __syncwarp();
  if (lane < qn) coul_eval<LOG>(K, q[lane].x, q[lane].y, out.acc, out.sacc, out.ov);
  __syncwarp();
  return out;
}

// The pair changes of the two changed particles A and B against the halo and
// the domain list, summed by a group of threads (thread i0 of `stride`; each
// thread's part is returned; the warp's queued Coulomb pairs are evaluated at
// the end), and the pair between A and B.  One loop over the halo
// and the list in shared memory; per 32 candidates it costs two distance tests
// and one compaction.
template <bool LOG, bool FLAT>
__device__ __forceinline__ PairSum sweep_pairs(const PairK &K, const SysParams &P, const TrialCtl &C, const Dom &Rg,
                                               const float4 *cpos, const unsigned char *hcls, int nlist, int i0,
                                               int stride, float2 *q) {
  const int lane = threadIdx.x & 31;
  const SweepPair sp = sweep_pair(K, Rg.wr + 16, C.c[0], C.c[1], Rg.strad);
  PairSum out{0, 0ull, 0};
  int qn = 0;
  if (i0 < 32 && queue_changed_pair<LOG, FLAT>(P, K, Rg.wr, C, q, out.acc, out.sacc, out.ov)) qn = 1;
  const int nhc = Rg.nhc, total = nhc + (Rg.in_smem ? nlist : 0);
  const int gap = Rg.hcs - nhc;  // from the on-chip halo to the list's slots
  const int skA = sp.skA >= 0 ? nhc + sp.skA : -1, skB = sp.skB >= 0 ? nhc + sp.skB : -1;
#pragma unroll 1
  for (int base = 0; base < total; base += stride) {
    const int u = base + i0;
    const bool v = u < total && u != skA && u != skB;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (v) p = cpos[u < nhc ? u : u + gap];
    offer2<LOG, FLAT>(P, K, Rg.wr, C, sp, v, p.x, p.y, p.z, p.w,
                      [&] { return u < nhc ? (int)hcls[u] : (Rg.L.info[u - nhc] >> INFO_CLS_SHIFT) & 3; }, q, qn,
                      out.acc, out.sacc, out.ov);
  }
  if (Rg.NH > nhc || !Rg.in_smem) {  // uniform over the CTA
    const PairSum g = sweep_rest<LOG, FLAT>(P, C, Rg, nlist, i0, stride, q, qn);
    out.acc += g.acc;
    out.sacc += g.sacc;
    out.ov |= g.ov;
  } else {
    __syncwarp();
    if (lane < qn) coul_eval<LOG>(K, q[lane].x, q[lane].y, out.acc, out.sacc, out.ov);
    __syncwarp();
  }
  return out;
}

// The same without the flat frame: regions wider than 0.4 L, i.e. small boxes
// and the global schedule.  Out of line, so that the flat loop is the only
// pair sweep in the trial loop's code.
template <bool LOG>
__device__ __noinline__ PairSum sweep_general(const SysParams &P, const TrialCtl &C, const Dom &Rg,
                                              const float4 *cpos, const unsigned char *hcls, int nlist, int i0,
                                              int stride, float2 *q) {
  const PairK K = pair_k(P);
  return sweep_pairs<LOG, false>(K, P, C, Rg, cpos, hcls, nlist, i0, stride, q);
}

// ---- Ewald reciprocal part (global schedule): the change of
// sum_k A_k |S(k)|^2 when the changed particles' charges dq enter S(k).  The
// phase exp(i 2 pi n u), u = x / L, is reduced exactly in integers: U = u in
// 0.32 fixed point (FP64), n U mod 2^32 is the fraction of n u; FP32 sincospi
// of that fraction gives the factor.  A reciprocal vector's factor is the
// product of its three axes' factors (the conjugate for negative n), y and x
// first (ew_xy).  The sums' fused products are fixed: contexts and batches,
// items and slices, logged and unlogged trials add the same bits, those of the
// sums before the vectors went by columns.
__device__ __forceinline__ uint32_t ew_frac32(float x, double invL) {
  return (uint32_t)(unsigned long long)llrint((double)x * invL * 4294967296.0);
}
__device__ __forceinline__ float2 ew_factor(uint32_t U, int n) {
  const uint32_t t = (uint32_t)n * U;
  float sn, cs;
  sincospif((float)t * (2.0f / 4294967296.0f), &sn, &cs);
  return make_float2(cs, sn);
}
__device__ __forceinline__ float2 ew_axis(const float2 *f, int n) {
  const float2 v = f[n < 0 ? -n : n];
  return make_float2(v.x, n < 0 ? -v.y : v.y);
}
__device__ __forceinline__ float2 ew_xy(float2 ex, float2 ey) { return cmul(ey, ex); }
__device__ __forceinline__ void ew_decode(int code, int &nx, int &ny, int &nz) {
  nx = (int)(signed char)(code & 255);
  ny = (int)(signed char)((code >> 8) & 255);
  nz = (int)(signed char)((code >> 16) & 255);
}

// the axis factors of the trial's two changed particles (f[c][axis][n], n <=
// kmax) and their charge changes dq[c] (0 where absent); threads tid of T
__device__ __noinline__ void ewald_factors(const SysParams &P, const TrialCtl &C, float2 *f, float *dq, int ewk, int tid,
                                           int T) {
  for (int i = tid; i < 6 * ewk; i += T) {
    const int c = i / (3 * ewk), ax = (i / ewk) % 3, n = i % ewk;
    const Desc &D = C.c[c];
    const float x = ax == 0 ? D.x : (ax == 1 ? D.y : D.z);
    f[i] = ew_factor(ew_frac32(x, P.invLd), n);
  }
  if (tid == 0) {
    dq[0] = (has(C, 0) ? C.qa_n : 0.0f) - (had(C, 0) ? C.qa_o : 0.0f);
    dq[1] = (has(C, 1) ? C.qb_n : 0.0f) - (had(C, 1) ? C.qb_o : 0.0f);
  }
}

// the two changed particles' factors of an item's column, and dS(k) of the
// trial for nz = +-|nz| from them
struct EwColumn {
  float2 a, b;  // e_x e_y of the changed particles
};
__device__ __forceinline__ EwColumn ew_column(const float2 *f, int ewk, int code) {
  int nx, ny, nz;
  ew_decode(code, nx, ny, nz);
  return EwColumn{ew_xy(ew_axis(f, nx), ew_axis(f + ewk, ny)), ew_xy(ew_axis(f + 3 * ewk, nx), ew_axis(f + 4 * ewk, ny))};
}
__device__ __forceinline__ float2 ewald_dS(const EwColumn &c, float2 za, float2 zb, const float *dq) {
  const float2 ea = cmul(c.a, za);
  const float2 eb = cmul(c.b, zb);
  return make_float2(sum2(dq[0], ea.x, dq[1], eb.x), sum2(dq[0], ea.y, dq[1], eb.y));
}
__device__ __forceinline__ float2 ew_conj(float2 v) { return make_float2(v.x, -v.y); }

// this thread's share of the reciprocal energy change, into 2^-32 fixed point
// (items tid, tid + T, ...; an item's vectors loaded ahead; sums of integers,
// so the order of the vectors does not matter)
template <bool WITH_S>
__device__ __noinline__ PairSum ewald_dE(const SysParams &P, const float2 *f, const float *dq, int ewk, int tid,
                                         int T) {
  PairSum out{0, 0ull, 0};
  const float *A = P.ek_A;
  const float2 *S32 = P.ek_Shi;
  const int4 *zt = P.ek_z;
  auto add = [&](float w, float2 s, float2 d) {
    const float term = __fmul_rn(w, __fmaf_rn(2.0f, sum2(s.x, d.x, s.y, d.y), sum2(d.x, d.x, d.y, d.y)));
    if (!(fabsf(term) < BIG_TERM)) {
      out.ov = 1;
    } else {
      out.acc += fix32(term);
      if (WITH_S) out.sacc += (unsigned long long)fix32(fabsf(term));
    }
  };
  for (int it = tid; it < P.ewald_items; it += T) {
    const int2 item = P.ek_item[it];
    const int z0 = item.x >> 16 << 2;
    float w[8];
    float2 sv[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int4 z = zt[z0 + k];
      const bool in = item.y < z.x, neg = in && z0 + k > 0;
      w[2 * k] = in ? A[z.y + item.y] : 0.0f;
      sv[2 * k] = in ? S32[z.y + item.y] : make_float2(0.0f, 0.0f);
      w[2 * k + 1] = neg ? A[z.z + item.y] : 0.0f;
      sv[2 * k + 1] = neg ? S32[z.z + item.y] : make_float2(0.0f, 0.0f);
    }
    const EwColumn c = ew_column(f, ewk, item.x);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (z0 + k >= ewk) break;
      const float2 za = f[2 * ewk + z0 + k], zb = f[5 * ewk + z0 + k];
      add(w[2 * k], sv[2 * k], ewald_dS(c, za, zb, dq));
      add(w[2 * k + 1], sv[2 * k + 1], ewald_dS(c, ew_conj(za), ew_conj(zb), dq));
    }
  }
  return out;
}

// hi + lo += d in FP32 with the rounding error kept (Knuth's two-sum, then
// Dekker's fast two-sum to renormalise: hi stays the FP32 value of the sum)
__device__ __forceinline__ void ew_add2(float &hi, float &lo, float d) {
  const float s = __fadd_rn(hi, d);
  const float bp = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(d, bp));
  const float l = __fadd_rn(lo, err);
  const float h = __fadd_rn(s, l);
  lo = __fsub_rn(l, __fsub_rn(h, s));
  hi = h;
}

// an accepted trial: S(k) += dS(k) for this thread's reciprocal vectors (the
// same items ewald_dE gave it)
__device__ __noinline__ void ewald_update(const SysParams &P, const float2 *f, const float *dq, int ewk, int tid,
                                          int T) {
  auto add = [&](int i, float2 d) {
    float2 hi = P.ek_Shi[i], lo = P.ek_Slo[i];
    ew_add2(hi.x, lo.x, d.x);
    ew_add2(hi.y, lo.y, d.y);
    P.ek_Shi[i] = hi;
    P.ek_Slo[i] = lo;
  };
  for (int it = tid; it < P.ewald_items; it += T) {
    const int2 item = P.ek_item[it];
    const int z0 = item.x >> 16 << 2;
    const EwColumn c = ew_column(f, ewk, item.x);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int4 z = P.ek_z[z0 + k];
      if (item.y >= z.x) break;  // (a column reaches every |nz| below its last)
      const float2 za = f[2 * ewk + z0 + k], zb = f[5 * ewk + z0 + k];
      add(z.y + item.y, ewald_dS(c, za, zb, dq));
      if (z0 + k > 0) add(z.z + item.y, ewald_dS(c, ew_conj(za), ew_conj(zb), dq));
    }
  }
}

// An accepted trial, by one warp: room for the ions an insertion adds -- their
// cells below the cell capacity and the list below its capacity (else -1 and
// nothing changes) -- then the site's charge state, the ions inserted (after
// every entry of their cells, as new ids are the largest) or deleted, the kind
// counts.  Returns the new list size.  Out of line: it runs only for accepted
// trials.  Lists that fit a warp (n + 2 <= 32) hold their order in the lanes
// meanwhile.
__device__ __noinline__ int try_commit(const SysParams &P, const Dom &D, int *misc, const TrialCtl &C,
                                       const TrialPre &q, const float4 *vel, int kk, int n) {
  const int lane = threadIdx.x & 31;
  const DomList &L = D.L;
  const int r = C.move >> 1;
  const bool fwd = (C.move & 1) == 0, salt = r == R_SALT;
  const int kn = r == R_ACID ? K_A0 : K_B0;
  const int nion = salt ? 2 : 1;
  // the ions of the move: kind of the last one (b); a salt move's first is the cation
  const int kB = salt || r == R_BASE ? P.kxm : P.kxp;
  const bool small = n + 2 <= 32;
  uint2 e = make_uint2(15u << ORD_KIND_SHIFT, 0x7fffffffu);
  if (small && lane < n) e = L.ord[lane];
  int at0 = 0, at1 = 0;  // places of the ions inserted
  if (fwd) {
    bool full = n + 2 > D.list_cap;
#pragma unroll 1
    for (int x = 2 - nion; x < 2; ++x) {
      const int rk = salt && x ? q.rankB : q.rankA;
      int below, upto;
      if (small) {
        below = __popc(__ballot_sync(FULL, (int)e.y < rk));
        upto = __popc(__ballot_sync(FULL, (int)e.y <= rk));
      } else {
        below = warp_lower(L.ord, n, rk);
        upto = warp_lower(L.ord, n, rk + 1);
      }
      if (x) at1 = upto;
      else at0 = upto;
      full = full || upto - below + 1 + (salt && x && q.rankB == q.rankA ? 1 : 0) > P.cap;
    }
    if (full) return -1;
    // the first ion of a salt move lies before the second unless its cell ranks higher
    if (salt && q.rankA <= q.rankB) at1 += 1;
  }
  if (!salt) {  // the site's charge state
    const int sl = slot_at(L, C.placeA), kd = fwd ? kn + 1 : kn, dlt = fwd ? 1 : -1;
    const unsigned ne = (unsigned)sl | ((unsigned)kd << ORD_KIND_SHIFT);
    __syncwarp();
    if (lane == 0) {
      L.info[sl] ^= INFO_ION_BIT;
      L.pos[sl].w = C.qa_n;
      L.ord[C.placeA].x = ne;
      misc[1 + kn] -= dlt;
      misc[2 + kn] += dlt;
    }
    if (lane == C.placeA) e.x = ne;
    __syncwarp();
  }
  // the ions, one after another: inserted in the order a, b; deleted from the
  // higher place down
#pragma unroll 1
  for (int y = 0; y < nion; ++y) {
    const bool swap = salt && !fwd && C.placeB < C.placeA;
    const int x = nion == 1 ? 1 : (fwd || swap ? y : 1 - y);
    const int kind = x ? kB : P.kxp;
    const int p = x ? (fwd ? at1 : C.placeB) : (fwd ? at0 : C.placeA);
    if (fwd) {
      const int f = misc[MISC_FREE];  // the last slot freed, or the next unused one
      const int sl = f > 0 ? f - 1 : misc[MISC_HW];
      const bool second = salt && x;
      const uint2 ne = make_uint2((unsigned)sl | ((unsigned)kind << ORD_KIND_SHIFT),
                                  (unsigned)(second ? q.rankB : q.rankA));
      __syncwarp();
      if (lane == 0) {
        if (f > 0) misc[MISC_FREE] = L.info[sl] >> INFO_SITE_SHIFT;
        else misc[MISC_HW] = sl + 1;
        const float X = second ? q.bx : q.ax, Y = second ? q.by : q.ay, Z = second ? q.bz : q.az;
        L.pos[sl] = make_float4(frame_x(X, D.strad, 0, P.halfL, P.Lf), frame_x(Y, D.strad, 1, P.halfL, P.Lf),
                                frame_x(Z, D.strad, 2, P.halfL, P.Lf), x ? C.qb_n : C.qa_n);
        L.vel[sl] = vel[second ? 1 : 0];
        L.id[sl] = new_id(D.phi, D.d, P.m, kk) + (second ? 1u : 0u);
        L.lnk[sl] = 0;
        L.info[sl] = (kind == P.kxp ? P.txp : P.txm) | (P.ion_cls << INFO_CLS_SHIFT);
        misc[1 + kind] += 1;
      }
      if (small) {
        const unsigned ex = __shfl_up_sync(FULL, e.x, 1), ey = __shfl_up_sync(FULL, e.y, 1);
        if (lane > p) e = make_uint2(ex, ey);
        if (lane == p) e = ne;
      } else {
        ord_open(L.ord, n, p);
        if (lane == 0) L.ord[p] = ne;
        __syncwarp();
      }
      n += 1;
    } else {
      const int sl = small ? (int)(__shfl_sync(FULL, e.x, p) & ORD_SLOT_MASK) : slot_at(L, p);
      __syncwarp();
      if (lane == 0) {
        L.pos[sl].w = 0.0f;
        L.info[sl] = INFO_FREE | (misc[MISC_FREE] << INFO_SITE_SHIFT);
        misc[MISC_FREE] = sl + 1;
        misc[1 + kind] -= 1;
      }
      if (small) {
        const unsigned ex = __shfl_down_sync(FULL, e.x, 1), ey = __shfl_down_sync(FULL, e.y, 1);
        if (lane >= p) e = make_uint2(ex, ey);
      } else {
        ord_close(L.ord, n, p);
      }
      n -= 1;
    }
    __syncwarp();
  }
  if (small && lane < n) L.ord[lane] = e;
  if (lane == 0) {
    misc[0] = n;
    misc[MISC_DIRTY] = 1;
  }
  __syncwarp();
  return n;
}

}  // namespace

// Shared memory of a domain's seat: the bytes of each array in order (every
// array starts on a 16-byte boundary); fills the layout, returns the total.
static size_t phase_layout(const PhaseCaps &C, const PhaseShape &S, int warps, int cta_warps, int groups, bool da,
                           PhaseLayout &Y) {
  const size_t dcs = C.dcs, chunk = S.chunk, nr3 = S.nr3 + 1, kc3 = S.kc3 + 1;
  const size_t bytes[PhaseLayout::N_OFF] = {
      sizeof(SysParams),
      sizeof(Dom),
      sizeof(float4) * (C.hcs + dcs),         // halo, then the list's positions
      sizeof(float4) * dcs,                   // velocities
      sizeof(unsigned long long) * dcs,       // ids
      sizeof(long long) * dcs,                // site constants
      sizeof(int) * dcs,                      // info words
      sizeof(uint2) * dcs,                    // canonical order
      (size_t)C.hcs,                          // halo classes
      sizeof(long long) * C.lns,              // log table
      sizeof(TrialPre) * chunk,
      sizeof(float4) * 2 * chunk,             // velocities of inserted ions
      sizeof(TrialCtl) * groups,
      sizeof(long long) * cta_warps,          // the warps' sums
      sizeof(unsigned long long) * cta_warps,
      sizeof(int) * cta_warps,
      sizeof(float2) * QCAP * warps,          // queues of Coulomb pairs
      sizeof(int) * MISC_TOTAL,
      sizeof(int) * nr3,                      // halo cells: counts, cells, prefix sums
      sizeof(int) * nr3,
      sizeof(int) * nr3,
      sizeof(int) * kc3,                      // domain cells: counts, then the cells; prefix sums
      sizeof(int) * kc3,
      sizeof(float2) * 6 * S.ewk,             // Ewald: axis factors, charge changes
      sizeof(float) * 4,
      da ? sizeof(int) * nr3 : 0,             // DA: region cell aggregates (ion charge, site charge, particles)
      da ? sizeof(int) * nr3 : 0,
      da ? sizeof(int) * nr3 : 0,
      da ? sizeof(int) * MLP_IN : 0,          // feature bins, surrogate layers
      da ? sizeof(float) * 2 * MLP_IN : 0,
      da ? sizeof(float) * 2 * MLP_H : 0,
      da ? sizeof(float) * 2 * MLP_H : 0};
  size_t at = 0;
  for (int pass = 0; pass < 2; ++pass)  // first the arrays whose place is the same in both of a launch's layouts
    for (int i = 0; i < PhaseLayout::N_OFF; ++i) {
      const bool sized = (i >= 2 && i <= 9) || (i >= 16 && i <= 22 && i != 17);
      if (sized != (pass == 1)) continue;
      Y.off[i] = (unsigned)at;
      at += (bytes[i] + 15) / 16 * 16;
    }
  Y.dcs = C.dcs;
  Y.hcs = C.hcs;
  Y.lns = C.lns;
  Y.chunk = S.chunk;
  Y.ewk = S.ewk;
  return at;
}

// ---------------------------------------------------------------------------
// One domain of one colour phase of replica `rep`: `rank` is its place in
// the colour's launch order.  Every thread of the CTA calls it; smem is the
// CTA's dynamic shared memory (phase_layout).
//
// Seat threads split into groups: with more than one, the groups take the next
// trials together, each as if those before it were rejected; the trials up to
// the first accepted one are then decided exactly as one after another, and
// the rest are evaluated again on the new state (so the outcomes do not depend
// on the number).
template <bool LOG, bool DA, bool SEATS>
__device__ __forceinline__ void phase_task(unsigned char *smem, const PhaseArgs &A, int which, const Seat<SEATS> seat,
                                           const SysParams *__restrict__ reps, uint32_t sweep, uint32_t sweep0,
                                           int colour, uint32_t key0, uint32_t key1_base, int rep, int rank) {
  const int tid = seat.tid, T = seat.n, GT = seat.gn, lane = tid & 31, warp = tid >> 5;
  const int group = seat.groups > 1 ? tid / GT : 0, gtid = tid - group * GT, gwarp = gtid >> 5;
  // (the offsets come from the launch's constant parameters)
#define CRMC_AT(i) (smem + A.lay[0].off[i])
#define CRMC_SIZED(i) (smem + A.lay[SEATS ? which : 0].off[i])
  SysParams &P = *(SysParams *)CRMC_AT(0);
  Dom &D = *(Dom *)CRMC_AT(1);
  float4 *cpos = (float4 *)CRMC_SIZED(2);  // halo [hcs], then the list's positions [dcs]
  unsigned char *hcls = CRMC_SIZED(8);
  long long *lntab_s = (long long *)CRMC_SIZED(9);
  TrialPre *tp = (TrialPre *)CRMC_AT(10);
  float4 *tvel = (float4 *)CRMC_AT(11);
  TrialCtl *ctls = (TrialCtl *)CRMC_AT(12);
  long long *red = (long long *)CRMC_AT(13);
  unsigned long long *reds = (unsigned long long *)CRMC_AT(14);
  int *redov = (int *)CRMC_AT(15);
  int *misc = (int *)CRMC_AT(17);  // [0] list size, [1 + kind] counts, [MISC_INIT + kind] at start, MISC_HW ...
  int *hcnt = (int *)CRMC_SIZED(18), *hcell = (int *)CRMC_SIZED(19), *hpre = (int *)CRMC_SIZED(20);
  int *dcnt = (int *)CRMC_SIZED(21), *dpre = (int *)CRMC_SIZED(22);
  float2 *ewf = (float2 *)CRMC_AT(23);
  float *ewq = (float *)CRMC_AT(24);
  int *aQi = nullptr, *aQs = nullptr, *aN = nullptr, *dfeat = nullptr;
  float *fv = nullptr, *hb0 = nullptr, *hb1 = nullptr;
  if (DA) {
    aQi = (int *)CRMC_AT(25);
    aQs = (int *)CRMC_AT(26);
    aN = (int *)CRMC_AT(27);
    dfeat = (int *)CRMC_AT(28);
    fv = (float *)CRMC_AT(29);
    hb0 = (float *)CRMC_AT(30);
    hb1 = (float *)CRMC_AT(31);
  }

  {
    const int4 *src = (const int4 *)&reps[rep];
    int4 *dst = (int4 *)&P;
    static_assert(sizeof(SysParams) % 16 == 0, "parameters copied 16 bytes at a time");
    for (int i = tid; i < (int)(sizeof(SysParams) / 16); i += T) dst[i] = src[i];
  }
  if (tid < MISC_TOTAL) misc[tid] = 0;
  seat.sync();
  if (rank >= P.nact) return;  // uniform over the CTA
  const int bdom = P.order ? P.order[colour * P.nact + rank] : rank;  // active-domain index
  const int k = P.k, h = P.h, nc = P.nc, nr = P.nr, m = P.m;
  const int KC = k * k * k, NR = nr * nr * nr;
  const uint32_t key1 = key1_base ^ P.key_xor;

  // ---- which domain
  int dd[3];
  if (P.global) {
    dd[0] = dd[1] = dd[2] = 0;
  } else {
    const int hn = P.nd >> 1;
    const int b = bdom;
    dd[0] = 2 * (b % hn) + (colour & 1);
    dd[1] = 2 * ((b / hn) % hn) + ((colour >> 1) & 1);
    dd[2] = 2 * (b / (hn * hn)) + ((colour >> 2) & 1);
  }
  const int d = dd[0] + P.nd * (dd[1] + P.nd * dd[2]);
  const uint32_t phi = sweep * (uint32_t)P.ncol + (uint32_t)colour;
  int off[3] = {0, 0, 0};
  if (!P.global) {
    const uint4 w = philox10(0u, 0u, sweep, 4u, key0, key1);
    off[0] = pick32(w.x, nc);
    off[1] = pick32(w.y, nc);
    off[2] = pick32(w.z, nc);
  }
  int org[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) org[i] = (off[i] + dd[i] * k) % nc;
  // flat frame (frame_x): a region spanning less than half the box along
  // every axis is compared without minimum-image tests; strad marks the
  // axes along which it wraps around the periodic boundary
  const bool flat = !P.global && 2.5f * (float)nr * P.af < P.Lf;
  int strad = 0;
  if (flat)
    for (int i = 0; i < 3; ++i) strad |= (org[i] < h || org[i] + k + h > nc) ? 1 << i : 0;

  // ---- the region's cells and their counts (four cells per thread at a
  // time, so that their loads are in flight together): the domain's own by
  // rank (the cells where their prefix sums will be), the halo's by region
  // index (zero at the domain's)
  const float rnr = 1.0f / (float)nr;
#pragma unroll 1
  for (int i0 = tid; i0 < NR; i0 += 4 * T) {
    int cl[4], cn[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = min(i0 + u * T, NR - 1), iyz = div_by(i, rnr), iz = div_by(iyz, rnr);
      const int ix = i - iyz * nr, iy = iyz - iz * nr;
      cl[u] = region_coord(ix, org[0], k, h, nr, nc) +
              nc * (region_coord(iy, org[1], k, h, nr, nc) + nc * region_coord(iz, org[2], k, h, nr, nc));
      // the domain's own cells by rank, the others marked
      const int r = ix < k && iy < k && iz < k ? ix + k * (iy + k * iz) : -1;
      cn[u] = P.cnt[cl[u]];
      cl[u] |= r >= 0 ? 0x80000000 : 0;
      if (r >= 0 && i0 + u * T < NR) {
        dpre[r] = cl[u] & 0x7fffffff;
        hcell[i] = r;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * T;
      if (i >= NR) break;
      const bool own = cl[u] < 0;
      hcnt[i] = own ? 0 : cn[u];
      if (own) dcnt[hcell[i]] = cn[u];
      hcell[i] = cl[u] & 0x7fffffff;
    }
  }
  // the WCA pre-check radii
  if (tid < 16) D.wr[tid] = wca_radius(P.wca[tid]);
  if (tid < 4)
    D.wr[16 + tid] = fmaxf(fmaxf(wca_radius(P.wca[4 * tid]), wca_radius(P.wca[4 * tid + 1])),
                           fmaxf(wca_radius(P.wca[4 * tid + 2]), wca_radius(P.wca[4 * tid + 3])));
  seat.sync();
  if (warp == 0) warp_scan<true>(dcnt, KC, dpre);
  if (warp == (T > 32 ? 1 : 0)) warp_scan<false>(hcnt, NR, hpre);
  seat.sync();
  int *dcell = dcnt;  // the domain's cells, from here on
  const int ND = dpre[KC], NH = hpre[NR];
  const int nhc = min(NH, A.lay[SEATS ? which : 0].hcs);
  // the list lives in shared memory unless the domain is unusually dense
  const bool in_smem = ND + 2 * m <= A.lay[SEATS ? which : 0].dcs;
  DomList L;
  L.pos = cpos + A.lay[SEATS ? which : 0].hcs; L.vel = (float4 *)CRMC_SIZED(3); L.id = (unsigned long long *)CRMC_SIZED(4); L.lnk = (long long *)CRMC_SIZED(5);
  L.info = (int *)CRMC_SIZED(6); L.ord = (uint2 *)CRMC_SIZED(7);
  if (!in_smem) {
    const size_t o = (size_t)(colour * P.nact + rank) * P.dcap_glob;  // this domain's region of the replica's scratch
    L.pos = P.gs_pos + o; L.vel = P.gs_vel + o; L.id = P.gs_id + o; L.lnk = P.gs_lnk + o;
    L.info = P.gs_info + o; L.ord = P.gs_ord + o;
    if (ND + 2 * m > P.dcap_glob) {  // cannot happen: a cell holds at most cap particles
      if (tid == 0) atomicOr(P.err, ERRB_CELL_OVERFLOW);
      return;
    }
  }
  const int lnmax_need = min(P.lnmax, ND + 2 * m + 2);
  const bool ln_in_smem = lnmax_need <= A.lay[SEATS ? which : 0].lns;
  const long long *lnt = ln_in_smem ? lntab_s : P.lntab_fx;
  if (tid == 0) {
    D.L = L;
    D.hpre = hpre;
    D.hcell = hcell;
    D.nhc = nhc;
    D.cpos_at = (int)A.lay[SEATS ? which : 0].off[2];
    D.hcls_at = (int)A.lay[SEATS ? which : 0].off[8];
    D.queue_at = (int)A.lay[SEATS ? which : 0].off[16];
    D.hcs = A.lay[SEATS ? which : 0].hcs;
    D.NH = NH;
    D.NR = NR;
    D.in_smem = in_smem ? 1 : 0;
    D.strad = strad;
    D.flat = flat ? 1 : 0;
    D.list_cap = in_smem ? A.lay[SEATS ? which : 0].dcs : P.dcap_glob;
    D.lnt = lnt;
    D.d = d;
    D.phi = phi;
    D.key0 = key0;
    D.key1 = key1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      D.org[i] = org[i];
      D.off[i] = off[i];
      D.dd[i] = dd[i];
    }
    D.log_dom = (long long)(sweep - sweep0) * P.per_sweep + (long long)colour * P.nact * m + (long long)bdom * m;
    misc[0] = ND;
    misc[MISC_HW] = ND;
  }
  // ---- the particles' slots, written by their cells: each halo entry's and
  // list entry's source slot (and rank) waits where the entry itself goes
  for (int i = tid; i < NR; i += T) {
    const int j0 = hpre[i], n = min(hcnt[i], max(nhc - j0, 0)), g = hcell[i] * P.cap;
    for (int q = 0; q < n; ++q) *(int *)&cpos[j0 + q] = g + q;
  }
  for (int r = tid; r < KC; r += T) {
    const int j0 = dpre[r], n = dpre[r + 1] - j0, g = dcell[r] * P.cap;
    for (int q = 0; q < n; ++q) L.ord[j0 + q] = make_uint2((unsigned)(g + q), (unsigned)r);
  }
  if (ln_in_smem)
    for (int i = tid; i < lnmax_need; i += T) lntab_s[i] = P.lntab_fx[i];
  seat.sync();
  // ---- the halo (it does not change during the phase)
  for (int j0 = tid; j0 < nhc; j0 += 4 * T) {
    float4 p[4];
    int inf[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + u * T;
      if (j < nhc) {
        const int g = *(const int *)&cpos[j];
        p[u] = P.pos[g];
        inf[u] = P.info[g];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + u * T;
      if (j < nhc) {
        cpos[j] = make_float4(frame_x(p[u].x, strad, 0, P.halfL, P.Lf), frame_x(p[u].y, strad, 1, P.halfL, P.Lf),
                              frame_x(p[u].z, strad, 2, P.halfL, P.Lf), p[u].w);
        hcls[j] = (unsigned char)((inf[u] >> INFO_CLS_SHIFT) & 3);
      }
    }
  }
  // ---- the list, in canonical order at first
  for (int j = tid; j < ND; j += T) {
    const uint2 o = L.ord[j];
    const int g = (int)o.x;
    const int info = P.info[g];
    const float4 p = P.pos[g], v = P.vel[g];
    const unsigned long long id = P.pid[g];
    const int t = info & INFO_TYPE_MASK, kd = min(kind_of(info), (int)K_OTHER);
    L.pos[j] = make_float4(frame_x(p.x, strad, 0, P.halfL, P.Lf), frame_x(p.y, strad, 1, P.halfL, P.Lf),
                           frame_x(p.z, strad, 2, P.halfL, P.Lf), p.w);
    L.vel[j] = v;
    L.id[j] = id;
    L.lnk[j] = (t == CR_ACID || t == CR_BASE) ? P.lnK_fx[info >> INFO_SITE_SHIFT] : 0ll;
    L.info[j] = info;
    L.ord[j] = make_uint2((unsigned)j | ((unsigned)kd << ORD_KIND_SHIFT), o.y);
    atomicAdd(&misc[1 + kd], 1);
  }
  if (DA) {  // region cell aggregates at the start of the phase
    for (int i = tid; i < NR; i += T) {
      const int cell = hcell[i], cn = P.cnt[cell];
      int qi = 0, qs = 0;
      for (int sl = 0; sl < cn; ++sl) {
        const int g = cell * P.cap + sl;
        const int t = P.info[g] & INFO_TYPE_MASK;
        const int q = __float2int_rn(P.pos[g].w);
        if (is_ion_type(t)) qi += q;
        else if (t == CR_ACID || t == CR_BASE) qs += q;
      }
      aQi[i] = qi;
      aQs[i] = qs;
      aN[i] = cn;
    }
  }
  seat.sync();
  if (tid < N_KIND) misc[MISC_INIT + tid] = misc[1 + tid];
  TrialCtl &ctl = ctls[group];
  // the CTA's statistics: lane l of each group's first warp counts entry l
  unsigned stat = 0u;

  for (int k0 = 0; k0 < P.m; k0 += A.lay[0].chunk) {
    const int nchunk = min(A.lay[0].chunk, P.m - k0);
    // ---- random numbers of the chunk
    draw_chunk<LOG, DA>(P, D, tp, tvel, k0, nchunk, tid, T);
    seat.sync();

    unsigned round = 0u;
    for (int t0 = 0; t0 < nchunk; round ^= 1u) {
      const int t = t0 + group, kk = k0 + t;
      const bool mine = t < nchunk;  // uniform over the group
      // ---- the group's first warp: proposal and participants; the selection
      // lives in shared memory across the sweep
      if (mine && gwarp == 0) select_trial<LOG, DA>(P, D, misc, tp[t], kk, ctl);
      seat.group_sync();
      // Ewald (global schedule): the changed particles' phase factors
      const bool ew = !DA && P.ewald_nk > 0 && ctl.nch;  // (one group: the shapes of Ewald systems)
      if (ew) {
        ewald_factors(P, ctl, ewf, ewq, A.lay[0].ewk, tid, T);
        seat.sync();
      }
      // ---- delayed acceptance (one group, no seats: its forms), stage 1:
      // surrogate features and MLP (all threads), decision in the first warp; a
      // rejection skips the pair sweep
      if (DA && mine && ctl.nch) {
        for (int i = gtid; i < MLP_IN; i += GT) dfeat[i] = 0;
        seat.group_sync();
        const int rka = ctl.rka, rkb = ctl.rkb;
        const int dqa = d_charge(ctl, 0), dqb = d_charge(ctl, 1);
        const int ea = d_presence(ctl, 0), eb = d_presence(ctl, 1);
        const int cat_a = (ctl.move >> 1) == R_SALT ? 0 : 8;  // feature group of a (0 ion, 8 site)
        for (int it = gtid; it < 250; it += GT) {  // 2 changed particles x 125 stencil cells
          const int sb = it >= 125 ? 1 : 0;
          const int c = it - 125 * sb;
          const int dx = c % 5 - 2, dy = (c / 5) % 5 - 2, dz = c / 25 - 2;
          const int ri = region_of(sb ? rkb : rka, dx, dy, dz, P.k, P.nr);
          const int sh = shell_of_n2(dx * dx + dy * dy + dz * dz);
          const int dq = sb ? dqb : dqa, eta = sb ? eb : ea;
          if (dq != 0) {
            const int qi = aQi[ri], qs = aQs[ri];
            if (qi) atomicAdd(&dfeat[24 * sb + sh], dq * qi);
            if (qs) atomicAdd(&dfeat[24 * sb + 8 + sh], dq * qs);
          }
          if (eta != 0 && aN[ri]) atomicAdd(&dfeat[24 * sb + 16 + sh], eta * aN[ri]);
        }
        seat.group_sync();
        if (gtid == 0) {  // the changed particles themselves do not count; the a-b pair term
          const TrialCtl &C = ctl;
          for (int sb = 0; sb < 2; ++sb) {
            const int rs = sb ? rkb : rka, dq = sb ? dqb : dqa, eta = sb ? eb : ea;
            for (int x = 0; x < 2; ++x) {
              if (!had(C, x)) continue;
              const int sh = shell_ranks(rs, x ? rkb : rka, P.k);
              if (sh < 0) continue;
              dfeat[24 * sb + (x ? 0 : cat_a) + sh] -= dq * q_old(C, x);
              dfeat[24 * sb + 16 + sh] -= eta;
            }
          }
          const int sh = shell_ranks(rka, rkb, P.k);
          if (sh >= 0) dfeat[sh] += q_new(C, 0) * q_new(C, 1) - q_old(C, 0) * q_old(C, 1);
        }
        seat.group_sync();
        for (int i = gtid; i < MLP_IN; i += GT) {
          const float f = (float)dfeat[i];
          fv[i] = f;
          fv[MLP_IN + i] = -f;
          if (LOG && P.feat_log) P.feat_log[(size_t)(D.log_dom + kk) * MLP_IN + i] = f;
        }
        seat.group_sync();
        mlp_layer((const uint4 *)(P.mlp_w + MLPW_W1), P.mlp_b, fv, MLP_IN, hb0, gtid, seat.gn);
        seat.group_sync();
        mlp_layer((const uint4 *)(P.mlp_w + MLPW_W2), P.mlp_b + MLP_H, hb0, MLP_H, hb1, gtid, seat.gn);
        seat.group_sync();
        mlp_layer((const uint4 *)(P.mlp_w + MLPW_W3), P.mlp_b + 2 * MLP_H, hb1, MLP_H, hb0, gtid, seat.gn);
        seat.group_sync();
        if (gwarp == 0) {
          float y = 0.0f;
          if (lane < 2) {
            y = __ldg(&P.mlp_b[3 * MLP_H]);
            const uint4 *w4 = (const uint4 *)(P.mlp_w + MLPW_W4);
            const float4 *hv = (const float4 *)(hb0 + lane * MLP_H);
#pragma unroll 4
            for (int kb = 0; kb < MLP_H / 8; ++kb) y = mlp_block(__ldg(&w4[kb]), hv[2 * kb], hv[2 * kb + 1], y);
          }
          const float y0 = __shfl_sync(FULL, y, 0), y1 = __shfl_sync(FULL, y, 1);
          const float sur = 0.5f * (y0 - y1);
          bool s1 = false;  // NaN: rejected, as a comparison with NaN is false
          long long sur_fx = 0;
          if (sur == sur) {
            sur_fx = __double2ll_rn((double)fminf(fmaxf(sur, -16384.0f), 16384.0f) * LNFIX);
            s1 = accept_fx(ctl.ln_ratio_fx - ctl.dself_fx - sur_fx, tp[t].lnu_f, tp[t].uhi, tp[t].ulo);
          }
          if (lane == 0) {
            ctl.go = s1 ? 1 : 0;
            ctl.sur = sur;
            ctl.sur_fx = sur_fx;
          }
        }
        seat.group_sync();
      } else if (DA && mine && LOG && P.feat_log) {
        for (int i = gtid; i < MLP_IN; i += GT) P.feat_log[(size_t)(D.log_dom + kk) * MLP_IN + i] = 0.0f;
      }
      // ---- the group: the pair-change sweep
      const int nch = !mine || (DA && !LOG && !ctl.go) ? 0 : ctl.nch;
      long long acc = 0;
      unsigned long long sacc = 0;
      int ov = 0;
      if (nch) {
        const int nlist = misc[MISC_HW];
        const float4 *cp = (const float4 *)(smem + D.cpos_at);
        const unsigned char *hc = smem + D.hcls_at;
        float2 *queue = (float2 *)(smem + D.queue_at) + warp * QCAP;
        const PairSum ps = D.flat ? sweep_pairs<LOG, true>(pair_k(P), P, ctl, D, cp, hc, nlist, gtid, GT, queue)
                                  : sweep_general<LOG>(P, ctl, D, cp, hc, nlist, gtid, GT, queue);
        acc = ps.acc;
        sacc = ps.sacc;
        ov = ps.ov;
        if (ew) {
          const PairSum e = ewald_dE<LOG>(P, ewf, ewq, A.lay[0].ewk, tid, T);
          acc += e.acc;
          sacc += e.sacc;
          ov |= e.ov;
        }
        acc = warp_sum_i64(acc);
        if (LOG) sacc = (unsigned long long)warp_sum_i64((long long)sacc);
        ov = __any_sync(FULL, ov) ? 1 : 0;
        if (GT > 32 && lane == 0) {
          red[warp] = acc;
          reds[warp] = sacc;
          redov[warp] = ov;
        }
      }
      if (GT > 32) seat.group_sync();
      // ---- the group's first warp: decision
      bool accept = false;
      int flags = 0;
      double dE = 0.0, Ssum = 0.0, lnA = -INFINITY, lnA2r = quiet_nan();  // records only
      const bool s1 = !DA || ctl.go != 0;
      if (mine && gwarp == 0) {
        const TrialPre &q = tp[t];
        const int s_nch = ctl.nch;
        const long long s_ln_ratio = ctl.ln_ratio_fx, s_dself = ctl.dself_fx;
        const float sur = DA ? ctl.sur : 0.0f;
        flags = ctl.flags;
        if (DA && LOG && s_nch) lnA = (double)s_ln_ratio / LNFIX - (double)s_dself / LNFIX - (double)sur;
        if (s_nch && (!DA || LOG || s1)) {
          long long tot = acc;
          unsigned long long stot = sacc;
          int anyov = ov;
          if (GT > 32) {
            const int gw = GT >> 5;
            tot = warp_sum_i64(lane < gw ? red[warp + lane] : 0ll);
            if (LOG) stot = (unsigned long long)warp_sum_i64(lane < gw ? (long long)reds[warp + lane] : 0ll);
            anyov = __any_sync(FULL, lane < gw && redov[warp + lane]) ? 1 : 0;
          }
          if (anyov) {
            if (!DA || s1) flags |= CR_TRIAL_OVERLAP;  // DA: only an exact evaluation that decides
            dE = INFINITY;
          } else {
            const long long totc = tot > DE_CLAMP32 ? DE_CLAMP32 : (tot < -DE_CLAMP32 ? -DE_CLAMP32 : tot);
            if (DA) {  // stage 2: ln u2 < dE~ - dE_pair
              if (s1) accept = accept_fx(ctl.sur_fx - (totc << 16), q.lnu2_f, q.u2hi, q.u2lo);
            } else {
              accept = accept_fx(s_ln_ratio - ((totc << 16) + s_dself), q.lnu_f, q.uhi, q.ulo);
            }
            if (LOG) {
              dE = (double)tot * FIX_INV + (double)s_dself / LNFIX;
              Ssum = (double)stot * FIX_INV + fabs((double)s_dself / LNFIX);
              if (!DA) lnA = (double)s_ln_ratio / LNFIX - dE;  // unclamped, for the record
              else lnA2r = (double)sur - (double)tot * FIX_INV;
            }
          }
        }
      }
      // ---- with several groups: the trials up to and including the first
      // accepted one are decided; the later ones were evaluated on a state
      // that it changes, and are taken up again in the next round
      bool decided = mine;
      int done = 1;
      unsigned won = 0u;
      if (seat.groups > 1) {
        int *res = misc + MISC_RES + round * MAX_GROUPS;
        if (gwarp == 0 && lane == 0) res[group] = accept ? 1 : 0;
        seat.sync();
        won = __ballot_sync(FULL, lane < seat.groups && res[lane] != 0);
        const int first = won ? __ffs(won) - 1 : seat.groups - 1;
        decided = mine && group <= first;
        accept = accept && group == first;
        done = min(first + 1, nchunk - t0);
      }
      // ---- commit, unless an insertion finds no room (checked before
      // anything changes)
      if (accept) {
        const int n2 = try_commit(P, D, misc, ctl, tp[t], tvel + 2 * t, kk, misc[0]);
        if (n2 < 0) {
          accept = false;
          if (lane == 0) atomicOr(P.err, ERRB_CELL_OVERFLOW);
        } else {
          flags |= CR_TRIAL_ACCEPTED;
          if (DA && lane == 0) {  // region aggregates follow the committed change
            const TrialCtl &C = ctl;
            for (int x = 0; x < 2; ++x) {
              const int ri = region_of(x ? C.rkb : C.rka, 0, 0, 0, P.k, P.nr);
              int *aq = (x == 0 && (C.move >> 1) != R_SALT) ? aQs : aQi;
              aq[ri] += d_charge(C, x);
              aN[ri] += d_presence(C, x);
            }
          }
        }
      }
      if (decided && gwarp == 0) {
        const unsigned hit = (1u << ctl.move) | (accept ? 64u << ctl.move : 0u) |
                             (flags & CR_TRIAL_NO_ELIGIBLE ? 1u << 12 : 0u) |
                             (flags & CR_TRIAL_EDGE ? 1u << 13 : 0u) | (flags & CR_TRIAL_OVERLAP ? 1u << 14 : 0u) |
                             (1u << 15);
        stat += (hit >> lane) & 1u;
        if (lane == 0) {
          ctl.ewacc = accept ? 1 : 0;
          if (LOG && P.log) {
            cr_trial rec;
            rec.move = ctl.move;
            rec.flags = flags;
            rec.id_a = ctl.id_a;
            rec.id_b = ctl.id_b;
            rec.dE = dE;
            rec.S = Ssum;
            rec.lnA = lnA;
            rec.lnu = tp[t].lnu;
            P.log[D.log_dom + kk] = rec;
            if (DA && P.dlog) {
              cr_trial_da dr;
              dr.dE_sur = ctl.nch ? ctl.sur : 0.0f;
              dr.stage = ctl.nch ? (s1 ? 2 : 1) : 0;
              dr.lnA2 = lnA2r;
              dr.lnu2 = ctl.nch ? tp[t].lnu2 : quiet_nan();
              P.dlog[D.log_dom + kk] = dr;
            }
          }
        }
      }
      t0 += done;
      if (won) seat.sync();  // the next selections see the committed state
      if (ew) {
        seat.sync();
        if (ctl.ewacc) ewald_update(P, ewf, ewq, A.lay[0].ewk, tid, T);
      }
      // (the other warps wait for the first one's next selection at the
      // group's barrier; what they read of this trial they have read)
    }
    seat.sync();  // the chunk's numbers have been read
  }
  // ---- write the domain back (id-sorted cells), if anything changed, and
  // publish the counts
  if (misc[MISC_DIRTY]) {
    const DomList L = D.L;
    const int n = misc[0], KC = P.k * P.k * P.k;
    for (int r = tid; r < KC; r += T) {
      int lo = 0, hi = n;  // first entry with rank >= r
      while (lo < hi) { const int mid = (lo + hi) >> 1; if ((int)L.ord[mid].y < r) lo = mid + 1; else hi = mid; }
      int lo2 = lo, hi2 = n;  // first entry with rank > r
      while (lo2 < hi2) { const int mid = (lo2 + hi2) >> 1; if ((int)L.ord[mid].y <= r) lo2 = mid + 1; else hi2 = mid; }
      const int cell = dcell[r];
      dcell[r] = cell * P.cap - lo;  // from a place in the list to the slot
      P.cnt[cell] = lo2 - lo;
    }
    seat.sync();
    for (int j = tid; j < n; j += T) {
      const uint2 o = L.ord[j];
      const int sl = (int)(o.x & ORD_SLOT_MASK);
      const int g = dcell[o.y] + j;
      const unsigned long long id = L.id[sl];
      P.pos[g] = raw_pos(L, sl, P.Lf);
      P.vel[g] = L.vel[sl];
      P.pid[g] = id;
      P.info[g] = L.info[sl];
      if (id < (unsigned long long)P.n_perm) P.perm_slot[id] = g;
    }
    if (tid < N_KIND && misc[1 + tid] != misc[MISC_INIT + tid])
      atomicAdd((unsigned long long *)&P.counts[tid],
                (unsigned long long)(long long)(misc[1 + tid] - misc[MISC_INIT + tid]));
  }
  if (gwarp == 0 && lane < 16 && stat) atomicAdd(&P.stats[lane], (unsigned long long)stat);
#undef CRMC_AT
#undef CRMC_SIZED
}

// ---------------------------------------------------------------------------
// the phase kernel.  Of a replica's domains (densest first) the first
// A.wide16 / 16 have a CTA each; the others share CTAs, one domain per seat of
// blockDim / A.seats threads.  Thread counts are run-time values, so that every
// seat runs the same code.
//
// What bounds it: one domain's chain of trials, each some 200 + instructions
// that one warp runs once while the others wait (of the 9.6 cycles between a
// warp's instructions 2.8 are spent at barriers, 2.2 on fixed latencies, 0.9 on
// global and 0.9 on shared loads, 0.5 on instruction fetch; issue active 34 %,
// 12.5 warps per SM; 64 threads per domain and longer code in the trial loop:
// 13.6 cycles, 3.8 at barriers, 3.2 on instruction fetch, 24 %).
// With one CTA of 64 threads per domain the densest domain of a colour, coils
// of a chain with 60 and more beads, lasted as long as two waves of the others.
// Seats give it four times the threads and the shared memory of four, from the
// same launch.  The same sweep of 13 polyelectrolyte boxes (125 domains a colour
// each): 0.96 ms with 64 threads per domain, 0.82 ms with 1/16 of the domains on
// 256 threads and the rest on seats of 64; 64 ragged single chains 0.76 ms with
// 128 threads, 0.65 ms with two seats; one box of 1,000 domains a colour 0.61 and
// 0.53 ms.  A box alone (125 domains for 152 SMs) runs fastest with 256 threads
// for every domain.
// ---------------------------------------------------------------------------
template <bool LOG, bool DA, bool SEATS>
__global__ void __launch_bounds__(512, 1)
    k_cr_phase(const SysParams *__restrict__ reps, const __grid_constant__ PhaseArgs A, uint32_t sweep,
               uint32_t sweep0, int colour, uint32_t key0, uint32_t key1_base, const StepDyn *dyn) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (dyn) {  // a captured cycle: this step's sweep counter and key
    const unsigned long long step = dyn->step, seed = dyn->sweep_seed0 + step;
    sweep = dyn->sweep0 + (uint32_t)step;
    key0 = (uint32_t)seed;
    key1_base = (uint32_t)(seed >> 32);
  }
  const int rep = (int)blockIdx.x, y = (int)blockIdx.y, T = (int)blockDim.x;
  int rank = y, which = 0, base = 0;
  Seat<SEATS> seat{(int)threadIdx.x, T, A.groups, T / A.groups, 0};
  if (SEATS) {
    const int wide = (reps[rep].nact * A.wide16 + 15) >> 4;
    if (y >= wide) {  // one of the CTA's seats
      const int n = T / A.seats, at = (int)threadIdx.x / n;
      rank = wide + (y - wide) * A.seats + at;
      seat = Seat<SEATS>{(int)threadIdx.x - at * n, n, 1, n, at};
      which = 1;
      base = at * (int)A.seat_bytes;
    }
  }
  phase_task<LOG, DA, SEATS>(smem + base, A, which, seat, reps, sweep, sweep0, colour, key0, key1_base, rep, rank);
}

// ---------------------------------------------------------------------------
// The persistent sweep: every colour of every replica of a batch in one
// launch.  CTAs claim tasks (colour c, replica r, domain rank i) in that
// order from a counter.  A domain's phase reads its region -- its own cells
// and the halo, which lies inside its 26 neighbouring domains -- and writes
// only its own cells, so the colour-by-colour schedule is reproduced exactly
// when each task starts after its neighbours of lower colours have finished
// (per-domain completion flags; Q.fine) or, for geometries whose halo reaches
// beyond the neighbouring domains, after its replica's whole previous colour
// (per-(replica, colour) counters).  Tasks of later colours thus start while
// distant domains of earlier colours still run, and no colour waits for the
// slowest domain of the batch.  A task is claimed only after every task it
// depends on was claimed, so the claims always make progress; each wait is
// nevertheless bounded in time, and a wait that runs out marks the replica's
// error word (ERRB_TIMEOUT), raises the launch's abort flag and skips the
// task, after which every remaining task is skipped without waiting.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// linear index of the domain of active rank i in colour c of replica P
__device__ __forceinline__ int task_domain(const SysParams &P, int c, int i, int (&dd)[3]) {
  const int b = P.order ? P.order[c * P.nact + i] : i;
  const int hn = P.nd >> 1;
  dd[0] = 2 * (b % hn) + (c & 1);
  dd[1] = 2 * ((b / hn) % hn) + ((c >> 1) & 1);
  dd[2] = 2 * (b / (hn * hn)) + ((c >> 2) & 1);
  return dd[0] + P.nd * (dd[1] + P.nd * dd[2]);
}

// bounded wait of one lane until *p >= need; false when the time ran out or
// the launch was aborted
__device__ __forceinline__ bool wait_at_least(const unsigned *p, unsigned need, const SweepSched &Q, int &timed_out) {
  const unsigned long long t0 = global_ns();
  while (ld_acquire_u32(p) < need) {
    if (*(volatile int *)Q.abort) return false;
    if (global_ns() - t0 > Q.wait_ns) {
      timed_out = 1;
      return false;
    }
    __nanosleep(64);
  }
  return true;
}

template <bool DA>
__global__ void __launch_bounds__(512, 1)
    k_cr_sweep(const SysParams *__restrict__ reps, const __grid_constant__ PhaseArgs A, uint32_t sweep,
               uint32_t sweep0, uint32_t key0, uint32_t key1_base, SweepSched Q, const StepDyn *dyn) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (dyn) {  // a captured cycle: this step's sweep counter and key
    const unsigned long long step = dyn->step, seed = dyn->sweep_seed0 + step;
    sweep = dyn->sweep0 + (uint32_t)step;
    key0 = (uint32_t)seed;
    key1_base = (uint32_t)(seed >> 32);
  }
  __shared__ int s_task, s_run, s_dom;
  const int lane = threadIdx.x & 31;
  const int per_colour = Q.rep_first[Q.n_rep];
  const int total = per_colour * Q.ncol;
  for (;;) {
    if (threadIdx.x < 32) {  // warp 0: claim a task and wait for what it depends on
      int t = 0;
      if (lane == 0) t = (int)atomicAdd(Q.next, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
      int run = 0, dom = -1;
      if (t < total) {
        const int c = t / per_colour, q = t - c * per_colour;
        int r = 0;
        while (Q.rep_first[r + 1] <= q) ++r;
        const SysParams &P = reps[r];
        int dd[3] = {0, 0, 0};
        if (Q.fine) dom = task_domain(P, c, q - Q.rep_first[r], dd);
        int ok = *(volatile int *)Q.abort ? 0 : 1, timed_out = 0;
        if (ok && c > 0) {
          if (Q.fine) {  // lane l < 26: neighbour l of the 3^3 block around the domain
            const int nd = P.nd;
            if (lane < 26) {
              const int o = lane < 13 ? lane : lane + 1;
              const int nx = (dd[0] + o % 3 - 1 + nd) % nd, ny = (dd[1] + (o / 3) % 3 - 1 + nd) % nd,
                        nz = (dd[2] + o / 9 - 1 + nd) % nd;
              const int col = (nx & 1) | ((ny & 1) << 1) | ((nz & 1) << 2);
              if (col < c) ok = wait_at_least(Q.flags + Q.dom_first[r] + nx + nd * (ny + nd * nz), 1u, Q, timed_out);
            }
          } else if (lane == 0) {  // the replica's whole previous colour
            const unsigned need = (unsigned)(Q.rep_first[r + 1] - Q.rep_first[r]);
            ok = wait_at_least(Q.done + r * Q.ncol + (c - 1), need, Q, timed_out);
          }
          ok = __all_sync(0xffffffffu, ok);
          if (__any_sync(0xffffffffu, timed_out) && lane == 0) {
            atomicOr(P.err, ERRB_TIMEOUT);
            atomicExch(Q.abort, 1);
          }
        }
        run = ok;
      }
      if (lane == 0) {
        s_task = t;
        s_run = run;
        s_dom = dom;
      }
    }
    __syncthreads();
    const int t = s_task;
    if (t >= total) break;
    const int c = t / per_colour, q = t - c * per_colour;
    int r = 0;
    while (Q.rep_first[r + 1] <= q) ++r;
    if (s_run)
      phase_task<false, DA, false>(smem, A, 0, Seat<false>{(int)threadIdx.x, (int)blockDim.x, A.groups, (int)blockDim.x / A.groups, 0},
                            reps, sweep, sweep0, c, key0, key1_base, r, q - Q.rep_first[r]);
    __syncthreads();  // the task's stores are done, its shared memory is free
    if (threadIdx.x == 0 && !(r == Q.withhold_rep && c == 0)) {
      __threadfence();
      if (Q.fine) st_release_u32(Q.flags + Q.dom_first[r] + s_dom, 1u);
      else atomicAdd(Q.done + r * Q.ncol + c, 1u);
    }
  }
}

// the launch's constant parameters: layouts of a CTA's domain and of a seat's
static PhaseArgs phase_args(const PhaseShape &S, const PhaseForm &F, bool da, size_t *smem) {
  PhaseArgs A{};
  A.seats = F.seats;
  A.groups = F.groups;
  A.wide16 = F.wide16;
  const int warps = F.threads / 32;
  const size_t wide = phase_layout(F.compact ? S.small : S.full, S, warps, warps, F.groups, da, A.lay[0]);
  size_t narrow = 0;
  if (F.seats > 1) narrow = phase_layout(S.small, S, warps / F.seats, warps, 1, da, A.lay[1]);
  A.seat_bytes = (unsigned)narrow;
  *smem = std::max(wide, narrow * (size_t)F.seats);
  return A;
}

size_t phase_smem_bytes(const PhaseShape &S, const PhaseForm &F, bool da) {
  size_t b = 0;
  phase_args(S, F, da, &b);
  return b;
}

template <bool DA>
static cudaError_t launch_sweep_t(const SysParams *d_reps, const PhaseShape &S, const PhaseForm &F, cudaStream_t s,
                                  uint32_t sweep, uint32_t sweep0, uint32_t k0, uint32_t k1, const SweepSched &Q,
                                  int max_ctas, const StepDyn *dyn) {
  static size_t attr_bytes = 0;
  size_t smem = 0;
  const PhaseArgs A = phase_args(S, F, DA, &smem);
  if (smem > attr_bytes) {
    cudaError_t e = cudaFuncSetAttribute(k_cr_sweep<DA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_bytes = smem;
  }
  int per_sm = 0;  // resident CTAs per SM at this block and shared-memory size
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cr_sweep<DA>, F.threads, smem);
  if (e != cudaSuccess) return e;
  per_sm = std::max(per_sm, 1);
  const int total = Q.tasks_total;
  int grid = std::min(total, per_sm * device_sms());
  if (max_ctas > 0) grid = std::min(grid, max_ctas);
  if (grid <= 0) return cudaSuccess;
  k_cr_sweep<DA><<<grid, F.threads, smem, s>>>(d_reps, A, sweep, sweep0, k0, k1, Q, dyn);
  return cudaGetLastError();
}

cudaError_t launch_sweep(const SysParams *d_reps, const PhaseShape &S, const PhaseForm &F, bool da, cudaStream_t s,
                         uint32_t sweep, uint32_t sweep0, uint32_t k0, uint32_t k1, const SweepSched &Q, int max_ctas,
                         const StepDyn *dyn) {
  return da ? launch_sweep_t<true>(d_reps, S, F, s, sweep, sweep0, k0, k1, Q, max_ctas, dyn)
            : launch_sweep_t<false>(d_reps, S, F, s, sweep, sweep0, k0, k1, Q, max_ctas, dyn);
}

// ---------------------------------------------------------------------------
// Launch order of the domains of one colour for one sweep, by decreasing
// expected time (ties by index).  A domain's time goes by the particles of its
// region (its cells and the halo around them: the sweep's candidates) and more
// by its own (near pairs of inserted ions, list scans: about five candidates'
// worth each); one whose list does not fit a seat's shared memory comes before
// all others, so that it gets a CTA's.  k_domain_cost: one warp sums a region's
// cell counts at the start of the sweep; k_domain_rank: each domain counts the
// costlier ones of its colour.  Only the order of independent CTAs changes,
// never a result.  Colours of more than ORDER_MAX_NACT domains keep the
// natural order (P.order is null).  (One CTA per replica and colour for both
// took 187 us for 8 x 1,000 domains and 25 us for 13 x 8 x 125;
// the two kernels 10 + 15 and 13 + 4 us: cycles of the large box 4.17 -> 3.20 ms,
// two nanoparticles, whose 1,000 sites crowd a few domains, 2.13 -> 1.88 ms.)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_domain_cost(const SysParams *__restrict__ reps, uint32_t sweep, uint32_t key0,
                                                     uint32_t key1_base, const StepDyn *dyn) {
  if (dyn) {  // a captured cycle: this step's sweep counter and key
    const unsigned long long step = dyn->step, seed = dyn->sweep_seed0 + step;
    sweep = dyn->sweep0 + (uint32_t)step;
    key0 = (uint32_t)seed;
    key1_base = (uint32_t)(seed >> 32);
  }
  const SysParams &P = reps[blockIdx.y];
  if (!P.order) return;
  const int lane = threadIdx.x & 31, task = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nact = P.nact, c = task / nact, b = task - c * nact;
  if (c >= P.ncol) return;
  const int nc = P.nc, nr = P.nr, h = P.h, k = P.k;
  const uint4 w = philox10(0u, 0u, sweep, 4u, key0, key1_base ^ P.key_xor);
  const int off[3] = {pick32(w.x, nc), pick32(w.y, nc), pick32(w.z, nc)};
  const int hn = P.nd >> 1, nr3 = nr * nr * nr;
  const int dd[3] = {2 * (b % hn) + (c & 1), 2 * ((b / hn) % hn) + ((c >> 1) & 1), 2 * (b / (hn * hn)) + ((c >> 2) & 1)};
  int o[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) o[i] = (off[i] + dd[i] * k) % nc;  // the domain's first cell
  const float rnr = 1.0f / (float)nr;
  int sum = 0, own = 0;
  for (int i = lane; i < nr3; i += 32) {
    const int iyz = div_by(i, rnr), iz = div_by(iyz, rnr), ix = i - iyz * nr, iy = iyz - iz * nr;
    const int n = P.cnt[region_coord(ix, o[0], k, h, nr, nc) +
                        nc * (region_coord(iy, o[1], k, h, nr, nc) + nc * region_coord(iz, o[2], k, h, nr, nc))];
    sum += n;
    own += ix < k && iy < k && iz < k ? n : 0;
  }
  sum = (int)__reduce_add_sync(FULL, (unsigned)sum);
  own = (int)__reduce_add_sync(FULL, (unsigned)own);
  if (lane == 0) P.cost[task] = min(sum + 4 * own, (1 << 24) - 1) + (own + 2 * P.m > P.list_small ? 1 << 24 : 0);
}

__global__ void __launch_bounds__(256) k_domain_rank(const SysParams *__restrict__ reps) {
  const SysParams &P = reps[blockIdx.z];
  const int c = blockIdx.y, nact = P.nact;
  if (!P.order || c >= P.ncol || (int)(blockIdx.x * blockDim.x) >= nact) return;
  __shared__ __align__(16) int cost[ORDER_MAX_NACT];
  const int pad = (nact + 3) & ~3;
  for (int i = threadIdx.x; i < pad; i += blockDim.x) cost[i] = i < nact ? P.cost[c * nact + i] : -1;
  __syncthreads();
  const int b = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (b >= nact) return;
  const int cb = cost[b];
  int rank = 0;
  for (int j = 0; j < pad; j += 4) {
    const int4 v = *(const int4 *)&cost[j];
    rank += (v.x > cb || (v.x == cb && j < b)) + (v.y > cb || (v.y == cb && j + 1 < b)) +
            (v.z > cb || (v.z == cb && j + 2 < b)) + (v.w > cb || (v.w == cb && j + 3 < b));
  }
  P.order[c * nact + rank] = b;
}

cudaError_t launch_domain_order(const SysParams *d_reps, int n_rep, int ncol, int nact, cudaStream_t s, uint32_t sweep,
                                uint32_t k0, uint32_t k1, const StepDyn *dyn) {
  if (nact > ORDER_MAX_NACT) nact = ORDER_MAX_NACT;  // contexts beyond keep P.order null
  k_domain_cost<<<dim3((unsigned)(ncol * nact + 7) / 8, (unsigned)n_rep), 256, 0, s>>>(d_reps, sweep, k0, k1, dyn);
  k_domain_rank<<<dim3((unsigned)(nact + 255) / 256, (unsigned)ncol, (unsigned)n_rep), 256, 0, s>>>(d_reps);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Ewald structure factor S(k) = sum_j q_j exp(i k.r_j) of every replica from
// scratch (at every sweep): k_ewald_list lists each replica's occupied slots
// (one CTA per replica, cells in order), k_ewald_sk gives each item (up to
// eight reciprocal vectors) or each vector a thread, the particles in tiles of
// 32 whose axis factors the CTA computes together in shared memory (FP32
// products summed per tile, tiles summed in FP64).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_ewald_list(const SysParams *__restrict__ reps) {
  const SysParams &P = reps[blockIdx.x];
  if (P.ewald_nk <= 0) return;
  __shared__ int warp_tot[8];
  __shared__ int base_s;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) base_s = 0;
  __syncthreads();
  for (int c0 = 0; c0 < P.ncell; c0 += 256) {
    const int c = c0 + (int)threadIdx.x;
    const int n = c < P.ncell ? P.cnt[c] : 0;
    int x = n;  // inclusive scan over the CTA
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    int before = base_s;
    for (int i = 0; i < w; ++i) before += warp_tot[i];
    const int start = before + x - n;
    for (int sl = 0; sl < n; ++sl) {
      if (start + sl < P.ek_cap) P.ek_list[start + sl] = c * P.cap + sl;
      else atomicOr(P.err, ERRB_CAPACITY);  // more particles than the context's capacity
    }
    __syncthreads();
    if (threadIdx.x == 255) base_s = start + n;
    __syncthreads();
  }
  if (threadIdx.x == 0) *P.ek_np = min(base_s, P.ek_cap);
}

constexpr int EW_TILE = 32;
constexpr int EW_KMAX = 32;

// FP32 pipes and shared-memory reads bound it where there are many boxes: a
// thread per vector took three factors from shared memory and two complex
// products for every particle, an item's thread forms e_x e_y once for up to
// eight vectors and reads each e_z, which is uniform over the warp, once for +nz
// and -nz (64 boxes of 1,150 particles, |n| <= 16, 8,578 vectors: 735 us with a
// vector per thread, 451 us).  A few boxes do not fill the SMs with items (one has
// 10 CTAs of them) and are bound by a thread's chain: there a thread takes one
// vector, in the order of nz, ny, nx (consecutive lanes read consecutive factors),
// and 256 threads share a tile's factors while such CTAs have an SM each, 512
// beyond (one box 138 us with 256, 145 with 512, 276 by items, 198 with a thread
// per column and |nz|; 8 boxes 163 and 154; 24 boxes 310 with 512, 344 by items;
// 32 boxes 407 and 363).
template <bool ITEMS, int THREADS>
__global__ void __launch_bounds__(THREADS) k_ewald_sk(const SysParams *__restrict__ reps) {
  constexpr int NV = ITEMS ? 8 : 1;  // vectors of a thread
  const SysParams &P = reps[blockIdx.y];
  const int n_work = ITEMS ? P.ewald_items : P.ewald_vec;
  if (P.ewald_nk <= 0 || (int)blockIdx.x * THREADS >= n_work) return;  // uniform over the CTA
  __shared__ float2 fac[EW_TILE][3][EW_KMAX + 4];
  __shared__ float qt[EW_TILE];
  __shared__ uint32_t ut[EW_TILE][3];
  const int ewk = P.ewald_kmax + 1, np = *P.ek_np;
  const int i = (int)blockIdx.x * THREADS + (int)threadIdx.x;
  const bool mine = i < n_work;
  int col = 0, z0 = 0, code = 0;
  if (mine) {
    if (ITEMS) {
      const int2 item = P.ek_item[i];
      code = item.x;
      col = item.y;
      z0 = item.x >> 16 << 2;
    } else {
      code = P.ek_vec[i].x;
    }
  }
  int nx, ny, nz;
  ew_decode(code, nx, ny, nz);
  double re[NV], im[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) re[k] = im[k] = 0.0;
  for (int t0 = 0; t0 < np; t0 += EW_TILE) {
    const int nt = min(EW_TILE, np - t0);
    if (threadIdx.x < 3 * nt) {  // the tile's coordinates as 0.32 fixed-point fractions of L
      const int p = threadIdx.x / 3, ax = threadIdx.x % 3;
      const float4 r = P.pos[P.ek_list[t0 + p]];
      ut[p][ax] = ew_frac32(ax == 0 ? r.x : (ax == 1 ? r.y : r.z), P.invLd);
      if (ax == 0) qt[p] = r.w;
    }
    __syncthreads();
    for (int v = threadIdx.x; v < nt * 3 * ewk; v += THREADS) {
      const int p = v / (3 * ewk), ax = (v / ewk) % 3, n = v % ewk;
      if (!ITEMS || qt[p] != 0.0f) fac[p][ax][n] = ew_factor(ut[p][ax], n);  // (few threads: the test costs more)
    }
    __syncthreads();
    if (mine) {
      float tr[NV], ti[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) tr[k] = ti[k] = 0.0f;
      for (int p = 0; p < nt; ++p) {
        const float q = qt[p];
        if (q == 0.0f) continue;
        const float2 xy = ew_xy(ew_axis(fac[p][0], nx), ew_axis(fac[p][1], ny));
        if constexpr (ITEMS) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {  // (places beyond kmax hold no factor and are not stored)
            const float2 ez = fac[p][2][z0 + k];
            const float2 ep = cmul(xy, ez), em = cmul(xy, ew_conj(ez));
            tr[2 * k] = __fmaf_rn(q, ep.x, tr[2 * k]);
            ti[2 * k] = __fmaf_rn(q, ep.y, ti[2 * k]);
            tr[2 * k + 1] = __fmaf_rn(q, em.x, tr[2 * k + 1]);
            ti[2 * k + 1] = __fmaf_rn(q, em.y, ti[2 * k + 1]);
          }
        } else {
          const float2 e = cmul(xy, ew_axis(fac[p][2], nz));
          tr[0] = __fmaf_rn(q, e.x, tr[0]);
          ti[0] = __fmaf_rn(q, e.y, ti[0]);
        }
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        re[k] += (double)tr[k];
        im[k] += (double)ti[k];
      }
    }
    __syncthreads();
  }
  if (!mine) return;
  // hi + lo at the vector's place (the trials), their FP32 sum in the order of
  // the vectors (the forces)
  auto store = [&](int place, int vec, double r, double m) {
    const float2 hi = make_float2((float)r, (float)m);
    const float2 lo = make_float2((float)(r - (double)hi.x), (float)(m - (double)hi.y));
    P.ek_Shi[place] = hi;
    P.ek_Slo[place] = lo;
    if (vec >= 0) P.ek_Sf[vec] = make_float2(__fadd_rn(hi.x, lo.x), __fadd_rn(hi.y, lo.y));
  };
  if constexpr (ITEMS) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int4 z = P.ek_z[z0 + k / 2];
      if (col >= z.x || ((k & 1) && z0 + k / 2 == 0)) continue;
      const int o = col + ((k & 1) ? z.z : z.y);
      store(o, P.ek_place[o], re[k], im[k]);
    }
  } else {
    store(P.ek_vec[i].z, i, re[0], im[0]);
  }
}

cudaError_t launch_ewald_sk(const SysParams *d_reps, int n_rep, int max_items, int max_vec, cudaStream_t s) {
  if (n_rep <= 0 || max_items <= 0) return cudaSuccess;
  k_ewald_list<<<n_rep, 256, 0, s>>>(d_reps);
  const unsigned R = (unsigned)n_rep;
  auto grid = [&](int n, int threads) { return dim3((unsigned)((n + threads - 1) / threads), R); };
  if ((long long)grid(max_items, 128).x * n_rep >= 2 * device_sms())
    k_ewald_sk<true, 128><<<grid(max_items, 128), 128, 0, s>>>(d_reps);
  else if ((long long)grid(max_vec, 256).x * n_rep > device_sms())
    k_ewald_sk<false, 512><<<grid(max_vec, 512), 512, 0, s>>>(d_reps);
  else
    k_ewald_sk<false, 256><<<grid(max_vec, 256), 256, 0, s>>>(d_reps);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <bool LOG, bool DA, bool SEATS>
static cudaError_t launch_phase_t(const SysParams *d_reps, int n_rep, int max_nact, const PhaseShape &S,
                                  const PhaseForm &F, cudaStream_t s, uint32_t sweep, uint32_t sweep0, int colour,
                                  uint32_t k0, uint32_t k1, const StepDyn *dyn) {
  static size_t attr_bytes = 0;
  size_t smem = 0;
  const PhaseArgs A = phase_args(S, F, DA, &smem);
  if (smem > attr_bytes) {
    cudaError_t e =
        cudaFuncSetAttribute(k_cr_phase<LOG, DA, SEATS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_bytes = smem;
  }
  int gy = max_nact;  // CTAs of the replica with the most domains (no fewer for any smaller one)
  if (SEATS) {
    const int wide = (max_nact * F.wide16 + 15) >> 4;
    gy = wide + (max_nact - wide + F.seats - 1) / F.seats;
  }
  k_cr_phase<LOG, DA, SEATS>
      <<<dim3(n_rep, gy), F.threads, smem, s>>>(d_reps, A, sweep, sweep0, colour, k0, k1, dyn);
  return cudaGetLastError();
}

cudaError_t launch_phase(const SysParams *d_reps, int n_rep, int max_nact, const PhaseShape &S, const PhaseForm &F,
                         bool log, bool da, cudaStream_t s, uint32_t sweep, uint32_t sweep0, int colour, uint32_t k0,
                         uint32_t k1, const StepDyn *dyn) {
  // (a logged sweep takes the form without its seats: the records do not depend on it)
  const PhaseForm G = log && F.seats > 1 ? PhaseForm{128, 1, 1, 16, 0} : F;
#define CRMC_CASE(LL, DD, SS)                 \
  if (log == LL && da == DD && (G.seats > 1) == SS) \
    return launch_phase_t<LL, DD, SS>(d_reps, n_rep, max_nact, S, G, s, sweep, sweep0, colour, k0, k1, dyn);
  CRMC_CASE(false, false, false)
  CRMC_CASE(false, false, true)
  CRMC_CASE(true, false, false)
  CRMC_CASE(false, true, false)
  CRMC_CASE(true, true, false)
#undef CRMC_CASE
  return cudaErrorInvalidValue;
}

// Forms the autotuner picks from.  Compact forms size the shared-memory list
// and halo for most domains rather than the densest (denser ones spill to
// global memory), so that more CTAs fit on an SM; forms with seats give the
// densest domains a CTA each.
static const PhaseForm kForms[] = {
    // threads, seats (of 64 or 128 threads), groups (of 32), wide16, compact
    {64, 1, 1, 16, 1},  {128, 1, 1, 16, 0}, {256, 1, 1, 16, 0}, {512, 1, 1, 16, 0}, {128, 1, 4, 16, 0}, {256, 1, 8, 16, 0},
    {128, 2, 1, 2, 0},  {256, 4, 1, 1, 0},  {256, 4, 1, 2, 0},  {256, 4, 1, 4, 0},  {256, 2, 1, 2, 0},  {512, 4, 1, 4, 0}};
// forms with a delayed-acceptance variant (the surrogate runs on >= 128 threads)
static const PhaseForm kFormsDA[] = {
    {128, 1, 1, 16, 0}, {256, 1, 1, 16, 0}, {512, 1, 1, 16, 0}, {128, 1, 1, 16, 1}, {256, 1, 1, 16, 1}};

int phase_form_count(bool da) { return da ? (int)std::size(kFormsDA) : (int)std::size(kForms); }
const PhaseForm &phase_form(int i, bool da) { return da ? kFormsDA[i] : kForms[i]; }

// the second value of the pair that names a form: 0 for whole CTAs with the
// full capacities; the other forms' values lie above 16
int phase_form_code(const PhaseForm &F) {
  if (F == PhaseForm{F.threads, 1, 1, 16, 0}) return 0;
  return F.seats | F.groups << 4 | F.compact << 8 | F.wide16 << 12;
}

bool phase_form_named(int threads, int regs, bool da, PhaseForm *F) {
  if (regs >= 16) {
    for (int i = 0; i < phase_form_count(da); ++i) {
      *F = phase_form(i, da);
      if (F->threads == threads && phase_form_code(*F) == regs) return true;
    }
    return false;
  }
  *F = PhaseForm{threads, 1, 1, 16, 0};
  if (regs != 0) return !da && ((threads == 128 && regs == 4) || (threads == 256 && regs == 2) || (threads == 512 && regs == 1));
  if (da) return threads == 128 || threads == 256 || threads == 512;
  return threads == 32 || threads == 64 || threads == 128 || threads == 256 || threads == 512;
}

}  // namespace crmc
