// Particle-parallel kernels: manufactured sampling (Sec. 3.2), state
// load/store, K-averaged NTC collisions (Algorithm 1, Eq. avg_outcome) with
// the hard-sphere source (Eq. vel_change_1c) or the odd-power one (Eqs.
// vel_change_3, fn), the velocity-Verlet kick and drift (Eq.
// velocity_verlet with the sources of Eq. eom_mms, for the travelling-wave
// and the paper's manufactured problem) and the error norms of Sec. 4.3.
#include "pic_internal.cuh"
#include "ntc_fp64.cuh"

namespace pic {
namespace {

constexpr int kThreads = 256;

inline int blocks_for(int64_t n, int t = kThreads) {
  int64_t b = (n + t - 1) / t;
  return (int)(b < 1 ? 1 : b);
}

// --------------------------------------------------------------------------
// Sampling: xi from the particle's Philox stream, x = x^M(t0), v = v^M.
// Written in pid order into the current buffer.
// --------------------------------------------------------------------------
struct SampleArgs {
  Params P;
  TimeTerms tt;
  double *x0, *x1, *x2, *v0, *v1, *v2, *vm0, *vm1, *vm2;
  uint32_t* pid;
};

__global__ void __launch_bounds__(kThreads) k_sample(SampleArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.P.np) return;
  const Params& P = a.P;
  const U4 b0 = sample_block(P, (uint64_t)i, 0), b1 = sample_block(P, (uint64_t)i, 1),
           b2 = sample_block(P, (uint64_t)i, 2);
  const double xi[6] = {unif52(b0.x, b0.y), unif52(b0.z, b0.w), unif52(b1.x, b1.y),
                        unif52(b1.z, b1.w), unif52(b2.x, b2.y), unif52(b2.z, b2.w)};
  if (P.dist == PIC_DIST_PAPER) {
    double s;
    // x^M(t0) per axis; v^M(t0) = vh(t0) tau(xi), tau kept in the v^M arrays
    double c;
    a.x0[i] = wrap_unit(xm_solve_gen(a.tt, 0, xi[0], &s, &c));
    a.x1[i] = wrap_unit(xm_solve_gen(a.tt, 1, xi[1], &s, &c));
    a.x2[i] = wrap_unit(xm_solve_gen(a.tt, 2, xi[2], &s, &c));
    const double t0 = tau_inv(xi[3]), t1 = tau_inv(xi[4]), t2 = tau_inv(xi[5]);
    a.v0[i] = t0 * a.tt.vh[0]; a.v1[i] = t1 * a.tt.vh[1]; a.v2[i] = t2 * a.tt.vh[2];
    a.vm0[i] = t0; a.vm1[i] = t1; a.vm2[i] = t2;
    a.pid[i] = (uint32_t)i;
    return;
  }
  const double X0 = xm_table(P, a.tt, xi[0]);
  const double X1 = xm_table(P, a.tt, xi[1]);
  const double X2 = xm_table(P, a.tt, xi[2]);
  const double V0 = P.vmean[0] + P.vsig * normal_quantile(P, xi[3]);
  const double V1 = P.vmean[1] + P.vsig * normal_quantile(P, xi[4]);
  const double V2 = P.vmean[2] + P.vsig * normal_quantile(P, xi[5]);
  a.x0[i] = wrap_unit(X0); a.x1[i] = wrap_unit(X1); a.x2[i] = wrap_unit(X2);
  a.v0[i] = V0; a.v1[i] = V1; a.v2[i] = V2;
  a.vm0[i] = V0; a.vm1[i] = V1; a.vm2[i] = V2;
  a.pid[i] = (uint32_t)i;
}

// Load a caller state (x and v, each [N_p][3] in pid order) into SoA.
struct LoadArgs {
  Params P;
  TimeTerms tt;
  const double *xs, *vs;  // device memory or mapped pinned host memory
  double *x0, *x1, *x2, *v0, *v1, *v2, *vm0, *vm1, *vm2;
  uint32_t* pid;
};

__global__ void __launch_bounds__(kThreads) k_load_state(LoadArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.P.np) return;
  const Params& P = a.P;
  const U4 b0 = sample_block(P, (uint64_t)i, 0), b1 = sample_block(P, (uint64_t)i, 1),
           b2 = sample_block(P, (uint64_t)i, 2);
  const double xi[6] = {unif52(b0.x, b0.y), unif52(b0.z, b0.w), unif52(b1.x, b1.y),
                        unif52(b1.z, b1.w), unif52(b2.x, b2.y), unif52(b2.z, b2.w)};
  if (P.dist == PIC_DIST_PAPER) {
    a.vm0[i] = tau_inv(xi[3]); a.vm1[i] = tau_inv(xi[4]); a.vm2[i] = tau_inv(xi[5]);
  } else {
    a.vm0[i] = P.vmean[0] + P.vsig * normal_quantile(P, xi[3]);
    a.vm1[i] = P.vmean[1] + P.vsig * normal_quantile(P, xi[4]);
    a.vm2[i] = P.vmean[2] + P.vsig * normal_quantile(P, xi[5]);
  }
  const double* xs = a.xs;
  const double* vs = a.vs;
  a.x0[i] = xs[3 * i]; a.x1[i] = xs[3 * i + 1]; a.x2[i] = xs[3 * i + 2];
  a.v0[i] = vs[3 * i]; a.v1[i] = vs[3 * i + 1]; a.v2[i] = vs[3 * i + 2];
  a.pid[i] = (uint32_t)i;
}

struct StoreArgs {
  int64_t np;
  const double *x0, *x1, *x2, *v0, *v1, *v2;
  const uint32_t* pid;
  double* xv;
};

__global__ void __launch_bounds__(kThreads) k_store_state(StoreArgs a) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= a.np) return;
  const int64_t p = a.pid[j];
  a.xv[3 * p] = a.x0[j]; a.xv[3 * p + 1] = a.x1[j]; a.xv[3 * p + 2] = a.x2[j];
  double* vs = a.xv + 3 * a.np;
  vs[3 * p] = a.v0[j]; vs[3 * p + 1] = a.v1[j]; vs[3 * p + 2] = a.v2[j];
}

struct StoreDvArgs {
  int64_t np;
  const double *d0, *d1, *d2, *m0, *m1, *m2;
  const uint32_t* pid;
  double *dv, *dvm;
};

__global__ void __launch_bounds__(kThreads) k_store_dv(StoreDvArgs a) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= a.np) return;
  const int64_t p = a.pid[j];
  a.dv[3 * p] = a.d0[j]; a.dv[3 * p + 1] = a.d1[j]; a.dv[3 * p + 2] = a.d2[j];
  a.dvm[3 * p] = a.m0[j]; a.dvm[3 * p + 1] = a.m1[j]; a.dvm[3 * p + 2] = a.m2[j];
}

// --------------------------------------------------------------------------
// K-averaged NTC collisions. One warp serves a group of G consecutive cells;
// lane l runs outcome (chunk Kc + l % Kc) of cell (l / Kc) of the group,
// sequentially over its candidate pairs with in-place updates (Algorithm 1).
// Then the lanes take the cells' particles: each adds its particle's changes
// in ascending outcome order and forms the analytic source.
//
// What bounds it is the FP64 pipe (two lanes an SM and clock), so as little
// as possible runs there, and that by full warps:
//  - the accept test runs in FP32 on a copy of the group's velocities in
//    shared memory, free of units, with a bound on its error; the one
//    candidate in a million it cannot decide is decided in FP64 as the paper
//    writes it (ntc_decide64), so every decision is the FP64 one;
//  - one candidate in eight is accepted: the lanes only test their
//    candidates and put the accepted pairs into a queue of the warp, which is
//    scattered 32 pairs at a time, whichever lanes they came from. A
//    candidate whose p or q is changed by a queued pair of its lane waits;
//  - the source's R(a) comes from a table of degree-7 polynomials in a^2
//    (hs_R64) instead of an exponential, an error function, a square root
//    and a division.
// Before, with the test and the source in FP64 and each lane scattering its
// own pairs, the FP64 pipe was 85% busy; a call now takes 0.32 ms instead of
// 1.36 (32^3 cells of 32, K = 16), 0.47 instead of 2.97 (12^3 cells of 101,
// K = 243) and 93 us instead of 158 (8^3 cells of 8, K = 16: latency of the few
// warps).
//
// Working velocities: bit l of mask[p] says that lane l has changed particle
// p of its cell. The first kList changed particles of a lane keep their
// velocity in a list in shared memory, any further ones in the lane's
// particle-indexed overlay in global memory. One word per lane holds the low
// bytes of its list's indices (0xff: unused), so that in cells of up to 255
// particles an entry is found by one zero-byte search.
// --------------------------------------------------------------------------
// Constants of the FP32 accept test (ntc_test32)
struct Test32 {
  double scale;         // of the velocities: 1, or a power of two
  int scaled;           // it is not 1
  float inv_gmax2;      // 1 / (scale g_max)^2
  float err;            // 2^-19 of it
  float tie;            // what a near tie (1e-12 in U) amounts to where U is below 1e-6
  float c0, c1, c2;     // sigma_k g_max^2k / (sigma g)_max
  int n_sigma;
};

// The velocities keep their units while g_max lies within 2^+-32; beyond, a power
// of two brings it there.
Test32 test32_of(const Params& P) {
  Test32 T;
  const int e = ilogb(P.gmax);
  T.scaled = abs(e) > 32;
  T.scale = T.scaled ? ldexp(1.0, -e) : 1.0;
  const double g = P.gmax * T.scale, g2 = P.gmax * P.gmax;
  T.inv_gmax2 = (float)(1.0 / (g * g));
  T.err = 0x1p-19f * T.inv_gmax2;
  T.n_sigma = P.n_sigma;
  T.tie = P.n_sigma == 0 ? 2e-18f : 2e-12f;
  T.c0 = (float)(P.sigma_n[0] / P.sg_max);
  T.c1 = (float)(P.sigma_n[1] * g2 / P.sg_max);
  T.c2 = (float)(P.sigma_n[2] * (g2 * g2) / P.sg_max);
  return T;
}

struct DsmcArgs {
  Params P;
  Test32 T;
  const double *v0, *v1, *v2;
  const int32_t* start;
  uint32_t c0;
  double *dv0, *dv1, *dv2;  // out: <dv> - <dv^M>, or <dv> when m0 != nullptr
  double *m0, *m1, *m2;     // out (optional): <dv^M>
  double* overlay;
  int max_ppc, G, Kc, nchunks;
  int stage;                // particles of a group whose velocities are staged
  int64_t ngroups;
  // parts > 1: a group's chunks of outcomes are shared by that many warps,
  // which leave their sums in partial ([parts][3][N_p]) for k_dsmc_merge
  int parts;
  double* partial;
  unsigned long long* queue;  // next (group, part) to take (zero at launch), or nullptr: a grid stride
  unsigned long long* counters;
  int* flags;
  double vh[3];             // PIC_DIST_PAPER: f_v scales at the call's time
  DLog lg;                  // decision log (mode 0: off)
  long long* hist;          // per-step history row: [1] candidates, [2] collisions, [3] g > g_max
};

// one warp a block: a launch of few groups still reaches every SM
constexpr int kDsmcThreads = 32;
constexpr int kList = 4;
constexpr int kOverlay = 7;     // slot number of a particle in the overlay
constexpr int kByteCell = 255;  // largest cell the byte keys are exact for
// accepted pairs queued before they are scattered: a pass takes 32, and a
// candidate adds at most 32 to a queue of 31
constexpr int kQueue = 64;

struct ListEntry {
  double v[3];
  long long p;
};
// A warp's shared memory; behind it the FP32 velocities [stage] and the
// masks [max_ppc].
struct Warp64 {
  ListEntry list[kList * 32];  // entry k of lane l at 32 k + l
  // p | q << 16; lane | slots of p and q << 8, 16 | kOld*; epsilon word; chi
  // word, or candidate + 1 with kChiSlot
  uint4 queue[kQueue];
  uint32_t keys[32];
  int len[32];
};
// of a queue entry: the slot of p or q held its velocity before; its chi word
// is still to be drawn
constexpr uint32_t kOldP = 1u << 24, kOldQ = 1u << 25, kChiSlot = 1u << 26;

struct Counts64 {
  uint32_t cand, coll, gmax, tie;  // per lane, flushed before they can overflow
};
constexpr uint32_t kFlushAt = 1u << 30;  // an outcome adds less than 2^31

__device__ __forceinline__ int key_find(uint32_t keys, int p) {
  const uint32_t x = keys ^ (((uint32_t)p & 0xffu) * 0x01010101u);
  const uint32_t z = (x - 0x01010101u) & ~x & 0x80808080u;
  return z ? (__ffs((int)z) - 8) >> 3 : -1;
}
__device__ __forceinline__ int list_find(const ListEntry* wl, int t, int p) {
  int k = -1;
#pragma unroll
  for (int i = 0; i < kList; ++i)
    if (i < t && wl[32 * i].p == p) k = i;
  return k;
}

// The same decision from FP32 velocities (each the FP64 one, in units of
// 1 / T.scale, rounded): 0 or 1, or -1 where FP64 has to decide. The test is
// on y = g^2 / g_max^2: U^2 < y, or for the odd-power sigma U < c0 + c1 y +
// c2 y^2. With S = sum (v_p^2 + v_q^2) the components' differences are off by at
// most 2^-23 (|v_p| + |v_q|), so y by less than 2^-19 S / g_max^2, the
// margin, and U^2 by less than 2^-20 of itself. y near or above one is left to
// FP64 too (its flag), and so is anything not finite (no comparison with it
// holds). Odd-power sigma: the same through its derivative.
//
// Nothing that matters lies below FP32's normal range whatever the units: U,
// y and c_k are numbers near one, g_max is within 2^+-32 of one in the units
// of the velocities (test32_of), so a subnormal square is 2^-85 of
// g_max^2 or less, and the near-tie term covers that.
__device__ __forceinline__ int ntc_test32(const Test32& T, uint32_t w, const float4& a, const float4& b) {
  const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  const float y = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) * T.inv_gmax2;
  const float U = fmaf((float)w, 0x1p-32f, 0x1p-33f);
  const float e = fmaf(T.err, a.w + b.w, T.tie);  // (|v_p|^2 + |v_q|^2)
  float lhs, rhs, margin;
  if (T.n_sigma == 0) {
    lhs = U * U;
    rhs = y;
    margin = fmaf(0x1p-19f, lhs, e);
  } else {
    lhs = U;
    rhs = fmaf(fmaf(T.c2, y, T.c1), y, T.c0);
    const float d = fmaf(2.f * fabsf(T.c2), y + e, fabsf(T.c1));
    margin = fmaf(d, e, fmaf(0x1p-19f, lhs + fabsf(T.c0) + y * d, T.tie));
  }
  if (fabsf(lhs - rhs) > margin && y + e < 1.f) return lhs < rhs ? 1 : 0;
  return -1;
}

// An FP64 velocity as the test takes it. The scaling is a call: in line, the
// multiplications take the FP64 pipe, predicated off as they are, also where
// there is none to do (12^3 cells of 101, K = 243: 1.37 ms a call, 1.19 so).
__device__ __noinline__ float4 rounded_scaled(double s, double x, double y, double z) {
  float4 f = make_float4((float)(x * s), (float)(y * s), (float)(z * s), 0.f);
  f.w = fmaf(f.x, f.x, fmaf(f.y, f.y, f.z * f.z));
  return f;
}
__device__ __forceinline__ float4 rounded(const Test32& T, double x, double y, double z) {
  if (T.scaled) return rounded_scaled(T.scale, x, y, z);
  float4 f = make_float4((float)x, (float)y, (float)z, 0.f);
  f.w = fmaf(f.x, f.x, fmaf(f.y, f.y, f.z * f.z));
  return f;
}

// Algorithm 1 for the warp's (cell, outcome) lanes: outcome o of cell `cell`
// (particles off .. off + c - 1) where run is set.
template <bool kVerify>
__device__ __forceinline__ void ntc_warp64(const DsmcArgs& a, uint32_t cell, uint32_t o, int off, int c, bool run,
                                           int lane, Warp64& W, const float4* stage, int gs, uint32_t* mask,
                                           double* wov, Counts64& cnt) {
  const Params& P = a.P;
  const DLog& lg = a.lg;
  const uint32_t c0 = a.c0;
  const bool log_all = kVerify && lg.mode == PIC_DLOG_ALL;
  long long npairs = 0;
  U4 bchi{0u, 0u, 0u, 0u}, b0{0u, 0u, 0u, 0u};
  if (run) {
    // the chi stream (c0, cell, slot, (o << 8) | 1): word 0 of slot 0 is the
    // N_pairs uniform, word (s + 1) mod 4 of slot (s + 1) / 4 the chi of
    // candidate s
    bchi = philox(c0, cell, 0u, (o << 8) | 1u, P.key0, P.key1);
    const double base = __dmul_rn(__dmul_rn((double)((long long)c * (long long)(c - 1)), P.pmax), 0.5);
    npairs = (long long)floor(__dadd_rn(base, unif32(bchi.x)));
    if (log_all) dlog_put(lg, c0, cell, o, -1, -1, -1, (int)npairs, PIC_DLOG_NPAIRS);
    if (npairs > 0) {
      // candidate s: block (c0, cell, s, o << 8) = (p, q, accept, epsilon)
      b0 = philox(c0, cell, 0u, o << 8, P.key0, P.key1);
      if (npairs > 0x7fffffffll) npairs = 0x7fffffffll;
      cnt.cand += (uint32_t)npairs;
    } else {
      npairs = 0;
    }
  }
  const uint32_t bit = 1u << lane;
  double* const ov = wov + (size_t)lane * a.max_ppc * 3;
  uint32_t keys = 0xffffffffu;   // low bytes of the list's indices
  int t = 0;                     // list entries
  bool spilled = false;          // some particle is in the overlay
  uint32_t waiting = 0u;         // bit k + 1: a queued pair will write slot k
  int s = 0, qn = 0;
  bool stuck = false;
  const int np = (int)npairs;
  // slot of particle x of this lane, or -1
  auto find = [&](int x) {
    int k = key_find(keys, x);
    if (c > kByteCell && k >= 0 && !(k < t && W.list[32 * k + lane].p == x)) k = list_find(W.list + lane, t, x);
    if (spilled && k < 0 && (mask[x] & bit)) k = kOverlay;
    return k;
  };
  // a slot for a particle that has none
  auto new_slot = [&](int x) {
    atomicOr(mask + x, bit);
    if (t == kList) {
      spilled = true;
      return kOverlay;
    }
    keys ^= (~(uint32_t)x & 0xffu) << (8 * t);
    W.list[32 * t + lane].p = x;
    return t++;
  };
  // working velocity of particle x in slot k (-1: none) of lane l, whose
  // cell's first particle is `at`
  auto velocity = [&](int x, int k, int l, int at, double* v) {
    if (k < 0) {
      v[0] = a.v0[at + x]; v[1] = a.v1[at + x]; v[2] = a.v2[at + x];
    } else {
      const double* e = k < kList ? W.list[32 * k + l].v : wov + ((size_t)l * a.max_ppc + x) * 3;
      v[0] = e[0]; v[1] = e[1]; v[2] = e[2];
    }
  };
  for (;;) {
    const bool go = s < np && !stuck;
    const int able = __popc(__ballot_sync(0xffffffffu, go));
    if (able <= 4 * __popc(__ballot_sync(0xffffffffu, stuck)) || qn >= 32) {
      if (qn == 0) break;  // no lane is stuck without a queued pair
      // scatter the queue
      __syncwarp();
      for (int e0 = 0; e0 < qn; e0 += 32) {
        const int e = e0 + lane;
        uint4 ec = make_uint4(0u, 0u, 0u, 0u);
        if (e < qn) ec = W.queue[e];
        const int owner = (int)(ec.y & 31u);
        // the owner's cell, outcome and first particle
        const uint32_t ocell = __shfl_sync(0xffffffffu, cell, owner), oo = __shfl_sync(0xffffffffu, o, owner);
        const int ooff = __shfl_sync(0xffffffffu, off, owner);
        if (e < qn) {
          const int p = (int)(ec.x & 0xffffu), q = (int)(ec.x >> 16);
          const int kp = (int)((ec.y >> 8) & 15u), kq = (int)((ec.y >> 16) & 15u);
          double vp[3], vq[3];
          velocity(p, ec.y & kOldP ? kp : -1, owner, ooff, vp);
          velocity(q, ec.y & kOldQ ? kq : -1, owner, ooff, vq);
          uint32_t wchi = ec.w;
          if (ec.y & kChiSlot) {
            const U4 b = philox(c0, ocell, ec.w >> 2, (oo << 8) | 1u, P.key0, P.key1);
            const uint32_t js = ec.w & 3u;
            wchi = js == 0u ? b.x : js == 1u ? b.y : js == 2u ? b.z : b.w;
          }
          const double dx = __dsub_rn(vp[0], vq[0]), dy = __dsub_rn(vp[1], vq[1]), dz = __dsub_rn(vp[2], vq[2]);
          const double g =
              __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
          double* wp = kp < kList ? W.list[32 * kp + owner].v : wov + ((size_t)owner * a.max_ppc + p) * 3;
          double* wq = kq < kList ? W.list[32 * kq + owner].v : wov + ((size_t)owner * a.max_ppc + q) * 3;
          if (kVerify && (P.verify & PIC_VERIFY_ERROR2)) {
            // injected Error 2: swap with probability 1/2 (coin = chi draw)
            const bool swap = unif32(wchi) < 0.5;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              wp[d] = swap ? vq[d] : vp[d];
              wq[d] = swap ? vp[d] : vq[d];
            }
          } else {
            double se, ce;
            sincospi(2.0 * unif32(ec.z), &se, &ce);
            double uchi = unif32(wchi);
            if (kVerify && (P.verify & PIC_VERIFY_ANISO)) uchi = aniso_u(uchi);
            const double cchi = __dsub_rn(1.0, __dmul_rn(2.0, uchi));
            const double schi = __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(cchi, cchi)));
            const double nv[3] = {__dmul_rn(ce, schi), __dmul_rn(se, schi), cchi};
            const bool err1 = kVerify && (P.verify & PIC_VERIFY_ERROR1);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const double gp = __dmul_rn(g, nv[d]);
              // Eq. v_cm; injected Error 1 flips the sign of v_q
              const double cm = __dmul_rn(err1 ? __dsub_rn(vp[d], vq[d]) : __dadd_rn(vp[d], vq[d]), 0.5);
              wp[d] = fma(gp, 0.5, cm);
              wq[d] = fma(gp, -0.5, cm);
            }
          }
          if (kVerify && P.ang_hist)
            record_angles(P.ang_hist, (P.verify & PIC_VERIFY_ANISO) != 0, g, __dsub_rn(wp[0], wq[0]),
                          __dsub_rn(wp[1], wq[1]), __dsub_rn(wp[2], wq[2]));
        }
      }
      __syncwarp();
      qn = 0;
      waiting = 0u;
      stuck = false;
      continue;
    }
    bool accept = false;
    uint32_t p = 0u, q = 0u, ww = 0u;
    int kp = -1, kq = -1;
    if (go) {
      p = draw_index(b0.x, (uint32_t)c);
      // q uniform over the other c - 1 particles: the distribution of
      // drawing again until q != p
      q = draw_index(b0.y, (uint32_t)(c - 1));
      q += q >= p ? 1u : 0u;
      kp = find((int)p);
      kq = find((int)q);
      stuck = ((waiting >> (kp + 1) | waiting >> (kq + 1)) & 1u) != 0u;
      if (!stuck) {
        const uint32_t wz = b0.z;
        ww = b0.w;
        ++s;
        if (s < np) b0 = philox(c0, cell, (uint32_t)s, o << 8, P.key0, P.key1);
        int d = -1;
        if (stage && kp < 0 && kq < 0) {
          d = ntc_test32(a.T, wz, stage[off - gs + (int)p], stage[off - gs + (int)q]);
        } else {
          double vp[3], vq[3];
          velocity((int)p, kp, lane, off, vp);
          velocity((int)q, kq, lane, off, vq);
          d = ntc_test32(a.T, wz, rounded(a.T, vp[0], vp[1], vp[2]), rounded(a.T, vq[0], vq[1], vq[2]));
        }
        if (d < 0) {
          double vp[3], vq[3];
          velocity((int)p, kp, lane, off, vp);
          velocity((int)q, kq, lane, off, vq);
          d = ntc_decide64(P, wz, __dsub_rn(vp[0], vq[0]), __dsub_rn(vp[1], vq[1]), __dsub_rn(vp[2], vq[2]));
        }
        if (d & 4) ++cnt.gmax;
        if (d & 2) ++cnt.tie;
        accept = (d & 1) != 0;
        if (log_all || ((d & 2) && lg.mode != PIC_DLOG_OFF))
          dlog_put(lg, c0, cell, o, s - 1, (int)p, (int)q, accept ? 1 : 0, d & 2 ? PIC_DLOG_TIE : 0);
      }
    }
    const unsigned acc = __ballot_sync(0xffffffffu, accept);
    if (accept) {
      uint32_t info = (uint32_t)lane | (kp >= 0 ? kOldP : 0u) | (kq >= 0 ? kOldQ : 0u) | (s > 3 ? kChiSlot : 0u);
      if (kp < 0) kp = new_slot((int)p);
      if (kq < 0) kq = new_slot((int)q);
      waiting |= 2u << kp | 2u << kq;
      info |= (uint32_t)kp << 8 | (uint32_t)kq << 16;
      const uint32_t wchi = s == 1 ? bchi.y : s == 2 ? bchi.z : s == 3 ? bchi.w : (uint32_t)s;
      W.queue[qn + __popc(acc & (bit - 1u))] = make_uint4(p | q << 16, info, ww, wchi);
      ++cnt.coll;
    }
    qn += __popc(acc);
  }
  W.keys[lane] = keys;
  W.len[lane] = t;
  __syncwarp();
}

// the warp's counts into the launch's totals
__device__ __forceinline__ void flush_counts(const DsmcArgs& a, Counts64& cnt, int lane) {
  const uint32_t v[4] = {cnt.cand, cnt.coll, cnt.gmax, cnt.tie};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned long long lo = __reduce_add_sync(0xffffffffu, v[k] & 0xffffu);
    const unsigned long long hi = __reduce_add_sync(0xffffffffu, v[k] >> 16);
    const unsigned long long tot = lo + (hi << 16);
    if (lane == 0 && tot) {
      atomicAdd(a.counters + k, tot);
      if (a.hist && k < 3) atomicAdd((unsigned long long*)a.hist + 1 + k, tot);
    }
  }
  cnt = {0u, 0u, 0u, 0u};
}

// the outputs of particle j (velocity w) of a cell of cc, from the sum of its
// changes over the outcomes
__device__ __forceinline__ void dsmc_finish(const DsmcArgs& a, int64_t j, int cc, const double* w, const double* acc,
                                            double invK) {
  const Params& P = a.P;
  double so[3];
  if (P.n_sigma == 0) {
    // Eq. vel_change_1c
    const double mx = P.vmean[0] - w[0], my = P.vmean[1] - w[1], mz = P.vmean[2] - w[2];
    const double u = fma(mx, mx, fma(my, my, mz * mz)) * (P.inv_vsig * P.inv_vsig);
    const double f = P.src_pref * (double)(cc - 1) * P.vsig * hs_R64(P, u);
    so[0] = f * mx; so[1] = f * my; so[2] = f * mz;
  } else {
    odd_source(P, a.vh, w[0], w[1], w[2], cc, so);
  }
  if (a.m0) {
    a.dv0[j] = acc[0] * invK; a.dv1[j] = acc[1] * invK; a.dv2[j] = acc[2] * invK;
    a.m0[j] = so[0]; a.m1[j] = so[1]; a.m2[j] = so[2];
  } else {
    a.dv0[j] = fma(acc[0], invK, -so[0]);
    a.dv1[j] = fma(acc[1], invK, -so[1]);
    a.dv2[j] = fma(acc[2], invK, -so[2]);
  }
}

// the parts' sums, in order, and the source: one warp a cell
constexpr int kMergeThreads = 128;
__global__ void __launch_bounds__(kMergeThreads) k_dsmc_merge(DsmcArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t cell = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (cell >= a.P.ncell) return;
  const int32_t s = a.start[cell], e = a.start[cell + 1];
  const double invK = 1.0 / (double)a.P.K;
  for (int32_t j = s + lane; j < e; j += 32) {
    double acc[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < a.parts; ++k)
#pragma unroll
      for (int d = 0; d < 3; ++d) acc[d] += a.partial[((int64_t)3 * k + d) * a.P.np + j];
    const double w[3] = {a.v0[j], a.v1[j], a.v2[j]};
    dsmc_finish(a, j, e - s, w, acc, invK);
  }
}

template <bool kVerify>
__global__ void __launch_bounds__(kDsmcThreads, 16) k_dsmc(DsmcArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Params& P = a.P;
  const int lane = threadIdx.x;
  Warp64& W = *reinterpret_cast<Warp64*>(smem);
  float4* const staged = reinterpret_cast<float4*>(&W + 1);
  uint32_t* const mask = reinterpret_cast<uint32_t*>(staged + a.stage);
  double* wov = a.overlay + (size_t)blockIdx.x * 32 * a.max_ppc * 3;
  for (int i = lane; i < a.max_ppc; i += 32) mask[i] = 0u;
  __syncwarp();
  Counts64 cnt = {0u, 0u, 0u, 0u};
  const double invK = 1.0 / (double)P.K;

  for (int64_t take = blockIdx.x;; take += gridDim.x) {
    int64_t item = take;
    if (a.queue) {
      unsigned long long q = 0;
      if (lane == 0) q = atomicAdd(a.queue, 1ull);
      item = (int64_t)__shfl_sync(0xffffffffu, q, 0);
    }
    if (item >= a.ngroups * a.parts) break;  // warp-uniform
    const int64_t grp = item / a.parts;
    const int part = (int)(item % a.parts);
    const int ch0 = (int)((int64_t)a.nchunks * part / a.parts), ch1 = (int)((int64_t)a.nchunks * (part + 1) / a.parts);
    // where the sums over the part's outcomes are kept
    double *d0 = a.dv0, *d1 = a.dv1, *d2 = a.dv2;
    if (a.parts > 1) {
      d0 = a.partial + (int64_t)3 * part * P.np;
      d1 = d0 + P.np;
      d2 = d1 + P.np;
    }
    const int64_t cell0 = grp * a.G;
    const int ncl = (int)min((int64_t)a.G, P.ncell - cell0);  // cells in this group
    const int mycl = lane / a.Kc;
    const bool lane_cell = mycl < ncl;
    int32_t s = 0, c = 0;
    if (lane_cell) {
      s = a.start[cell0 + mycl];
      c = a.start[cell0 + mycl + 1] - s;
    }
    const int cmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)c);
    const int32_t gs = a.start[cell0], gn = a.start[cell0 + ncl] - gs;
    const bool use_stage = gn <= a.stage;
    __syncwarp();
    if (use_stage)
      for (int i = lane; i < gn; i += 32) staged[i] = rounded(a.T, a.v0[gs + i], a.v1[gs + i], a.v2[gs + i]);
    __syncwarp();
    for (int ch = ch0; ch < ch1; ++ch) {
      const int o = ch * a.Kc + lane % a.Kc;
      bool run = lane_cell && o < P.K && c >= 2;
      if (run && c > a.max_ppc) {
        atomicOr(a.flags, 1);
        run = false;
      }
      ntc_warp64<kVerify>(a, (uint32_t)(cell0 + mycl), (uint32_t)o, s, c, run, lane, W,
                          use_stage ? staged : nullptr, gs, mask, wov, cnt);
      // sum this chunk's changes per particle in ascending outcome order
      const bool last = ch == a.nchunks - 1 && a.parts == 1;
      const uint32_t kseg = a.Kc == 32 ? 0xffffffffu : ((1u << a.Kc) - 1u);
      for (int jb = 0; jb < cmax; jb += 32) {
        const int jj = jb + lane;
        // cells above max_ppc have no masks (and no collisions)
        uint32_t word = 0u;
        if (jj < a.max_ppc) {
          word = mask[jj];
          mask[jj] = 0u;
        }
        for (int cl = 0; cl < ncl; ++cl) {
          const int32_t cs = __shfl_sync(0xffffffffu, s, cl * a.Kc);
          const int cc = __shfl_sync(0xffffffffu, c, cl * a.Kc);
          if (jj >= cc) continue;
          uint32_t mine = word & (kseg << (cl * a.Kc));
          if (!last && ch > ch0 && !mine) continue;  // nothing to add
          const int32_t j = cs + jj;
          const double w[3] = {a.v0[j], a.v1[j], a.v2[j]};
          double acc[3] = {0.0, 0.0, 0.0};
          if (ch > ch0) { acc[0] = d0[j]; acc[1] = d1[j]; acc[2] = d2[j]; }
          while (mine) {
            const int l = __ffs((int)mine) - 1;
            mine &= mine - 1u;
            // lane l's working velocity of particle jj: its list, else its overlay
            const int k = cc <= kByteCell ? key_find(W.keys[l], jj) : list_find(W.list + l, W.len[l], jj);
            const double* e = k >= 0 ? W.list[32 * k + l].v : wov + ((size_t)l * a.max_ppc + jj) * 3;
#pragma unroll
            for (int d = 0; d < 3; ++d) acc[d] = __dadd_rn(acc[d], __dsub_rn(e[d], w[d]));
          }
          if (last) {
            dsmc_finish(a, j, cc, w, acc, invK);
          } else {
            d0[j] = acc[0]; d1[j] = acc[1]; d2[j] = acc[2];
          }
        }
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, cnt.cand >= kFlushAt)) flush_counts(a, cnt, lane);
    }
  }
  flush_counts(a, cnt, lane);
}

// --------------------------------------------------------------------------
// Kick (and optionally drift) in sorted order:
//   v += 1/2 (dt q/m (E_p - E^M_p) + dv + dt vdot^M) (vdot^M = 0 for the
//   Gaussian f_v, vh'(t) tau for the paper's f_v),
//   x += dt (v + xdot^M - v^M) at t_half (drift), wrapped; new cell key.
//
// What bounds it is the FP64 pipe (an instruction of a warp takes the SM's 19
// cycles), so operations are what counts: sin and cos from a table and the
// angle's remainder (15, sincospi 22 and a reduction); the drift's xdot^M from
// a table of its one transcendental quantity, dG^{-1}/dT (xm_solve and xm_dot:
// a Hermite start, a Newton step with its sincospi, three divisions: 90);
// uniforms, cells and table indexes read off the bits of a sum with 2^52
// (a conversion takes the pipe like an addition). Per particle some 110
// FP64 instructions instead of 150 for the Lorentz term, 70 instead of 310
// for the drift. Two steps of 64^3 cells of 32 (a closing kick, one with
// drift): 9.2 ms before, 4.6 now.
// --------------------------------------------------------------------------
struct KickArgs {
  Params P;
  double *x0, *x1, *x2, *v0, *v1, *v2;
  const double *vm0, *vm1, *vm2;
  const uint32_t* pid;
  const double *dv0, *dv1, *dv2;
  const double *E0, *E1, *E2;
  double *L0, *L1, *L2;  // Lorentz term dt q/m (E_p - E^M_p)
  int lor_mode;          // 0: compute, 1: compute and store, 2: load
  double dt_qm;
  TimeTerms tE, th;
  TimeTerms t0, t1;      // t_n, t_{n+1} for the isolated-collision drift
  int drift;
  // the drift by table: T = 1.m - T0 with 1.m = xi + 1 - 2^-53, and
  // xdot^M = c - xslope dG^{-1}/dT(T)
  double T0, xslope;
  int32_t *key, *rank, *count;
};

__device__ __noinline__ void sincos_far(double d, double* s, double* c) { sincospi(2.0 * d, s, c); }

// sin and cos of 2 pi d: the table at the nearest kTrigM-th of
// a turn, and the remainder b, |b| <= pi / kTrigM, by Taylor's series (the
// first terms left out are b^7/5040 = 8e-18 and b^8/40320)
__device__ __forceinline__ void sincos_turn(const double2* tab, double d, double* s, double* c) {
  constexpr double w = kTwoPi / kTrigM, w2 = w * w;
  if (!below_pow2(d, 40)) return sincos_far(d, s, c);  // (or not finite)
  const double z = fma(d, (double)kTrigM, kRound52);
  const double2 t = __ldg(tab + (__double2loint(z) & (kTrigM - 1)));
  const double u = fma(d, (double)kTrigM, kRound52 - z);
  const double u2 = u * u;
  const double sb = u * fma(u2, fma(u2, w * w2 * w2 / 120.0, -w * w2 / 6.0), w);
  const double cb = u2 * fma(u2, fma(u2, -w2 * w2 * w2 / 720.0, w2 * w2 / 24.0), -0.5 * w2);  // cos - 1
  *s = fma(t.y, sb, fma(t.x, cb, t.x));
  *c = fma(-t.x, sb, fma(t.y, cb, t.y));
}

// cell_coord(x, n) without conversions where x lies in the box; xn = x n
// rounded, *whole the coordinate in FP64
__device__ __forceinline__ int cell_coord_fast(double x, double xn, int n, double* whole) {
  const double z = __dadd_rd(xn, kRound52);
  int i = __double2loint(z);
  *whole = __dsub_rn(z, kRound52);
  if ((unsigned)i >= (unsigned)n || !below_pow2(xn, 31)) {
    i = cell_coord(x, n);
    *whole = (double)i;
  }
  return i;
}

// dt q/m (E_p + E_app - E^M) at a particle
__device__ __forceinline__ void lorentz64(const KickArgs& a, const double* x, double* L) {
  const Params& P = a.P;
  const int n = P.n;
  double w1[3], w0[3];
  int i0[3], i1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double xn = __dmul_rn(x[d], (double)n);
    double whole;
    i0[d] = cell_coord_fast(x[d], xn, n, &whole);
    i1[d] = i0[d] + 1 == n ? 0 : i0[d] + 1;
    w1[d] = xn - whole;
    w0[d] = 1.0 - w1[d];
  }
  double e0 = P.E_app[0], e1 = P.E_app[1], e2 = P.E_app[2];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const double wyz = (b ? w1[1] : w0[1]) * (c ? w1[2] : w0[2]);
      const int64_t row = (int64_t)n * ((b ? i1[1] : i0[1]) + (int64_t)n * (c ? i1[2] : i0[2]));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int64_t node = row + (q ? i1[0] : i0[0]);
        const double w = (q ? w1[0] : w0[0]) * wyz;
        e0 = fma(w, __ldg(a.E0 + node), e0);
        e1 = fma(w, __ldg(a.E1 + node), e1);
        e2 = fma(w, __ldg(a.E2 + node), e2);
      }
    }
  // E^M = -amp (c0 s1 s2, s0 c1 s2, s0 s1 c2)
  const double2* tab =
      reinterpret_cast<const double2*>(P.ginv + 2 * (P.ginv_M + 1) + kQuantileDoubles + kR64Doubles + 8 * kSlopeM);
  double s0, c0, s1, c1, s2, c2;
  sincos_turn(tab, x[0] - P.phi_shift[0], &s0, &c0);
  sincos_turn(tab, x[1] - P.phi_shift[1], &s1, &c1);
  sincos_turn(tab, x[2] - P.phi_shift[2], &s2, &c2);
  const double as0 = a.tE.em_amp * s0;
  L[0] = a.dt_qm * fma(a.tE.em_amp * c0, s1 * s2, e0);
  L[1] = a.dt_qm * fma(as0 * c1, s2, e1);
  L[2] = a.dt_qm * fma(as0 * s1, c2, e2);
}

// kTable: the Gaussian f_v's drift by table; otherwise the paper's problem,
// the isolated-collision drift of Sec. 5.4 and an f_x too sharp for the table.
template <bool kTable>
__global__ void __launch_bounds__(kThreads) k_kick(KickArgs a) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const Params& P = a.P;
  if (j >= P.np) return;
  double x[3] = {a.x0[j], a.x1[j], a.x2[j]};
  double v[3] = {a.v0[j], a.v1[j], a.v2[j]};
  double L[3];
  if (a.lor_mode == 2) {
    L[0] = a.L0[j]; L[1] = a.L1[j]; L[2] = a.L2[j];
  } else {
    lorentz64(a, x, L);
    if (a.lor_mode == 1) {
      a.L0[j] = L[0]; a.L1[j] = L[1]; a.L2[j] = L[2];
    }
  }
  const bool paper = !kTable && P.dist == PIC_DIST_PAPER;
  double vm[3] = {0.0, 0.0, 0.0};
  if (a.drift || paper) { vm[0] = a.vm0[j]; vm[1] = a.vm1[j]; vm[2] = a.vm2[j]; }
  if (a.dv0) { L[0] += a.dv0[j]; L[1] += a.dv1[j]; L[2] += a.dv2[j]; }
  if (paper) {
    // v^M arrays hold tau: vdot^M(t) = vh'(t) tau (Eq. velocity_verlet)
#pragma unroll
    for (int d = 0; d < 3; ++d) L[d] += P.dt * (vm[d] * a.tE.dvh[d]);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) v[d] = fma(0.5, L[d], v[d]);
  a.v0[j] = v[0]; a.v1[j] = v[1]; a.v2[j] = v[2];
  if (!a.drift) return;
  const uint64_t p = a.pid[j];
  const U4 b0 = sample_block(P, p, 0), b1 = sample_block(P, p, 1);
  const uint32_t hi[3] = {b0.x, b0.z, b1.x}, lw[3] = {b0.y, b0.w, b1.y};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if constexpr (kTable) {
      // unif52's 52 bits as the mantissa of a number in [1, 2)
      const double m = __hiloint2double((int)(0x3ff00000u | hi[d] >> 12), (int)(hi[d] << 20 | lw[d] >> 12));
      const double T = m - a.T0;
      const double z = fma(T, (double)kSlopeM, kRound52);
      const double u = fma(T, (double)kSlopeM, kRound52 - z);
      const double g = poly7(P.ginv + 2 * (P.ginv_M + 1) + kQuantileDoubles + kR64Doubles,
                             __double2loint(z) & (kSlopeM - 1), u);
      x[d] = wrap_unit(fma(P.dt, (v[d] - vm[d]) + fma(-a.xslope, g, P.fx_speed), x[d]));
    } else {
      const double xi = unif52(hi[d], lw[d]);
      double s;
      if (paper) {
        double c;
        xm_solve_gen(a.th, d, xi, &s, &c);
        const double xd = xm_dot_gen(a.th, d, s, c);
        x[d] = wrap_unit(x[d] + P.dt * (v[d] + xd - vm[d] * a.th.vh[d]));
      } else if (P.verify & PIC_VERIFY_ISOLATE) {
        // exact manufactured increment x^M(t_{n+1}) - x^M(t_n) (Sec. 5.4)
        const double dxm = xm_solve(P, a.t1, xi, &s) - xm_solve(P, a.t0, xi, &s);
        x[d] = wrap_unit(x[d] + (P.dt * (v[d] - vm[d]) + dxm));
      } else {
        xm_solve(P, a.th, xi, &s);
        const double xd = xm_dot(P, a.th, s);
        x[d] = wrap_unit(x[d] + P.dt * (v[d] + xd - vm[d]));
      }
    }
  }
  a.x0[j] = x[0]; a.x1[j] = x[1]; a.x2[j] = x[2];
  const int n = P.n;
  double whole;
  int ci[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) ci[d] = cell_coord_fast(x[d], __dmul_rn(x[d], (double)n), n, &whole);
  const int32_t k = ci[0] + n * (ci[1] + n * ci[2]);
  a.key[j] = k;
  a.rank[j] = cell_slot(a.count, k);
}

// --------------------------------------------------------------------------
// Error norms (Sec. 4.3): per-block partial sums of squares and maxima of
// e = alpha - alpha^M for x, y, z (minimum image), u, v, w; then phi over
// nodes; a single block combines the partials in fixed order.
// --------------------------------------------------------------------------
struct ErrArgs {
  Params P;
  TimeTerms tt;
  const double *x0, *x1, *x2, *v0, *v1, *v2, *vm0, *vm1, *vm2;
  const uint32_t* pid;
  const double* phi;
  double* part;  // [blocks][14]: 7 sums then 7 maxima
  int pblocks;   // blocks over particles; the rest cover nodes
  double* out;
};

__device__ __forceinline__ void block_reduce_14(double* vals, double* sh) {
  // vals[0..6] summed, vals[7..13] max-reduced; result in thread 0
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 14; ++q) {
    double x = vals[q];
    for (int off = 16; off > 0; off >>= 1) {
      const double y = __shfl_down_sync(0xffffffffu, x, off);
      x = q < 7 ? x + y : fmax(x, y);
    }
    if (lane == 0) sh[w * 14 + q] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 0; q < 14; ++q) {
      double x = sh[q];
      for (int ww = 1; ww < (int)(blockDim.x >> 5); ++ww) x = q < 7 ? x + sh[ww * 14 + q] : fmax(x, sh[ww * 14 + q]);
      vals[q] = x;
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_err_partial(ErrArgs a) {
  __shared__ double sh[(kThreads / 32) * 14];
  const Params& P = a.P;
  double vals[14];
#pragma unroll
  for (int q = 0; q < 14; ++q) vals[q] = 0.0;
  if ((int)blockIdx.x < a.pblocks) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < P.np) {
      const uint64_t p = a.pid[j];
      const U4 b0 = sample_block(P, p, 0), b1 = sample_block(P, p, 1);
      const double xi[3] = {unif52(b0.x, b0.y), unif52(b0.z, b0.w), unif52(b1.x, b1.y)};
      const double xs[3] = {a.x0[j], a.x1[j], a.x2[j]};
      const double vs[3] = {a.v0[j], a.v1[j], a.v2[j]};
      const double vms[3] = {a.vm0[j], a.vm1[j], a.vm2[j]};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        double s, c;
        const bool paper = P.dist == PIC_DIST_PAPER;
        const double xm = paper ? xm_solve_gen(a.tt, d, xi[d], &s, &c) : xm_table(P, a.tt, xi[d]);
        double e = xs[d] - xm;
        e -= floor(e + 0.5);
        vals[d] = e * e;
        vals[7 + d] = fabs(e);
        const double ev = vs[d] - (paper ? vms[d] * a.tt.vh[d] : vms[d]);
        vals[3 + d] = ev * ev;
        vals[10 + d] = fabs(ev);
      }
    }
  } else {
    const int64_t id = (int64_t)(blockIdx.x - a.pblocks) * blockDim.x + threadIdx.x;
    if (id < P.ncell) {
      const int n = P.n;
      const int i = (int)(id % n), jj = (int)((id / n) % n), k = (int)(id / ((int64_t)n * n));
      const double X = i * P.h, Y = jj * P.h, Z = k * P.h;
      double s0, s1, s2;
      s0 = sinpi(2.0 * (X - P.phi_shift[0]));
      s1 = sinpi(2.0 * (Y - P.phi_shift[1]));
      s2 = sinpi(2.0 * (Z - P.phi_shift[2]));
      const double phiM = a.tt.em_amp / kTwoPi * s0 * s1 * s2;
      const double e = a.phi[id] - phiM;
      vals[6] = e * e;
      vals[13] = fabs(e);
    }
  }
  block_reduce_14(vals, sh);
  if (threadIdx.x == 0)
    for (int q = 0; q < 14; ++q) a.part[(size_t)blockIdx.x * 14 + q] = vals[q];
}

constexpr int kFinalThreads = 512;

// one block: each thread sums a fixed strided subset, then a fixed tree
__global__ void __launch_bounds__(kFinalThreads) k_err_final(ErrArgs a, int nblocks) {
  __shared__ double sh[kFinalThreads];
  for (int q = 0; q < 14; ++q) {
    double x = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
      const double y = a.part[(size_t)b * 14 + q];
      x = q < 7 ? x + y : fmax(x, y);
    }
    sh[threadIdx.x] = x;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sh[threadIdx.x] = q < 7 ? sh[threadIdx.x] + sh[threadIdx.x + w]
                                                       : fmax(sh[threadIdx.x], sh[threadIdx.x + w]);
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      double r = sh[0];
      if (q < 6) r = sqrt(r / (double)a.P.np);
      else if (q == 6) r = sqrt(r / (double)a.P.ncell);
      a.out[q] = r;
    }
    __syncthreads();
  }
}

}  // namespace

// ---------------------------------------------------------------------------
cudaError_t launch_sample(pic_ctx* c, double t0) {
  SampleArgs a;
  a.P = c->P;
  a.tt = time_terms(c->P, t0);
  const int b = c->cur;
  a.x0 = c->x[b][0]; a.x1 = c->x[b][1]; a.x2 = c->x[b][2];
  a.v0 = c->v[b][0]; a.v1 = c->v[b][1]; a.v2 = c->v[b][2];
  a.vm0 = c->vm[b][0]; a.vm1 = c->vm[b][1]; a.vm2 = c->vm[b][2];
  a.pid = c->pid[b];
  prof_begin(c);
  k_sample<<<blocks_for(c->P.np), kThreads, 0, c->stream>>>(a);
  prof_end(c, KC_SAMPLE);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t launch_load_state(pic_ctx* c, const double* x, const double* v, double t) {
  LoadArgs a;
  a.P = c->P;
  a.tt = time_terms(c->P, t);
  a.xs = x;
  a.vs = v;
  const int b = c->cur;
  a.x0 = c->x[b][0]; a.x1 = c->x[b][1]; a.x2 = c->x[b][2];
  a.v0 = c->v[b][0]; a.v1 = c->v[b][1]; a.v2 = c->v[b][2];
  a.vm0 = c->vm[b][0]; a.vm1 = c->vm[b][1]; a.vm2 = c->vm[b][2];
  a.pid = c->pid[b];
  prof_begin(c);
  k_load_state<<<blocks_for(c->P.np), kThreads, 0, c->stream>>>(a);
  prof_end(c, KC_OTHER);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t launch_store_state(pic_ctx* c, double* xv) {
  StoreArgs a;
  a.np = c->P.np;
  const int b = c->cur;
  a.x0 = c->x[b][0]; a.x1 = c->x[b][1]; a.x2 = c->x[b][2];
  a.v0 = c->v[b][0]; a.v1 = c->v[b][1]; a.v2 = c->v[b][2];
  a.pid = c->pid[b];
  a.xv = xv;
  prof_begin(c);
  k_store_state<<<blocks_for(c->P.np), kThreads, 0, c->stream>>>(a);
  prof_end(c, KC_OTHER);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t launch_store_dv(pic_ctx* c, double* dv, double* dvm) {
  StoreDvArgs a;
  a.np = c->P.np;
  a.d0 = c->dv[0]; a.d1 = c->dv[1]; a.d2 = c->dv[2];
  a.m0 = c->dvm[0]; a.m1 = c->dvm[1]; a.m2 = c->dvm[2];
  a.pid = c->pid[c->cur];
  a.dv = dv;
  a.dvm = dvm;
  prof_begin(c);
  k_store_dv<<<blocks_for(c->P.np), kThreads, 0, c->stream>>>(a);
  prof_end(c, KC_OTHER);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t launch_dsmc(pic_ctx* c, uint32_t c0, bool separate, double t_src) {
  DsmcArgs a;
  a.P = c->P;
  const TimeTerms ts = time_terms(c->P, t_src);
  for (int d = 0; d < 3; ++d) a.vh[d] = ts.vh[d];
  const int b = c->cur;
  a.v0 = c->v[b][0]; a.v1 = c->v[b][1]; a.v2 = c->v[b][2];
  a.start = c->start;
  a.c0 = c0;
  a.dv0 = c->dv[0]; a.dv1 = c->dv[1]; a.dv2 = c->dv[2];
  if (separate) { a.m0 = c->dvm[0]; a.m1 = c->dvm[1]; a.m2 = c->dvm[2]; }
  else { a.m0 = a.m1 = a.m2 = nullptr; }
  a.overlay = c->overlay;
  a.max_ppc = c->cfg.max_ppc;
  a.G = c->dsmc_G;
  a.Kc = c->dsmc_Kc;
  a.nchunks = (c->P.K + c->dsmc_Kc - 1) / c->dsmc_Kc;
  a.stage = c->dsmc_stage;
  a.T = test32_of(c->P);
  a.ngroups = c->dsmc_groups;
  a.parts = c->dsmc_parts;
  a.partial = c->dsmc_partial;
  // more work than warps: taken from a queue, since a cell's work varies
  a.queue = a.ngroups * a.parts > c->dsmc_grid ? c->dsmc_queue : nullptr;
  a.counters = c->counters;
  a.flags = c->flags;
  a.lg = DLog{c->dlog, c->dlog_n, (long long)c->dlog_cap, c->dlog ? c->dlog_mode : 0};
  a.hist = c->hist_row;
  prof_begin(c);
  if (a.queue) {
    const cudaError_t eq = cudaMemsetAsync(c->dsmc_queue, 0, 8, c->stream);
    if (eq != cudaSuccess) return eq;
  }
  if (c->P.verify || a.lg.mode == PIC_DLOG_ALL)
    k_dsmc<true><<<c->dsmc_grid, kDsmcThreads, c->dsmc_smem, c->stream>>>(a);
  else
    k_dsmc<false><<<c->dsmc_grid, kDsmcThreads, c->dsmc_smem, c->stream>>>(a);
  if (a.parts > 1) {
    k_dsmc_merge<<<blocks_for(32 * c->P.ncell, kMergeThreads), kMergeThreads, 0, c->stream>>>(a);
    c->launches++;
  }
  prof_end(c, KC_DSMC);
  c->launches++;
  return cudaGetLastError();
}

int dsmc_threads() { return kDsmcThreads; }
size_t dsmc_smem_bytes(int max_ppc, int stage) {
  return sizeof(Warp64) + (size_t)stage * sizeof(float4) + (size_t)max_ppc * 4;
}
const void* dsmc_kernel_ptr(bool verify) {
  return verify ? (const void*)k_dsmc<true> : (const void*)k_dsmc<false>;
}

cudaError_t launch_kick(pic_ctx* c, double tE, bool with_coll, bool drift, double th, double tn1) {
  KickArgs a;
  a.P = c->P;
  const int b = c->cur;
  a.x0 = c->x[b][0]; a.x1 = c->x[b][1]; a.x2 = c->x[b][2];
  a.v0 = c->v[b][0]; a.v1 = c->v[b][1]; a.v2 = c->v[b][2];
  a.vm0 = c->vm[b][0]; a.vm1 = c->vm[b][1]; a.vm2 = c->vm[b][2];
  a.pid = c->pid[b];
  if (with_coll) { a.dv0 = c->dv[0]; a.dv1 = c->dv[1]; a.dv2 = c->dv[2]; }
  else { a.dv0 = a.dv1 = a.dv2 = nullptr; }
  a.E0 = c->E[0]; a.E1 = c->E[1]; a.E2 = c->E[2];
  a.L0 = c->lor[0]; a.L1 = c->lor[1]; a.L2 = c->lor[2];
  // the kick without drift closes a step at the time level where the next
  // step's first kick starts: keep its Lorentz term for that kick
  a.lor_mode = drift ? (c->lor_valid ? 2 : 0) : 1;
  a.tE = time_terms(c->P, tE);
  a.th = time_terms(c->P, th);
  a.t0 = time_terms(c->P, tE);
  a.t1 = time_terms(c->P, tn1);
  a.drift = drift ? 1 : 0;
  const Params& P = c->P;
  a.dt_qm = P.dt * P.qm_eff;
  a.T0 = (1.0 - 0x1p-53) + (a.th.ct + P.fx_amp_over_2pi * a.th.cos2ct);
  // A c (S + s) / (1 + A S) with s = sin(2 pi c t) is c - c (1 - A s) / (1 + A S)
  a.xslope = P.fx_speed * (1.0 - P.fx_amp * a.th.sin2ct);
  a.key = c->key;
  a.rank = c->rank;
  a.count = c->count;
  const bool table = P.dist == PIC_DIST_CONFIG && !(P.verify & PIC_VERIFY_ISOLATE) && P.xm_table &&
                     fabs(a.T0) < 0x1p30;  // (beyond, T has no digits left to look up)
  prof_begin(c);
  if (table) k_kick<true><<<blocks_for(P.np), kThreads, 0, c->stream>>>(a);
  else k_kick<false><<<blocks_for(P.np), kThreads, 0, c->stream>>>(a);
  prof_end(c, KC_KICK);
  c->launches++;
  c->lor_valid = !drift;
  return cudaGetLastError();
}

cudaError_t launch_errors(pic_ctx* c, double t) {
  ErrArgs a;
  a.P = c->P;
  a.tt = time_terms(c->P, t);
  const int b = c->cur;
  a.x0 = c->x[b][0]; a.x1 = c->x[b][1]; a.x2 = c->x[b][2];
  a.v0 = c->v[b][0]; a.v1 = c->v[b][1]; a.v2 = c->v[b][2];
  a.vm0 = c->vm[b][0]; a.vm1 = c->vm[b][1]; a.vm2 = c->vm[b][2];
  a.pid = c->pid[b];
  a.phi = c->phi;
  a.part = c->err_part;
  a.pblocks = blocks_for(c->P.np);
  a.out = c->err_out;
  const int nb = a.pblocks + blocks_for(c->P.ncell);
  prof_begin(c);
  k_err_partial<<<nb, kThreads, 0, c->stream>>>(a);
  k_err_final<<<1, kFinalThreads, 0, c->stream>>>(a, nb);
  prof_end(c, KC_ERR);
  c->launches += 2;
  return cudaGetLastError();
}

int err_blocks_needed(int64_t np, int64_t ncell) { return blocks_for(np) + blocks_for(ncell); }

cudaError_t launch_err_final(pic_ctx* c, int nb) {
  ErrArgs a;
  a.P = c->P;
  a.part = c->err_part;
  a.out = c->err_out;
  k_err_final<<<1, kFinalThreads, 0, c->stream>>>(a, nb);
  c->launches++;
  return cudaGetLastError();
}

}  // namespace pic

namespace pic {
TimeTerms time_terms(const Params& P, double t) {
  TimeTerms tt;
  tt.t = t;
  tt.ct = P.fx_speed * t;
  tt.cos2ct = cos(kTwoPi * tt.ct);
  tt.sin2ct = sin(kTwoPi * tt.ct);
  tt.em_amp = kTwoPi * P.phi_amp * exp(t / (2.0 * P.phi_T));
  for (int d = 0; d < 3; ++d) {
    tt.fA[d] = tt.fs[d] = tt.fdA[d] = tt.fds[d] = tt.fsn[d] = 0.0;
    tt.fcs[d] = 1.0;
    tt.vh[d] = tt.dvh[d] = 0.0;
  }
  if (P.dist == PIC_DIST_PAPER) {
    // Sec. 5.2 on the unit cube, T = t_ref
    const double T = P.t_ref, e = exp(t / T), vb = P.vbar;
    tt.fA[0] = e / 5.0;  tt.fs[0] = 0.0;
    tt.fA[1] = 1.0 / 5.0; tt.fs[1] = 3.0 * e / 20.0;
    tt.fA[2] = -e / 6.0; tt.fs[2] = -e / 15.0;
    for (int d = 0; d < 3; ++d) {
      tt.fdA[d] = d == 1 ? 0.0 : tt.fA[d] / T;
      tt.fds[d] = tt.fs[d] / T;
      tt.fcs[d] = cos(kTwoPi * tt.fs[d]);
      tt.fsn[d] = sin(kTwoPi * tt.fs[d]);
    }
    tt.vh[0] = vb * (1.0 + sin(kPi * t / (2.0 * T)) / 5.0);
    tt.vh[1] = vb * (1.0 + cos(kPi * t / T) / 5.0);
    tt.vh[2] = vb * (1.0 + sin(3.0 * kPi * t / (2.0 * T)) / 5.0);
    tt.dvh[0] = vb * (kPi / (2.0 * T)) * cos(kPi * t / (2.0 * T)) / 5.0;
    tt.dvh[1] = -vb * (kPi / T) * sin(kPi * t / T) / 5.0;
    tt.dvh[2] = vb * (3.0 * kPi / (2.0 * T)) * cos(3.0 * kPi * t / (2.0 * T)) / 5.0;
  }
  return tt;
}
}  // namespace pic
