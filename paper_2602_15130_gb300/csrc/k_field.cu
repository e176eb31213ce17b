// Field solve of Eq. poisson_mms on the periodic node mesh:
//   rhs : rho at nodes from the per-cell CIC partials, b = rho/eps0 -
//         Lap phi^M - rho^M/eps0 and per-block partial sums of b;
//   cg  : one cooperative persistent kernel: conjugate gradients on
//         -Lap_h phi = b - mean(b) (7-point, warm start), zero-mean
//         projection and E = -grad_h phi by central differences.
// All reductions are per-block partials combined in a fixed order, so a
// solve is deterministic for a given grid. Waits over the grid are bounded
// (grid_exchange.cuh).
#include <type_traits>

#include "grid_exchange.cuh"
#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kThreads = 256;

inline int blocks_for(int64_t n, int t = kThreads) {
  int64_t b = (n + t - 1) / t;
  return (int)(b < 1 ? 1 : b);
}

// fixed-shape block sum (sh holds at least 33 doubles); thread 0 adds the
// warp totals and the result is broadcast to every thread
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += sh[i];
    sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

struct RhsArgs {
  Params P;
  TimeTerms tt;
  const double* corner;
  double *rho, *b, *part;
  float* b32;  // precision form: b in FP32 (b may then be null)
};

__global__ void __launch_bounds__(kThreads) k_rhs(RhsArgs a) {
  __shared__ double sh[40];
  const Params& P = a.P;
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double bv = 0.0;
  if (id < P.ncell) {
    const int n = P.n;
    const int i = (int)(id % n), j = (int)((id / n) % n), k = (int)(id / ((int64_t)n * n));
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int ii = i - q < 0 ? n - 1 : i - q, jj = j - b < 0 ? n - 1 : j - b, kk = k - c < 0 ? n - 1 : k - c;
          s += a.corner[(int64_t)(q + 2 * b + 4 * c) * P.ncell + ii + (int64_t)n * (jj + (int64_t)n * kk)];
        }
    const double rho = P.rho_scale * s;
    const double X = i * P.h, Y = j * P.h, Z = k * P.h;
    const double ct = a.tt.ct;
    const double phiM = a.tt.em_amp / kTwoPi * sinpi(2.0 * (X - P.phi_shift[0])) *
                        sinpi(2.0 * (Y - P.phi_shift[1])) * sinpi(2.0 * (Z - P.phi_shift[2]));
    const double lap_phiM = -3.0 * kTwoPi * kTwoPi * phiM;
    const double rhoM =
        P.dist == PIC_DIST_PAPER
            ? P.q_eff * P.nphys * (1.0 + a.tt.fA[0] * sinpi(2.0 * (X - a.tt.fs[0]))) *
                  (1.0 + a.tt.fA[1] * sinpi(2.0 * (Y - a.tt.fs[1]))) * (1.0 + a.tt.fA[2] * sinpi(2.0 * (Z - a.tt.fs[2])))
            : P.q_eff * P.nphys * (1.0 + P.fx_amp * sinpi(2.0 * (X - ct))) * (1.0 + P.fx_amp * sinpi(2.0 * (Y - ct))) *
                  (1.0 + P.fx_amp * sinpi(2.0 * (Z - ct)));
    bv = rho / P.eps0 - lap_phiM - rhoM / P.eps0;
    a.rho[id] = rho;
    if (a.b) a.b[id] = bv;
    if (a.b32) a.b32[id] = (float)bv;
  }
  const double tot = block_sum(bv, sh);
  if (threadIdx.x == 0) a.part[blockIdx.x] = tot;
}

// Precision form: the same RHS with the manufactured terms in FP32 (the
// FP64 pipe is slow on this part); the corner sums, rho and the block
// partial of the mean stay FP64.
struct Rhs32Consts {
  float h, two_pi_over, lap_scale;   // h, phi^M amplitude / (2 pi) * e^{t/2T}, -3 (2 pi)^2
  float shift[3], ct, fx_amp;
  float rhoM_scale, inv_eps0;         // q N, 1/eps0
  int paper;                          // PIC_DIST_PAPER: per-axis amplitude fA and phase fs
  float fA[3], fs[3];
};

__global__ void __launch_bounds__(kThreads) k_rhs32(RhsArgs a, Rhs32Consts k) {
  __shared__ double sh[40];
  const Params& P = a.P;
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double bsum = 0.0;
  if (id < P.ncell) {
    const int n = P.n;
    const int i = (int)(id % n), j = (int)((id / n) % n), kk0 = (int)(id / ((int64_t)n * n));
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int ii = i - q < 0 ? n - 1 : i - q, jj = j - b < 0 ? n - 1 : j - b, kk = kk0 - c < 0 ? n - 1 : kk0 - c;
          s += a.corner[(int64_t)(q + 2 * b + 4 * c) * P.ncell + ii + (int64_t)n * (jj + (int64_t)n * kk)];
        }
    const double rho = P.rho_scale * s;
    const float X = (float)i * k.h, Y = (float)j * k.h, Z = (float)kk0 * k.h;
    const float phiM = k.two_pi_over * sinpif(2.f * (X - k.shift[0])) * sinpif(2.f * (Y - k.shift[1])) *
                       sinpif(2.f * (Z - k.shift[2]));
    const float rhoM =
        k.paper ? k.rhoM_scale * (1.f + k.fA[0] * sinpif(2.f * (X - k.fs[0]))) *
                      (1.f + k.fA[1] * sinpif(2.f * (Y - k.fs[1]))) * (1.f + k.fA[2] * sinpif(2.f * (Z - k.fs[2])))
                : k.rhoM_scale * (1.f + k.fx_amp * sinpif(2.f * (X - k.ct))) *
                      (1.f + k.fx_amp * sinpif(2.f * (Y - k.ct))) * (1.f + k.fx_amp * sinpif(2.f * (Z - k.ct)));
    const float bv = (float)(rho * (double)k.inv_eps0) - k.lap_scale * phiM - rhoM * k.inv_eps0;
    a.rho[id] = rho;
    a.b32[id] = bv;
    bsum = (double)bv;
  }
  const double tot = block_sum(bsum, sh);
  if (threadIdx.x == 0) a.part[blockIdx.x] = tot;
}

struct CgArgs {
  int n;
  int64_t ncell;
  double inv_h2, two_h;
  const double* b;
  double *x, *r, *p0, *p1, *q;
  const double* rhs_part;  // block partial sums of b, or nullptr: summed here
  int rhs_blocks;
  GridSlot* slots;         // exchange_slots(gridDim.x) of them
  unsigned launch;         // the launch's number: never zero, never the same twice on these slots
  int* info;    // [0] iterations [1] status (1 = no convergence) [2] number of a launch that timed out
  int* flags;   // sticky context flags
  double* res;
  int skip_block = -1;  // failure injection: this block leaves before its first exchange
  double tol;
  int maxit;
  double *E0, *E1, *E2;
  long long* hist = nullptr;  // per-step history row: [0] iterations
};

// periodic neighbours of node id = i + n (j + n k), 32-bit indices (n^3 <
// 2^31): x+, x-, y+, y-, z+, z-
struct Nbr {
  int xp, xm, yp, ym, zp, zm;
};
__device__ __forceinline__ Nbr neighbours(int id, int i, int j, int k, int n, int nn) {
  Nbr b;
  b.xp = i == n - 1 ? id - (n - 1) : id + 1;
  b.xm = i == 0 ? id + (n - 1) : id - 1;
  b.yp = j == n - 1 ? id - (n - 1) * n : id + n;
  b.ym = j == 0 ? id + (n - 1) * n : id - n;
  b.zp = k == n - 1 ? id - (n - 1) * nn : id + nn;
  b.zm = k == 0 ? id + (n - 1) * nn : id - nn;
  return b;
}

// Launch shape of the solve. The FP64 pipe does two lanes per SM and clock,
// so a warp's FP64 instruction holds it for 19 cycles (measured): the nodes are spread
// over every SM, one block each, with as few threads as hold them (32 at
// least), npt nodes a thread in registers (1, 2, 4 or 8; 0: more than that,
// the vectors stay in memory).
//
// With the vectors in memory (n >= 86 on 152 SMs) a solve is bound by L2: 1,024
// threads for the loads in flight, and the grid's threads on consecutive nodes,
// so that the blocks' stencils meet in L2 at the same time. us an iteration at
// 86^3, 100^3, 128^3 and 144^3: 27.3, 34.8, 59.1, 88.4; with 512 threads and a
// contiguous range a block 28.1, 38.4, 70.6, 117; with 1,024 and ranges 26.6,
// 34.3, 60.7, 95.1. Loads through L1 made no difference.
constexpr int kCgThreads = 512;
constexpr int kCgThreadsMem = 1024;

struct CgShape {
  int npt, threads, grid;
};
inline CgShape cg_shape(int64_t m, int sms) {
  CgShape s;
  if (sms > kMaxExchangeBlocks) sms = kMaxExchangeBlocks;
  const int64_t per = (m + sms - 1) / sms;  // nodes an SM
  s.npt = per <= kCgThreads ? 1 : per <= 2 * kCgThreads ? 2 : per <= 4 * kCgThreads ? 4 : per <= 8 * kCgThreads ? 8 : 0;
  if (s.npt == 0) {
    s.threads = kCgThreadsMem;
    s.grid = sms;
    return s;
  }
  s.threads = (int)(((per + s.npt - 1) / s.npt + 31) / 32 * 32);
  s.grid = (int)((m + (int64_t)s.npt * s.threads - 1) / ((int64_t)s.npt * s.threads));
  return s;
}

// Conjugate gradients, the textbook recurrence. What bounds a small solve is
// the two reductions over the grid that an iteration cannot do without:
//  - a reduction and the barrier that goes with it are one exchange
//    (grid_exchange.cuh), and inside a block the FP64 additions are done by
//    one warp (a shuffle tree in every warp costs warps x 5 x 19 cycles of
//    the FP64 pipe);
//  - p's update needs no barrier of its own where a thread holds one node
//    (m <= 512 nodes an SM): every thread forms its neighbours' new p from
//    their r and old p (the same arithmetic, p double-buffered). From two
//    nodes a thread on, those six extra FP64 operations a node cost more
//    than the third exchange.
// Per iteration at 32^3, 48^3 and 64^3 nodes, with the solve's launch: 11.9,
// 17.8 and 23 us before (256- or 1024-thread blocks, an atomic-counter
// barrier, three barriers, shuffle trees in every warp), 9.1, 11.4 and 15 us
// now, two thirds of it in the exchanges.

// The stopping rule ||r|| <= thresh = tol ||b||: the squares decide where
// they are clearly apart (an FP64 square root takes 600 cycles).
__device__ __forceinline__ bool done(double bb, double rr, double thresh, double lo2, double hi2) {
  if (bb == 0.0 || rr < lo2) return true;
  if (rr > hi2) return false;
  return sqrt(rr) <= thresh;
}

template <int NPT>
__global__ void __launch_bounds__(NPT > 0 ? kCgThreads : kCgThreadsMem) k_cg(CgArgs a) {
  constexpr bool kRegs = NPT > 0, kRecompute = NPT == 1;
  constexpr int kN = kRegs ? NPT : 1;
  __shared__ double sh[2 * (kRegs ? kCgThreads : kCgThreadsMem)];
  __shared__ double scal[2];  // scalars formed once per block by thread 0
  __shared__ int stop, ok_sh;
  // the others then wait for an arrival that never comes, until the bound
  if ((int)blockIdx.x == a.skip_block) return;
  const int n = a.n, nn = a.n * a.n;
  const int m = (int)a.ncell;
  const int t = threadIdx.x, T = blockDim.x, G = gridDim.x;
  const int64_t lo64 = (int64_t)blockIdx.x * (NPT * T);  // (in registers: the block's nodes)
  const int lo = (int)(lo64 < m ? lo64 : m), hi = lo64 + NPT * T < m ? (int)(lo64 + NPT * T) : m;
  GridExchange X{a.slots, G, a.launch, 0u, a.info + 2, a.flags, &ok_sh};
  double xr[kN], rr_[kN], pr[kN], qr[kN];
  int ijk[kN];  // the node's coordinates, 10 bits each
  // f(k, id, i, j, l) for every node of the thread: register slot k, node id
  // with coordinates (i, j, l)
  auto each = [&](auto f) {
    if constexpr (kRegs) {
#pragma unroll
      for (int k = 0; k < kN; ++k) {
        const int id = lo + t + k * T;
        if (id < hi) f(k, id, ijk[k] & 1023, (ijk[k] >> 10) & 1023, ijk[k] >> 20);
      }
    } else {
      for (int64_t i = (int64_t)blockIdx.x * T + t; i < m; i += G * T) {
        const int id = (int)i;
        f(0, id, id % n, (id / n) % n, id / nn);
      }
    }
  };
  if constexpr (kRegs) {
#pragma unroll
    for (int k = 0; k < kN; ++k) {
      const int id = lo + t + k * T;
      ijk[k] = (id % n) | ((id / n) % n) << 10 | (id / nn) << 20;
    }
  }
  double tot[2];

  // the mean of b
  if (a.rhs_part) {
    if (t < 32) {
      double s = 0.0;
      for (int i = t; i < a.rhs_blocks; i += 32) s += a.rhs_part[i];
      s = warp_sum_d(s);
      if (t == 0) scal[0] = s / (double)m;
    }
    __syncthreads();
  } else {
    double s = 0.0;
    each([&](int, int id, int, int, int) { s += a.b[id]; });
    X.sum<1, false>(&s, tot, sh);
    if (t == 0) scal[0] = tot[0] / (double)m;
    __syncthreads();
    if (!ok_sh) return;
  }
  const double mean_b = scal[0];
  // r = b - A x, ||r||^2 and ||b||^2
  double loc[2] = {0.0, 0.0};
  each([&](int k, int id, int i, int j, int l) {
    const Nbr q = neighbours(id, i, j, l, n, nn);
    const double bv = a.b[id] - mean_b;
    const double* x = a.x;
    const double xc = x[id];
    const double nb = x[q.xp] + x[q.xm] + x[q.yp] + x[q.ym] + x[q.zp] + x[q.zm];
    const double rv = bv - (6.0 * xc - nb) * a.inv_h2;
    a.r[id] = rv;
    if constexpr (kRegs) {
      xr[k] = xc;
      rr_[k] = rv;
    }
    loc[0] += rv * rv;
    loc[1] += bv * bv;
  });
  double rr = 0.0, bb = 0.0, thresh = 0.0, lo2 = 0.0, hi2 = 0.0;  // thread 0
  int it = 0, status = 0;
  // every sum ends with thread 0's scalars published by one block barrier
  X.sum<2, true>(loc, tot, sh);
  if (t == 0) {
    rr = tot[0];
    bb = tot[1];
    thresh = a.tol * sqrt(bb);
    lo2 = thresh * thresh * (1.0 - 1e-12);
    hi2 = thresh * thresh * (1.0 + 1e-12);
    stop = done(bb, rr, thresh, lo2, hi2) ? 1 : (it >= a.maxit ? 2 : 0);
  }
  __syncthreads();
  if (!ok_sh) return;
  double beta = 0.0;
  double *p = a.p0, *p_new = kRecompute ? a.p1 : a.p0;
  while (true) {
    if (stop == 1) break;
    if (stop == 2) { status = 1; break; }
    // p = r + beta p, then q = A p and p.q
    double pq = 0.0;
    if constexpr (kRecompute) {
      each([&](int k, int id, int i, int j, int l) {
        const Nbr q = neighbours(id, i, j, l, n, nn);
        const double* r = a.r;
        const double pc = it == 0 ? rr_[k] : rr_[k] + beta * pr[k];
        double v[6] = {__ldcg(r + q.xp), __ldcg(r + q.xm), __ldcg(r + q.yp),
                       __ldcg(r + q.ym), __ldcg(r + q.zp), __ldcg(r + q.zm)};
        if (it > 0) {
          const double o[6] = {__ldcg(p + q.xp), __ldcg(p + q.xm), __ldcg(p + q.yp),
                               __ldcg(p + q.ym), __ldcg(p + q.zp), __ldcg(p + q.zm)};
#pragma unroll
          for (int e = 0; e < 6; ++e) v[e] = v[e] + beta * o[e];
        }
        p_new[id] = pc;
        pr[k] = pc;
        const double qv = (6.0 * pc - (v[0] + v[1] + v[2] + v[3] + v[4] + v[5])) * a.inv_h2;
        qr[k] = qv;
        pq += pc * qv;
      });
      double* s = p;
      p = p_new;
      p_new = s;
    } else {
      each([&](int k, int id, int, int, int) {
        const double rv = kRegs ? rr_[k] : a.r[id];
        const double pc = it == 0 ? rv : rv + beta * (kRegs ? pr[k] : p[id]);
        p[id] = pc;
        if constexpr (kRegs) pr[k] = pc;
      });
      X.sum<0, true>(nullptr, nullptr, sh);
      __syncthreads();
      if (!ok_sh) return;
      each([&](int k, int id, int i, int j, int l) {
        const Nbr q = neighbours(id, i, j, l, n, nn);
        const double nb = __ldcg(p + q.xp) + __ldcg(p + q.xm) + __ldcg(p + q.yp) + __ldcg(p + q.ym) +
                          __ldcg(p + q.zp) + __ldcg(p + q.zm);
        const double pc = kRegs ? pr[k] : p[id];
        const double qv = (6.0 * pc - nb) * a.inv_h2;
        if constexpr (kRegs) qr[k] = qv;
        else a.q[id] = qv;
        pq += pc * qv;
      });
    }
    X.sum<1, false>(&pq, tot, sh);
    if (t == 0) scal[0] = rr / tot[0];
    __syncthreads();
    if (!ok_sh) return;
    const double alpha = scal[0];
    double rn = 0.0;
    each([&](int k, int id, int, int, int) {
      if constexpr (kRegs) {
        xr[k] += alpha * pr[k];
        rr_[k] = rr_[k] - alpha * qr[k];
        a.r[id] = rr_[k];
        rn += rr_[k] * rr_[k];
      } else {
        a.x[id] += alpha * p[id];
        const double rv = a.r[id] - alpha * a.q[id];
        a.r[id] = rv;
        rn += rv * rv;
      }
    });
    ++it;
    X.sum<1, kRecompute>(&rn, tot, sh);  // with r (and p) for the neighbours' p
    if (t == 0) {
      scal[1] = tot[0] / rr;
      rr = tot[0];
      stop = done(bb, rr, thresh, lo2, hi2) ? 1 : (it >= a.maxit ? 2 : 0);
    }
    __syncthreads();
    if (!ok_sh) return;
    beta = scal[1];
  }
  // zero-mean projection
  double xs = 0.0;
  each([&](int k, int id, int, int, int) { xs += kRegs ? xr[k] : a.x[id]; });
  X.sum<1, false>(&xs, tot, sh);
  if (t == 0) scal[0] = tot[0] / (double)m;
  __syncthreads();
  if (!ok_sh) return;
  const double mean_x = scal[0];
  each([&](int k, int id, int, int, int) { a.x[id] = (kRegs ? xr[k] : a.x[id]) - mean_x; });
  X.sum<0, true>(nullptr, nullptr, sh);
  __syncthreads();
  if (!ok_sh) return;
  // E = -grad_h phi, second-order central differences
  each([&](int, int id, int i, int j, int l) {
    const Nbr q = neighbours(id, i, j, l, n, nn);
    const double* x = a.x;
    a.E0[id] = -(__ldcg(x + q.xp) - __ldcg(x + q.xm)) / a.two_h;
    a.E1[id] = -(__ldcg(x + q.yp) - __ldcg(x + q.ym)) / a.two_h;
    a.E2[id] = -(__ldcg(x + q.zp) - __ldcg(x + q.zm)) / a.two_h;
  });
  if (blockIdx.x == 0 && t == 0) {
    a.info[0] = it;
    a.info[1] = status;
    if (a.hist) a.hist[0] = it;
    a.res[0] = bb > 0.0 ? sqrt(rr) / sqrt(bb) : 0.0;
    if (status) atomicOr(a.flags, 2);
    atomicMax(a.flags + 1, it);
  }
}

const void* cg_kernel(int npt) {
  return npt == 1   ? (const void*)k_cg<1>
         : npt == 2 ? (const void*)k_cg<2>
         : npt == 4 ? (const void*)k_cg<4>
         : npt == 8 ? (const void*)k_cg<8>
                    : (const void*)k_cg<0>;
}

// The solve on one cluster of 16 blocks, one node a thread, for meshes of at
// most 8,192 nodes (n <= 20): a block's p lives in its shared memory,
// neighbours in other blocks are read there, and a sum over the cluster is
// 16 stores into every block's shared memory and one cluster barrier (400
// cycles; 2,080 with the sums, where an exchange over the whole grid takes
// 5,000). With more nodes the cluster's 16 FP64 pipes take longer than the
// exchanges over all SMs cost: per iteration at 8^3 and 24^3 nodes (there
// two nodes a thread) 4.4 and 7.9 us against 6.2 and 7.4 us on the grid.
constexpr int kClusterBlocks = 16;
constexpr int64_t kClusterNodes = (int64_t)kClusterBlocks * kCgThreads;

__device__ __forceinline__ uint32_t cluster_address(const void* shared, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(shared)), "r"(rank));
  return a;
}
__device__ __forceinline__ double ld_cluster(uint32_t a) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kCgThreads) k_cg_cluster(CgArgs a) {
  __shared__ double sh[2 * kCgThreads];
  __shared__ double ps[kCgThreads];                      // this block's p
  __shared__ double part[2][2][kClusterBlocks];          // every block's partials, alternating
  __shared__ double scal[2];
  __shared__ int stop;
  const int n = a.n, nn = a.n * a.n, m = (int)a.ncell;
  const int t = threadIdx.x, T = blockDim.x;
  const int id = (int)blockIdx.x * T + t;
  const bool own = id < m;
  uint32_t nbr[6];  // the neighbours' p: x+, x-, y+, y-, z+, z-
  {
    const Nbr q = neighbours(id, id % n, (id / n) % n, id / nn, n, nn);
    const int o[6] = {q.xp, q.xm, q.yp, q.ym, q.zp, q.zm};
#pragma unroll
    for (int e = 0; e < 6; ++e) nbr[e] = own ? cluster_address(ps + o[e] % T, (uint32_t)(o[e] / T)) : 0u;
  }
  auto nbr_sum = [&]() {
    double v[6];
#pragma unroll
    for (int e = 0; e < 6; ++e) v[e] = ld_cluster(nbr[e]);
    return v[0] + v[1] + v[2] + v[3] + v[4] + v[5];
  };
  // Totals over the cluster of two values per thread (or one), in warp 0;
  // the caller follows with a __syncthreads.
  int set = 0;
  double tot[2];
  auto sum = [&](auto two, double u, double v) {
    constexpr int kV = decltype(two)::value ? 2 : 1;
    set ^= 1;
    sh[t] = u;
    if (kV == 2) sh[T + t] = v;
    __syncthreads();
    if (t < 32) {
#pragma unroll
      for (int q = 0; q < kV; ++q) {
        double s = sh[q * T + t];
        for (int w = t + 32; w < T; w += 32) s += sh[q * T + w];
        s = warp_sum_d(s);
        if (t < kClusterBlocks) st_cluster(cluster_address(&part[set][q][blockIdx.x], (uint32_t)t), s);
      }
    }
    cluster_barrier();
    if (t < 32) {
#pragma unroll
      for (int q = 0; q < kV; ++q) {
        double s = part[set][q][t & (kClusterBlocks - 1)];
#pragma unroll
        for (int off = kClusterBlocks / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        tot[q] = s;
      }
    }
  };

  cluster_barrier();  // every block's shared memory is there
  if (a.rhs_part) {
    if (t < 32) {
      double s = 0.0;
      for (int i = t; i < a.rhs_blocks; i += 32) s += a.rhs_part[i];
      s = warp_sum_d(s);
      if (t == 0) scal[0] = s / (double)m;
    }
  } else {
    sum(std::false_type{}, own ? a.b[id] : 0.0, 0.0);
    if (t == 0) scal[0] = tot[0] / (double)m;
  }
  __syncthreads();
  const double mean_b = scal[0];
  // r = b - A x
  double xr = 0.0, rv = 0.0, pr = 0.0, qr = 0.0, bv = 0.0;
  if (own) {
    xr = a.x[id];
    ps[t] = xr;
  }
  cluster_barrier();
  if (own) {
    bv = a.b[id] - mean_b;
    rv = bv - (6.0 * xr - nbr_sum()) * a.inv_h2;
  }
  double rr = 0.0, bb = 0.0, thresh = 0.0, lo2 = 0.0, hi2 = 0.0;  // thread 0
  int it = 0, status = 0;
  sum(std::true_type{}, rv * rv, bv * bv);
  if (t == 0) {
    rr = tot[0];
    bb = tot[1];
    thresh = a.tol * sqrt(bb);
    lo2 = thresh * thresh * (1.0 - 1e-12);
    hi2 = thresh * thresh * (1.0 + 1e-12);
    stop = done(bb, rr, thresh, lo2, hi2) ? 1 : (it >= a.maxit ? 2 : 0);
  }
  __syncthreads();
  double beta = 0.0;
  while (true) {
    if (stop == 1) break;
    if (stop == 2) { status = 1; break; }
    if (own) {
      pr = it == 0 ? rv : rv + beta * pr;
      ps[t] = pr;
    }
    cluster_barrier();
    if (own) qr = (6.0 * pr - nbr_sum()) * a.inv_h2;
    sum(std::false_type{}, pr * qr, 0.0);
    if (t == 0) scal[0] = rr / tot[0];
    __syncthreads();
    const double alpha = scal[0];
    if (own) {
      xr += alpha * pr;
      rv = rv - alpha * qr;
    }
    ++it;
    sum(std::false_type{}, rv * rv, 0.0);
    if (t == 0) {
      scal[1] = tot[0] / rr;
      rr = tot[0];
      stop = done(bb, rr, thresh, lo2, hi2) ? 1 : (it >= a.maxit ? 2 : 0);
    }
    __syncthreads();
    beta = scal[1];
  }
  // zero-mean projection and E
  sum(std::false_type{}, xr, 0.0);
  if (t == 0) scal[0] = tot[0] / (double)m;
  __syncthreads();
  const double mean_x = scal[0];
  if (own) {
    a.x[id] = xr - mean_x;
    ps[t] = xr - mean_x;
  }
  cluster_barrier();
  if (own) {
    a.E0[id] = -(ld_cluster(nbr[0]) - ld_cluster(nbr[1])) / a.two_h;
    a.E1[id] = -(ld_cluster(nbr[2]) - ld_cluster(nbr[3])) / a.two_h;
    a.E2[id] = -(ld_cluster(nbr[4]) - ld_cluster(nbr[5])) / a.two_h;
  }
  if (blockIdx.x == 0 && t == 0) {
    a.info[0] = it;
    a.info[1] = status;
    if (a.hist) a.hist[0] = it;
    a.res[0] = bb > 0.0 ? sqrt(rr) / sqrt(bb) : 0.0;
    if (status) atomicOr(a.flags, 2);
    atomicMax(a.flags + 1, it);
  }
  cluster_barrier();  // no block leaves while another reads its shared memory
}

int cluster_threads(int64_t m) { return (int)(((m + kClusterBlocks - 1) / kClusterBlocks + 31) / 32 * 32); }

// Launch the solve: on one cluster (cg_cluster_fits), else on a cooperative
// grid over the SMs (always with a failure injection, whose wait is bounded
// there).
cudaError_t launch_solve(const CgArgs& args, bool cluster, int sms, cudaStream_t stream) {
  CgArgs a = args;
  void* argv[] = {&a};
  if (cluster && a.skip_block < 0) {
    const ClusterLaunch l(kClusterBlocks, cluster_threads(a.ncell), stream);
    return cudaLaunchKernelExC(&l.cfg, (const void*)k_cg_cluster, argv);
  }
  const CgShape s = cg_shape(a.ncell, sms);
  return cudaLaunchCooperativeKernel(cg_kernel(s.npt), dim3(s.grid), dim3(s.threads), argv, 0, stream);
}

struct StoreFieldArgs {
  int64_t ncell;
  const double *rho, *phi, *E0, *E1, *E2;
  double *orho, *ophi, *oE;
};

__global__ void __launch_bounds__(kThreads) k_store_field(StoreFieldArgs a) {
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= a.ncell) return;
  if (a.orho) a.orho[id] = a.rho[id];
  if (a.ophi) a.ophi[id] = a.phi[id];
  if (a.oE) {
    a.oE[3 * id] = a.E0[id];
    a.oE[3 * id + 1] = a.E1[id];
    a.oE[3 * id + 2] = a.E2[id];
  }
}

}  // namespace

int rhs_blocks_needed(int64_t ncell) { return blocks_for(ncell); }

cudaError_t launch_rhs(pic_ctx* c, double t) {
  RhsArgs a;
  a.P = c->P;
  a.tt = time_terms(c->P, t);
  a.corner = c->corner;
  a.rho = c->rho;
  a.b = c->mixed ? nullptr : c->b;
  a.b32 = c->mixed ? c->bf : nullptr;
  a.part = c->rhs_part;
  prof_begin(c);
  if (c->mixed) {
    Rhs32Consts k;
    k.h = (float)c->P.h;
    k.two_pi_over = (float)(a.tt.em_amp / kTwoPi);
    k.lap_scale = (float)(-3.0 * kTwoPi * kTwoPi);
    for (int d = 0; d < 3; ++d) k.shift[d] = (float)c->P.phi_shift[d];
    k.ct = (float)(a.tt.ct - floor(a.tt.ct));
    k.fx_amp = (float)c->P.fx_amp;
    k.rhoM_scale = (float)(c->P.q_eff * c->P.nphys);
    k.inv_eps0 = (float)(1.0 / c->P.eps0);
    k.paper = c->P.dist == PIC_DIST_PAPER;
    for (int d = 0; d < 3; ++d) {
      k.fA[d] = (float)a.tt.fA[d];
      k.fs[d] = (float)(a.tt.fs[d] - floor(a.tt.fs[d]));
    }
    k_rhs32<<<(int)c->rhs_blocks, kThreads, 0, c->stream>>>(a, k);
  } else {
    k_rhs<<<(int)c->rhs_blocks, kThreads, 0, c->stream>>>(a);
  }
  prof_end(c, KC_RHS);
  c->launches++;
  return cudaGetLastError();
}

bool cg_cluster_fits(int64_t m, cudaStream_t stream) {
  return m <= kClusterNodes && ClusterLaunch(kClusterBlocks, cluster_threads(m), stream).fits((const void*)k_cg_cluster);
}
int cg_blocks(int64_t m, int sms) { return cg_shape(m, sms).grid; }
// bytes of the exchange inboxes a context of this grid holds
size_t cg_slot_bytes(int grid) { return exchange_slots((size_t)grid) * sizeof(GridSlot); }

cudaError_t launch_cg_on(pic_ctx* c, const double* b, double* x, const double* rhs_part, int rhs_blocks, double* E0,
                         double* E1, double* E2) {
  CgArgs a;
  a.n = c->P.n;
  a.ncell = c->P.ncell;
  a.inv_h2 = (double)c->P.n * (double)c->P.n;
  a.two_h = 2.0 * c->P.h;
  a.b = b;
  a.x = x;
  a.r = c->cg_r;
  a.p0 = c->cg_p[0];
  a.p1 = c->cg_p[1];
  a.q = c->cg_q;
  a.rhs_part = rhs_part;
  a.rhs_blocks = rhs_blocks;
  a.slots = reinterpret_cast<GridSlot*>(c->cg_red);
  a.launch = ++c->cg_launch;
  a.info = c->cg_info;
  a.flags = c->flags;
  a.res = c->cg_res;
  a.tol = c->cfg.cg_tol;
  a.maxit = c->cfg.cg_maxit;
  a.E0 = E0;
  a.E1 = E1;
  a.E2 = E2;
  a.skip_block = c->stall_next_cg ? c->cg_grid - 1 : -1;
  a.hist = c->hist_row;
  c->stall_next_cg = false;
  prof_begin(c);
  cudaError_t e = launch_solve(a, c->cg_cluster, c->num_sms, c->stream);
  prof_end(c, KC_CG);
  c->launches++;
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t launch_cg(pic_ctx* c) {
  return launch_cg_on(c, c->b, c->phi, c->rhs_part, (int)c->rhs_blocks, c->E[0], c->E[1], c->E[2]);
}

cudaError_t launch_store_field(pic_ctx* c, double* rho, double* phi, double* E) {
  StoreFieldArgs a;
  a.ncell = c->P.ncell;
  a.rho = c->rho;
  a.phi = c->phi;
  a.E0 = c->E[0];
  a.E1 = c->E[1];
  a.E2 = c->E[2];
  a.orho = rho;
  a.ophi = phi;
  a.oE = E;
  prof_begin(c);
  k_store_field<<<blocks_for(a.ncell), kThreads, 0, c->stream>>>(a);
  prof_end(c, KC_OTHER);
  c->launches++;
  return cudaGetLastError();
}

}  // namespace pic

// ---------------------------------------------------------------------------
// Allocation-free Poisson solve (pic_poisson_solve_noalloc).
//
// Some callers cannot allocate device memory at solve time: code running
// under a memory budget fixed at start-up, or a host framework that forbids
// cudaMalloc/cudaFree on its hot path because they synchronise the device.
// For them the CG scratch lives in this one fixed array in the library's own
// device memory: every GPU that loads the library holds it until the process
// exits. Host code must not use the array's name as a device address; it
// looks the address up once per device with cudaGetSymbolAddress.
// ---------------------------------------------------------------------------
#include <mutex>

namespace pic {
namespace {

constexpr int64_t kNoallocMaxNodes = 48 * 48 * 48;   // largest mesh: 48^3 nodes
// layout in doubles: r, p0, p1, q [4 N]; the exchange slots (two doubles
// each); 16 words of status / residual
constexpr int64_t kNoallocSlots = exchange_slots(kMaxExchangeBlocks);
constexpr int64_t kNoallocDoubles = 4 * kNoallocMaxNodes + 2 * kNoallocSlots + 16;

static __device__ __align__(256) double g_noalloc_scratch[kNoallocDoubles];

std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[64] = {nullptr};
unsigned g_noalloc_launch[64] = {0};

}  // namespace
}  // namespace pic

extern "C" pic_status pic_poisson_solve_noalloc(int32_t n, const double* b, double* phi, double* E, double tol,
                                                int32_t maxit, void* cuda_stream, int32_t* iters, double* rel_res) {
  using namespace pic;
  if (n < 2 || b == nullptr || phi == nullptr || E == nullptr || !(tol > 0.0) || maxit < 1) return PIC_EINVAL;
  const int64_t m = (int64_t)n * n * n;
  if (m > kNoallocMaxNodes) return PIC_EINVAL;  // beyond the fixed scratch: n <= 48
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return PIC_ECUDA;
  }
  // b, phi and E must be device memory of the current device
  const void* ptrs[3] = {b, phi, E};
  for (const void* p : ptrs) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
      cudaGetLastError();
      return PIC_EINVAL;
    }
    if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) return PIC_EINVAL;
    // device memory of another GPU would be read across the link, or fault
    // without peer access: only the current device's memory is accepted
    if (at.type == cudaMemoryTypeDevice && at.device != dev) return PIC_EINVAL;
  }
  // one-time set-up per device: the scratch array's device address
  double* base = nullptr;
  unsigned launch = 0;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) {
        cudaGetLastError();
        return PIC_ECUDA;
      }
      g_noalloc_ptr[dev] = (double*)p;
    }
    base = g_noalloc_ptr[dev];
    launch = ++g_noalloc_launch[dev];
  }
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return PIC_ECUDA;
  }

  double* slots = base + 4 * kNoallocMaxNodes;
  int* words = (int*)(slots + 2 * kNoallocSlots);   // [0..2] info, [4,5] flags
  double* res = (double*)(words + 8);

  CgArgs a;
  a.n = n;
  a.ncell = m;
  a.inv_h2 = (double)n * (double)n;
  a.two_h = 2.0 * (1.0 / (double)n);
  a.b = b;
  a.x = phi;
  a.r = base;
  a.p0 = base + kNoallocMaxNodes;
  a.p1 = base + 2 * kNoallocMaxNodes;
  a.q = base + 3 * kNoallocMaxNodes;
  a.rhs_part = nullptr;
  a.rhs_blocks = 0;
  a.slots = reinterpret_cast<GridSlot*>(slots);
  a.launch = launch;
  a.info = words;
  a.flags = words + 4;
  a.res = res;
  a.tol = tol;
  a.maxit = maxit;
  a.E0 = E;
  a.E1 = E + m;
  a.E2 = E + 2 * m;
  // the array keeps the last call's contents: clear the status words
  cudaError_t e = cudaMemsetAsync(words, 0, 8 * sizeof(int), stream);
  if (e == cudaSuccess) e = launch_solve(a, cg_cluster_fits(m, stream), sms, stream);
  int info[3] = {0, 0, 0};
  double r = 0.0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(info, words, sizeof(info), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&r, res, sizeof(double), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return PIC_ECUDA;
  }
  if (iters) *iters = info[0];
  if (rel_res) *rel_res = r;
  if (info[2]) return PIC_ETIMEOUT;
  if (info[1]) return PIC_ENOCONV;
  return PIC_OK;
}
