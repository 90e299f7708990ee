// The two solves of a small flow's step.
//
// Direct pressure solve of small systems (Section 3, Eq. pressure_Poisson; the
// paper factorises its implicit matrices once, too): the dense inverse of the
// scaled operator A_f = A + es 1^T is built once per plan, and a solve is a
// product with it inside iterative refinement on the sparse operator, in one
// cooperative launch.
//
// Resident viscous solve: both components' BiCGSTAB in one cooperative launch.
#include <algorithm>
#include <cmath>

#include "gridsync.cuh"
#include "psolve.cuh"

namespace rbffd {

namespace {

constexpr int kPT = 1024;      // threads per block, one block per SM
constexpr int kPW = kPT / 32;  // warps per block
constexpr int kMaxSweeps = 8;
constexpr int kOwn = 32;  // rows a block of the inversion owns, at most

// T = A + es 1^T, one block per row
__global__ void __launch_bounds__(256)
    k_dense_fill(int n, int64_t ld, int k, const int32_t* __restrict__ idx,
                 const double* __restrict__ w, const double* __restrict__ es,
                 double* __restrict__ T, int ldt) {
  const int i = blockIdx.x;
  for (int j = threadIdx.x; j < n; j += blockDim.x) T[(int64_t)i * ldt + j] = es[i];
  __syncthreads();
  if (threadIdx.x == 0)  // a padded row may repeat a column
    for (int s = 0; s < k; ++s) T[(int64_t)i * ldt + idx[s * ld + i]] += w[s * ld + i];
}

struct InvArgs {
  int n, ldt;
  double* T;
  int* prow;             // [n] pivot row of step k
  double* cand_v;        // [2][gridDim.x] each block's best pivot candidate
  int* cand_r;           // [2][gridDim.x]
  double* partials;
  unsigned int* arrivals;  // [kBarrierWords], zero at launch
  long long polls;
  int* status;             // 0 on entry; 1: singular, 2: non-finite
};

// Gauss-Jordan exchange with partial pivoting, in place: step k exchanges
// row p (the largest |T[i][k]| among the rows not yet used) with column k.
// Block b owns rows b, b + gridDim.x, ...; rows are never moved.  One barrier
// per step: every block reads row p as step k - 1 left it, and its owner
// rescales it while it applies step k + 1.
//
// What bounds it: n^2 FP64 FMAs and one pass over the matrix (in L2 up to about
// n = 3,500) per step, 4.1 us for the FMAs at n = 1,600, and the barrier and the
// pivot search.  A blocked form would save memory traffic, not FP64
// instructions.
__global__ void __launch_bounds__(kPT, 1) k_dense_invert(const __grid_constant__ InvArgs a) {
  __shared__ double sh[kNVMax * kPT];
  __shared__ double part[kNVMax * 4];
  __shared__ double f[kOwn], cv[kOwn], s_inv;
  __shared__ int used[kOwn], okf, s_p, s_bad;
  Grid<kPT> g{sh, part, &okf, a.partials, a.arrivals, a.polls};
  const int tid = threadIdx.x, n = a.n, nb = gridDim.x, blk = blockIdx.x;
  const int own = blk < n ? (n - blk + nb - 1) / nb : 0;
  if (tid < kOwn) {
    used[tid] = 0;
    cv[tid] = tid < own ? fabs(a.T[(int64_t)(blk + tid * nb) * a.ldt]) : -1.0;
  }
  if (tid == 0) s_bad = 0;
  int pend = -1, kprev = 0;  // own row still to be rescaled by the last step's pivot
  double inv_prev = 0.0;
  for (int k = 0; k < n; ++k) {
    __syncthreads();
    if (tid < 32) {  // this block's candidate: largest magnitude, lowest row on ties
      double v = tid < own && !used[tid] ? cv[tid] : -1.0;
      if (!(v == v)) v = INFINITY;  // NaN: picked, then caught below
      int r = blk + tid * nb;
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int orr = __shfl_xor_sync(0xffffffffu, r, o);
        if (ov > v || (ov == v && orr < r)) {
          v = ov;
          r = orr;
        }
      }
      if (tid == 0) {
        a.cand_v[(k & 1) * nb + blk] = v;
        a.cand_r[(k & 1) * nb + blk] = r;
      }
    }
    if (!g.sync()) return;
    if (tid < 32) {
      double v = -2.0;
      int r = n;
      for (int b = tid; b < nb; b += 32) {
        const double ov = a.cand_v[(k & 1) * nb + b];
        const int orr = a.cand_r[(k & 1) * nb + b];
        if (ov > v || (ov == v && orr < r)) {
          v = ov;
          r = orr;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int orr = __shfl_xor_sync(0xffffffffu, r, o);
        if (ov > v || (ov == v && orr < r)) {
          v = ov;
          r = orr;
        }
      }
      if (tid == 0) {
        s_p = r;
        // rows are scaled to a unit diagonal: a pivot this small is rounding
        s_bad = !isfinite(v) ? 2 : (v > 1e-13 ? 0 : 1);
        if (!s_bad) s_inv = 1.0 / a.T[(int64_t)r * a.ldt + k];
      }
    }
    // the multipliers of the own rows in column k, before it is overwritten
    if (tid >= 32 && tid < 32 + own) {
      const int q = tid - 32;
      double v = a.T[(int64_t)(blk + q * nb) * a.ldt + k];
      if (q == pend) v = -v * inv_prev;  // k != kprev
      f[q] = v;
    }
    __syncthreads();
    if (s_bad) {
      if (blk == 0 && tid == 0) *a.status = s_bad;
      return;
    }
    const int p = s_p;
    const double inv = s_inv;
    const int qp = p % nb == blk ? p / nb : -1;
    const double* Tp = a.T + (int64_t)p * a.ldt;
    for (int j = tid; j < n; j += kPT) {
      const double t = j == k ? inv : -Tp[j] * inv;
      double* col = a.T + (int64_t)blk * a.ldt + j;
      const int64_t step = (int64_t)nb * a.ldt;
#pragma unroll 4
      for (int q = 0; q < own; ++q) {
        if (q == qp) continue;
        double old = j == k ? 0.0 : col[q * step];
        if (q == pend && j != k) old = j == kprev ? inv_prev : -old * inv_prev;
        const double v = fma(f[q], t, old);
        col[q * step] = v;
        if (j == k + 1) cv[q] = fabs(v);
      }
    }
    if (tid == 0) {
      if (qp >= 0) used[qp] = 1;
      if (blk == 0) a.prow[k] = p;
    }
    pend = qp;
    inv_prev = inv;
    kprev = k;
  }
  if (!g.sync()) return;  // the other blocks still read the last pivot row in their last step
  if (pend >= 0) {
    double* row = a.T + (int64_t)(blk + pend * nb) * a.ldt;
    for (int j = tid; j < n; j += kPT) row[j] = j == kprev ? inv_prev : -row[j] * inv_prev;
  }
}

// out[k][prow[j]] = T[prow[k]][j], rows padded with zeros to ldt
__global__ void __launch_bounds__(256)
    k_dense_order(int n, int ldt, const int* __restrict__ prow, const double* __restrict__ T,
                  double* __restrict__ out) {
  const int k = blockIdx.x;
  const double* row = T + (int64_t)prow[k] * ldt;
  for (int j = threadIdx.x; j < n; j += blockDim.x) out[(int64_t)k * ldt + prow[j]] = row[j];
}

struct DArgs {
  int M, rows, k, ldt;
  int64_t ld;
  const int32_t* idx;
  const double *w, *es, *inv;
  const double* b;
  double *x, *r;  // r: ldt values, zero beyond M
  double tol2;
  double* partials;
  unsigned int* arrivals;  // [kBarrierWords], zero between launches
  long long polls;
  PSolveResult* res;
  int* fail;  // null, or see psolve.cuh
  int step;
};

// what ended the step: the code of a wait outranks the others
template <typename A>
__device__ __forceinline__ void set_fail(const A& a, int code) {
  atomicMax(a.fail, (a.step << 4) | code);
}
// a barrier that ran out of its bounded wait
template <typename A>
__device__ __forceinline__ void give_up(const A& a) {
  if (a.fail && threadIdx.x == 0) set_fail(a, kFailWait);
}

// Refinement: r = b - A_f x, x += A_f^-1 r until (r, r) <= tol^2 (b, b).  A
// block owns `rows` consecutive rows, in the residual (one thread per row) and
// in the product (one warp per row, r in shared memory).  What bounds it: the
// product's M^2 FP64 FMAs (4.1 us at 1,600 rows on the FP64 pipe) and the
// latency of its four phases.
template <int K>
__global__ void __launch_bounds__(kPT, 1) k_dsolve(const __grid_constant__ DArgs a) {
  if (a.fail && *a.fail) return;
  __shared__ __align__(16) double sh[kNVMax * kPT];
  static_assert(kNVMax * kPT >= kDenseMax, "the residual is staged in sh");
  __shared__ double part[kNVMax * 4];
  __shared__ double s_sig, s_rr, s_bb;
  __shared__ int okf;
  Grid<kPT> g{sh, part, &okf, a.partials, a.arrivals, a.polls};
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = min(a.M, a.rows * (int)blockIdx.x), r1 = min(a.M, r0 + a.rows);
  const int active = min(kPT, (a.rows + 31) / 32 * 32);
  {
    double sx = 0.0;
    for (int i = r0 + tid; i < r1; i += kPT) sx += a.x[i];
    const double v[1] = {sx};
    if (!g.reduce<1>(v, active, [&](const double* t) { s_sig = t[0]; })) return give_up(a);
  }
  double prev = INFINITY;
  for (int sweep = 0;; ++sweep) {
    double d0 = 0.0, d1 = 0.0;
    const double sig = s_sig;
    for (int i = r0 + tid; i < r1; i += kPT) {
      double ax = 0.0;
      if constexpr (K > 0) {
#pragma unroll
        for (int s = 0; s < K; ++s)
          ax += __ldg(a.w + s * a.ld + i) * a.x[__ldg(a.idx + s * a.ld + i)];
      } else {
#pragma unroll 4
        for (int s = 0; s < a.k; ++s)
          ax += __ldg(a.w + s * a.ld + i) * a.x[__ldg(a.idx + s * a.ld + i)];
      }
      const double bi = a.b[i], ri = bi - (ax + __ldg(a.es + i) * sig);
      a.r[i] = ri;
      d0 += ri * ri;
      d1 += bi * bi;
    }
    const double v[2] = {d0, d1};
    const bool ok = g.reduce<2>(v, active, [&](const double* t) {
      s_rr = t[0];
      s_bb = t[1];
    });
    if (!ok) return give_up(a);
    const double rr = s_rr, bb = s_bb;
    const bool conv = rr <= a.tol2 * bb, fin = isfinite(rr);
    // a sweep that does not halve the residual has reached the rounding level
    const bool stalled = sweep > 0 && !(rr < 0.25 * prev);
    if (conv || !fin || stalled || sweep >= kMaxSweeps) {
      if (blockIdx.x == 0 && tid == 0) {
        a.res->iters = sweep;
        a.res->status = conv ? 0 : (fin ? 5 : 2);
        a.res->relres = bb > 0 ? sqrt(rr / bb) : sqrt(rr);
        a.res->converged = conv;
        if (a.fail && !conv) set_fail(a, kFailPressure);
      }
      return leave(a.arrivals);
    }
    prev = rr;
    // x += inv r: the rows' products need all of r, read once per block
    for (int j = tid; j < a.ldt; j += kPT) sh[j] = a.r[j];
    __syncthreads();
    double sx = 0.0;
    for (int i = r0 + warp; i < r1; i += kPW) {
      const double2* row = reinterpret_cast<const double2*>(a.inv + (int64_t)i * a.ldt);
      const double2* r2 = reinterpret_cast<const double2*>(sh);
      double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
      for (int j = lane; j < a.ldt / 2; j += 32) {
        const double2 u = __ldg(row + j), q = r2[j];
        s0 = fma(u.x, q.x, s0);
        s1 = fma(u.y, q.y, s1);
      }
      const double s = warp_sum(s0 + s1);
      if (lane == 0) {
        const double xi = a.x[i] + s;
        a.x[i] = xi;
        sx += xi;
      }
    }
    __syncthreads();  // sh is reused by the reduction
    const double vx[1] = {sx};
    if (!g.reduce<1>(vx, kPT, [&](const double* t) { s_sig = t[0]; })) return give_up(a);
  }
}

// ---------------------------------------------------------- viscous solves
constexpr int kVT = 512;  // threads per block
constexpr int kVL = 4;    // threads per row
// Rows of a block, where there are SMs for so few: fewer blocks make the
// barrier lighter, fewer rows the phases (8, 16, 32, 64 rows: 20 steps of 1,600
// nodes 5.67, 5.69, 5.63, 5.57 ms, four of the 2,700-node wake 1.47, 1.45, 1.44,
// 1.49; 5.13 and 1.37 since the sums of a warp meet before those of a block).
constexpr int kVRows = 32;
constexpr int kVNV = 6;

struct VArgs {
  int N, rows, k;
  int64_t ld;
  const int32_t* idx;
  const double* w[2];
  double* x[2];
  const double* b[2];
  double *p, *s;  // [N][2], both components side by side
  double tol2, accept2;
  int maxit;
  double* partials;        // [2][kVNV][gridDim.x]
  unsigned int* arrivals;  // [kBarrierWords], zero between launches
  long long polls;
  PSolveResult* res;
  int* fail;
  int step;
};

struct VScal {
  double rho[2], rr[2], ss[2], bb[2], rhs[2], alpha[2], omega[2], beta[2];
  int active[2], mode[2], status, iters, total, go, iterate;
  int its[2];  // iterations of each component, over all restarts
};

// What bounds it: latency, four phases an iteration (a barrier of 1.3 us, the
// reduction behind it, one gather from L2): 141 us with cold caches for the 6.5
// iterations of a solve at 1,600 rows, 227 us with the vectors and weights in
// memory and one thread per row.  As separate launches an iteration took five
// kernels and the solve two or three waits of the host.
//
// Layout: kVL threads per row, each with its share of the row's slots in
// registers for the whole solve (K > 0), two of them with one component's
// vectors; only p and s, which other rows gather, are in memory, the two
// components side by side so that a gather is one 16-byte load.
//
// Fewer reductions than the textbook form: (rh, r) = (rh, s) - omega (rh, t),
// so x, r and p are one pass; (r, r) = (s, s) - omega (t, s), raised by 1e-14
// (s, s), more than the rounding of the difference, so that it never claims a
// convergence that the vectors do not have.  A component that has converged
// keeps its x while the other one goes on.
template <int K>
__global__ void __launch_bounds__(kVT, 1) k_vsolve(const __grid_constant__ VArgs a) {
  if (*a.fail) return;
  constexpr int NS = K > 0 ? (K + kVL - 1) / kVL : 1;
  __shared__ double wsum[kVNV * (kVT / 32)];
  __shared__ VScal S;
  __shared__ int okf;
  Grid<kVT, kVNV> g{nullptr, nullptr, &okf, a.partials, a.arrivals, a.polls};
  const int tid = threadIdx.x, sub = tid & (kVL - 1), c = sub & 1;
  const int i = a.rows * (int)blockIdx.x + tid / kVL;
  const bool mine = tid / kVL < a.rows && i < a.N;
  const bool own = mine && sub < 2;
  const int active = min(kVT, (a.rows * kVL + 31) / 32 * 32);  // whole warps
  const bool same = a.w[0] == a.w[1];
  int jj[NS] = {};
  double w0[NS] = {}, w1[NS] = {};
  if constexpr (K > 0) {
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      const int s = sub + kVL * t;
      if (!mine || s >= K) continue;
      jj[t] = a.idx[s * a.ld + i];
      w0[t] = a.w[0][s * a.ld + i];
      w1[t] = same ? w0[t] : a.w[1][s * a.ld + i];
    }
  }
  // this thread's component of the row's off-diagonal sum; at(j) gives both
  // components' entries of column j
  auto row = [&](auto at) {
    double s0 = 0.0, s1 = 0.0;
    if constexpr (K > 0) {
#pragma unroll
      for (int t = 0; t < NS; ++t) {
        const double2 q = at(jj[t]);
        s0 = fma(w0[t], q.x, s0);
        s1 = fma(w1[t], q.y, s1);
      }
    } else if (mine) {
      for (int s = sub; s < a.k; s += kVL) {
        const double2 q = at(__ldg(a.idx + s * a.ld + i));
        s0 = fma(__ldg(a.w[0] + s * a.ld + i), q.x, s0);
        s1 = fma(__ldg(a.w[1] + s * a.ld + i), q.y, s1);
      }
    }
    double y = c ? s1 : s0;
    y += __shfl_xor_sync(0xffffffffu, c ? s0 : s1, 1);
    return y + __shfl_xor_sync(0xffffffffu, y, 2);
  };
  // Grid-wide sums of n values of each component, handed to fin as
  // [component][value]; only threads that own a component of a row hold values.
  // In the warp they meet over the rows alone: three FP64 adds per value, where
  // adding two components' values over all lanes would take ten.
  auto sum = [&](auto& d, auto fin) -> bool {
    constexpr int n = sizeof(d) / sizeof(double);
    if (tid < active) {
#pragma unroll
      for (int o = kVL; o < 32; o *= 2) {
#pragma unroll
        for (int j = 0; j < n; ++j) d[j] += __shfl_xor_sync(0xffffffffu, d[j], o);
      }
      if ((tid & 31) < 2) {
#pragma unroll
        for (int j = 0; j < n; ++j) wsum[(c * n + j) * (kVT / 32) + tid / 32] = d[j];
      }
    }
    __syncthreads();
    double t = 0.0;
    if (tid < 2 * n)
      for (int w = 0; w < active / 32; ++w) t += wsum[tid * (kVT / 32) + w];
    return g.template spread<2 * n>(t, fin);
  };
  const double2* P = reinterpret_cast<const double2*>(a.p);
  const double2* Sv = reinterpret_cast<const double2*>(a.s);
  const double b = mine ? a.b[c][i] : 0.0, x0 = mine ? a.x[c][i] : 0.0;
  double x = x0, r = 0.0, rh = 0.0, p = 0.0, v = 0.0, s = 0.0, t = 0.0;
  if (tid == 0) S.total = S.its[0] = S.its[1] = 0;
  for (int cyc = 0;; ++cyc) {
    {
      const uint32_t seed = cyc ? 0x51ED27u + (uint32_t)cyc : 0u;
      double d[3] = {};
      if (tid < active) {
        r = b - (x + row([&](int j) { return make_double2(a.x[0][j], a.x[1][j]); }));
        rh = seed ? (double)shadow_sign(i, seed) * r : r;
        p = r;
        if (own) {
          a.p[2 * i + c] = p;
          d[0] = r * r;
          d[1] = b * b;
          d[2] = rh * r;
        }
      }
      const bool ok = sum(d, [&](const double* q6) {
        S.status = 0;
        S.iters = 0;
        S.go = 0;
        for (int q = 0; q < 2; ++q) {
          S.rr[q] = q6[3 * q];
          S.bb[q] = q6[3 * q + 1];
          S.rho[q] = q6[3 * q + 2];
          if (!isfinite(S.rr[q])) S.status = 2;
          S.active[q] = isfinite(S.rr[q]) && S.rr[q] > a.tol2 * S.bb[q] && S.rho[q] != 0.0;
          S.go |= S.active[q];
        }
        if (a.maxit - S.total <= 0) S.go = 0;
      });
      if (!ok) return give_up(a);
    }
    bool run = S.go != 0;
    while (run) {
      {  // v = H p; (rh, v)
        double d[1] = {};
        if (tid < active) {
          v = p + row([&](int j) { return P[j]; });
          if (own) d[0] = rh * v;
        }
        const bool ok = sum(d, [&](const double* q2) {
          S.go = 0;
          for (int q = 0; q < 2; ++q) {
            S.mode[q] = 0;
            if (!S.active[q]) continue;
            if (q2[q] == 0.0 || !isfinite(q2[q])) {
              S.active[q] = 0;
              S.status = isfinite(q2[q]) ? 1 : 2;
            } else {
              S.alpha[q] = S.rho[q] / q2[q];
              S.go = 1;
            }
          }
        });
        if (!ok) return give_up(a);
        if (!S.go) break;
      }
      const double al = S.alpha[c];
      {  // s = r - alpha v; (s, s), (rh, s)
        double d[2] = {};
        if (own && S.active[c]) {
          s = r - al * v;
          a.s[2 * i + c] = s;
          d[0] = s * s;
          d[1] = rh * s;
        }
        const bool ok = sum(d, [&](const double* q4) {
          S.iterate = 0;
          for (int q = 0; q < 2; ++q) {
            if (!S.active[q]) continue;
            S.ss[q] = q4[2 * q];
            S.rhs[q] = q4[2 * q + 1];
            if (S.ss[q] <= a.tol2 * S.bb[q]) {
              S.rr[q] = S.ss[q];
              S.its[q] += 1;
              S.mode[q] = 1;
              S.active[q] = 0;
            } else {
              S.mode[q] = 2;
              S.iterate = 1;
            }
          }
          if (!S.iterate) {
            S.iters += 1;
            S.go = 0;
          }
        });
        if (!ok) return give_up(a);
      }
      if (S.iterate) {  // t = H s; (t, s), (t, t), (rh, t)
        double d[3] = {};
        if (tid < active) {
          t = s + row([&](int j) { return Sv[j]; });
          if (own) {
            d[0] = t * s;
            d[1] = t * t;
            d[2] = rh * t;
          }
        }
        const bool ok = sum(d, [&](const double* q6) {
          S.iters += 1;
          int any = 0;
          for (int q = 0; q < 2; ++q) {
            if (S.mode[q] != 2) continue;
            S.its[q] += 1;
            const double ts = q6[3 * q], tt = q6[3 * q + 1];
            S.active[q] = 0;
            if (!(tt > 0.0) || !isfinite(ts)) {
              S.mode[q] = 0;
              S.status = isfinite(tt) ? 3 : 2;
              continue;
            }
            const double om = ts / tt, rn = S.rhs[q] - om * q6[3 * q + 2];
            const double rr = fmax(S.ss[q] - om * ts, 0.0) + 1e-14 * S.ss[q];
            S.beta[q] = (rn / S.rho[q]) * (S.alpha[q] / om);
            S.omega[q] = om;
            S.rho[q] = rn;
            S.rr[q] = rr;
            if (!isfinite(S.ss[q]) || !isfinite(om))
              S.status = 2;
            else if (rr > 1e8 * S.bb[q] && S.bb[q] > 0.0)
              S.status = 5;
            else if (rr <= a.tol2 * S.bb[q])
              ;
            else if (rn == 0.0 || om == 0.0)
              S.status = 4;
            else
              any = S.active[q] = 1;
          }
          S.go = any && S.total + S.iters < a.maxit;
        });
        if (!ok) return give_up(a);
      }
      // x, r, p
      const int mode = S.mode[c];
      run = S.go != 0;
      if (mode == 1) {
        x += al * p;
      } else if (mode == 2) {
        const double om = S.omega[c];
        x += al * p + om * s;
        r = s - om * t;
        p = r + S.beta[c] * (p - om * v);
        if (own) a.p[2 * i + c] = p;
      }
      if (run && !g.sync()) return give_up(a);
    }
    bool conv = true, near = true;
    for (int q = 0; q < 2; ++q) {
      conv = conv && S.rr[q] <= a.tol2 * S.bb[q];
      near = near && S.rr[q] <= a.accept2 * S.bb[q];
    }
    const int st = S.status, tot = S.total + S.iters;
    const bool again = st == 1 || st == 3 || st == 4 || st == 5;
    const bool end = conv || !again || tot >= a.maxit || cyc >= 400;
    if (!end && st == 5) x = x0;  // the recurrence has blown up: from the initial iterate
    if (own) a.x[c][i] = x;
    if (end) {
      if (blockIdx.x == 0 && tid == 0) {
        double worst = 0.0;
        for (int q = 0; q < 2; ++q)
          worst = fmax(worst, S.bb[q] > 0 ? sqrt(S.rr[q] / S.bb[q]) : sqrt(S.rr[q]));
        // an open flow's components are systems of their own, whose iterations
        // add up; a closed flow's are two right sides of one
        a.res->iters = same ? tot : S.its[0] + S.its[1];
        a.res->status = st;
        a.res->relres = worst;
        a.res->converged = conv;
        if (st == 2 || (!conv && !near)) set_fail(a, kFailViscous);
      }
      return leave(a.arrivals);
    }
    // the restart's residual reads x of other blocks
    if (!g.sync()) return give_up(a);
    if (tid == 0) S.total = tot;
  }
}

}  // namespace

long long barrier_polls(const rbffd_ctx* ctx) {
  return ctx->barrier_limit < 0 ? kPolls : std::min<long long>(ctx->barrier_limit, kPolls);
}

struct VSolve {
  std::vector<void*> allocs;
  int grid = 0;
  VArgs a{};
};

void vsolve_free(VSolve* v) {
  if (!v) return;
  for (void* q : v->allocs) cudaFree(q);
  delete v;
}

static const void* vsolve_kernel(int k) {
  return k == 28 ? (const void*)k_vsolve<28> : (const void*)k_vsolve<0>;
}

int vsolve_build(rbffd_ctx* ctx, int64_t N, int64_t ld, int k, const int32_t* idx,
                 const double* wu, const double* wv, VSolve** out, cudaStream_t st) {
  *out = nullptr;
  // a block's threads hold its rows' vectors
  if (N > (int64_t)sm_count() * (kVT / kVL)) return RBFFD_OK;
  VSolve* v = new VSolve();
  VArgs& a = v->a;
  a.N = (int)N;
  a.rows = (int)std::max<int64_t>(kVRows, (N + sm_count() - 1) / sm_count());
  v->grid = (int)((N + a.rows - 1) / a.rows);
  a.k = k;
  a.ld = ld;
  a.idx = idx;
  a.w[0] = wu;
  a.w[1] = wv;
  auto get = [&](void** p, size_t bytes) {
    int rc = check_cuda(ctx, solver_malloc(ctx, p, bytes), "viscous solve alloc");
    if (rc) return rc;
    v->allocs.push_back(*p);
    return check_cuda(ctx, cudaMemsetAsync(*p, 0, bytes, st), "memset");
  };
  int rc = get((void**)&a.p, sizeof(double) * 2 * N);
  if (!rc) rc = get((void**)&a.s, sizeof(double) * 2 * N);
  if (!rc) rc = get((void**)&a.partials, sizeof(double) * 2 * kVNV * v->grid);
  if (!rc) rc = get((void**)&a.arrivals, kBarrierWords * sizeof(unsigned int));
  if (rc || !coop_fits(vsolve_kernel(k), v->grid, kVT, 0)) {
    cudaStreamSynchronize(st);
    vsolve_free(v);
    return solver_left_out(ctx, rc);
  }
  *out = v;
  return RBFFD_OK;
}

cudaError_t vsolve_enqueue(VSolve* v, double* const* x, const double* const* b, double tol,
                           double accept, int maxit, PSolveResult* res, int* fail, int step,
                           long long polls, cudaStream_t st) {
  VArgs a = v->a;
  a.polls = polls;
  for (int q = 0; q < 2; ++q) {
    a.x[q] = x[q];
    a.b[q] = b[q];
  }
  a.tol2 = tol * tol;
  a.accept2 = accept * accept;
  a.maxit = maxit;
  a.res = res;
  a.fail = fail;
  a.step = step;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(vsolve_kernel(a.k), dim3(v->grid), dim3(kVT), args, 0, st);
}

struct DSolve {
  std::vector<void*> allocs;
  int grid = 0;
  DArgs a{};
};

void dsolve_free(DSolve* d) {
  if (!d) return;
  for (void* q : d->allocs) cudaFree(q);
  delete d;
}

namespace {

template <typename T>
int d_alloc(rbffd_ctx* ctx, DSolve* d, T** out, size_t count, cudaStream_t st) {
  void* ptr = nullptr;
  const int rc =
      check_cuda(ctx, solver_malloc(ctx, &ptr, sizeof(T) * count), "direct solve alloc");
  if (rc) return rc;
  d->allocs.push_back(ptr);
  *out = (T*)ptr;
  return check_cuda(ctx, cudaMemsetAsync(ptr, 0, sizeof(T) * count, st), "memset");
}

const void* dsolve_kernel(int k) {
  return k == 28 ? (const void*)k_dsolve<28> : (const void*)k_dsolve<0>;
}

int invert(rbffd_ctx* ctx, DSolve* d, const InvArgs& in, const double* es, double* out, int* h_status,
           cudaStream_t st) {
  DArgs& a = d->a;
  k_dense_fill<<<a.M, 256, 0, st>>>(a.M, a.ld, a.k, a.idx, a.w, es, in.T, a.ldt);
  int rc = check_cuda(ctx, cudaGetLastError(), "dense operator");
  if (rc) return rc;
  InvArgs arg = in;
  void* args[] = {&arg};
  rc = check_cuda(ctx, cudaLaunchCooperativeKernel((const void*)k_dense_invert, dim3(d->grid),
                                                   dim3(kPT), args, 0, st), "dense inverse");
  if (rc) return rc;
  int* h = (int*)ctx->host_pinned;
  unsigned int* gave_up = (unsigned int*)(h + 1);
  rc = check_cuda(ctx, cudaMemcpyAsync(h, in.status, sizeof(int), cudaMemcpyDeviceToHost, st),
                  "inverse status");
  if (!rc)
    rc = check_cuda(ctx, cudaMemcpyAsync(gave_up, in.arrivals + 2, sizeof(unsigned int),
                                         cudaMemcpyDeviceToHost, st), "inverse status");
  if (!rc) rc = check_cuda(ctx, cudaStreamSynchronize(st), "dense inverse sync");
  if (rc) return rc;
  *h_status = *h;
  if (*gave_up)
    return set_error(ctx, RBFFD_ERR_CUDA, "dense inverse: grid barrier not reached (bounded wait)");
  if (*h == 0) {
    k_dense_order<<<a.M, 256, 0, st>>>(a.M, a.ldt, in.prow, in.T, out);
    rc = check_cuda(ctx, cudaGetLastError(), "dense inverse order");
  }
  return rc;
}

}  // namespace

int dsolve_build(rbffd_ctx* ctx, int64_t M, int64_t ld, int k, const int32_t* idx,
                 const double* w, const double* es, DSolve** out, cudaStream_t st) {
  *out = nullptr;
  DSolve* d = new DSolve();
  d->grid = sm_count();
  DArgs& a = d->a;
  a.M = (int)M;
  a.rows = (int)((M + d->grid - 1) / d->grid);
  a.k = k;
  a.ld = ld;
  a.ldt = (int)round_up(M, 2);
  a.idx = idx;
  a.w = w;
  a.es = es;
  InvArgs in{};
  in.n = a.M;
  in.ldt = a.ldt;
  const size_t nn = (size_t)M * a.ldt;
  double* inv = nullptr;
  int rc = 0, bad = 0;
  // fewer SMs than the ownership tables assume, or than the grids need
  if (a.rows > kOwn || !coop_fits((const void*)k_dense_invert, d->grid, kPT, 0) ||
      !coop_fits(dsolve_kernel(k), d->grid, kPT, 0))
    bad = 1;
  if (!bad) rc = d_alloc(ctx, d, &inv, nn, st);
  if (!rc && !bad) rc = d_alloc(ctx, d, &in.T, nn, st);
  void* work = in.T;
  if (!rc && !bad) rc = d_alloc(ctx, d, &in.prow, (size_t)M, st);
  if (!rc && !bad) rc = d_alloc(ctx, d, &in.cand_v, (size_t)2 * d->grid, st);
  if (!rc && !bad) rc = d_alloc(ctx, d, &in.cand_r, (size_t)2 * d->grid, st);
  if (!rc && !bad) rc = d_alloc(ctx, d, &in.status, 1, st);
  if (!rc && !bad) rc = d_alloc(ctx, d, &a.partials, (size_t)2 * kNVMax * d->grid, st);
  SolveStatus* status = nullptr;
  if (!rc && !bad) rc = d_alloc(ctx, d, &status, 1, st);
  if (!rc && !bad) rc = d_alloc(ctx, d, &a.r, (size_t)a.ldt, st);
  if (status) {
    a.res = &status->res;
    a.arrivals = status->bar;
  }
  in.partials = a.partials;
  in.arrivals = a.arrivals;
  in.polls = barrier_polls(ctx);
  a.inv = inv;
  if (!rc && !bad) rc = invert(ctx, d, in, es, inv, &bad, st);
  if (!rc && !bad) rc = check_cuda(ctx, cudaStreamSynchronize(st), "dense inverse sync");
  if (rc || bad) {
    cudaStreamSynchronize(st);
    dsolve_free(d);
    // singular to working precision, or no room: the Krylov solve takes over
    return solver_left_out(ctx, rc);
  }
  for (void*& q : d->allocs)  // the inversion's matrix is not needed any more
    if (q == work) {
      cudaFree(q);
      q = nullptr;
    }
  *out = d;
  return RBFFD_OK;
}

cudaError_t dsolve_enqueue(DSolve* d, double* x, const double* b, double tol, PSolveResult* res,
                           int* fail, int step, long long polls, cudaStream_t st) {
  DArgs a = d->a;
  a.polls = polls;
  a.x = x;
  a.b = b;
  a.tol2 = tol * tol;
  a.res = res;
  a.fail = fail;
  a.step = step;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(dsolve_kernel(a.k), dim3(d->grid), dim3(kPT), args, 0, st);
}

cudaError_t small_reset(VSolve* v, DSolve* d, int* fail, cudaStream_t st) {
  constexpr size_t words = kBarrierWords * sizeof(unsigned int);
  cudaError_t e = cudaMemsetAsync(v->a.arrivals, 0, words, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(d->a.arrivals, 0, words, st);
  return e == cudaSuccess ? cudaMemsetAsync(fail, 0, sizeof(int), st) : e;
}

int dsolve_run(rbffd_ctx* ctx, DSolve* d, double* x, const double* b, double tol,
               PSolveResult* res, int64_t* launches, cudaStream_t st) {
  SolveStatus* h = (SolveStatus*)ctx->host_pinned;
  const DArgs& a = d->a;
  int rc = check_cuda(ctx, cudaMemsetAsync(a.arrivals, 0, kBarrierWords * sizeof(unsigned int), st),
                      "memset");
  if (!rc)
    rc = check_cuda(ctx, dsolve_enqueue(d, x, b, tol, a.res, nullptr, 0, barrier_polls(ctx), st),
                    "direct pressure solve");
  if (!rc)
    rc = check_cuda(ctx, cudaMemcpyAsync(h, a.res, sizeof(SolveStatus), cudaMemcpyDeviceToHost, st),
                    "direct solve result");
  if (!rc) rc = check_cuda(ctx, cudaStreamSynchronize(st), "direct solve sync");
  if (rc) return rc;
  *launches += 1;
  if (h->bar[2])
    return set_error(ctx, RBFFD_ERR_CUDA, "direct solve: grid barrier not reached (bounded wait)");
  *res = h->res;
  return RBFFD_OK;
}

}  // namespace rbffd
