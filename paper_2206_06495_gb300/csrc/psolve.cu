// The preconditioned pressure solve (Section 3, Eq. pressure_Poisson) as one
// resident kernel: BiCGSTAB, its V-cycles and its restarts run in a single
// cooperative launch of one block per SM, with a grid barrier between dependent
// phases.
//
// What bounds it: an iteration is a chain of about 2 (2 nlev + 1) dependent
// phases.  As launches of a replayed graph a phase costs 2.5 us at the least
// and 5 to 14 us on the coarse levels, whose reductions and dense product were
// spread over 1,216 blocks whatever their size; here it costs a barrier (about
// 1.3 us) and its own memory latency.  Large sets are bound by the operator's
// stream (336 B a row, twice per iteration) and the level-0 graph rows.
//
// Layout: everything is in the hierarchy's level-0 order, in which each
// aggregate's rows are consecutive, so that the V-cycle needs no permuting
// passes; x and b are permuted once on the way in and out.  A block owns a
// contiguous share of the rows for the whole solve.
//
// Fewer phases than the textbook form: (c . s) and (c . p), which the rank-one
// completion of the preconditioner needs before each V-cycle, follow from
// (c . v) and (c . t) of the products, and (rh, r) = (rh, s) - omega (rh, t),
// so that x, r and p and the next V-cycle's input are one pass.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "gridsync.cuh"
#include "psolve.cuh"

namespace rbffd {

namespace {

// Threads per block (one block per SM).  512 where the phases are bound by
// latency: with 1,024, 64 registers a thread spill, and the spilled addresses
// are reloaded through L2 in every phase (each barrier empties L1), 0.7 us a
// phase (FP64 100k rows: 94 against 104 us an iteration; MIXED 250k: 123 against
// 140).  1,024 where they are bound by the streams and need the loads in
// flight (FP64 1M rows: 0.38 against 0.46 ms).  The line: milliseconds of a step
// for each pressure iteration with 512 and with 1,024, FP64 0.161 and 0.182 at
// 200k rows, 0.195 and 0.189 at 250k, 0.228 and 0.203 at 300k; MIXED 0.142 and
// 0.161, 0.152 and 0.169, 0.189 and 0.176.
constexpr int kSmallPT = 512, kLargePT = 1024;
constexpr int64_t kLargeRows = 300000;
constexpr int kCycle = 50;            // iterations before a restart from the true residual
constexpr int kMaxCycles = 400;       // restarts of one solve before giving up
// shared memory for static rows: a block's 227 KB less what the reductions take
constexpr size_t stage_room(int pt) { return 226 * 1024 - sizeof(double) * kNVMax * pt; }

// One level of the hierarchy as the kernel reads it (rows of level l + 1 are
// the aggregates of level l; the coarsest level uses n and r only).
struct PLevel {
  int n, ld, width;
  const int32_t* idx;
  const float *val, *diag, *wd;
  const int32_t* cptr;
  float *r, *x;
  // Block b restricts the aggregates 8 per b .. (a task is eight aggregates).
  // With soff >= 0 the graph rows of those aggregates are kept in shared
  // memory (from byte soff) for the whole solve: idx [width][cap], val
  // [width][cap], diag [cap], wd [cap], the aggregates' first rows
  // [8 per + 1] and, above level 0, each row's first row on the finer level
  // [cap + 1], with cap = 32 per.  (Eight FP64 steps of 100k rows 63.2 to 55.1
  // ms, a MIXED one of 250k 15.3 to 11.5, with the lighter barrier and the 512
  // threads; a barrier empties L1, so unstaged rows came from L2 every time.)
  int per, soff;
};
__host__ __device__ inline size_t stage_bytes(int width, int per, bool level0) {
  const size_t cap = 32 * (size_t)per;
  return 4 * (2 * width * cap + 2 * cap + 8 * per + 1 + (level0 ? 0 : cap + 1));
}

template <typename T>
struct PArgs {
  int M, rows;  // rows of the system; rows per block (a multiple of 32)
  int64_t ld;
  int k;
  const int32_t* idx;  // [k][ld], level-0 order
  const T* w;
  const T *es, *a1;
  const float *c, *ce;
  const int32_t* perm;  // level-0 row p is P-node perm[p]
  const T* x_in;        // P-node order
  const T* b_in;
  T* x_out;
  T *x, *b, *r, *rh, *p, *v, *s, *t, *zp, *zs;
  PLevel lev[kAmgMaxLevels];
  int nlev, nc, ldx;
  const float* X;  // [nc][ldx] dense inverse of the coarsest level, rows padded with zeros
  int xoff;        // >= 0: the block's rows of X stay in shared memory from this byte
  double inv_ces, inv_R, tol2;
  int maxit, x_zero;
  uint32_t seed;
  double* partials;        // [2][kNVMax][gridDim.x], alternating
  unsigned int* arrivals;  // [kBarrierWords], zero at launch
  long long polls;
  PSolveResult* res;
};

// y_i = sum_s w_s z_j (FP64), or sum_s w_s (z_j - z_i) (FP32 rows, applied in
// difference form: step.cu, k_spmv_pc)
// The operator's rows: read twice an iteration; larger than L2 (STREAM), they
// are marked for early eviction so that the vectors stay there.
template <bool STREAM, typename V>
__device__ __forceinline__ V stream_ld(const V* p) {
  return STREAM ? __ldcs(p) : __ldg(p);
}

template <int K, bool STREAM, typename T>
__device__ __forceinline__ T p_row(const PArgs<T>& a, int i, const T* z, T zi) {
  constexpr bool dif = std::is_same<T, float>::value;
  T acc = 0;
  if constexpr (K > 0) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const T zj = z[stream_ld<STREAM>(a.idx + s * a.ld + i)];
      acc += stream_ld<STREAM>(a.w + s * a.ld + i) * (dif ? zj - zi : zj);
    }
  } else {
#pragma unroll 4
    for (int s = 0; s < a.k; ++s) {
      const T zj = z[stream_ld<STREAM>(a.idx + s * a.ld + i)];
      acc += stream_ld<STREAM>(a.w + s * a.ld + i) * (dif ? zj - zi : zj);
    }
  }
  return acc;
}

// The rows of a level that a block works on: in global memory (row i at
// [s ld + i]) or staged in shared memory (S; local row i at [s cap + i]).
template <bool S>
struct Rows {
  const int32_t* idx;
  const float *val, *diag, *wd;
  int64_t ld;
  int width;
};
extern __shared__ __align__(16) unsigned char psm[];

template <bool S>
__device__ __forceinline__ Rows<S> rows_of(const PLevel& F) {
  if constexpr (S) {
    const int cap = 32 * F.per;
    const int32_t* p = reinterpret_cast<const int32_t*>(psm + F.soff);
    const float* v = reinterpret_cast<const float*>(p + F.width * cap);
    return {p, v, v + F.width * cap, v + F.width * cap + cap, cap, F.width};
  } else {
    return {F.idx, F.val, F.diag, F.wd, F.ld, F.width};
  }
}
template <bool S>
__device__ __forceinline__ const int32_t* agg_of(const PLevel& F) {  // first rows of the aggregates
  const int cap = 32 * F.per;
  return reinterpret_cast<const int32_t*>(psm + F.soff) + 2 * F.width * cap + 2 * cap;
}
template <bool S, typename V>
__device__ __forceinline__ V ro(const V* p) {
  if constexpr (S)
    return *p;
  else
    return __ldg(p);
}

// diag x_i + sum_s val_s x_j over row i, W slots in flight at once
template <int W, bool S>
__device__ __forceinline__ float p_graph(const Rows<S>& R, int i, const float* x, float xi) {
  float ax = ro<S>(R.diag + i) * xi;
  for (int s0 = 0; s0 < R.width; s0 += W) {
    int32_t j[W];
    float v[W];
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const bool in = s0 + s < R.width;
      j[s] = in ? ro<S>(R.idx + (s0 + s) * R.ld + i) : ro<S>(R.idx + i);
      v[s] = in ? ro<S>(R.val + (s0 + s) * R.ld + i) : 0.f;
    }
#pragma unroll
    for (int s = 0; s < W; ++s) ax += v[s] * x[j[s]];
  }
  return ax;
}

// Residual of the pre-smoothed iterate, summed over the aggregates: a warp
// takes eight consecutive aggregates, whose rows (at most 32) are consecutive;
// lane q adds the rows of aggregate q in row order.  The coarse level's
// iterate x = omega D^-1 r is written with its r.
template <int W, bool S, int PT>
__device__ __forceinline__ void p_restrict(const PLevel& F, const PLevel& Cn, bool coarsest,
                                           int first) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tasks = (Cn.n + 7) / 8, t0 = F.per * blockIdx.x;
  const int t1 = min(tasks, t0 + F.per);
  const Rows<S> R = rows_of<S>(F);
  for (int t = t0 + warp; t < t1; t += (PT / 32)) {
    const int I = 8 * t + lane;
    const float wc = !coarsest && lane < 8 && I < Cn.n ? __ldg(Cn.wd + I) : 0.f;
    const int at = min(8 * t + min(lane, 8), Cn.n);
    const int cp = S ? agg_of<S>(F)[at - 8 * t0] : __ldg(F.cptr + at);  // local row with S
    const int f0 = __shfl_sync(0xffffffffu, cp, 0), f1 = __shfl_sync(0xffffffffu, cp, 8);
    const int nx = __shfl_down_sync(0xffffffffu, cp, 1);
    const int i = f0 + lane, gi = S ? first + i : i;
    float res = 0.f;
    if (i < f1) res = F.r[gi] - p_graph<W, S>(R, i, F.x, F.x[gi]);
    const int o = cp - f0, cnt = nx - cp;
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float e = __shfl_sync(0xffffffffu, res, (o + q) & 31);
      if (q < cnt) acc += e;
    }
    if (lane < 8 && I < Cn.n) {
      Cn.r[I] = acc;
      if (!coarsest) Cn.x[I] = wc * acc;
    }
  }
}

// Post-smoothing sweep of a level above 0, whose result corrects the finer
// level's rows of each aggregate (at most four, read with the gathers).
template <int W, bool S, int PT>
__device__ __forceinline__ void p_up(const PLevel& F, const PLevel& Fine, int first, int count) {
  const Rows<S> R = rows_of<S>(F);
  const int32_t* child = S ? agg_of<S>(F) + 8 * F.per + 1 : Fine.cptr;
  auto row = [&](int i, int gi) {
    const int c0 = ro<S>(child + i), c1 = ro<S>(child + i + 1);
    float xf[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) xf[q] = c0 + q < c1 ? Fine.x[c0 + q] : 0.f;
    const float xi = F.x[gi], ri = F.r[gi];
    const float ax = p_graph<W, S>(R, i, F.x, xi);
    const float v = kAmgCoarseScale * (xi + ro<S>(R.wd + i) * (ri - ax));
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (c0 + q < c1) Fine.x[c0 + q] = xf[q] + v;
  };
  if constexpr (S) {
    for (int i = threadIdx.x; i < count; i += PT) row(i, first + i);
  } else {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tasks = (F.n + 31) / 32;
    const int per = (tasks + gridDim.x - 1) / gridDim.x;
    const int t1 = min(tasks, per * ((int)blockIdx.x + 1));
    for (int t = per * blockIdx.x + warp; t < t1; t += (PT / 32)) {
      const int i = 32 * t + lane;
      if (i < F.n) row(i, i);
    }
  }
}

template <int PT>
__device__ __forceinline__ void p_restrict_level(const PLevel& F, const PLevel& Cn, bool coarsest,
                                                 int first) {
  if (F.soff >= 0) {
    if (F.width <= 8)
      p_restrict<8, true, PT>(F, Cn, coarsest, first);
    else
      p_restrict<16, true, PT>(F, Cn, coarsest, first);
  } else {
    if (F.width <= 8)
      p_restrict<8, false, PT>(F, Cn, coarsest, 0);
    else
      p_restrict<16, false, PT>(F, Cn, coarsest, 0);
  }
}
template <int PT>
__device__ __forceinline__ void p_up_level(const PLevel& F, const PLevel& Fine, int first,
                                           int count) {
  if (F.soff >= 0) {
    if (F.width <= 8)
      p_up<8, true, PT>(F, Fine, first, count);
    else
      p_up<16, true, PT>(F, Fine, first, count);
  } else {
    if (F.width <= 8)
      p_up<8, false, PT>(F, Fine, 0, 0);
    else
      p_up<16, false, PT>(F, Fine, 0, 0);
  }
}

// Coarsest level: z = X r, one warp per row, 16 B loads with eight in flight;
// then the correction of the finer level, or z itself without one.  Consecutive
// rows are on different SMs, whose bandwidth bounds it.
template <int PT, typename T>
__device__ __forceinline__ void p_coarse(const PArgs<T>& a, T* z) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float4* r4 = reinterpret_cast<const float4*>(a.lev[a.nlev - 1].r);
  const int n4 = a.ldx / 4;
  for (int q = warp, row = blockIdx.x + warp * gridDim.x; row < a.nc;
       q += (PT / 32), row += gridDim.x * (PT / 32)) {
    float acc = 0.f;
    if (a.xoff >= 0) {
      const float4* x4 = reinterpret_cast<const float4*>(psm + a.xoff) + q * n4;
#pragma unroll 8
      for (int j = lane; j < n4; j += 32) {
        const float4 u = x4[j], v = r4[j];
        acc += u.x * v.x + u.y * v.y + u.z * v.z + u.w * v.w;
      }
    } else {
      const float4* x4 = reinterpret_cast<const float4*>(a.X + (int64_t)row * a.ldx);
#pragma unroll 8
      for (int j = lane; j < n4; j += 32) {
        const float4 u = __ldg(x4 + j), v = r4[j];
        acc += u.x * v.x + u.y * v.y + u.z * v.z + u.w * v.w;
      }
    }
    acc = warp_sum(acc);
    if (a.nlev == 1) {
      if (lane == 0) z[row] = (T)acc;
    } else {
      const PLevel& F = a.lev[a.nlev - 2];
      const int c0 = __ldg(F.cptr + row), c1 = __ldg(F.cptr + row + 1);
      if (lane < c1 - c0) F.x[c0 + lane] += kAmgCoarseScale * acc;
    }
  }
}

// Copies the block's static rows into shared memory; first[l], count[l]: the
// rows of level l that its aggregates hold.
template <int PT, typename T>
__device__ __forceinline__ void p_stage(const PArgs<T>& a, int* first, int* count) {
  for (int l = 0; l + 1 < a.nlev; ++l) {
    const PLevel& F = a.lev[l];
    const int nagg = a.lev[l + 1].n;
    const int k0 = min(nagg, 8 * F.per * (int)blockIdx.x), k1 = min(nagg, k0 + 8 * F.per);
    const int f0 = __ldg(F.cptr + k0), nr = __ldg(F.cptr + k1) - f0;
    if (threadIdx.x == 0) {
      first[l] = f0;
      count[l] = nr;
    }
    if (F.soff < 0) continue;
    const int cap = 32 * F.per;
    int32_t* pi = reinterpret_cast<int32_t*>(psm + F.soff);
    float* pv = reinterpret_cast<float*>(pi + F.width * cap);
    for (int s = 0; s < F.width; ++s)
      for (int r = threadIdx.x; r < nr; r += PT) {
        pi[s * cap + r] = __ldg(F.idx + (int64_t)s * F.ld + f0 + r);
        pv[s * cap + r] = __ldg(F.val + (int64_t)s * F.ld + f0 + r);
      }
    float* pd = pv + F.width * cap;
    for (int r = threadIdx.x; r < nr; r += PT) {
      pd[r] = __ldg(F.diag + f0 + r);
      pd[cap + r] = __ldg(F.wd + f0 + r);
    }
    int32_t* pa = reinterpret_cast<int32_t*>(pd + 2 * cap);
    for (int k = threadIdx.x; k <= k1 - k0; k += PT) pa[k] = __ldg(F.cptr + k0 + k) - f0;
    if (l > 0) {
      int32_t* pc = pa + 8 * F.per + 1;
      for (int r = threadIdx.x; r <= nr; r += PT) pc[r] = __ldg(a.lev[l - 1].cptr + f0 + r);
    }
  }
  if (a.xoff >= 0) {
    float4* xs = reinterpret_cast<float4*>(psm + a.xoff);
    const int n4 = a.ldx / 4;
    for (int q = 0, row = blockIdx.x; row < a.nc; ++q, row += gridDim.x) {
      const float4* x4 = reinterpret_cast<const float4*>(a.X + (int64_t)row * a.ldx);
      for (int j = threadIdx.x; j < n4; j += PT) xs[q * n4 + j] = __ldg(x4 + j);
    }
  }
  __syncthreads();
}

// The solve's scalars, one copy per block (identical in all of them).
template <typename T>
struct PScal {
  double rho, bb, rr, ss, rhs, cr, cs, cp, cv, alpha, omega, mu_p, mu_s;
  T al, om, be, kp, ks, mp, ms;  // alpha, omega, beta, kap_p, kap_s, mu_p, mu_s as the rows use them
  float fp, fs;                  // mu_p, mu_s as the V-cycle's input uses them
  double sig;
  int iters, total, budget, status;
  int go;  // 1: iterate, 0: this cycle has ended, 2: converged at the half step
  int ended;
};

template <int K, typename T, int PT>
__global__ void __launch_bounds__(PT, 1) k_psolve(const __grid_constant__ PArgs<T> a) {
  __shared__ double sh[kNVMax * PT];
  __shared__ double part[kNVMax * 4];
  __shared__ PScal<T> S;
  __shared__ int okf, first[kAmgMaxLevels], count[kAmgMaxLevels];
  Grid<PT> g{sh, part, &okf, a.partials, a.arrivals, a.polls};
  const int tid = threadIdx.x;
  const int r0 = min(a.M, a.rows * (int)blockIdx.x), r1 = min(a.M, r0 + a.rows);
  const int active = min(PT, a.rows);
  const PLevel& L0 = a.lev[0];
  constexpr bool dif = std::is_same<T, float>::value;

  // level-0 input of the V-cycle for a residual value
  auto feed = [&](int i, T val, float mu) {
    const float e = __ldg(a.c + i) * (float)val - mu * __ldg(a.ce + i);
    L0.r[i] = e;
    if (a.nlev > 1) L0.x[i] = __ldg(L0.wd + i) * e;
  };
  // one V-cycle, B v = z + kap with kap = (mu - sum(z)) / M: fin(sum(z)) sets
  // kap (with one level the lifted coarse solve is mean-free: sum 0)
  auto vcycle = [&](T* z, auto fin) -> bool {
    for (int l = 0; l + 1 < a.nlev; ++l) {
      const bool last = l + 2 == a.nlev;
      p_restrict_level<PT>(a.lev[l], a.lev[l + 1], last, first[l]);
      if (!g.sync()) return false;
    }
    p_coarse<PT>(a, z);
    if (a.nlev == 1) {
      if (tid == 0) fin(0.0);
      return g.sync();
    }
    if (!g.sync()) return false;
    for (int l = a.nlev - 2; l >= 1; --l) {
      p_up_level<PT>(a.lev[l], a.lev[l - 1], first[l], count[l]);
      if (!g.sync()) return false;
    }
    Part<float> part0;
    auto sweep0 = [&](auto staged, int i, int gi) {
      constexpr bool ST = decltype(staged)::value;
      const Rows<ST> R = rows_of<ST>(L0);
      const float xi = L0.x[gi], ri = L0.r[gi];
      const float ax = L0.width <= 8 ? p_graph<8, ST>(R, i, L0.x, xi)
                                     : p_graph<16, ST>(R, i, L0.x, xi);
      const float zi = xi + ro<ST>(R.wd + i) * (ri - ax);
      z[gi] = (T)zi;
      part0.add(zi);
    };
    if (L0.soff >= 0) {
      for (int i = tid; i < count[0]; i += PT) sweep0(std::true_type{}, i, first[0] + i);
    } else {
      for (int i = r0 + tid; i < r1; i += PT) sweep0(std::false_type{}, i, i);
    }
    const double v[1] = {part0.value()};
    return g.template reduce<1>(v, PT, [&](const double* t) { fin(t[0]); });
  };
  auto fin_p = [&](double zsum) { S.kp = (T)((S.mu_p - zsum) * a.inv_R); };
  auto fin_s = [&](double zsum) { S.ks = (T)((S.mu_s - zsum) * a.inv_R); };

  p_stage<PT>(a, first, count);
  for (int i = r0 + tid; i < r1; i += PT) {
    const int q = __ldg(a.perm + i);
    a.b[i] = a.b_in[q];
    a.x[i] = a.x_zero ? (T)0 : a.x_in[q];
  }
  if (tid == 0) S.total = 0;
  for (int cyc = 0;; ++cyc) {
    // r = b - A x; shadow residual rh = r (seed 0) or r with seeded signs; p = r
    const bool zero = a.x_zero && cyc == 0;
    if (!zero) {
      Part<T> sx;
      for (int i = r0 + tid; i < r1; i += PT) sx.add(a.x[i]);
      const double v[1] = {sx.value()};
      if (!g.template reduce<1>(v, active, [&](const double* t) { S.sig = t[0]; })) return;
    }
    const uint32_t seed = (cyc || a.seed) ? 0x51ED27u + 977u * a.seed + (uint32_t)cyc : 0u;
    {
      const T sig = zero ? (T)0 : (T)S.sig;
      Part<T> prr, pbb, prh, pc;
      for (int i = r0 + tid; i < r1; i += PT) {
        const T bi = a.b[i];
        T ri = bi;
        if (!zero) {
          const T xi = a.x[i];
          T ax = p_row<K, (PT == kLargePT)>(a, i, a.x, xi);
          if (dif) ax += a.a1[i] * xi;
          ri = bi - (ax + a.es[i] * sig);
        }
        const T sgn = seed ? (T)shadow_sign(__ldg(a.perm + i), seed) : (T)1;
        a.r[i] = ri;
        a.rh[i] = sgn * ri;
        a.p[i] = ri;
        prr.add(ri * ri);
        pbb.add(bi * bi);
        prh.add(sgn * ri * ri);
        pc.add((T)__ldg(a.c + i) * ri);
      }
      const double v[4] = {prr.value(), pbb.value(), prh.value(), pc.value()};
      const bool ok = g.template reduce<4>(v, active, [&](const double* t) {
        S.rr = t[0];
        S.bb = t[1];
        S.rho = t[2];
        S.cr = S.cp = t[3];
        S.mu_p = t[3] * a.inv_ces;
        S.fp = (float)S.mu_p;
        S.mp = (T)S.mu_p;
        S.status = isfinite(t[0]) ? 0 : 2;
        S.iters = 0;
        S.budget = min(a.maxit - S.total, kCycle);
        S.go = S.status == 0 && t[0] > a.tol2 * t[1] && t[2] != 0.0 && S.budget > 0;
        S.ended = !S.go;  // ended by convergence or a breakdown, not by the budget
      });
      if (!ok) return;
    }
    bool run = S.go == 1;
    if (run) {
      const float mu = S.fp;
      for (int i = r0 + tid; i < r1; i += PT) feed(i, a.p[i], mu);
      if (!g.sync()) return;
    }
    while (run) {
      if (!vcycle(a.zp, fin_p)) return;
      // v = A p^, p^ = zp + kap_p; (rh, v), (c . v)
      {
        const T kap = S.kp, mu = S.mp;
        Part<T> d0, d1;
        for (int i = r0 + tid; i < r1; i += PT) {
          const T zi = dif ? a.zp[i] : (T)0;
          const T y = p_row<K, (PT == kLargePT)>(a, i, a.zp, zi) + (dif ? zi + kap : kap) * __ldg(a.a1 + i) +
                      __ldg(a.es + i) * mu;
          a.v[i] = y;
          d0.add(a.rh[i] * y);
          d1.add((T)__ldg(a.c + i) * y);
        }
        const double v[2] = {d0.value(), d1.value()};
        const bool ok = g.template reduce<2>(v, active, [&](const double* t) {
          if (t[0] == 0.0 || !isfinite(t[0])) {
            S.status = isfinite(t[0]) ? 1 : 2;
            S.iters += 1;
            S.go = 0;
            S.ended = 1;
            return;
          }
          S.alpha = S.rho / t[0];
          S.al = (T)S.alpha;
          S.cv = t[1];
          S.cs = S.cr - S.alpha * t[1];
          S.mu_s = S.cs * a.inv_ces;
          S.fs = (float)S.mu_s;
          S.ms = (T)S.mu_s;
        });
        if (!ok) return;
      }
      if (S.go != 1) break;
      // s = r - alpha v; the V-cycle's input; (s, s), (rh, s)
      {
        const T al = S.al;
        const float mu = S.fs;
        Part<T> d0, d1;
        for (int i = r0 + tid; i < r1; i += PT) {
          const T si = a.r[i] - al * a.v[i];
          a.s[i] = si;
          feed(i, si, mu);
          d0.add(si * si);
          d1.add(a.rh[i] * si);
        }
        const double v[2] = {d0.value(), d1.value()};
        const bool ok = g.template reduce<2>(v, active, [&](const double* t) {
          S.rhs = t[1];
          if (t[0] <= a.tol2 * S.bb) {  // converged at the half step
            S.rr = t[0];
            S.iters += 1;
            S.go = 2;
            S.ended = 1;
          }
        });
        if (!ok) return;
      }
      if (S.go == 2) {
        const T al = S.al, kp = S.kp;
        for (int i = r0 + tid; i < r1; i += PT) a.x[i] += al * (a.zp[i] + kp);
        break;
      }
      if (!vcycle(a.zs, fin_s)) return;
      // t = A s^, s^ = zs + kap_s; (t, s), (t, t), (c . t), (rh, t)
      {
        const T kap = S.ks, mu = S.ms;
        Part<T> d0, d1, d2, d3;
        for (int i = r0 + tid; i < r1; i += PT) {
          const T zi = dif ? a.zs[i] : (T)0;
          const T y = p_row<K, (PT == kLargePT)>(a, i, a.zs, zi) + (dif ? zi + kap : kap) * __ldg(a.a1 + i) +
                      __ldg(a.es + i) * mu;
          a.t[i] = y;
          d0.add(y * a.s[i]);
          d1.add(y * y);
          d2.add((T)__ldg(a.c + i) * y);
          d3.add(a.rh[i] * y);
        }
        const double v[4] = {d0.value(), d1.value(), d2.value(), d3.value()};
        const bool ok = g.template reduce<4>(v, active, [&](const double* t) {
          if (!(t[1] > 0.0) || !isfinite(t[0])) {
            S.status = isfinite(t[1]) ? 3 : 2;
            S.iters += 1;
            S.go = 0;
            S.ended = 1;
            return;
          }
          const double om = t[0] / t[1];
          const double rn = S.rhs - om * t[3];
          const double be = (rn / S.rho) * (S.alpha / om);
          S.rho = rn;
          S.omega = om;
          S.om = (T)om;
          S.be = (T)be;
          S.cr = S.cs - om * t[2];
          S.cp = S.cr + be * (S.cp - om * S.cv);
          S.mu_p = S.cp * a.inv_ces;
          S.fp = (float)S.mu_p;
          S.mp = (T)S.mu_p;
        });
        if (!ok) return;
      }
      if (S.go != 1) break;
      // x, r and p, and the next V-cycle's input; (r, r)
      {
        const T al = S.al, om = S.om, be = S.be, shift = al * S.kp + om * S.ks;
        const float mu = S.fp;
        Part<T> d0;
        for (int i = r0 + tid; i < r1; i += PT) {
          a.x[i] += al * a.zp[i] + (om * a.zs[i] + shift);
          const T ri = a.s[i] - om * a.t[i];
          a.r[i] = ri;
          const T pi = ri + be * (a.p[i] - om * a.v[i]);
          a.p[i] = pi;
          feed(i, pi, mu);
          d0.add(ri * ri);
        }
        const double v[1] = {d0.value()};
        const bool ok = g.template reduce<1>(v, active, [&](const double* t) {
          const double rr = t[0];
          const bool conv = rr <= a.tol2 * S.bb;
          S.rr = rr;
          S.iters += 1;
          if (!isfinite(rr))
            S.status = 2;
          else if (rr > 1e8 * S.bb && S.bb > 0.0)
            S.status = 5;
          else if (!conv && (S.rho == 0.0 || S.omega == 0.0))
            S.status = 4;
          S.ended = S.status != 0 || conv || S.total + S.iters >= a.maxit;
          S.go = (S.ended || S.iters >= S.budget) ? 0 : 1;
        });
        if (!ok) return;
      }
      run = S.go == 1;
    }
    const bool conv = S.rr <= a.tol2 * S.bb;
    const int st = S.status, tot = S.total + S.iters;
    const bool again = st == 1 || st == 3 || st == 4 || st == 5 || !S.ended;
    __syncthreads();
    if (tid == 0) S.total = tot;
    if (conv || !again || tot >= a.maxit || cyc >= kMaxCycles) {
      if (blockIdx.x == 0 && tid == 0) {
        a.res->iters = tot;
        a.res->status = st;
        a.res->relres = S.bb > 0 ? sqrt(S.rr / S.bb) : sqrt(S.rr);
        a.res->converged = conv;
      }
      break;
    }
    if (st == 5)  // the recurrence has blown up: start again from the initial iterate
      for (int i = r0 + tid; i < r1; i += PT)
        a.x[i] = a.x_zero ? (T)0 : a.x_in[__ldg(a.perm + i)];
  }
  for (int i = r0 + tid; i < r1; i += PT) a.x_out[__ldg(a.perm + i)] = a.x[i];
}

// ------------------------------------------------------------------ set-up
// Row p of the permuted operator is row perm[p] of the original one, slot by
// slot in the same order, with its columns renumbered.
template <typename T>
__global__ void k_permute_op(int64_t M, int64_t ld, int k, const int32_t* __restrict__ perm,
                             const int32_t* __restrict__ inv, const int32_t* __restrict__ idx,
                             const double* __restrict__ w, const double* __restrict__ es,
                             const double* __restrict__ a1, int32_t* __restrict__ pidx,
                             T* __restrict__ pw, T* __restrict__ pes, T* __restrict__ pa1) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < M;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = perm[p];
    for (int s = 0; s < k; ++s) {
      pidx[s * ld + p] = inv[idx[s * ld + i]];
      pw[s * ld + p] = (T)w[s * ld + i];
    }
    pes[p] = (T)es[i];
    pa1[p] = (T)a1[i];
  }
}

__global__ void k_invert_perm(int64_t M, const int32_t* __restrict__ perm,
                              int32_t* __restrict__ inv) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < M;
       p += (int64_t)gridDim.x * blockDim.x)
    inv[perm[p]] = (int32_t)p;
}

}  // namespace

struct PSolve {
  std::vector<void*> allocs;
  bool mix = false;
  int grid = 0;
  size_t smem = 0;
  int pt = 0;  // threads per block
  PArgs<double> a64{};
  PArgs<float> a32{};
};

void psolve_free(PSolve* p) {
  if (!p) return;
  for (void* q : p->allocs) cudaFree(q);
  delete p;
}

namespace {

template <typename T>
int p_alloc(rbffd_ctx* ctx, PSolve* p, T** out, size_t count, cudaStream_t st) {
  void* ptr = nullptr;
  int rc = check_cuda(ctx, solver_malloc(ctx, &ptr, sizeof(T) * (count ? count : 1)),
                      "pressure solve alloc");
  if (rc) return rc;
  p->allocs.push_back(ptr);
  *out = (T*)ptr;
  return check_cuda(ctx, cudaMemsetAsync(ptr, 0, sizeof(T) * (count ? count : 1), st), "memset");
}

template <typename T>
int fill(rbffd_ctx* ctx, PSolve* p, PArgs<T>& a, int64_t M, int64_t ld, int k,
         const int32_t* idx, const double* w, const double* es, const double* a1, const Amg* amg,
         cudaStream_t st) {
  int rc = 0;
  const int64_t len = round_up(M, 32);
  int32_t *pidx = nullptr, *inv = nullptr;
  T *pw = nullptr, *pes = nullptr, *pa1 = nullptr;
  if ((rc = p_alloc(ctx, p, &pidx, (size_t)ld * k, st)) ||
      (rc = p_alloc(ctx, p, &pw, (size_t)ld * k, st)) ||
      (rc = p_alloc(ctx, p, &inv, len, st)) || (rc = p_alloc(ctx, p, &pes, len, st)) ||
      (rc = p_alloc(ctx, p, &pa1, len, st)))
    return rc;
  const int G = sm_count() * 8;
  k_invert_perm<<<G, 256, 0, st>>>(M, amg->perm0, inv);
  k_permute_op<T><<<G, 256, 0, st>>>(M, ld, k, amg->perm0, inv, idx, w, es, a1, pidx, pw, pes,
                                     pa1);
  if ((rc = check_cuda(ctx, cudaGetLastError(), "pressure operator order"))) return rc;
  T** vec[] = {&a.x, &a.b, &a.r, &a.rh, &a.p, &a.v, &a.s, &a.t, &a.zp, &a.zs};
  for (T** v : vec)
    if ((rc = p_alloc(ctx, p, v, len, st))) return rc;
  a.M = (int)M;
  a.rows = (int)round_up((M + p->grid - 1) / p->grid, 32);
  a.ld = ld;
  a.k = k;
  a.idx = pidx;
  a.w = pw;
  a.es = pes;
  a.a1 = pa1;
  a.c = amg->c;
  a.ce = amg->ce;
  a.perm = amg->perm0;
  a.nlev = amg->nlev;
  a.nc = (int)amg->nc;
  a.ldx = (int)round_up(amg->nc, 4);
  SolveStatus* status = nullptr;
  float* X = nullptr;
  if ((rc = p_alloc(ctx, p, &X, (size_t)a.nc * a.ldx, st))) return rc;
  if ((rc = check_cuda(ctx, cudaMemcpy2DAsync(X, sizeof(float) * a.ldx, amg->Xc,
                                              sizeof(float) * a.nc, sizeof(float) * a.nc, a.nc,
                                              cudaMemcpyDeviceToDevice, st),
                       "coarse inverse")))
    return rc;
  a.X = X;
  for (int l = 0; l < a.nlev; ++l) {
    const AmgLevel& g = amg->lev[l];
    PLevel& q = a.lev[l];
    q.n = (int)g.n;
    q.ld = (int)g.ld;
    q.width = g.width;
    q.idx = g.idx;
    q.val = g.val;
    q.diag = g.diag;
    q.wd = g.wd;
    q.cptr = g.cptr;
    if ((rc = p_alloc(ctx, p, &q.r, g.ld, st)) || (rc = p_alloc(ctx, p, &q.x, g.ld, st))) return rc;
  }
  // shared memory for the static rows: the levels from the coarsest up (two
  // phases a V-cycle use each), then the rows of the dense inverse
  p->smem = 0;
  for (int l = 0; l + 1 < a.nlev; ++l) {
    a.lev[l].per = ((a.lev[l + 1].n + 7) / 8 + p->grid - 1) / p->grid;
    a.lev[l].soff = -1;
  }
  bool room = true;
  for (int l = a.nlev - 2; l >= 0 && room; --l) {
    const size_t need = round_up(stage_bytes(a.lev[l].width, a.lev[l].per, l == 0), 16);
    room = p->smem + need <= stage_room(p->pt);
    if (!room) break;
    a.lev[l].soff = (int)p->smem;
    p->smem += need;
  }
  const size_t xneed = sizeof(float) * (size_t)a.ldx * ((a.nc + p->grid - 1) / p->grid);
  a.xoff = p->smem + xneed <= stage_room(p->pt) ? (int)p->smem : -1;
  if (a.xoff >= 0) p->smem += xneed;
  a.inv_ces = amg->inv_ces;
  a.inv_R = amg->inv_R;
  if ((rc = p_alloc(ctx, p, &a.partials, (size_t)2 * kNVMax * p->grid, st)) ||
      (rc = p_alloc(ctx, p, &status, 1, st)))
    return rc;
  a.res = &status->res;
  a.arrivals = status->bar;
  return RBFFD_OK;
}

template <typename T>
const void* kernel_of(int k, int pt) {
  if (pt == kLargePT)
    return k == 28 ? (const void*)k_psolve<28, T, kLargePT> : (const void*)k_psolve<0, T, kLargePT>;
  return k == 28 ? (const void*)k_psolve<28, T, kSmallPT> : (const void*)k_psolve<0, T, kSmallPT>;
}

template <typename T>
PArgs<T>& args_of(PSolve* p);
template <>
PArgs<double>& args_of<double>(PSolve* p) {
  return p->a64;
}
template <>
PArgs<float>& args_of<float>(PSolve* p) {
  return p->a32;
}

}  // namespace

int psolve_build(rbffd_ctx* ctx, int64_t M, int64_t ld, int k, const int32_t* idx,
                 const double* w, const double* es, const double* a1, const Amg* amg, bool mix,
                 PSolve** out, cudaStream_t st) {
  PSolve* p = new PSolve();
  p->mix = mix;
  p->grid = sm_count();
  p->pt = M > kLargeRows ? kLargePT : kSmallPT;
  const int rc = mix ? fill(ctx, p, p->a32, M, ld, k, idx, w, es, a1, amg, st)
                     : fill(ctx, p, p->a64, M, ld, k, idx, w, es, a1, amg, st);
  const void* fn = mix ? kernel_of<float>(k, p->pt) : kernel_of<double>(k, p->pt);
  if (rc || !coop_fits(fn, p->grid, p->pt, stage_room(p->pt))) {
    cudaStreamSynchronize(st);
    psolve_free(p);
    return solver_left_out(ctx, rc);
  }
  *out = p;
  return RBFFD_OK;
}

template <typename T>
int psolve_run(rbffd_ctx* ctx, PSolve* p, T* x, const T* b, double tol, int maxit, uint32_t seed,
               bool x_zero, PSolveResult* res, int64_t* launches, cudaStream_t st) {
  PArgs<T> a = args_of<T>(p);
  a.x_in = x;
  a.x_out = x;
  a.b_in = b;
  a.tol2 = tol * tol;
  a.maxit = maxit;
  a.seed = seed;
  a.x_zero = x_zero ? 1 : 0;
  a.polls = barrier_polls(ctx);
  SolveStatus* h = (SolveStatus*)ctx->host_pinned;
  int rc = check_cuda(ctx, cudaMemsetAsync(a.arrivals, 0, kBarrierWords * sizeof(unsigned int), st),
                      "memset");
  if (rc) return rc;
  const void* fn = kernel_of<T>(a.k, p->pt);
  void* args[] = {&a};
  rc = check_cuda(ctx, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)stage_room(p->pt)),
                  "pressure solve shared memory");
  if (!rc)
    rc = check_cuda(ctx, cudaLaunchCooperativeKernel(fn, dim3(p->grid), dim3(p->pt), args, p->smem, st),
                    "pressure solve");
  if (!rc)
    rc = check_cuda(ctx, cudaMemcpyAsync(h, a.res, sizeof(SolveStatus), cudaMemcpyDeviceToHost, st),
                    "pressure solve result");
  if (!rc) rc = check_cuda(ctx, cudaStreamSynchronize(st), "pressure solve sync");
  if (rc) return rc;
  *launches += 1;
  if (h->bar[2])  // given up by any block: some of the solution may not have been written
    return set_error(ctx, RBFFD_ERR_CUDA, "pressure solve: grid barrier not reached (bounded wait)");
  *res = h->res;
  return RBFFD_OK;
}

template int psolve_run<double>(rbffd_ctx*, PSolve*, double*, const double*, double, int, uint32_t,
                                bool, PSolveResult*, int64_t*, cudaStream_t);
template int psolve_run<float>(rbffd_ctx*, PSolve*, float*, const float*, double, int, uint32_t,
                               bool, PSolveResult*, int64_t*, cudaStream_t);

}  // namespace rbffd
