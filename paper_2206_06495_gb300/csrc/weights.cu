// Batched PHS+poly stencil weights (Section 2.1, Eq. rbf_poly_compact).
//
// One warp owns one stencil.  The augmented system [A P; P^T 0] (size
// S = n + (q+1)(q+2)/2) and its right-hand sides (one column per requested
// operator) live column-major in the warp's slice of shared memory, with an
// odd leading dimension so that a warp touching one column hits 32 banks.
// The warp factors the system by Gaussian elimination with partial pivoting
// (pivot: largest magnitude, lowest row on ties) applied to the right-hand
// sides in the same sweep, then back-substitutes.  Every elimination update is
// spread over the 32 lanes as a flat list of (row, column) pairs, so lanes stay
// busy down to the last columns.  All arithmetic is FP64.
//
// What bounds it: the FP64 pipe, which retires one warp-wide instruction in 16
// cycles of an SM, so what counts is FP64 instructions per stencil, whatever
// number of lanes they use.  For S = 38 and three operators the elimination
// and the back substitution issue about 800; the rest is kept small: the
// pivot search, the thresholds and the maxima compare bit patterns as
// integers, reciprocals and roots are formed from hardware seeds in 4 and 6
// instructions, each power of a coordinate is formed once per node, and the
// right-hand sides share one root per node: 1,200 FP64 instructions a stencil
// against 1,890 before, with the same weights bit for bit, but for a reciprocal
// or a root in some 2e9 that misses the correct rounding (1.08M stencils with
// three operators: 77.7 against 89.6 ms; the pipe is 85 % busy).
//
// Local coordinates (the "shift and scale" of the implementation the paper
// follows): stencil nodes are shifted to the alpha-node and divided by the
// largest centre-to-node distance s; derivative weights are divided by s (first
// derivatives) or s^2 (Laplacian) afterwards.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace rbffd {
namespace {

constexpr int kMaxWarpsPerBlock = 17;
constexpr size_t kSmemBlock = 227 * 1024;  // shared memory a block may take
constexpr size_t kSmemSm = 228 * 1024;     // of an SM, which adds 1 KB to each block's
constexpr int kMaxDegree = 5;  // largest q accepted by the ABI

// x^e, e >= 1
__device__ __forceinline__ double ipow(double x, int e) {
  double r = x;
  for (int i = 1; i < e; ++i) r *= x;
  return r;
}

// 1/a for a normal a whose reciprocal is normal, within one unit in the last
// place: a hardware seed (about 20 bits), a Newton step, and a second one with
// an exact residual (Markstein's correction), which leaves 2^-80 before the
// rounding, so that all but one in some 2e9 random arguments are rounded to
// nearest.  (With the compiler's division and root instead, 1.08M stencils with
// three operators take 84.5 against 80.7 ms; the listed weights have the same
// bits.)
__device__ __forceinline__ double recip(double a) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  y = fma(y, fma(-a, y, 1.0), y);
  return fma(y, fma(-a, y, 1.0), y);
}

// sqrt(a), within one unit in the last place and as rarely not rounded to
// nearest, for a >= 2^-1000 (below it the compiled root: the halves below are
// exponent decrements).  From a seed y of 1/sqrt(a) with
// a y^2 = 1 - e, Newton steps for the root, t + t e / 2 (t = a y), and for
// 1 / (2 sqrt(a)), y / 2 + y e / 4, then the correction with an exact residual.
__device__ __forceinline__ double half(double x) {
  return __hiloint2double(__double2hiint(x) - 0x00100000, __double2loint(x));
}
__device__ __forceinline__ double root(double a) {
  if (__double2hiint(a) < 0x01700000) return sqrt(a);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double t = a * y, e = fma(-t, y, 1.0), h = half(y);
  const double g = fma(half(h), e, h), s = fma(half(t), e, t);
  return fma(fma(-s, s, a), g, s);
}

// a^2 + b^2, the square of b rounded on its own
__device__ __forceinline__ double norm2(double a, double b) {
  return __fma_rn(a, a, __dmul_rn(b, b));
}

// r^m for odd m from r^2: r^(m-1) * r
__device__ __forceinline__ double phs_from_r2(double r2, int m) {
  return m > 1 ? ipow(r2, (m - 1) / 2) * root(r2) : root(r2);
}

// Right-hand side of operator `op` (bit index 0..3 = INTERP, DX, DY, LAP) in
// the row of monomial (a, b).
__device__ __forceinline__ double rhs_poly(int op, int a, int b) {
  switch (op) {
    case 0:
      return (a == 0 && b == 0) ? 1.0 : 0.0;
    case 1:
      return (a == 1 && b == 0) ? 1.0 : 0.0;
    case 2:
      return (a == 0 && b == 1) ? 1.0 : 0.0;
    default:
      return ((a == 2 && b == 0) || (a == 0 && b == 2)) ? 2.0 : 0.0;
  }
}

// (a, b) of the t-th monomial in graded lexicographic order 1, x, y, x^2, xy, y^2, ...
__device__ __forceinline__ void monomial(int t, int& a, int& b) {
  int d = 0;
  while ((d + 1) * (d + 2) / 2 <= t) ++d;
  int r = t - d * (d + 1) / 2;
  b = r;
  a = d - r;
}

// Magnitude of a double as an ordered integer key: for non-negative values
// the IEEE bit pattern orders like the value, so the pivot search compares
// integers instead of spending FP64 instructions (NaN, with the largest
// patterns, wins and is then caught as a singular pivot).
__device__ __forceinline__ unsigned long long mag_key(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long k) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, k, o);
    k = x > k ? x : k;
  }
  return k;
}
constexpr unsigned long long kInfKey = 0x7ff0000000000000ull;

// largest column sum of |T| (S columns of S rows): lanes take columns
__device__ __forceinline__ double norm1(const double* T, int S, int LD, int lane) {
  double m = 0.0;
  for (int c = lane; c < S; c += 32) {
    double s0 = 0.0, s1 = 0.0;
    int r = 0;
    for (; r + 1 < S; r += 2) {
      s0 += fabs(T[c * LD + r]);
      s1 += fabs(T[c * LD + r + 1]);
    }
    if (r < S) s0 += fabs(T[c * LD + r]);
    m = fmax(m, s0 + s1);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  return m;
}

// One warp per stencil.  COND = false: the weights of the requested operators,
// written to w.  COND = true: the 1-norm condition number ||A_aug||_1
// ||A_aug^-1||_1 of the same local system, written to w[i]; the inverse is
// formed in place by Gauss-Jordan elimination with the same pivoting (S^3
// multiply-adds instead of the 4 S^3 / 3 of an elimination that carries the
// unit vectors along, and half the shared memory: 99,856 systems of 38 rows
// in 14.2 against 24.4 ms).  Its columns end up permuted, which the 1-norm does
// not see.
template <bool COND>
__global__ void __launch_bounds__(kMaxWarpsPerBlock * 32)
    weights_kernel(const double* __restrict__ ax, const double* __restrict__ ay, int64_t na,
                   const double* __restrict__ bx, const double* __restrict__ by,
                   const int32_t* __restrict__ idx, int64_t ld, int n, int m, int q, int nrhs,
                   int4 ops, int LD, double* __restrict__ w,
                   unsigned long long* __restrict__ bad) {
  extern __shared__ double smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int np = q < 0 ? 0 : (q + 1) * (q + 2) / 2;
  const int S = n + np, NC = S + nrhs;
  double* Am = smem + (size_t)wib * (LD * NC + 2 * n + S);
  double* xs = Am + LD * NC;
  double* ys = xs + n;
  double* invd = ys + n;  // reciprocals of U's diagonal
  const int op_of[4] = {ops.x, ops.y, ops.z, ops.w};
  const int wpb = blockDim.x >> 5;
  const int64_t gw = (int64_t)blockIdx.x * wpb + wib;
  const int64_t nwarps = (int64_t)gridDim.x * wpb;
  const int npair = n * (n - 1) / 2;
  for (int64_t i = gw; i < na; i += nwarps) {
    const double cx = ax[i], cy = ay[i];
    unsigned long long rk = 0ull;
    for (int s = lane; s < n; s += 32) {
      const int j = idx[s * ld + i];
      const double X = bx[j] - cx, Y = by[j] - cy;
      xs[s] = X;
      ys[s] = Y;
      const unsigned long long k = mag_key(norm2(X, Y));
      rk = k > rk ? k : rk;
    }
    const double isc = 1.0 / sqrt(__longlong_as_double((long long)warp_max(rk)));
    __syncwarp();
    // ---- assemble [A P; P^T 0 | rhs] column-major: element (r, c) at Am[c*LD + r].
    // Node by node: local coordinates, monomials (row of P and column of P^T)
    // and the operators' right-hand sides.
    unsigned long long ak = 0ull;  // largest entry of A and P
    for (int s = lane; s < n; s += 32) {
      const double X = xs[s] * isc, Y = ys[s] * isc;
      xs[s] = X;
      ys[s] = Y;
      Am[s * LD + s] = 0.0;  // phi(0)
      // x^a y^b with the powers of x in px; y^b grows with b
      double px[kMaxDegree + 1] = {1.0, X};
#pragma unroll
      for (int a = 2; a <= kMaxDegree; ++a) px[a] = px[a - 1] * X;
      double py = 1.0;
#pragma unroll
      for (int b = 0; b <= kMaxDegree; ++b) {
        if (b > 1) py *= Y;
        if (b == 1) py = Y;
#pragma unroll
        for (int a = 0; a + b <= kMaxDegree; ++a) {
          if (a + b > q) continue;
          const int t = (a + b) * (a + b + 1) / 2 + b;
          const double v = b == 0 ? px[a] : (a == 0 ? py : px[a] * py);
          Am[(n + t) * LD + s] = v;
          Am[s * LD + n + t] = v;
          const unsigned long long k = mag_key(v);
          ak = k > ak ? k : ak;
        }
      }
      if (!COND) {
        const double r2 = norm2(X, Y);
        const double base = phs_from_r2(r2, m - 2);
        for (int o = 0; o < nrhs; ++o) {
          double v;
          switch (op_of[o]) {
            case 0:  // phi(|0 - x_j|)
              v = phs_from_r2(r2, m);
              break;
            case 1:  // d/dx |x - x_j|^m at x = 0: -m r^(m-2) x_j
              v = -m * base * X;
              break;
            case 2:
              v = -m * base * Y;
              break;
            default:  // 2-D Laplacian of r^m: m^2 r^(m-2)
              v = (double)(m * m) * base;
          }
          Am[(S + o) * LD + s] = v;
        }
      }
    }
    for (int e = lane; e < np * np; e += 32) {
      const int c = e / np, r = e - c * np;
      Am[(n + c) * LD + n + r] = 0.0;
    }
    if (!COND) {
      for (int e = lane; e < np * nrhs; e += 32) {
        const int o = e / np, t = e - o * np;
        int a, b;
        monomial(t, a, b);
        Am[(S + o) * LD + n + t] = rhs_poly(op_of[o], a, b);
      }
    }
    __syncwarp();
    // A is symmetric: each pair (r < c) is evaluated once and stored twice
    for (int p = lane; p < npair; p += 32) {
      int c = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f);
      while (c * (c - 1) / 2 > p) --c;
      while (c * (c + 1) / 2 <= p) ++c;
      const int r = p - c * (c - 1) / 2;
      const double dx = xs[r] - xs[c], dy = ys[r] - ys[c];
      const double r2 = norm2(dx, dy);
      const double v = phs_from_r2(r2, m);
      Am[c * LD + r] = v;
      Am[r * LD + c] = v;
      const unsigned long long k = mag_key(v);
      ak = k > ak ? k : ak;
    }
    const unsigned long long tiny =
        mag_key(1e-14 * __longlong_as_double((long long)warp_max(ak)));
    __syncwarp();
    const double anorm = COND ? norm1(Am, S, LD, lane) : 0.0;
    // ---- elimination with partial pivoting
    bool singular = false;
    for (int kk = 0; kk < S; ++kk) {
      unsigned long long bk = 0ull;
      int br = S;
      for (int r = kk + lane; r < S; r += 32) {
        const unsigned long long key = mag_key(Am[kk * LD + r]);
        if (br == S || key > bk) {
          bk = key;
          br = r;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
        const int orr = __shfl_xor_sync(0xffffffffu, br, o);
        if (ok > bk || (ok == bk && orr < br)) {
          bk = ok;
          br = orr;
        }
      }
      if (!(bk > tiny) || bk >= kInfKey) {
        singular = true;
        break;
      }
      const double inv = recip(Am[kk * LD + br]);
      __syncwarp();  // every lane has the pivot before the exchange overwrites it
      if (br != kk) {
        for (int c = (COND ? 0 : kk) + lane; c < NC; c += 32) {
          const double t = Am[c * LD + kk];
          Am[c * LD + kk] = Am[c * LD + br];
          Am[c * LD + br] = t;
        }
      }
      __syncwarp();
      if (COND) {
        // exchange step: pivot row scaled, the other rows updated, then the
        // pivot column
        for (int c = lane; c < S; c += 32)
          if (c != kk) Am[c * LD + kk] *= inv;
        __syncwarp();
        const int R = S - 1;
        for (int p = lane; p < R * R; p += 32) {
          int c = p / R, r = p - c * R;
          c += c >= kk;
          r += r >= kk;
          Am[c * LD + r] -= Am[kk * LD + r] * Am[c * LD + kk];
        }
        __syncwarp();
        for (int r = lane; r < S; r += 32)
          Am[kk * LD + r] = r == kk ? inv : -Am[kk * LD + r] * inv;
      } else {
        if (lane == 0) invd[kk] = inv;
        for (int r = kk + 1 + lane; r < S; r += 32) Am[kk * LD + r] *= inv;
        __syncwarp();
        const int R = S - 1 - kk, C = NC - 1 - kk;
        for (int p = lane; p < R * C; p += 32) {
          const int c = kk + 1 + p / R, r = kk + 1 + (p - (p / R) * R);
          Am[c * LD + r] -= Am[kk * LD + r] * Am[c * LD + kk];
        }
      }
      __syncwarp();
    }
    if (singular) {
      if (lane == 0) atomicMin(bad, (unsigned long long)i);
      if (COND) {
        if (lane == 0) w[i] = INFINITY;
      } else {
        for (int e = lane; e < nrhs * n; e += 32) {
          const int o = e / n, s = e - o * n;
          w[(int64_t)o * n * ld + (int64_t)s * ld + i] = 0.0;
        }
      }
      __syncwarp();
      continue;
    }
    if (COND) {
      const double inorm = norm1(Am, S, LD, lane);
      if (lane == 0) w[i] = anorm * inorm;
      __syncwarp();
      continue;
    }
    // ---- back substitution on the upper triangle, all right-hand sides
    for (int c = S - 1; !COND && c >= 0; --c) {
      const double ic = invd[c];
      for (int o = lane; o < nrhs; o += 32) Am[(S + o) * LD + c] *= ic;
      __syncwarp();
      for (int p = lane; p < c * nrhs; p += 32) {
        const int o = p / c, r = p - o * c;
        Am[(S + o) * LD + r] -= Am[c * LD + r] * Am[(S + o) * LD + c];
      }
      __syncwarp();
    }
    // ---- unscale and store w (the first n entries of each solution)
    for (int e = lane; e < nrhs * n; e += 32) {
      const int o = e / n, s = e - o * n;
      const int op = op_of[o];
      double v = Am[(S + o) * LD + s];
      if (op == 1 || op == 2) v *= isc;
      else if (op == 3) v *= isc * isc;
      w[(int64_t)o * n * ld + (int64_t)s * ld + i] = v;
    }
    __syncwarp();
  }
}

// shared memory of one warp (the system with its right-hand sides, the local
// coordinates and the pivot reciprocals) and the launch shape
struct WShape {
  int LD, wpb;
  size_t smem;
};
// Warps per block: the number that leaves most warps resident on an SM (17 in
// one block for S = 38, against 16 in four blocks of four), the smallest
// such number.
inline WShape weights_shape(int n, int S, int nrhs) {
  WShape sh;
  sh.LD = (S % 2) ? S : S + 1;
  const size_t per_warp = sizeof(double) * ((size_t)sh.LD * (S + nrhs) + 2 * n + S);
  size_t best = 0;
  sh.wpb = 1;
  for (int w = 1; w <= kMaxWarpsPerBlock && per_warp * w <= kSmemBlock; ++w) {
    const size_t resident = w * (kSmemSm / (per_warp * w + 1024));
    if (resident > best) {
      best = resident;
      sh.wpb = w;
    }
  }
  sh.smem = per_warp * sh.wpb;
  return sh;
}

}  // namespace

int weights_build(rbffd_ctx* ctx, const double* ax, const double* ay, int64_t na, const double* bx,
                  const double* by, const int32_t* idx, int64_t ld, uint32_t op_mask, double* w,
                  int64_t* bad_node, cudaStream_t st) {
  const int n = ctx->prm.n, m = ctx->prm.m, q = ctx->prm.q;
  const int np = q < 0 ? 0 : (q + 1) * (q + 2) / 2;
  const int S = n + np;
  int opv[4] = {0, 0, 0, 0};
  int nrhs = 0;
  for (int b = 0; b < 4; ++b)
    if (op_mask & (1u << b)) opv[nrhs++] = b;
  const WShape sh = weights_shape(n, S, nrhs);
  const int LD = sh.LD, wpb = sh.wpb;
  const size_t smem = sh.smem;
  int rc = check_cuda(ctx,
                      cudaFuncSetAttribute(weights_kernel<false>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                      "weights smem attribute");
  if (rc) return rc;
  void* base = nullptr;
  rc = ctx_scratch(ctx, 256, &base);
  if (rc) return rc;
  unsigned long long* d_bad = (unsigned long long*)base;
  rc = check_cuda(ctx, cudaMemsetAsync(d_bad, 0xff, sizeof(unsigned long long), st), "memset");
  if (rc) return rc;
  const int sms = sm_count();
  const int64_t need = (na + wpb - 1) / wpb;
  const int blocks = (int)std::min<int64_t>(need, (int64_t)sms * 16);
  weights_kernel<false><<<blocks, wpb * 32, smem, st>>>(
      ax, ay, na, bx, by, idx, ld, n, m, q, nrhs, make_int4(opv[0], opv[1], opv[2], opv[3]), LD,
      w, d_bad);
  rc = check_cuda(ctx, cudaGetLastError(), "weights kernel");
  if (rc) return rc;
  unsigned long long* h_bad = (unsigned long long*)ctx->host_pinned;
  rc = check_cuda(ctx, cudaMemcpyAsync(h_bad, d_bad, sizeof(*h_bad), cudaMemcpyDeviceToHost, st),
                  "status copy");
  if (rc) return rc;
  rc = check_cuda(ctx, cudaStreamSynchronize(st), "weights sync");
  if (rc) return rc;
  if (*h_bad != ~0ull) {
    if (bad_node) *bad_node = (int64_t)*h_bad;
    return set_error(ctx, RBFFD_ERR_SINGULAR_STENCIL, "singular stencil system at alpha-node %lld",
                     (long long)*h_bad);
  }
  return RBFFD_OK;
}

}  // namespace rbffd

namespace rbffd {

// The weight solves of weights_build with the singular-stencil status word in
// caller-provided device memory (no context, no allocation).  Returns an
// RBFFD status code; bad_node (host, may be null) as in weights_build.
int weights_build_scratch(int n, int m, int q, const double* ax, const double* ay, int64_t na,
                          const double* bx, const double* by, const int32_t* idx, int64_t ld,
                          uint32_t op_mask, double* w, unsigned long long* d_bad,
                          int64_t* bad_node, cudaStream_t st) {
  const int np = q < 0 ? 0 : (q + 1) * (q + 2) / 2;
  const int S = n + np;
  int opv[4] = {0, 0, 0, 0};
  int nrhs = 0;
  for (int b = 0; b < 4; ++b)
    if (op_mask & (1u << b)) opv[nrhs++] = b;
  const WShape sh = weights_shape(n, S, nrhs);
  const int LD = sh.LD, wpb = sh.wpb;
  const size_t smem = sh.smem;
  if (cudaFuncSetAttribute(weights_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess)
    return RBFFD_ERR_CUDA;
  // the status word keeps the previous call's value: reset it
  if (cudaMemsetAsync(d_bad, 0xff, sizeof(unsigned long long), st) != cudaSuccess)
    return RBFFD_ERR_CUDA;
  const int sms = sm_count();
  const int64_t need = (na + wpb - 1) / wpb;
  const int blocks = (int)std::min<int64_t>(need, (int64_t)sms * 16);
  weights_kernel<false><<<blocks, wpb * 32, smem, st>>>(ax, ay, na, bx, by, idx, ld, n, m, q,
                                                        nrhs,
                                                        make_int4(opv[0], opv[1], opv[2], opv[3]),
                                                        LD, w, d_bad);
  unsigned long long h_bad = 0;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&h_bad, d_bad, sizeof(h_bad), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return RBFFD_ERR_CUDA;
  if (h_bad != ~0ull) {
    if (bad_node) *bad_node = (int64_t)h_bad;
    return RBFFD_ERR_SINGULAR_STENCIL;
  }
  return RBFFD_OK;
}

}  // namespace rbffd

namespace rbffd {

// 1-norm condition numbers of the local systems the weight solves factor
// (rbffd_stencil_condition): the weight kernel in its COND mode.
int cond_build(rbffd_ctx* ctx, const double* ax, const double* ay, int64_t na, const double* bx,
               const double* by, const int32_t* idx, int64_t ld, double* cond,
               cudaStream_t st) {
  const int n = ctx->prm.n, m = ctx->prm.m, q = ctx->prm.q;
  const int np = q < 0 ? 0 : (q + 1) * (q + 2) / 2;
  const int S = n + np;
  const WShape sh = weights_shape(n, S, 0);
  int rc = check_cuda(ctx,
                      cudaFuncSetAttribute(weights_kernel<true>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sh.smem),
                      "condition smem attribute");
  if (rc) return rc;
  void* base = nullptr;
  rc = ctx_scratch(ctx, 256, &base);
  if (rc) return rc;
  unsigned long long* d_bad = (unsigned long long*)base;
  rc = check_cuda(ctx, cudaMemsetAsync(d_bad, 0xff, sizeof(unsigned long long), st), "memset");
  if (rc) return rc;
  const int64_t need = (na + sh.wpb - 1) / sh.wpb;
  const int blocks = (int)std::min<int64_t>(need, (int64_t)sm_count() * 16);
  weights_kernel<true><<<blocks, sh.wpb * 32, sh.smem, st>>>(
      ax, ay, na, bx, by, idx, ld, n, m, q, 0, make_int4(0, 0, 0, 0), sh.LD, cond, d_bad);
  rc = check_cuda(ctx, cudaGetLastError(), "condition kernel");
  if (rc) return rc;
  return check_cuda(ctx, cudaStreamSynchronize(st), "condition sync");
}

}  // namespace rbffd
