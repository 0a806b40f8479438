// Batched Gaussian-process likelihood and gradient in lockstep: every member of a
// batch takes the same block step in one launch.
//
// One CTA per GP (batched.cu) is bound by the FP64 units of the SM that holds it
// (under two multiply-adds per cycle: 0.2 s for a GP of order 1024 whatever the
// batch) and, for less GPs than SMs, by its largest member.  Here the sweep of
// 128-wide blocks is the outer loop and the members are the grid: the panel
// solves (products with the block's inverse), the trailing updates, the adjoint's
// updates and its symbolic step are products on BF16 slices at FP64 accuracy
// (f64x.cu), which leaves the diagonal blocks (128^3 / 6 multiply-adds twice), the
// covariance and the gradient's sums to the FP64 units, spread over all SMs.
//
// Members lie in the workspace in one layout: order and leading dimension P (the
// batch's largest order in whole blocks), rows and columns past the member's own
// order continued by the identity in the factor and by zeros in the adjoint, so
// that every step has whole blocks and a member is described by its number of
// blocks alone.  The caller's Kws holds the covariance until the last kernel has
// read it for the gradient and puts the factor there.  Members are taken in order
// of size, largest first, in passes of as many as the workspace holds.
//
// 512 GPs of orders 64 .. 1024: 200 ms one CTA per GP, 42 ms here: 18 ms products
// (195 launches; few 128-deep chunks per output tile, so their epilogues' instructions
// bound them), 8 ms splits (3 TB/s), 5 ms covariance and 7 ms diagonal blocks (FP64
// units), 2 ms gradient.  96 of orders 32 .. 512: 12.6 -> 3.7 ms.  Accuracy: the
// likelihood's error against 64 bits is that of the kernel it replaces (5.9e-13).
#include "common.cuh"

#include <algorithm>

namespace gpc {
namespace {

constexpr int SB = 128;  // block
constexpr size_t kStepCap = size_t(8) << 30;

#define TRY(x)                        \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

struct Member {
  int batch, d, nmax, P, z0;
  const int *n;
  const long long *offK, *rowX;
  const double *X, *y, *hyp;
  double *K;
  const int *order;  // of the whole batch; this pass begins at z0
  int *info;
};
__device__ __forceinline__ int member_index(const Member &m) { return __ldg(m.order + m.z0 + blockIdx.z); }
__device__ __forceinline__ int member_order(const Member &m, int gi) {
  const int n = __ldg(m.n + gi);
  return n < 1 || n > m.nmax ? 0 : n;  // sizes travel in device memory
}

// Blocks of every member of the pass (0: an order out of range), and its info; err: no product has given up yet.
__global__ void steps_init_kernel(Member m, int count, int *nblk, int *nrow, int *err) {
  const int z = blockIdx.x * blockDim.x + threadIdx.x;
  if (z == 0) *err = GPC_OK;
  if (z >= count) return;
  const int gi = m.order[m.z0 + z], n = m.n[gi];
  const bool bad = n < 1 || n > m.nmax;
  nblk[z] = bad ? 0 : (n + SB - 1) / SB;
  nrow[z] = bad ? 0 : n;
  m.info[2 * gi] = -1;
  m.info[2 * gi + 1] = bad ? GPC_ERR_INVALID_ARG : GPC_OK;
}

// Covariance, lower triangle, into the workspace (continued by the identity to
// whole blocks) and into Kws.  A warp per row, lanes along it.
__global__ void __launch_bounds__(256) steps_cov_kernel(Member m, double *Lw, long long sL) {
  const int gi = member_index(m), n = member_order(m, gi), i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= (n + SB - 1) / SB * SB) return;
  const int lane = threadIdx.x & 31, d = m.d;
  double *Li = Lw + blockIdx.z * sL + (long long)i * m.P;
  if (i >= n) {
    for (int j = lane; j <= i; j += 32) Li[j] = i == j ? 1.0 : 0.0;
    return;
  }
  const double *X = m.X + __ldg(m.rowX + gi) * d, *xi = X + (long long)i * d;
  const double al = m.hyp[3 * gi], rho = m.hyp[3 * gi + 1], sig = m.hyp[3 * gi + 2];
  const double a2 = al * al, inv2r2 = 1.0 / (2.0 * rho * rho), dg = a2 + sig * sig;
  double *Ki = m.K + __ldg(m.offK + gi) + (long long)i * n;
  for (int j = lane; j <= i; j += 32) {
    double v = dg;
    if (j < i) {
      double r2 = 0.0;
      for (int q = 0; q < d; ++q) {
        const double df = xi[q] - X[(long long)j * d + q];
        r2 = fma(df, df, r2);
      }
      v = a2 * exp(-r2 * inv2r2);
    }
    Li[j] = v;
    Ki[j] = v;
  }
}

__device__ double block_sum(double v, double *red) {  // 512 threads
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < (int)blockDim.x / 32; ++w) s += red[w];
  return s;
}

// z = L^-1 y, alpha = L^-T z and the value, with the stored block inverses, the
// vectors in shared memory.  A CTA per member: per block a product with the
// inverse (four threads per row) and the update of the rows below (four threads
// per row) or of the columns to the left (a thread per column).  Bound by the
// latency of the chain of blocks; members share the SMs.
constexpr int SV_T = 512;
__global__ void __launch_bounds__(SV_T)
steps_solve_kernel(Member m, const double *Lw, long long sL, const double *inv, long long sinv, double *zv, double *av,
                   double *value) {
  extern __shared__ double xs[];  // P entries, then w[SB], red[SV_T / 32]
  double *w = xs + m.P, *red = w + SB;
  const int gi = member_index(m), n = member_order(m, gi), t = threadIdx.x;
  if (n == 0) return;
  const int nblk = (n + SB - 1) / SB, np = nblk * SB;
  const double *L = Lw + blockIdx.z * sL, *Di0 = inv + blockIdx.z * sinv, *y = m.y + __ldg(m.rowX + gi);
  const long long ld = m.P;
  double *z = zv + (size_t)blockIdx.z * m.P, *alpha = av + (size_t)blockIdx.z * m.P;
  for (int i = t; i < np; i += SV_T) xs[i] = i < n ? y[i] : 0.0;
  __syncthreads();
  const int r = t >> 2, h = t & 3;
  for (int s = 0; s < nblk; ++s) {
    const int i0 = s * SB;
    const double *Di = Di0 + (size_t)s * SB * SB;
    double a = 0.0, b = 0.0;
    for (int c = h; c <= r; c += 8) {
      a = fma(Di[r * SB + c], xs[i0 + c], a);
      if (c + 4 <= r) b = fma(Di[r * SB + c + 4], xs[i0 + c + 4], b);
    }
    a += b;
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    __syncthreads();
    if (h == 0) {
      xs[i0 + r] = a;
      z[i0 + r] = a;
    }
    __syncthreads();
    for (int i = i0 + SB + r; i < np; i += SV_T / 4) {
      const double *row = L + i * ld + i0;
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll 4
      for (int c = h; c < SB; c += 16) {
        a0 = fma(row[c], xs[i0 + c], a0);
        a1 = fma(row[c + 4], xs[i0 + c + 4], a1);
        a2 = fma(row[c + 8], xs[i0 + c + 8], a2);
        a3 = fma(row[c + 12], xs[i0 + c + 12], a3);
      }
      a0 = (a0 + a1) + (a2 + a3);
      a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
      a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
      if (h == 0) xs[i] -= a0;
    }
    __syncthreads();
  }
  for (int s = nblk - 1; s >= 0; --s) {
    const int i0 = s * SB;
    const double *Di = Di0 + (size_t)s * SB * SB;
    const int c = t & (SB - 1), q = t >> 7;  // column c of the inverse, every fourth row
    double a = 0.0;
    for (int k = c + ((q - c) & 3); k < SB; k += 4) a = fma(Di[k * SB + c], xs[i0 + k], a);
    __syncthreads();
    if (q == 0) w[c] = a;
    __syncthreads();
    if (q == 1) w[c] += a;
    __syncthreads();
    if (q == 2) w[c] += a;
    __syncthreads();
    if (q == 3) xs[i0 + c] = w[c] + a;
    __syncthreads();
    for (int col = t; col < i0; col += SV_T) {
      const double *p = L + i0 * ld + col;
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll 4
      for (int k = 0; k < SB; k += 4) {
        a0 = fma(p[k * ld], xs[i0 + k], a0);
        a1 = fma(p[(k + 1) * ld], xs[i0 + k + 1], a1);
        a2 = fma(p[(k + 2) * ld], xs[i0 + k + 2], a2);
        a3 = fma(p[(k + 3) * ld], xs[i0 + k + 3], a3);
      }
      xs[col] -= (a0 + a1) + (a2 + a3);
    }
    __syncthreads();
  }
  double lsum = 0.0, q = 0.0;
  for (int i = t; i < np; i += SV_T) {
    alpha[i] = xs[i];
    if (i < n) {
      lsum += log(L[i * ld + i]);
      q = fma(y[i], xs[i], q);
    }
  }
  lsum = block_sum(lsum, red);
  q = block_sum(q, red);
  if (t == 0)
    value[gi] = m.info[2 * gi + 1] != GPC_OK ? __longlong_as_double(0x7ff8000000000000LL)
                                             : -0.5 * q - lsum - 0.5 * (double)n * 1.8378770664093454835606594728112;
}

// Lbar = tril(alpha z^T) - diag(1/L_ii), zeros in the rest of the diagonal blocks and past the member's order.
__global__ void __launch_bounds__(256)
steps_lbar_kernel(Member m, const double *Lw, double *Kb, long long sL, const double *zv, const double *av) {
  const int gi = member_index(m), n = member_order(m, gi), i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= (n + SB - 1) / SB * SB) return;
  const double *z = zv + (size_t)blockIdx.z * m.P;
  const double ai = av[(size_t)blockIdx.z * m.P + i];
  const long long at = blockIdx.z * sL + (long long)i * m.P;
  for (int j = threadIdx.x & 31; j < i / SB * SB + SB; j += 32) {
    double v = 0.0;
    if (j <= i && i < n) {
      v = ai * z[j];
      if (i == j) v -= 1.0 / Lw[at + i];
    }
    Kb[at + j] = v;
  }
}

// The gradient's sums over 8 rows: of kb k off the diagonal, of kb k r^2 and of
// the diagonal's kb (which the sweep leaves twice as large); then the factor
// takes the covariance's place in Kws.
__global__ void __launch_bounds__(256)
steps_grad_kernel(Member m, const double *Lw, const double *Kb, long long sL, double *part) {
  __shared__ double red[8][3];
  const int gi = member_index(m), n = member_order(m, gi), w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + w, d = m.d;
  if (blockIdx.x * 8 >= n) return;
  double sk = 0.0, skr = 0.0, sd = 0.0;
  if (i < n) {
    const double *X = m.X + __ldg(m.rowX + gi) * d, *xi = X + (long long)i * d;
    double *Ki = m.K + __ldg(m.offK + gi) + (long long)i * n;
    const long long at = blockIdx.z * sL + (long long)i * m.P;
    for (int j = lane; j < n; j += 32) {
      if (j > i) {
        Ki[j] = 0.0;
        continue;
      }
      const double kb = Kb[at + j], k = Ki[j];
      Ki[j] = Lw[at + j];
      if (j == i) {
        sd += 0.5 * kb;
      } else {
        double r2 = 0.0;
        for (int q = 0; q < d; ++q) {
          const double df = xi[q] - X[(long long)j * d + q];
          r2 = fma(df, df, r2);
        }
        sk = fma(kb, k, sk);
        skr = fma(kb, k * r2, skr);
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    sk += __shfl_xor_sync(0xffffffffu, sk, o);
    skr += __shfl_xor_sync(0xffffffffu, skr, o);
    sd += __shfl_xor_sync(0xffffffffu, sd, o);
  }
  if (lane == 0) {
    red[w][0] = sk;
    red[w][1] = skr;
    red[w][2] = sd;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s += red[q][threadIdx.x];
    part[((size_t)blockIdx.z * (m.P / 8) + blockIdx.x) * 3 + threadIdx.x] = s;
  }
}

// The gradient from the sums.  A product whose bounded wait gave up (err) served
// every member of the pass: those still fine take its status, and NaN results.
__global__ void __launch_bounds__(96)
steps_grad_sum_kernel(Member m, const double *part, double *value, double *grad3, const int *err) {
  __shared__ double tot[3];
  const int gi = member_index(m), n = member_order(m, gi), w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (n == 0) return;
  double s = 0.0;
  for (int b = lane; b < (n + 7) / 8; b += 32) s += part[((size_t)blockIdx.z * (m.P / 8) + b) * 3 + w];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) tot[w] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    const double al = m.hyp[3 * gi], rho = m.hyp[3 * gi + 1], sig = m.hyp[3 * gi + 2];
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    if (*err != GPC_OK && m.info[2 * gi + 1] == GPC_OK) {
      m.info[2 * gi + 1] = *err;
      value[gi] = nan;
    }
    const bool bad = m.info[2 * gi + 1] != GPC_OK;
    grad3[3 * gi] = bad ? nan : 2.0 * (tot[0] + tot[2] * (al * al)) / al;
    grad3[3 * gi + 1] = bad ? nan : tot[1] / (rho * rho * rho);
    grad3[3 * gi + 2] = bad ? nan : 2.0 * sig * tot[2];
  }
}

// Workspace of one pass of `count` members.
struct StepWs {
  double *L, *Kb, *inv, *m, *t, *z, *a, *part;
  void *lt, *sc, *sdc, *sx, *si, *sy;
  int *rexp, *cexp, *xexp, *iexp, *yexp, *bexp, *nblk, *n, *err;
  size_t bytes;
};
StepWs carve(void *ws, int count, int nmax) {
  const size_t Z = count, nb = (nmax + SB - 1) / SB, P = nb * SB;
  size_t p = 0;
  auto take = [&](size_t bytes) {
    void *q = (char *)ws + p;
    p += align_up(bytes, 1024);
    return q;
  };
  StepWs w;
  w.L = (double *)take(Z * P * P * 8);
  w.Kb = (double *)take(Z * P * P * 8);
  w.inv = (double *)take(Z * nb * SB * SB * 8);
  w.m = (double *)take(Z * SB * SB * 8);
  w.t = (double *)take(Z * SB * SB * 8);
  w.z = (double *)take(Z * P * 8);
  w.a = (double *)take(Z * P * 8);
  w.part = (double *)take(Z * (P / 8) * 3 * 8);
  w.lt = take(Z * P * P * 2 * kF64xSlices);
  w.sc = take(Z * P * SB * 2 * kF64xSlices);
  w.sdc = take(Z * P * SB * 2 * kF64xSlices);
  w.sx = take(Z * P * SB * 2 * kF64xWide);
  w.si = take(Z * SB * SB * 2 * kF64xWide);
  w.sy = take(Z * SB * SB * 2 * kF64xWide);
  w.rexp = (int *)take(Z * P * 4);
  w.cexp = (int *)take(Z * P * 4);
  w.xexp = (int *)take(Z * P * 4);
  w.iexp = (int *)take(Z * P * 4);
  w.yexp = (int *)take(Z * P * 4);
  w.bexp = (int *)take(Z * 4);
  w.nblk = (int *)take(Z * 4);
  w.n = (int *)take((Z + 1) * 4);
  w.err = w.n + Z;
  w.bytes = p;
  return w;
}

}  // namespace

// Members of a pass that a workspace of `bytes` holds.
int batched_steps_members(int batch, int nmax, size_t bytes) {
  const size_t one = carve(nullptr, 1, nmax).bytes;
  int z = (int)std::min<size_t>(batch, bytes / one + 1);
  while (z > 0 && carve(nullptr, z, nmax).bytes > bytes) --z;
  return z;
}
size_t batched_steps_bytes(int batch, int nmax, size_t floor) {
  const size_t cap = std::max(kStepCap, floor);
  const size_t all = carve(nullptr, batch, nmax).bytes;
  return all <= cap ? all : carve(nullptr, std::max(1, batched_steps_members(batch, nmax, cap)), nmax).bytes;
}

cudaError_t batched_steps(int batch, const int *n, const long long *offK, const long long *rowX, int d, const double *X,
                          const double *y, const double *hyp, double *K, double *value, double *grad3, int *info,
                          int nmax, const int *order, void *ws, size_t ws_bytes, cudaStream_t s) {
  const int per = batched_steps_members(batch, nmax, ws_bytes);
  if (per < 1) return cudaErrorInvalidValue;
  const int nb = (nmax + SB - 1) / SB, P = nb * SB;
  const long long sL = (long long)P * P, sinv = (long long)nb * SB * SB, sb = SB * SB;
  const size_t solve_smem = ((size_t)P + SB + SV_T / 32) * sizeof(double);
  for (int z0 = 0; z0 < batch; z0 += per) {
    const int Z = std::min(per, batch - z0);
    const StepWs w = carve(ws, Z, nmax);
    Member m{batch, d, nmax, P, z0, n, offK, rowX, X, y, hyp, K, order, info};
    const dim3 rows(P / 8, 1, Z), one(1, 1, Z);
    const double mem = 8.0 * Z * P * (P + 1.0);
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 8.0 * Z, s,
               launch_k(steps_init_kernel, (unsigned)((Z + 255) / 256), 256, 0, s, m, Z, w.nblk, w.n, w.err));
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, mem, s, launch_k(steps_cov_kernel, rows, 256, 0, s, m, w.L, sL));
    F64xBatch b;
    b.count = Z;
    b.nblk = w.nblk;
    b.n = w.n;
    auto split = [&](int act, int mb, int kb, const F64xBatchSplit &q) {
      b.act = act;
      b.mb = mb;
      b.kb = kb;
      return f64x_split_batch(b, q, s);
    };
    auto product = [&](int act, int mb, int nb_, int kb, const F64xBatchGemm &g) {
      b.act = act;
      b.mb = mb;
      b.nb = nb_;
      b.kb = kb;
      return f64x_gemm_batch(b, g, w.err, s);
    };
    // Operand of whole 128 x 128 blocks or panels with each row's own scale
    auto rows_split = [&](const double *src, long long rs, long long ks, long long stride, int M, void *out, int tri,
                          bool wide, int *exps, int rows_per) {
      F64xBatchSplit q = {};
      q.src = src;
      q.rs = rs;
      q.ks = ks;
      q.stride = stride;
      q.M = M;
      q.K = SB;
      q.out = out;
      q.rows = rows_per;
      q.kpad = SB;
      q.tri = tri;
      q.wide = wide;
      q.vec = P;
      q.rexp_out = exps;
      return q;
    };
    auto wide_product = [&](const void *A, int a_rows, const int *ra, const void *B, const int *rb, int M, bool lower,
                            double *C, long long ldc, long long sC) {
      F64xBatchGemm g = {};
      g.A = A;
      g.a_rows = a_rows;
      g.a_kpad = SB;
      g.B = B;
      g.b_rows = SB;
      g.b_kpad = SB;
      g.M = M;
      g.N = SB;
      g.chunks = 1;
      g.lower = lower;
      g.wide = true;
      g.ra = ra;
      g.rb = rb;
      g.vec = P;
      g.C = C;
      g.ldc = ldc;
      g.sC = sC;
      return g;
    };
    // ---- factorisation, left-looking: a block column takes all earlier ones' products
    // at once, so that a tile's output is read and rounded once (right-looking, with one
    // 128-deep chunk per visit, 512 GPs of orders 64 .. 1024 took 44.8 ms instead of 43.1).  The slices of L's block columns collect in the
    // buffer of the adjoint's, rows scaled by the diagonal (mixed.cu).
    TRY(f64x_diag_exps_batch(b, P, w.L, P, sL, P, w.rexp, s));
    for (int ib = 0; ib < nb; ++ib) {
      const int j = ib * SB, k = j + SB, M = P - k;
      double *D = w.L + (long long)j * P + j, *Di = w.inv + (size_t)ib * sb;
      if (ib > 0) {
        F64xBatchGemm g = {};
        g.A = g.B = w.lt;
        g.a_rows = g.b_rows = g.a_kpad = g.b_kpad = P;
        g.a_row0 = g.b_row0 = j;
        g.M = P - j;
        g.N = SB;
        g.chunks = ib;
        g.lower = true;
        g.ra = g.rb = w.rexp + j;
        g.vec = P;
        g.C = D;
        g.ldc = P;
        g.sC = sL;
        TRY(product(ib, ib, -1, -1, g));
      }
      TRY(diag_batch(b, D, P, sL, ib, Di, sinv, order + z0, info, s));
      if (M <= 0) continue;
      double *A21 = D + (long long)SB * P;
      TRY(split(ib + 1, -1, -1, rows_split(Di, SB, 1, sinv, SB, w.si, 2, true, w.iexp, SB)));
      TRY(split(ib + 1, ib + 1, -1, rows_split(A21, P, 1, sL, M, w.sx, 0, true, w.xexp, P)));
      TRY(product(ib + 1, ib + 1, -1, -1, wide_product(w.sx, P, w.xexp, w.si, w.iexp, M, false, A21, P, sL)));
      F64xBatchSplit q = rows_split(A21, P, 1, sL, M, (unsigned short *)w.lt + (long long)k * P, 0, false, nullptr, P);
      q.kpad = P;
      q.chunk0 = ib;
      q.rexps = w.rexp + k;
      q.saturate = true;
      TRY(split(ib + 1, ib + 1, -1, q));
    }
    // ---- solves, value and the upstream adjoint
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, mem, s,
               launch_k(steps_solve_kernel, one, SV_T, solve_smem, s, m, (const double *)w.L, sL, (const double *)w.inv,
                        sinv, w.z, w.a, value));
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 0.5 * mem, s,
               launch_k(steps_lbar_kernel, rows, 256, 0, s, m, (const double *)w.L, w.Kb, sL, (const double *)w.z,
                        (const double *)w.a));
    // ---- adjoint sweep (chol_adjoint_mixed's products and scales, mixed.cu)
    TRY(f64x_lower_exps_batch(b, P, w.L, P, sL, P, w.rexp, w.cexp, s));
    if (nb > 1) {
      F64xBatchSplit q = {};  // operand row t = column t of L, scaled rows
      q.src = w.L;
      q.rs = 1;
      q.ks = P;
      q.stride = sL;
      q.M = q.K = P;
      q.out = w.lt;
      q.rows = q.kpad = P;
      q.tri = 1;
      q.vec = P;
      q.rexps = w.cexp;
      q.kexp = w.rexp;
      q.kexp_minus = true;
      q.skip_zero = true;  // every product reads rows below its columns only
      TRY(split(0, 0, 0, q));
    }
    for (int ib = nb - 1; ib >= 0; --ib) {
      const int j = ib * SB, k = j + SB, M = P - k;
      double *Dbar = w.Kb + (long long)j * P + j, *Cbar = Dbar + (long long)SB * P;
      const double *D = w.L + (long long)j * P + j, *Di = w.inv + (size_t)ib * sb;
      TRY(split(ib, -1, -1, rows_split(Di, 1, SB, sinv, SB, w.si, 1, true, w.iexp, SB)));  // columns of the inverse
      if (M > 0) {  // Cbar <- Cbar D^-1
        TRY(split(ib + 1, ib + 1, -1, rows_split(Cbar, P, 1, sL, M, w.sx, 0, true, w.xexp, P)));
        TRY(product(ib + 1, ib + 1, -1, -1, wide_product(w.sx, P, w.xexp, w.si, w.iexp, M, false, Cbar, P, sL)));
      }
      {  // the block column's rows, and its common scale
        F64xBatchSplit q = rows_split(Dbar, P, 1, sL, M + SB, w.sc, 0, false, w.xexp, P);
        q.kexp = w.rexp + j;
        q.block_out = w.bexp;
        q.row_exps = w.rexp + j;
        TRY(split(ib, ib, -1, q));
      }
      F64xBatchSplit col = {};  // the block column's columns: K = rows
      col.rs = 1;
      col.ks = P;
      col.stride = sL;
      col.M = SB;
      col.out = w.sdc;
      col.rows = SB;
      col.kpad = P;
      col.vec = P;
      col.rexp = w.bexp;
      col.rexp_sub = w.rexp + j;
      F64xBatchGemm g = {};  // products with L's columns
      g.B = w.lt;
      g.b_rows = g.b_kpad = P;
      g.vec = P;
      g.ldc = P;
      g.sC = sL;
      if (M > 0) {
        col.src = Cbar;
        col.K = M;
        col.chunk0 = 1;
        col.kexp = w.rexp + k;
        TRY(split(ib + 1, -1, ib + 1, col));
        g.A = w.sdc;  // Dbar -= Cbar^T C
        g.a_rows = SB;
        g.a_kpad = P;
        g.a_k0 = SB;
        g.b_row0 = j;
        g.b_k0 = k;
        g.M = g.N = SB;
        g.chunks = nb - ib - 1;
        g.lower = true;
        g.ra = w.bexp;
        g.ra_sub = w.rexp + j;
        g.rb = w.cexp + j;
        g.C = Dbar;
        TRY(product(ib + 1, -1, -1, ib + 1, g));
        if (j > 0) {  // Bbar -= Cbar R
          g.A = w.sc;
          g.a_rows = P;
          g.a_kpad = SB;
          g.a_row0 = SB;
          g.a_k0 = 0;
          g.b_row0 = 0;
          g.b_k0 = j;
          g.M = M;
          g.N = j;
          g.chunks = 1;
          g.lower = false;
          g.ra = w.xexp + SB;
          g.ra_sub = nullptr;
          g.rb = w.cexp;
          g.C = w.Kb + (long long)k * P;
          TRY(product(ib + 1, ib + 1, -1, -1, g));
        }
      }
      // Dbar <- D^-T sym(tril(D^T Dbar)) D^-1
      TRY(split(ib, -1, -1, rows_split(D, 1, P, sL, SB, w.sx, 1, true, w.xexp, SB)));
      TRY(split(ib, -1, -1, rows_split(Dbar, 1, P, sL, SB, w.sy, 1, true, w.yexp, SB)));
      TRY(product(ib, -1, -1, -1, wide_product(w.sx, SB, w.xexp, w.sy, w.yexp, SB, true, w.m, SB, sb)));
      TRY(split(ib, -1, -1, rows_split(w.m, SB, 1, sb, SB, w.sy, 3, true, w.yexp, SB)));
      TRY(product(ib, -1, -1, -1, wide_product(w.sy, SB, w.yexp, w.si, w.iexp, SB, false, w.t, SB, sb)));
      TRY(split(ib, -1, -1, rows_split(w.t, 1, SB, sb, SB, w.sy, 0, true, w.yexp, SB)));
      TRY(product(ib, -1, -1, -1, wide_product(w.si, SB, w.iexp, w.sy, w.yexp, SB, true, Dbar, P, sL)));
      if (j > 0) {  // Rbar -= [Dbar; Cbar]^T [R; B]
        col.src = Dbar;
        col.rs = P;  // symmetric, from its lower triangle
        col.ks = 1;
        col.tri = 3;
        col.K = SB;
        col.chunk0 = 0;
        col.kexp = w.rexp + j;
        TRY(split(ib, -1, -1, col));
        g.A = w.sdc;
        g.a_rows = SB;
        g.a_kpad = P;
        g.a_row0 = 0;
        g.a_k0 = 0;
        g.b_row0 = 0;
        g.b_k0 = j;
        g.M = SB;
        g.N = j;
        g.chunks = nb - ib;
        g.lower = false;
        g.ra = w.bexp;
        g.ra_sub = w.rexp + j;
        g.rb = w.cexp;
        g.C = w.Kb + (long long)j * P;
        TRY(product(ib, -1, -1, ib, g));
      }
    }
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 2.0 * mem, s,
               launch_k(steps_grad_kernel, rows, 256, 0, s, m, (const double *)w.L, (const double *)w.Kb, sL, w.part));
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 0.0, s,
               launch_k(steps_grad_sum_kernel, one, 96, 0, s, m, (const double *)w.part, value, grad3,
                        (const int *)w.err));
  }
  return cudaGetLastError();
}

}  // namespace gpc
