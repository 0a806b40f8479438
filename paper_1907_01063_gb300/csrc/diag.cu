// Diagonal-block kernels and elementwise helpers of the blocked factorisation.
//
// The small-block factorisation of Section 3.3 (potrf_la_kernel,
// potrf_diag_kernel, potrf_lookahead_kernel in double-float storage; potrf_batch_kernel for batches in lockstep), the panel solve against a factored block
// (trsm_quad_kernel, trsm_rows_kernel) and the inverses of all diagonal blocks
// (trtri_cols_kernel; the per-block inverses of Section 3.2).
#include "common.cuh"

#include <algorithm>

namespace gpc {
namespace {

// All diagonal-block inverses of L at once.  Block 0 is rows [0, first),
// block ib >= 1 is [first + (ib - 1) b, first + ib b).  With ldo == 0 the
// inverse of block ib goes to out + ib * b * b with leading dimension equal to
// its size; otherwise to its diagonal position in an n x n matrix out with
// leading dimension ldo (out may be L itself: the CTAs of a block form a cluster
// then and meet between their reads and their writes).  (The
// per-block inverses of Section 3.2, computed as a batch.)
//
// FP64 work bounds it: one SM's rate makes a whole 128 block 106 us (nb^3 / 6
// multiply-adds at 1.6 per cycle), and a batch of a few blocks would leave the
// other SMs idle.  The columns of an inverse are independent, so a CTA takes 8
// columns of one block (16 CTAs per 128 block).  trtri16_kernel first inverts
// every 16 x 16 diagonal sub-block (a warp each, lane = column and row parity)
// into its final place; trtri_cols_kernel then solves L X = E over 16-row blocks,
// a warp per block: X_K = Dinv_K R_K by 128 threads (a product of one warp would
// hold its sub-partition's FP64 pipe 2.5 us), then every later warp subtracts
// L_IK X_K (one m16n8k16 instruction, its fragment of L loaded one step ahead).
// Measured (both launches; one CTA per block before): 480 -> 42 us for two 128
// blocks (n = 256), 500 -> 69 us for 32 (n = 4096).
constexpr int TI_NB = 16, TI_COLS = 8, TI_WARPS = kMaxBlock / TI_NB;

__device__ __forceinline__ void dmma_16816(double (&c)[4], const double (&a)[8], const double (&b)[4]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, "
      "{%4,%5,%6,%7,%8,%9,%10,%11}, {%12,%13,%14,%15}, {%0,%1,%2,%3};\n"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(a[4]), "d"(a[5]), "d"(a[6]), "d"(a[7]),
        "d"(b[0]), "d"(b[1]), "d"(b[2]), "d"(b[3]));
}

struct TriBatch {  // grid.z members (zero: one)
  const int *n;
  int ib;
  long long sL, so;
};
// Rows of block ib of a member of order n: the rest of its 128 is the identity.
__device__ __forceinline__ int member_rows(const int *n, int z, int ib) { return min(kMaxBlock, __ldg(n + z) - ib * kMaxBlock); }
struct TriBlock {
  int j0, nb;
  double *dst;
  long long ldd;
};
__device__ __forceinline__ TriBlock tri_block(int ib, int n, int first, int b, double *out, long long ldo) {
  TriBlock t;
  t.j0 = (ib == 0) ? 0 : first + (ib - 1) * b;
  t.nb = (ib == 0) ? first : min(b, n - t.j0);
  t.dst = ldo ? out + (long long)t.j0 * ldo + t.j0 : out + (size_t)ib * b * b;
  t.ldd = ldo ? ldo : t.nb;
  return t;
}

// grid.x blocks, grid.y sub-blocks of a block in twos (64 threads)
__global__ void __launch_bounds__(64)
trtri16_kernel(int n, const double *L, long long ldl, int first, int b, double *out, long long ldo, TriBatch q) {
  if (q.n) n = first = member_rows(q.n, blockIdx.z, q.ib);
  if (n <= 0) return;
  L += blockIdx.z * q.sL;
  out += blockIdx.z * q.so;
  __shared__ double sub_s[2][TI_NB][TI_NB + 1];
  const TriBlock t = tri_block(blockIdx.x, n, first, b, out, ldo);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, r0 = (2 * blockIdx.y + w) * TI_NB;
  if (r0 >= t.nb) return;
  double(*sub)[TI_NB + 1] = sub_s[w];
  const double *A = L + (long long)(t.j0 + r0) * ldl + t.j0 + r0;
  const int m = min(TI_NB, t.nb - r0);
#pragma unroll
  for (int q = 0; q < 8; ++q) {  // padded with the identity
    const int i = 2 * q + (lane >> 4), j = lane & 15;
    sub[i][j] = (i < m && j <= i) ? A[(long long)i * ldl + j] : (i == j ? 1.0 : 0.0);
  }
  __syncwarp();
  const int j = lane & 15, h = lane >> 4;
  double x[8], rd[TI_NB];
  const double d = 1.0 / sub[j][j];
#pragma unroll
  for (int k = 0; k < TI_NB; ++k) rd[k] = __shfl_sync(0xffffffffu, d, k);
#pragma unroll
  for (int u = 0; u < 8; ++u) x[u] = (2 * u + h == j) ? 1.0 : 0.0;
#pragma unroll
  for (int k = 0; k < TI_NB; ++k) {
    const double xk = __shfl_sync(0xffffffffu, x[k >> 1], j | ((k & 1) << 4)) * rd[k];
    if (h == (k & 1)) x[k >> 1] = xk;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (2 * u + 1 <= k) continue;
      const int i = 2 * u + h;
      if (i > k) x[u] = fma(-sub[i][k], xk, x[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = 2 * u + h;
    if (i < m && j < m) t.dst[(long long)(r0 + i) * t.ldd + r0 + j] = (i >= j) ? x[u] : 0.0;
  }
}

__global__ void __launch_bounds__(32 * TI_WARPS, 2)
trtri_cols_kernel(int n, const double *L, long long ldl, int first, int b, double *out, long long ldo, TriBatch q) {
  if (q.n) n = first = member_rows(q.n, blockIdx.z, q.ib);
  if (n <= 0) return;
  L += blockIdx.z * q.sL;
  out += blockIdx.z * q.so;
  __shared__ double dinv[TI_WARPS][TI_NB][TI_NB + 1];
  __shared__ double rhs[TI_NB][TI_COLS + 1];
  __shared__ double xs[TI_WARPS][TI_NB][TI_COLS + 1];
  const TriBlock t = tri_block(blockIdx.x, n, first, b, out, ldo);
  const int nb = t.nb, c0 = blockIdx.y * TI_COLS;
  const double *A = L + (long long)t.j0 * ldl + t.j0;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
  const int k0 = c0 / TI_NB, r0 = w * TI_NB;  // first row block with entries; this warp's rows
  const bool live = w >= k0 && r0 < nb && c0 < nb;
  if (live) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = 2 * q + (lane >> 4), j = lane & 15;
      dinv[w][i][j] = (r0 + i < nb && r0 + j < nb) ? t.dst[(long long)(r0 + i) * t.ldd + r0 + j] : (i == j ? 1.0 : 0.0);
    }
  }
  auto load = [&](int K, double(&a)[8]) {  // L_wK as an A fragment
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = r0 + g + 8 * (i & 1), col = K * TI_NB + tg + 4 * (i >> 1);
      a[i] = row < nb ? A[(long long)row * ldl + col] : 0.0;
    }
  };
  double a[8];
  if (live && w > k0) load(k0, a);
  double acc[4] = {0.0, 0.0, 0.0, 0.0};  // rows g, g + 8; columns 2 tg, 2 tg + 1
  __syncthreads();
  const int last = c0 < nb ? (nb - 1) / TI_NB : k0 - 1;
  for (int K = k0; K <= last; ++K) {
    if (w == K) {  // the identity's columns c0 .. c0 + 7 minus the products so far
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int row = g + ((r >> 1) << 3), col = 2 * tg + (r & 1);
        rhs[row][col] = ((r0 + row == c0 + col) ? 1.0 : 0.0) - acc[r];
      }
    }
    __syncthreads();
    if (threadIdx.x < TI_NB * TI_COLS) {
      const int r = threadIdx.x >> 3, c = threadIdx.x & 7;
      double p[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int q = 0; q < TI_NB; ++q) p[q & 3] = fma(dinv[K][r][q], rhs[q][c], p[q & 3]);
      xs[K][r][c] = (p[0] + p[1]) + (p[2] + p[3]);
    }
    __syncthreads();
    if (live && w > K) {
      double bb[4], an[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) bb[i] = xs[K][tg + 4 * i][g];
      if (K + 1 < w) load(K + 1, an);
      dmma_16816(acc, a, bb);
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = an[i];
    }
  }
  // every CTA of the block's cluster has read L (a cluster of one unless out is L)
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  for (int idx = threadIdx.x; idx < nb * TI_COLS; idx += blockDim.x) {
    const int i = idx >> 3, c = idx & 7;
    // the diagonal sub-blocks are in place already
    if (c0 + c < nb && i >> 4 != k0) t.dst[(long long)i * t.ldd + c0 + c] = (i >> 4 > k0) ? xs[i >> 4][i & 15][c] : 0.0;
  }
  if (q.n)  // the identity past the member's order
    for (int idx = threadIdx.x; idx < kMaxBlock * TI_COLS; idx += blockDim.x) {
      const int i = idx >> 3, c = c0 + (idx & 7);
      if (i >= nb || c >= nb) t.dst[(long long)i * t.ldd + c] = i == c ? 1.0 : 0.0;
    }
}

// The mixed path's diagonal-block inverses (block ib at out + ib b^2, leading
// dimension its size), one CTA per block, in place in shared memory by a backward
// column sweep: with L = [[l, 0], [x, L2]],
// L^{-1} = [[1/l, 0], [-L2^{-1} x / l, L2^{-1}]], every entry one chain of
// multiply-adds.  Kept for its order of operations, as potrf_lookahead_kernel
// below (480 us a launch against 42 to 69 of the kernels above).
__global__ void __launch_bounds__(256)
trtri_sweep_kernel(int n, const double *L, long long ldl, int first, int b, double *out) {
  extern __shared__ double sm[];
  __shared__ double col[kMaxBlock];
  const TriBlock t = tri_block(blockIdx.x, n, first, b, out, 0);
  const int nb = t.nb, ld = nb + 1;
  const double *A = L + (long long)t.j0 * ldl + t.j0;
  for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
    const int i = idx / nb, j = idx - i * nb;
    sm[i * ld + j] = (j <= i) ? A[(long long)i * ldl + j] : 0.0;
  }
  __syncthreads();
  for (int j = nb - 1; j >= 0; --j) {
    const double ljj = sm[j * ld + j];
    for (int i = j + 1 + threadIdx.x; i < nb; i += blockDim.x) {
      double v = 0.0;
      for (int k = j + 1; k <= i; ++k) v = fma(sm[i * ld + k], sm[k * ld + j], v);
      col[i] = -v / ljj;
    }
    __syncthreads();
    for (int i = j + 1 + threadIdx.x; i < nb; i += blockDim.x) sm[i * ld + j] = col[i];
    if (threadIdx.x == 0) sm[j * ld + j] = 1.0 / ljj;
    __syncthreads();
  }
  for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
    const int i = idx / nb, j = idx - i * nb;
    t.dst[(long long)i * t.ldd + j] = (j <= i) ? sm[i * ld + j] : 0.0;
  }
}

// An FP64 entry, or a double-float one (FP32 hi + lo in the same 8 bytes) when df.
__device__ __forceinline__ double load_entry(const double *p, int df) {
  if (df) {
    const float2 v = *reinterpret_cast<const float2 *>(p);
    return exact_f64(v.x) + exact_f64(v.y);
  }
  return *p;
}

// Cholesky factor of one nb x nb diagonal block, nb <= NB (the small-block step
// of Section 3.3), in panels of 8 columns without square roots: A = X D^-1 X^T
// with X = L sqrt(D), so the chain from pivot to pivot is one reciprocal, one
// multiply and one multiply-add, and all square roots are taken at the end.
// FP64 instructions are what counts here: each holds its sub-partition's FP64
// pipe for 64 cycles whatever its active lanes, and a dependent one follows after
// 67.  Per panel p:
//   1. warp 0 factors the 8 x 8 diagonal tile (lane = row and column mod 4: at
//      most six FP64 instructions per column, three of them the reciprocal);
//      meanwhile the other warps, which hold the trailing 8 x 8 tiles in registers
//      (two entries per lane, dealt in column order), apply panel p-1 to theirs,
//      the tiles of column p first, which they store;
//   2. every warp solves 16 of the rows below (two lanes per row, 20 FP64
//      instructions) and stores them as X and as W = X D^-1;
//   3. the next diagonal tile takes its update -X W^T and is stored.
// Three barriers per panel.  The trailing updates are plain multiply-adds: the
// tensor instruction m8n8k4 takes 611 cycles against 512 for the same 256 of
// them, and takes them even when its predicate is off.  Writes L11 in place with the upper part of the block
// zeroed; the first failing pivot is recorded in info (GPC_ERR_NOT_PD, or
// GPC_ERR_NAN for NaN/Inf) and the rest of the block is written back unfinished.
// Measured: 64 rows 74 -> 51 us against a column-by-column lookahead with one
// pivot warp (square roots and two row halves on the chain), 128 rows 250 -> 170.
// 1/x within 2 ulp for x and 1/x normal: the hardware seed and one third-order
// Householder step for the reciprocal, y (1 + e + e^2) with e = 1 - x y (pinned
// beside the other refinements by gpc_test_recip_cubic's test).
__device__ __forceinline__ double recip_cubic(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// Positive and normal with a normal reciprocal (x < 2^1022), by the high word (a
// comparison of FP64 values would take the FP64 pipe).
__device__ __forceinline__ bool plain_pivot(double x) {
  return (unsigned)(__double2hiint(x) - 0x00100000) < 0x7FC00000u;
}

constexpr int kPotrfW = 12;  // row of W: 8 entries, padded against bank conflicts
template <int NB>
constexpr size_t potrf_smem() {
  return ((size_t)NB * (NB + 4) + (size_t)NB * kPotrfW + 8 * 9 + NB) * sizeof(double);
}

template <int NB>
__device__ __forceinline__ void potrf_block(int nb, double *A, long long lda, int *info, int pivot_offset) {
  constexpr int LD = NB + 4, NT = NB / 8, NW = NB / 16, OWN = NW - 1, TILES = NT * (NT - 1) / 2,
                SLOTS = (TILES + OWN - 1) / OWN;
  extern __shared__ double sm[];
  double *M = sm, *W = sm + NB * LD, *Wd = W + NB * kPotrfW, *pinv_s = Wd + 8 * 9;
  __shared__ int fail;  // failing column, or NB
  // Pivots beyond plain_pivot: 1/d is pinv sc sc, sc a power of two applied in two
  // steps, since 1/d itself would overflow (denormal pivots) or lose its digits.
  __shared__ double sc_s[NB];
  __shared__ int scaled;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tr = lane >> 2, tc = lane & 3;  // row and column pair of an 8 x 8 tile
  if (threadIdx.x == 0) {
    fail = NB;
    scaled = 0;
  }
  if (threadIdx.x < NB) sc_s[threadIdx.x] = 1.0;
#pragma unroll 16
  for (int idx = threadIdx.x; idx < NB * NB; idx += 32 * NW) {
    const int r = idx / NB, c = idx - r * NB;  // rows past nb: the identity
    M[r * LD + c] = (r < nb && c < nb) ? (c <= r ? A[(long long)r * lda + c] : 0.0) : (r == c ? 1.0 : 0.0);
  }
  __syncthreads();
  // tiles (ti, tk), 1 <= tk <= ti, in column order: slot s of owner o = w - 1 is number s OWN + o
  double acc[SLOTS][2];
  int ti[SLOTS], tk[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    int t = s * OWN + w - 1, k = 1;
    if (w == 0 || t >= TILES) {
      ti[s] = tk[s] = -1;
      continue;
    }
    while (t >= NT - k) t -= NT - k++;
    tk[s] = k;
    ti[s] = k + t;
    const double *src = M + (8 * ti[s] + tr) * LD + 8 * k + 2 * tc;
    acc[s][0] = src[0];
    acc[s][1] = src[1];
  }
  auto update = [&](int s, int p) {  // tile s -= X W^T of panel p
    const double *x = M + (8 * ti[s] + tr) * LD + 8 * p, *v = W + (8 * tk[s] + 2 * tc) * kPotrfW;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      acc[s][0] = fma(-x[q], v[q], acc[s][0]);
      acc[s][1] = fma(-x[q], v[kPotrfW + q], acc[s][1]);
    }
  };
  auto store = [&](int s) {
    double *dst = M + (8 * ti[s] + tr) * LD + 8 * tk[s] + 2 * tc;
    dst[0] = acc[s][0];
    dst[1] = acc[s][1];
  };
  const int np = (nb + 7) / 8;
  for (int p = 0; p < np; ++p) {
    if (w == 0) {
      const int i = tr, q = tc;
      double *D = M + (8 * p + i) * LD + 8 * p + q;
      double a0 = D[0], a1 = D[4];
      bool ok = true;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double aj = j < 4 ? a0 : a1;
        const double d = __shfl_sync(0xffffffffu, aj, j * 4 + (j & 3));
        const bool fine = plain_pivot(d);
        if (ok && !fine && !(d > 0.0 && d <= 1.79769313486231570e308)) {
          ok = false;
          if (lane == 0) {
            fail = 8 * p + j;
            if (info && info[1] == 0) {
              info[0] = pivot_offset + 8 * p + j;
              info[1] = (d != d || d > 1.79769313486231570e308) ? GPC_ERR_NAN : GPC_ERR_NOT_PD;
            }
          }
        }
        if (!ok) continue;
        const double aij = __shfl_sync(0xffffffffu, aj, (lane & ~3) | (j & 3));
        const double k0 = __shfl_sync(0xffffffffu, aj, q * 4 + (j & 3));
        const double k1 = __shfl_sync(0xffffffffu, aj, (q + 4) * 4 + (j & 3));
        double pinv, t;
        if (fine) {
          pinv = recip_cubic(d);
          t = aij * pinv;
        } else {
          const double sc = d < 1.0 ? 0x1p270 : 0x1p-270;
          pinv = 1.0 / (d * sc * sc);
          t = aij * sc * pinv * sc;
          if (lane == 0) {
            sc_s[8 * p + j] = sc;
            scaled = 1;
          }
        }
        if (j < 3 && q > j) a0 = fma(-t, k0, a0);
        if (j < 7 && q + 4 > j) a1 = fma(-t, k1, a1);
        if (q == (j & 3)) Wd[i * 9 + j] = t;
        if (lane == 0) pinv_s[8 * p + j] = pinv;
      }
      D[0] = a0;
      D[4] = a1;
    } else if (p > 0) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (tk[s] == p && ti[s] > p) {
          update(s, p - 1);
          store(s);
        }
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (tk[s] > p) update(s, p - 1);
    }
    __syncthreads();
    if (fail < NB || p == np - 1) break;
    const int row = 8 * (p + 1) + 16 * w + (lane >> 1), h = lane & 1;
    if (8 * (p + 1) + 16 * w < NB) {
      double *xr = M + (row < NB ? row : NB - 1) * LD + 8 * p + h;
      double x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = xr[2 * u];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double xj = __shfl_sync(0xffffffffu, x[j >> 1], (lane & ~1) | (j & 1));
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (2 * u + 1 <= j) continue;
          if (2 * u + h > j) x[u] = fma(-xj, Wd[(2 * u + h) * 9 + j], x[u]);
        }
      }
      if (row < NB) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          xr[2 * u] = x[u];
          const int c = 8 * p + 2 * u + h;
          W[row * kPotrfW + 2 * u + h] = scaled ? x[u] * sc_s[c] * pinv_s[c] * sc_s[c] : x[u] * pinv_s[c];
        }
      }
    }
    __syncthreads();
    if (w > 0) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (tk[s] == p + 1 && ti[s] == p + 1) {
          update(s, p);
          store(s);
        }
    }
    __syncthreads();
  }
  // L = X D^-1/2; the diagonal holds D
  const int last = fail;
  double *rs = W;
  __syncthreads();
  if (threadIdx.x < NB) rs[threadIdx.x] = threadIdx.x < last ? rsqrt_nr(M[threadIdx.x * (LD + 1)]) : 1.0;
  __syncthreads();
#pragma unroll 8
  for (int idx = threadIdx.x; idx < NB * NB; idx += 32 * NW) {
    const int r = idx / NB, c = idx - r * NB;
    if (r < nb && c < nb) A[(long long)r * lda + c] = (c <= r) ? M[r * LD + c] * rs[c] : 0.0;
  }
}

// Blocks of up to 64 rows.
__global__ void __launch_bounds__(128)
potrf_la_kernel(int nb, double *A, long long lda, int *info, int pivot_offset) {
  potrf_block<64>(nb, A, lda, info, pivot_offset);
}
// Blocks of 65 to 128 rows.
__global__ void __launch_bounds__(256)
potrf_diag_kernel(int nb, double *A, long long lda, int *info, int pivot_offset) {
  potrf_block<128>(nb, A, lda, info, pivot_offset);
}

// Whole 128 blocks, one per member (grid.x).
__global__ void __launch_bounds__(256)
potrf_batch_kernel(double *A, long long lda, long long sA, const int *n, int ib, const int *order, int *info) {
  const int z = blockIdx.x, nb = member_rows(n, z, ib);
  if (nb <= 0) return;
  potrf_block<128>(nb, A + z * sA, lda, info + 2 * __ldg(order + z), ib * 128);
}

// The factor of a diagonal block in double-float storage, nb <= 64 (the mixed
// path's), with a one-column lookahead.  Column k+1 is finished (pivot, 1/sqrt,
// scaling) by one warp while six other warps apply column k to the rest of the
// block:
//   * warp 0 (the pivot warp): for column k+1 it applies the column-k update
//     itself, takes r = 1/sqrt(pivot), writes the final column to shared memory
//     and publishes col_ready = k+1;
//   * warps 1-3 and 5-7 (the updaters, u = 0..5) own whole columns j = u mod 6,
//     lane l holding rows j + l and j + l + 32 in registers; at step k, once
//     column k is final, the owner of column k+2 updates and stores it first and
//     marks rounds[k+1], then every warp updates its later columns (rounds[0]:
//     columns 0 and 1 stored as loaded, one mark per warp);
//   * warp 4 idles, so the pivot warp has its SM sub-partition to itself.
// Every wait is a bounded spin on a shared-memory word; a wait that runs out
// records GPC_ERR_TIMEOUT and stops the block.
//
// The mixed path keeps this order of operations although potrf_block is faster
// (74 against 51 us for 64 rows).  Its products keep 40 bits, so a last-bit change
// of a factor's entry decides anew how the entries that follow are rounded, and
// the hyperparameter gradient, whose sums cancel to 1/60 and less, moves by its
// own error: by 7e-9 of its size at n = 16384 in one draw, where callers compare
// runs to 1e-9.
constexpr int PL_NB = 64, PL_LD = PL_NB + 1, PL_W = 6, PL_COLS = (PL_NB + PL_W - 1) / PL_W;
constexpr long long PL_SPIN = 1LL << 24;

__global__ void __launch_bounds__(256)
potrf_lookahead_kernel(int nb, double *A, long long lda, int *info, int pivot_offset, int *gerr) {
  __shared__ double M[PL_NB * PL_LD];
  __shared__ int col_ready, stop;
  __shared__ int rounds[PL_NB];  // rounds[r]: marks of round r
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    col_ready = -1;
    stop = 0;
  }
  if (threadIdx.x < PL_NB) rounds[threadIdx.x] = 0;
  const bool updater = warp != 0 && warp != 4;
  const int uw = updater ? warp - 1 - (warp > 4) : 0;
  double a0[PL_COLS], a1[PL_COLS];  // column uw + 6 c: rows j + lane, j + lane + 32
  if (updater) {
#pragma unroll
    for (int c = 0; c < PL_COLS; ++c) {
      const int j = uw + PL_W * c, r0 = j + lane, r1 = r0 + 32;
      a0[c] = (j < nb && r0 < nb) ? load_entry(A + (long long)r0 * lda + j, 1) : 0.0;
      a1[c] = (j < nb && r1 < nb) ? load_entry(A + (long long)r1 * lda + j, 1) : 0.0;
    }
  }
  __syncthreads();
  volatile int *vready = &col_ready, *vstop = &stop;
  // Polls: the updaters back off between polls, so that their loads do not
  // queue in front of the pivot warp's shared-memory accesses.
  auto spin_ge = [&](volatile int *w, int target) -> bool {
    for (long long it = 0; it < PL_SPIN; ++it) {
      if (*w >= target) return true;
      if (*vstop) return false;
      if (updater) __nanosleep(64);
    }
    return false;
  };
  auto give_up = [&]() {  // a wait ran out: report and stop the block
    if (info && info[1] == 0) info[1] = GPC_ERR_TIMEOUT;
    record_error(gerr, GPC_ERR_TIMEOUT);
    *vstop = 1;
  };
  if (updater) {
    // round 0: columns 0 and 1 as loaded (owned by updaters 0 and 1)
    if (uw <= 1 && uw < nb) {
      const int j = uw, r0 = j + lane, r1 = r0 + 32;
      if (r0 < nb) M[r0 * PL_LD + j] = a0[0];
      if (r1 < nb) M[r1 * PL_LD + j] = a1[0];
    }
    __threadfence_block();
    __syncwarp();
    if (lane == 0) atomicAdd(&rounds[0], 1);
  }
  if (warp == 0) {
    // ---- pivot warp: lanes own rows lane and lane + 32
    for (int c = 0; c < nb; ++c) {
      // column c comes from round max(c - 1, 0)
      if (!spin_ge((volatile int *)&rounds[max(c - 1, 0)], c <= 1 ? PL_W : 1)) {
        if (!*vstop && lane == 0) give_up();
        break;
      }
      __threadfence_block();
      const int i0 = lane, i1 = lane + 32;
      double v0 = (i0 >= c && i0 < nb) ? M[i0 * PL_LD + c] : 0.0;
      double v1 = (i1 >= c && i1 < nb) ? M[i1 * PL_LD + c] : 0.0;
      if (c > 0) {  // the update by column c - 1, finished by this warp just before
        const double lc = M[c * PL_LD + c - 1];
        if (i0 >= c && i0 < nb) v0 = fma(-M[i0 * PL_LD + c - 1], lc, v0);
        if (i1 >= c && i1 < nb) v1 = fma(-M[i1 * PL_LD + c - 1], lc, v1);
      }
      const double pv = (c < 32) ? __shfl_sync(0xffffffffu, v0, c) : __shfl_sync(0xffffffffu, v1, c - 32);
      if (!(pv > 0.0 && pv <= 1.79769313486231570e308)) {
        if (lane == 0) {
          if (info && info[1] == 0) {
            info[0] = pivot_offset + c;
            info[1] = (pv != pv || pv > 1.79769313486231570e308) ? GPC_ERR_NAN : GPC_ERR_NOT_PD;
          }
          *vstop = 1;
        }
        break;
      }
      const double r = rsqrt_nr(pv);  // every lane: no broadcast on the chain
      if (i0 >= c && i0 < nb) M[i0 * PL_LD + c] = (i0 == c) ? pv * r : v0 * r;
      if (i1 >= c && i1 < nb) M[i1 * PL_LD + c] = (i1 == c) ? pv * r : v1 * r;
      __threadfence_block();
      __syncwarp();
      if (lane == 0) *vready = c;
    }
  } else if (updater) {
    // ---- updaters: step k applies column k to columns k + 2 .. nb - 1
    for (int k = 0; k + 2 < nb; ++k) {
      if (!spin_ge(vready, k)) {
        if (!*vstop && lane == 0) give_up();
        break;
      }
      __threadfence_block();
#pragma unroll
      for (int c = 0; c < PL_COLS; ++c) {
        const int j = uw + PL_W * c;
        if (j == k + 2) {  // warp-uniform: the column the pivot warp needs next
          const double ljk = M[j * PL_LD + k];
          const int r0 = j + lane, r1 = r0 + 32;
          if (r0 < nb) {
            a0[c] = fma(-M[r0 * PL_LD + k], ljk, a0[c]);
            M[r0 * PL_LD + j] = a0[c];
          }
          if (r1 < nb) {
            a1[c] = fma(-M[r1 * PL_LD + k], ljk, a1[c]);
            M[r1 * PL_LD + j] = a1[c];
          }
          __threadfence_block();
          __syncwarp();
          if (lane == 0) atomicAdd(&rounds[k + 1], 1);
        }
      }
#pragma unroll
      for (int c = 0; c < PL_COLS; ++c) {
        const int j = uw + PL_W * c;
        if (j > k + 2 && j < nb) {  // warp-uniform
          const double ljk = M[j * PL_LD + k];
          const int r0 = j + lane, r1 = r0 + 32;
          if (r0 < nb) a0[c] = fma(-M[r0 * PL_LD + k], ljk, a0[c]);
          if (j + 32 < nb && r1 < nb) a1[c] = fma(-M[r1 * PL_LD + k], ljk, a1[c]);
        }
      }
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
    const int r = idx / nb, c = idx - r * nb;
    A[(long long)r * lda + c] = (c <= r) ? M[r * PL_LD + c] : 0.0;
  }
}

// Row-parallel triangular solve of an m x nb panel X (in place) against the
// nb x nb lower block T (Section 3.3's panel step, by substitution instead of
// a product with the inverse):
//   mode 0: X <- X T^{-T}  (forward panel L21 = A21 L11^{-T}; columns ascending)
//   mode 1: X <- X T^{-1}  (adjoint panel Cbar D^{-1}; columns descending)
// One CTA per ROWS rows, the rows in shared memory; T is read through L1.
// Thread (r, g) owns the columns k = g (mod 256 / ROWS) of row r; the owner of
// the next column scales it right after its last update, so one barrier per
// column suffices.  Fewer rows per CTA for short panels keep every SM busy.
template <int ROWS>
__global__ void __launch_bounds__(256)
trsm_rows_kernel(int m, int nb, double *X, long long ldx, const double *T, long long ldt, int mode, int df) {
  constexpr int CG = 256 / ROWS;
  __shared__ double xs[ROWS][kMaxBlock + 1];
  __shared__ double rdiag[kMaxBlock];
  const int r0 = blockIdx.x * ROWS, rows = min(ROWS, m - r0);
  for (int idx = threadIdx.x; idx < ROWS * nb; idx += blockDim.x) {
    const int r = idx / nb, c = idx - r * nb;
    xs[r][c] = (r < rows) ? load_entry(X + (long long)(r0 + r) * ldx + c, df) : 0.0;
  }
  for (int j = threadIdx.x; j < nb; j += blockDim.x) rdiag[j] = 1.0 / __ldg(&T[(long long)j * ldt + j]);
  __syncthreads();
  const int r = threadIdx.x % ROWS, cg = threadIdx.x / ROWS;
  const int jfirst = mode == 0 ? 0 : nb - 1;
  if (cg == jfirst % CG) xs[r][jfirst] *= rdiag[jfirst];
  __syncthreads();
  for (int step = 0; step < nb; ++step) {
    const int j = mode == 0 ? step : nb - 1 - step;
    const double xj = xs[r][j];
    if (mode == 0) {
      int k = j + 1 + ((cg - (j + 1)) % CG + CG) % CG;
      if (k == j + 1 && k < nb) {  // the next column: last update, then scale
        xs[r][k] = fma(-xj, __ldg(&T[(long long)k * ldt + j]), xs[r][k]) * rdiag[k];
        k += CG;
      }
      for (; k < nb; k += CG) xs[r][k] = fma(-xj, __ldg(&T[(long long)k * ldt + j]), xs[r][k]);
    } else {
      const int kl = j - 1;
      for (int k = cg; k < kl; k += CG) xs[r][k] = fma(-xj, __ldg(&T[(long long)j * ldt + k]), xs[r][k]);
      if (kl >= 0 && kl % CG == cg)
        xs[r][kl] = fma(-xj, __ldg(&T[(long long)j * ldt + kl]), xs[r][kl]) * rdiag[kl];
    }
    __syncthreads();
  }
  for (int idx = threadIdx.x; idx < ROWS * nb; idx += blockDim.x) {
    const int rr = idx / nb, c = idx - rr * nb;
    if (rr < rows) X[(long long)(r0 + rr) * ldx + c] = xs[rr][c];
  }
}

// The same panel solve with TPR threads per row (4 or 16 by panel height)
// and no block barriers, for the block sizes the factorisations use (NB = 64
// or 128).  Thread t of a row holds columns k = TPR c + t (c < NB / TPR) in
// registers; at step j the owner of column j (final by then) passes it to the
// row's other threads with a warp shuffle, every thread updates its columns
// still to be solved, and the owner of the next column scales it.  Columns
// are dealt round-robin so the shrinking work stays balanced; the loops are
// unrolled at compile time so the row stays in registers.  The FP64 pipe, not
// synchronisation, bounds it: one FP64 warp instruction holds a sub-partition's
// FP64 unit for about 64 cycles, so a short panel (the 64 x 64 solve of a
// diagonal block's halves) is spread over 16 threads per row and more warps.
// Every element sees the same operations in the same order for any TPR.
constexpr int TQ_THREADS = 64;  // 16 rows per CTA at TPR = 4: enough CTAs that every SM gets an even share
template <int NB, int MODE, int TPR>
__global__ void __launch_bounds__(TQ_THREADS)
trsm_quad_kernel(int m, double *X, long long ldx, const double *T, long long ldt, int df) {
  constexpr int C = NB / TPR;
  __shared__ double rdiag[NB];
  for (int k = threadIdx.x; k < NB; k += blockDim.x) rdiag[k] = 1.0 / __ldg(&T[(long long)k * ldt + k]);
  __syncthreads();
  const int lane = threadIdx.x & 31, t = lane & (TPR - 1), src0 = lane & ~(TPR - 1);
  const int row = blockIdx.x * (TQ_THREADS / TPR) + (threadIdx.x / TPR);
  const bool live = row < m;
  double *xr = X + (long long)(live ? row : 0) * ldx;
  double x[C];
#pragma unroll
  for (int c = 0; c < C; ++c) x[c] = live ? load_entry(xr + TPR * c + t, df) : 0.0;
  if (MODE == 0) {  // X <- X T^{-T}: columns ascending, x_k -= x_j T[k][j] for k > j
    if (t == 0) x[0] *= rdiag[0];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const double xj = __shfl_sync(0xffffffffu, x[j / TPR], src0 | (j % TPR));
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (TPR * c + TPR - 1 <= j) continue;  // every column of this group is already final
        const int k = TPR * c + t;
        const double tv = __ldg(&T[(long long)k * ldt + j]);
        if (TPR * c > j || k > j) x[c] = fma(-xj, tv, x[c]);
      }
      if (j + 1 < NB && t == ((j + 1) % TPR)) x[(j + 1) / TPR] *= rdiag[j + 1];
    }
  } else {  // X <- X T^{-1}: columns descending, x_k -= x_j T[j][k] for k < j
    if (t == ((NB - 1) % TPR)) x[C - 1] *= rdiag[NB - 1];
#pragma unroll
    for (int j = NB - 1; j >= 0; --j) {
      const double xj = __shfl_sync(0xffffffffu, x[j / TPR], src0 | (j % TPR));
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (TPR * c >= j) continue;  // every column of this group is at or past j
        const int k = TPR * c + t;
        const double tv = __ldg(&T[(long long)j * ldt + k]);
        if (TPR * c + TPR - 1 < j || k < j) x[c] = fma(-xj, tv, x[c]);
      }
      if (j > 0 && t == ((j - 1) % TPR)) x[(j - 1) / TPR] *= rdiag[j - 1];
    }
  }
  if (live) {
#pragma unroll
    for (int c = 0; c < C; ++c) xr[TPR * c + t] = x[c];
  }
}

// emax (null, or zero on entry): the largest biased exponent of the lower triangle.
__global__ void __launch_bounds__(256)
copy_lower_kernel(int n, const double *src, long long lds, double *dst, long long ldd, int *emax) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (idx < (long long)n * n) {
    const int i = (int)(idx / n), j = (int)(idx - (long long)i * n);
    if (j <= i) v = src[(long long)i * lds + j];
    dst[(long long)i * ldd + j] = v;
  }
  if (!emax) return;
  __shared__ int es[8];  // one look at *emax per CTA: one per warp cost 0.2 ms at n = 6007
  const int e = __reduce_max_sync(0xffffffffu, (__double2hiint(v) >> 20) & 0x7FF);
  if ((threadIdx.x & 31) == 0) es[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x != 0) return;
  int m = es[0];
  for (int w = 1; w < 8; ++w) m = max(m, es[w]);
  if (m > *(volatile int *)emax) atomicMax(emax, m);
}

// The lower triangle times 2^shift where *emax is below kTinyExponent; otherwise nothing.
constexpr int kTinyExponent = 123;  // 2^-900
__global__ void __launch_bounds__(256)
rescale_tiny_kernel(int n, double *A, long long lda, int shift, const int *emax) {
  if (*emax >= kTinyExponent) return;
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = threadIdx.x; j <= i; j += 256) A[(long long)i * lda + j] = scalbn(A[(long long)i * lda + j], shift);
}

__global__ void copy_rect_kernel(int m, int c, const double *src, long long lds, double *dst,
                                 long long ldd) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)m * c) return;
  const int i = (int)(idx / c), j = (int)(idx - (long long)i * c);
  dst[(long long)i * ldd + j] = src[(long long)i * lds + j];
}

__global__ void phi_block_kernel(int nb, double *A, long long lda) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nb * nb) return;
  const int i = idx / nb, j = idx - i * nb;
  double *p = A + (long long)i * lda + j;
  if (j > i) *p = 0.0;
  else if (j == i) *p *= 0.5;
}

__global__ void lower_to_symmetric_half_kernel(int n, double *A, long long lda) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * n) return;
  const int i = (int)(idx / n), j = (int)(idx - (long long)i * n);
  if (j >= i) return;
  const double v = 0.5 * A[(long long)i * lda + j];
  A[(long long)i * lda + j] = v;
  A[(long long)j * lda + i] = v;
}

__global__ void reset_info_kernel(int *info) {
  info[0] = -1;
  info[1] = GPC_OK;
}

// Test hook: the pivots' reciprocals.
__global__ void recip_cubic_probe_kernel(int n, const double *x, double *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = recip_cubic(x[i]);
}

unsigned blocks_for(long long total, int threads) { return (unsigned)((total + threads - 1) / threads); }

// Test hook: the refined reciprocals next to CUDA's own 1.0 / x and rsqrt(x).
__global__ void recip_rsqrt_probe_kernel(int n, const double *x, double *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  out[4 * i + 0] = recip_nr(v);
  out[4 * i + 1] = 1.0 / v;
  out[4 * i + 2] = rsqrt_nr(v);
  out[4 * i + 3] = rsqrt(v);
}

}  // namespace

cudaError_t trtri_batched(int n, const double *L, long long ldl, int first, int b, double *out,
                          cudaStream_t s, long long ldo) {
  if (n <= 0) return cudaSuccess;
  if (b > kMaxBlock || first < 1 || first > b) return cudaErrorInvalidValue;
  const int nblk = 1 + (n - first + b - 1) / b;
  const bool in_place = (const double *)out == L;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nblk, (unsigned)((b + TI_COLS - 1) / TI_COLS));
  cfg.blockDim = dim3(32 * TI_WARPS);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (in_place) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {  // up to 16 CTAs per cluster
      cudaError_t e = cudaFuncSetAttribute(trtri_cols_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
      attr_set[dev] = true;
    }
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = cfg.gridDim.y;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  GPC_LAUNCH(GPC_TRACE_DIAG, (double)n * TI_NB * TI_NB / 3.0, 16.0 * (double)n * TI_NB, s,
             trtri16_kernel<<<dim3((unsigned)nblk, (unsigned)((b + 31) / 32)), 64, 0, s>>>(n, L, ldl, first, b, out, ldo,
                                                                                                 TriBatch{}));
  if (b <= TI_NB) return cudaGetLastError();
  cudaError_t le = cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_DIAG, (double)n * b * b / 3.0, 16.0 * (double)n * b, s,
             le = cudaLaunchKernelEx(&cfg, trtri_cols_kernel, n, L, ldl, first, b, out, ldo, TriBatch{}));
  return le;
}

cudaError_t trtri_sweep(int n, const double *L, long long ldl, int first, int b, double *out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (b > kMaxBlock || first < 1 || first > b) return cudaErrorInvalidValue;
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(trtri_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)((size_t)kMaxBlock * (kMaxBlock + 1) * sizeof(double)));
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  const int nblk = 1 + (n - first + b - 1) / b;
  const size_t smem = (size_t)b * (b + 1) * sizeof(double);
  GPC_LAUNCH(GPC_TRACE_DIAG, (double)n * b * b / 3.0, 16.0 * (double)n * b, s,
             trtri_sweep_kernel<<<nblk, 256, smem, s>>>(n, L, ldl, first, b, out));
  return cudaGetLastError();
}

cudaError_t potrf_diag(int nb, double *A, long long lda, int *info, int pivot_offset, cudaStream_t s, bool df) {
  if (nb <= 0) return cudaSuccess;
  if (nb > (df ? PL_NB : kMaxBlock)) return cudaErrorInvalidValue;
  if (df) {
    GPC_LAUNCH(GPC_TRACE_DIAG, (double)nb * nb * nb / 3.0, 16.0 * nb * nb, s,
               launch_k(potrf_lookahead_kernel, 1, 256, 0, s, nb, A, lda, info, pivot_offset, error_word()));
    return cudaGetLastError();
  }
  if (nb <= 64) {
    GPC_LAUNCH(GPC_TRACE_DIAG, (double)nb * nb * nb / 3.0, 16.0 * nb * nb, s,
               launch_k(potrf_la_kernel, 1, 128, potrf_smem<64>(), s, nb, A, lda, info, pivot_offset));
    return cudaGetLastError();
  }
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(potrf_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)potrf_smem<128>());
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  GPC_LAUNCH(GPC_TRACE_DIAG, (double)nb * nb * nb / 3.0, 16.0 * nb * nb, s,
             launch_k(potrf_diag_kernel, 1, 256, potrf_smem<128>(), s, nb, A, lda, info, pivot_offset));
  return cudaGetLastError();
}

cudaError_t diag_batch(const F64xBatch &b, double *A, long long lda, long long sA, int ib, double *out, long long so,
                       const int *order, int *info, cudaStream_t s) {
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    cudaError_t e =
        cudaFuncSetAttribute(potrf_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)potrf_smem<128>());
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  constexpr int nb = kMaxBlock;
  const double work = (double)b.count * nb * nb * nb / 3.0, bytes = 16.0 * b.count * nb * nb;
  const TriBatch q{b.n, ib, sA, so};
  GPC_LAUNCH(GPC_TRACE_DIAG, work, bytes, s,
             potrf_batch_kernel<<<b.count, 256, potrf_smem<128>(), s>>>(A, lda, sA, b.n, ib, order, info));
  GPC_LAUNCH(GPC_TRACE_DIAG, 0.0, bytes, s,
             trtri16_kernel<<<dim3(1, nb / 32, (unsigned)b.count), 64, 0, s>>>(nb, A, lda, nb, nb, out, nb, q));
  GPC_LAUNCH(GPC_TRACE_DIAG, work, bytes, s,
             trtri_cols_kernel<<<dim3(1, nb / TI_COLS, (unsigned)b.count), 32 * TI_WARPS, 0, s>>>(nb, A, lda, nb, nb, out,
                                                                                                  nb, q));
  return cudaGetLastError();
}

// The panel solves run beside the split products' CTAs (one product CTA per
// SM holds ~219 KB of shared memory, leaving room for a small solve CTA).  An
// SM runs CTAs of one shared-memory configuration at a time, so the solve
// kernels ask for the same maximal shared-memory carveout as the products.
bool g_trsm_carveout[64];
cudaError_t trsm_carveout() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaSuccess;
  if (g_trsm_carveout[dev]) return cudaSuccess;
  const void *fns[] = {(const void *)trsm_quad_kernel<64, 0, 4>, (const void *)trsm_quad_kernel<64, 1, 4>,
                       (const void *)trsm_quad_kernel<128, 0, 4>, (const void *)trsm_quad_kernel<128, 1, 4>,
                       (const void *)trsm_quad_kernel<64, 0, 16>, (const void *)trsm_quad_kernel<64, 1, 16>,
                       (const void *)trsm_quad_kernel<128, 0, 16>, (const void *)trsm_quad_kernel<128, 1, 16>,
                       (const void *)trsm_rows_kernel<8>, (const void *)trsm_rows_kernel<16>,
                       (const void *)trsm_rows_kernel<32>};
  for (const void *f : fns) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  g_trsm_carveout[dev] = true;
  return cudaSuccess;
}

cudaError_t trsm_rows(int m, int nb, double *X, long long ldx, const double *T, long long ldt, int mode,
                      cudaStream_t s, bool df) {
  if (m <= 0 || nb <= 0) return cudaSuccess;
  if (nb > kMaxBlock) return cudaErrorInvalidValue;
  if (cudaError_t ce = trsm_carveout(); ce != cudaSuccess) return ce;
  const double fl = (double)m * nb * nb, by = 16.0 * (double)m * nb + 4.0 * nb * nb;
  if (nb == 64 || nb == 128) {
    // A warp issues 224 FP64 instructions for its 2 rows with 16 threads per row
    // and 608 for 8 rows with 4 (NB = 64; the same proportion at 128): as long as
    // all warps run at once, the wider split is the faster (m = 1000: 31 us with
    // 4 threads per row, 18 with 16).  Eight threads per row gained nothing above.
    const int tpr = m <= 8 * sm_count() ? 16 : 4;
    const unsigned qgrid = (unsigned)((m + TQ_THREADS / tpr - 1) / (TQ_THREADS / tpr));
#define GPC_TRSM_QUAD(NB_, MODE_, TPR_)                                                                      \
  GPC_LAUNCH(GPC_TRACE_TRSM, fl, by, s,                                                                     \
             launch_k(trsm_quad_kernel<NB_, MODE_, TPR_>, qgrid, TQ_THREADS, 0, s, m, X, ldx, T, ldt, df))
#define GPC_TRSM_TPR(TPR_)                                \
  do {                                                    \
    if (nb == 64 && mode == 0) GPC_TRSM_QUAD(64, 0, TPR_);  \
    else if (nb == 64) GPC_TRSM_QUAD(64, 1, TPR_);          \
    else if (mode == 0) GPC_TRSM_QUAD(128, 0, TPR_);        \
    else GPC_TRSM_QUAD(128, 1, TPR_);                       \
  } while (0)
    if (tpr == 16) GPC_TRSM_TPR(16);
    else GPC_TRSM_TPR(4);
#undef GPC_TRSM_TPR
#undef GPC_TRSM_QUAD
    return cudaGetLastError();
  }
  // other block sizes: 32 rows per CTA when that still gives two CTAs per SM, else 16 or 8
  const int sms = sm_count();
  if ((m + 31) / 32 >= 2 * sms) {
    GPC_LAUNCH(GPC_TRACE_TRSM, (double)m * nb * nb, 16.0 * (double)m * nb + 4.0 * nb * nb, s,
               launch_k(trsm_rows_kernel<32>, (m + 31) / 32, 256, 0, s, m, nb, X, ldx, T, ldt, mode,
                        df ? 1 : 0));
  } else if ((m + 15) / 16 >= sms) {
    GPC_LAUNCH(GPC_TRACE_TRSM, (double)m * nb * nb, 16.0 * (double)m * nb + 4.0 * nb * nb, s,
               launch_k(trsm_rows_kernel<16>, (m + 15) / 16, 256, 0, s, m, nb, X, ldx, T, ldt, mode,
                        df ? 1 : 0));
  } else {
    GPC_LAUNCH(GPC_TRACE_TRSM, (double)m * nb * nb, 16.0 * (double)m * nb + 4.0 * nb * nb, s,
               launch_k(trsm_rows_kernel<8>, (m + 7) / 8, 256, 0, s, m, nb, X, ldx, T, ldt, mode,
                        df ? 1 : 0));
  }
  return cudaGetLastError();
}

cudaError_t copy_lower(int n, const double *src, long long lds, double *dst, long long ldd, cudaStream_t s, int *emax) {
  if (n <= 0) return cudaSuccess;
  if (emax)
    if (cudaError_t e = cudaMemsetAsync(emax, 0, sizeof(int), s); e != cudaSuccess) return e;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 8.0 * (double)n * n * 1.5, s,
             copy_lower_kernel<<<blocks_for((long long)n * n, 256), 256, 0, s>>>(n, src, lds, dst, ldd, emax));
  return cudaGetLastError();
}

cudaError_t rescale_tiny(int n, double *A, long long lda, int shift, const int *emax, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 0.0, s,
             rescale_tiny_kernel<<<std::min(n, 4 * sm_count()), 256, 0, s>>>(n, A, lda, shift, emax));
  return cudaGetLastError();
}

cudaError_t copy_rect(int m, int c, const double *src, long long lds, double *dst, long long ldd,
                      cudaStream_t s) {
  if (m <= 0 || c <= 0) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 16.0 * (double)m * c, s,
             copy_rect_kernel<<<blocks_for((long long)m * c, 256), 256, 0, s>>>(m, c, src, lds, dst, ldd));
  return cudaGetLastError();
}

cudaError_t phi_block(int nb, double *A, long long lda, cudaStream_t s) {
  if (nb <= 0) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 16.0 * (double)nb * nb, s,
             phi_block_kernel<<<blocks_for((long long)nb * nb, 256), 256, 0, s>>>(nb, A, lda));
  return cudaGetLastError();
}

cudaError_t lower_to_symmetric_half(int n, double *A, long long lda, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 16.0 * (double)n * n, s,
             lower_to_symmetric_half_kernel<<<blocks_for((long long)n * n, 256), 256, 0, s>>>(n, A, lda));
  return cudaGetLastError();
}

cudaError_t recip_rsqrt_probe(int n, const double *x, double *out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 40.0 * n, s, recip_rsqrt_probe_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, x, out));
  return cudaGetLastError();
}

cudaError_t recip_cubic_probe(int n, const double *x, double *out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 16.0 * n, s, recip_cubic_probe_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, x, out));
  return cudaGetLastError();
}

cudaError_t reset_info(int *info, cudaStream_t s) {
  if (!info) return cudaSuccess;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 8.0, s, reset_info_kernel<<<1, 1, 0, s>>>(info));
  return cudaGetLastError();
}

}  // namespace gpc
