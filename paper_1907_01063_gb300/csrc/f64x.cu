// FP64-accurate products on the fifth-generation tensor cores (tcgen05).
//
// On this part FP64 multiply-adds run at about 1.1 TFLOP/s in every form (DFMA
// or DMMA), 1/1700 of the BF16 tensor rate, so an FP64 product is evaluated
// with an error-free split of its operands into BF16 slices (the Ozaki scheme:
// Ozaki, Ogita, Oishi & Rump, 2012), with enough slices that the result is at
// least as accurate as the FP64 multiply-add chain it stands for.
//
// Splitting.  Every operand row r is scaled by a power of two 2^-E_r (its
// largest entry, or another bound the caller has) and its K index is cut into
// chunks of 128.  For every (row, chunk) the entries are rounded to the grid
// 2^(e - 8 S), e the chunk's exponent, and written with S balanced base-256
// digits (the first in [0, 256], the others in [-128, 127]); slice p holds
// digit p times 2^(e - 8 p), exact in BF16.  S = 7 (56 bits) or 8 (64 bits):
// an entry within 3 (11) bits of its chunk's largest is held exactly.
//
// Products.  The slice products A_p B_q^T are summed on tcgen05 into seven FP32
// TMEM accumulators by p + q (1-based): G2, .., G8, pairs with p + q > 8 (S = 7)
// or > 9 (S = 8, G9 joins G8) dropped.  Over a chunk |G2| <= 2^23, |G3| <= 2^23,
// |G4|, |G5|, |G6| < 2^24 in units of their slice scales, so these are integer
// sums the tensor core forms exactly; G7 and G8 lie 2^-40 and more below G2.
//
// Accumulation.  The epilogue keeps every output as three FP32 numbers
// (A, B, C): after each chunk G2 enters A, and G3..G6 enter B, through exact
// two-sums whose errors go one place down, and G7, G8 go into C.  The output
// read at the start of a work item (C += product) enters the same sum exactly,
// and the result is rounded to FP64 once, with integer field moves: three FP64
// additions per output would take 15 000 cycles per 128 x 64 tile on the FP64
// pipe (1.6 operations per cycle per SM), 1.6 times the MMAs of a chunk.
//
// When it is as good as FP64.  Writing a' = a 2^-E for the scaled operands,
// the split loses at most about 2^-55 (S = 7), 2^-62.5 (S = 8) per product
// term, absolutely, where the FP64 chain's bound is K 2^-53 sum |a'||b'|.  The
// factorisation and its adjoint only need the bound relative to the scales
// (2^E_i 2^E_j bounds |K_ij| by the diagonal; see mixed.cu).  A general product
// is checked: an S = 1 pass forms sum |a'||b'| from the magnitudes' leading eight bits
// for every output, and a 32 x 32 block with an output below the threshold (or with
// an infinity, a NaN or denormal rows) is left to the FP64 kernel, which
// computes just those blocks in the following launch.
//
// Kernel structure: persistent CTAs of 10 warps: warp 0 issues TMA loads of
// slice tiles (64B-swizzled, K-major, 32 wide, two stages of 84 or 96 KiB),
// warp 1 issues the MMAs, warps 2..9 are the epilogue.  Seven accumulators of
// 64 columns leave no room for a second set, so the fold releases the groups
// one by one (G8 first) and the MMAs of the next chunk's first stage are issued
// in that order (a_7 b_1, then a_6 .., a_1 ..), each waiting only for its own
// accumulators.  Every wait is bounded in time, as in ozaki.cu.
//
// What bounds it: the shared-memory port (11 to 19 operand passes of 4 KiB of A
// and 28 or 36 of 2 KiB of B per K = 16 step against 896 or 1152 cycles of MMA)
// and the fold between chunks.  Measured: 4096^3 in 3.4 ms (S = 8, the product
// launch 3.2 ms = 1546 BF16 TFLOP/s, 0.88 of the sustained rate) against 125 ms
// for the FP64 kernel; 2000 x 1537 x 1025 and its reverse mode 0.96 against
// 21.0 ms; largest error over sampled outputs 1.1e-17 sum |a||b| at 4096^3
// against 3.2e-16.
#include "common.cuh"
#include "tc.cuh"

#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

namespace gpc {
namespace {

using namespace tc;

constexpr int FX_BM = 128, FX_BN = 64, FX_BK = 32, FX_CHUNK = 128;
constexpr int FX_EPI_WARPS = 8;
constexpr int FX_THREADS = 64 + 32 * FX_EPI_WARPS;
constexpr int FX_GROUPS = 7;
constexpr int FX_A_PLANE = FX_BM * FX_BK * 2;  // 8 KiB
constexpr int FX_B_PLANE = FX_BN * FX_BK * 2;  // 4 KiB
constexpr int FX_EPI_COLS = 8;                 // columns per pass of an epilogue buffer
constexpr int FX_EPI_BUF = 3 * 32 * FX_EPI_COLS * 4;  // three FP32 planes of 32 rows per warp (columns XOR-swizzled)
constexpr int fx_stages(int S) { return S == 1 ? 4 : 2; }
constexpr int fx_smem(int S) {
  return fx_stages(S) * S * (FX_A_PLANE + FX_B_PLANE) + (S == 1 ? 0 : FX_EPI_WARPS * FX_EPI_BUF) + 1024 + 1024;
}
static_assert(fx_smem(8) <= 232448, "shared memory of one CTA");

// codes of a row's largest magnitude (row_codes_kernel)
constexpr int kCodeZero = 0;     // every entry is zero
constexpr int kCodeTiny = 64;    // biased exponents up to this: too close to the denormals to be split exactly
constexpr int kCodeBad = 2047;   // an infinity or a NaN
__device__ __forceinline__ int code_exponent(int code) { return code == kCodeZero ? 0 : code - 1022; }
__device__ __forceinline__ bool code_bad(int code) {
  return code >= kCodeBad || (code > kCodeZero && code <= kCodeTiny);
}

struct FxParams {
  int M, N, chunks, qpc, kstages;  // qpc: stages per chunk; kstages: stages in all (0: chunks * qpc)
  int a_row0, b_row0, a_k0, b_k0;
  int lower;                       // entries with col <= row
  int kskip, ksh_m, ksh_n;         // known-zero K ranges (Gemm::kskip), shifted by the panel's offsets
  int splits, tiles_m, tiles_n, per_batch, num_work;
  int sub;                         // 4: four CTAs per tile, each with 8 columns of every epilogue warp's 32 (else 1)
  int a_rows, b_rows;              // slice rows per batch entry
  int accumulate;
  const int *ra, *rb;              // scale exponents of the output's rows and columns (null: 0), ...
  int ra_mul;                      // 0: one exponent for all rows, less ra_sub[row]
  const int *ra_sub;
  int sub_stride;
  int ra_codes, rb_codes;          // ... or row_codes_kernel codes
  const int *nblk;                 // non-null: F64xBatch
  int act, mb, nb, kb;
  int ra_stride, rb_stride;        // per batch entry
  double *C;
  long long ldc, sC;
  double *partial;
  unsigned char *flags;            // per 32 x 32 block: safe by the row counts (1) or the check (2); 0 = left to FP64
  int flag_ld;
  long long flag_stride;
  float theta;
  int *err, *gerr;
  unsigned long long wait_ns;
  int no_loads;
};

__device__ __forceinline__ int row_exp(const int *e, int codes, int i) {
  if (!e) return 0;
  const int v = __ldg(e + i);
  return codes ? code_exponent(v) : (v < -100000 ? 0 : v);
}

// ------------------------------------------------------------------ work list
struct Work {
  int b, tm, tn, c0, c1, split;
  bool none, skip;  // none: the tile's whole K range is known zeros
};
template <bool CHECK>
__device__ __forceinline__ Work work_item(const FxParams &p, int w) {
  Work k;
  k.split = w % p.splits;
  int t = w / p.splits;
  k.b = t / p.per_batch;
  t -= k.b * p.per_batch;
  if (p.lower) {
    // rows of tiles hold 2 tm + 2 tiles until tiles_n caps them
    int tm = 0;
    for (;;) {
      const int cnt = min(p.tiles_n, (tm * FX_BM + FX_BM - 1) / FX_BN + 1);
      if (t < cnt) break;
      t -= cnt;
      ++tm;
    }
    k.tm = tm;
    k.tn = t;
  } else {
    k.tm = t / p.tiles_n;
    k.tn = t - k.tm * p.tiles_n;
  }
  const int m0 = k.tm * FX_BM, n0 = k.tn * FX_BN;
  int lo = 0, hi = p.chunks;
  if (p.kskip == KSKIP_ROWS) lo = max(0, m0 + p.ksh_m) / FX_CHUNK;
  if (p.kskip == KSKIP_COLS) lo = max(0, n0 + p.ksh_n) / FX_CHUNK;
  if (p.kskip == KSKIP_ROWS_END) hi = min(hi, max(0, m0 + FX_BM + p.ksh_m + FX_CHUNK - 1) / FX_CHUNK);
  if (p.kskip == KSKIP_COLS_END) hi = min(hi, max(0, n0 + FX_BN + p.ksh_n + FX_CHUNK - 1) / FX_CHUNK);
  lo = min(lo, hi);
  k.skip = false;
  if (p.nblk) {
    const int blocks = __ldg(p.nblk + k.b);
    if (p.kb >= 0) hi = min(hi, max(0, blocks - p.kb));
    k.skip = blocks <= p.act || (p.mb >= 0 && m0 >= FX_CHUNK * (blocks - p.mb)) ||
             (p.nb >= 0 && n0 >= FX_CHUNK * (blocks - p.nb));
  }
  const int per = (hi - lo + p.splits - 1) / p.splits;
  k.c0 = min(hi, lo + k.split * per);
  k.c1 = min(hi, k.c0 + per);
  k.none = lo >= hi;
  // The check skips tiles the row counts show to be safe (bit 0, not written by
  // this launch, so every warp of every K range decides alike), the product the
  // tiles left to the FP64 kernel.
  if (p.flags) {
    const volatile unsigned char *f = p.flags + (size_t)k.b * p.flag_stride + (size_t)(4 * k.tm) * p.flag_ld + 2 * k.tn;
    bool all = true;
    for (int q = 0; q < 4 && all; ++q)
      for (int h = 0; h < 2; ++h)
        if (m0 + 32 * q < p.M && n0 + 32 * h < p.N && (CHECK ? !(f[(size_t)q * p.flag_ld + h] & 1) : f[(size_t)q * p.flag_ld + h] != 0))
          all = false;
    k.skip = all;
  }
  return k;
}
__device__ __forceinline__ int chunk_stages(const FxParams &p, int c) {
  return p.kstages > 0 ? min(p.qpc, p.kstages - 4 * c) : p.qpc;
}

// ------------------------------------------------------------------ triples
__device__ __forceinline__ void two_sum1(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// x 2^-sh as three FP32 numbers (24 + 15 + 14 bits of the mantissa, exact) when
// its exponent lies in [-70, 100]; false otherwise (nothing is written).
__device__ __forceinline__ bool f64_to_triple(double x, int sh, float &a, float &b, float &c) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7FF) - 1023 - sh;
  if ((u << 1) == 0) {
    a = b = c = 0.f;
    return true;
  }
  if (e < -70 || e > 100 || e + sh == 1024 || e + sh == -1023) return false;  // also Inf, NaN, denormals
  const uint32_t s = (uint32_t)(u >> 63) << 31;
  const uint32_t m23 = (uint32_t)(u >> 29) & 0x7FFFFFu;
  const uint32_t n1 = (uint32_t)(u >> 14) & 0x7FFFu, n2 = (uint32_t)u & 0x3FFFu;
  a = __uint_as_float(s | ((uint32_t)(e + 127) << 23) | m23);
  b = __fmul_rn(__fsub_rn(__uint_as_float(0x4B000000u | n1), 8388608.0f),
                __uint_as_float(s | ((uint32_t)(e - 38 + 127) << 23)));
  c = __fmul_rn(__fsub_rn(__uint_as_float(0x4B000000u | n2), 8388608.0f),
                __uint_as_float(s | ((uint32_t)(e - 52 + 127) << 23)));
  return true;
}
// (a + b + c) 2^sh rounded to FP64.  The three are made non-overlapping
// (h, m, l), h's fields are moved to FP64 and m + l, an integer of at most 29
// bits in units of the result's last place, is added to the bit pattern (just
// below a power of two the unit is half as large).  Results near the ends of
// the exponent range take FP64 arithmetic.
__device__ __forceinline__ double triple_to_f64(float a, float b, float c, int sh) {
  float h, t, m, l;
  two_sum1(a, b, h, t);
  two_sum1(t, c, m, l);
  two_sum1(h, m, h, m);
  two_sum1(m, l, m, l);
  const uint32_t hb = __float_as_uint(h);
  if (h == 0.f) return __longlong_as_double((long long)((unsigned long long)hb << 32));
  const int eb = (int)(hb >> 23) & 0xFF;
  if (eb >= 54 && eb <= 254 && (unsigned)(eb + 896 + sh - 2) <= 2042u) {
    const uint32_t sign = hb & 0x80000000u;
    const bool edge = (hb & 0x7FFFFFu) == 0u && m != 0.f && ((hb ^ __float_as_uint(m)) & 0x80000000u) != 0u;
    const float sc = __uint_as_float((uint32_t)(306 - eb + (edge ? 1 : 0)) << 23);  // 2^(52 - exponent of h)
    const float q = __uint_as_float(__float_as_uint(__fmul_rn(m, sc)) ^ sign);
    const float ql = __uint_as_float(__float_as_uint(__fmul_rn(l, sc)) ^ sign);
    const float ta = __fmaf_rn(q, 0x1p-14f, 12582912.0f);
    const float ra = __fsub_rn(ta, 12582912.0f);
    const float rem = __fmaf_rn(-16384.0f, ra, q);
    const float tb = __fadd_rn(__fadd_rn(rem, ql), 12582912.0f);
    const int d = ((__float_as_int(ta) - 0x4B400000) << 14) + (__float_as_int(tb) - 0x4B400000);
    const unsigned long long bits = ((unsigned long long)sign << 32) |
                                    ((unsigned long long)(uint32_t)(eb + 896 + sh) << 52) |
                                    ((unsigned long long)(hb & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)bits + (long long)d);
  }
  return scalbn((double)h + ((double)m + (double)l), sh);
}

// s + e == a + b, or a - b, exactly.
template <bool NEG>
__device__ __forceinline__ void fold2(f2x a, f2x b, f2x &s, f2x &e) {
  if (NEG) two_diff2(a, b, s, e);
  else two_sum2(a, b, s, e);
}

// ------------------------------------------------------------------ MMAs
// Products a_p b_0 .. a_p b_{c-1} (0-based) into groups p .. p + c - 1.
__device__ __forceinline__ void mma_run(uint32_t tacc, int group, int count, uint64_t da, uint64_t db, uint32_t acc) {
  constexpr uint64_t pb = FX_B_PLANE >> 4;
  const uint32_t d = tacc + (uint32_t)(group * FX_BN);
  if (count > 4) {
    mma_bf16(d, da, db, idesc_n(256), acc);
    mma_bf16(d + 4 * FX_BN, da, db + 4 * pb, idesc_n(64 * (count - 4)), acc);
  } else if (count > 0) {
    mma_bf16(d, da, db, idesc_n(64 * count), acc);
  }
}
template <int S, int P>
__device__ __forceinline__ void mma_plane(uint32_t tacc, uint64_t da0, uint64_t db, bool init) {
  constexpr uint64_t pa = FX_A_PLANE >> 4, pb = FX_B_PLANE >> 4;
  const uint64_t da = da0 + (uint64_t)P * pa;
  if constexpr (P < FX_GROUPS) {
    if (init) {  // group P is written for the first time, the later ones hold a_{P+1} .. already
      mma_run(tacc, P, 1, da, db, 0u);
      mma_run(tacc, P + 1, FX_GROUPS - 1 - P, da, db + pb, 1u);
    } else {
      mma_run(tacc, P, FX_GROUPS - P, da, db, 1u);
    }
  }
  if constexpr (S > FX_GROUPS)  // p + q = 9 joins the last group
    mma_run(tacc, FX_GROUPS - 1, 1, da, db + (uint64_t)(FX_GROUPS - P) * pb, 1u);
}
template <int S>
__device__ __forceinline__ void mma_kstep(uint32_t tacc, uint64_t da, uint64_t db) {
  mma_plane<S, 0>(tacc, da, db, false);
  mma_plane<S, 1>(tacc, da, db, false);
  mma_plane<S, 2>(tacc, da, db, false);
  mma_plane<S, 3>(tacc, da, db, false);
  mma_plane<S, 4>(tacc, da, db, false);
  mma_plane<S, 5>(tacc, da, db, false);
  mma_plane<S, 6>(tacc, da, db, false);
  if constexpr (S > FX_GROUPS) mma_plane<S, 7>(tacc, da, db, false);
}

__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&r)[32]) {
  uint32_t v[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr));
#pragma unroll
  for (int i = 0; i < 32; ++i) r[i] = __uint_as_float(v[i]);
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, float (&r)[8]) {
  uint32_t v[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(addr));
#pragma unroll
  for (int i = 0; i < 8; ++i) r[i] = __uint_as_float(v[i]);
}
__device__ __forceinline__ void pin8(float (&r)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) asm volatile("" : "+f"(r[i]));
}
__device__ __forceinline__ void pin32(float (&r)[32]) {
#pragma unroll
  for (int i = 0; i < 32; ++i) asm volatile("" : "+f"(r[i]));
}

// The output tile of a work item into L2, 512 bytes per row (16-byte pieces inside
// the row only), so that the epilogue's loads at the item's start do not wait for HBM.
__device__ __forceinline__ void prefetch_output(const FxParams &p, const Work &k) {
  const int r0 = k.tm * FX_BM, n0 = k.tn * FX_BN;
  const int rows = min(FX_BM, p.M - r0), cols = min(FX_BN, p.N - n0);
  const double *base = p.C + (long long)k.b * p.sC + (long long)r0 * p.ldc + n0;
  for (int r = 0; r < rows; ++r) {
    const uintptr_t a = ((uintptr_t)(base + (long long)r * p.ldc) + 15) & ~(uintptr_t)15;
    const uintptr_t e = (uintptr_t)(base + (long long)r * p.ldc + cols) & ~(uintptr_t)15;
    if (e > a)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(e - a)) : "memory");
  }
}

// ------------------------------------------------------------------ the product
// S slices; CHECK (S = 1): sums of the magnitudes' products against theta, into flags.
template <int S, bool NEG, bool CHECK>
__global__ void __launch_bounds__(FX_THREADS, 1)
f64x_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, FxParams p) {
  constexpr int STAGES = fx_stages(S), A_STAGE = S * FX_A_PLANE, B_STAGE = S * FX_B_PLANE;
  constexpr int NG = CHECK ? 1 : FX_GROUPS;
  constexpr int TCOLS = CHECK ? 64 : 512;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *sA = smem;
  unsigned char *sB = smem + STAGES * A_STAGE;
  float *epi_buf = (float *)(sB + STAGES * B_STAGE);
  uint64_t *bars = (uint64_t *)((unsigned char *)epi_buf + (CHECK ? 0 : FX_EPI_WARPS * FX_EPI_BUF));
  // bars: full[STAGES], empty[STAGES], tfull, gfree[NG], drain
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES), tfull = smem_u32(bars + 2 * STAGES);
  const uint32_t gfree0 = smem_u32(bars + 2 * STAGES + 1), drain = smem_u32(bars + 2 * STAGES + 1 + NG);
  volatile int *abort_flag = (volatile int *)(bars + 2 * STAGES + 2 + NG);
  uint32_t *tmem_slot = (uint32_t *)(bars + 2 * STAGES + 3 + NG);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    mbar_init(tfull, 1);
    for (int i = 0; i < NG; ++i) mbar_init(gfree0 + 8 * i, FX_EPI_WARPS);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = *tmem_slot;
  auto report = [&]() {
    *abort_flag = 1;
    if (p.err) atomicExch(p.err, GPC_ERR_TIMEOUT);
    record_error(p.gerr, GPC_ERR_TIMEOUT);
  };

  if (warp == 0) {
    // ---------------- TMA producer
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
      int stage = 0;
      uint32_t phase = 0;
      long long issued = 0;
      bool ok = true;
      for (int w = blockIdx.x; w < p.num_work && ok && !p.no_loads; w += gridDim.x) {
        const Work k = work_item<CHECK>(p, CHECK ? w : w / p.sub);
        if (k.skip) continue;
        if (!CHECK && p.accumulate && !p.partial) prefetch_output(p, k);
        const int ya = p.a_row0 + k.b * p.a_rows + k.tm * FX_BM, yb = p.b_row0 + k.b * p.b_rows + k.tn * FX_BN;
        for (int c = k.c0; c < k.c1 && ok; ++c) {
          const int ns = chunk_stages(p, c);
          for (int h = 0; h < ns; ++h) {
            if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag, p.wait_ns)) { ok = false; break; }
            mbar_expect_tx(full0 + 8 * stage, A_STAGE + B_STAGE);
            tma_load_3d(smem_u32(sA + stage * A_STAGE), &tmA, p.a_k0 + c * FX_CHUNK + h * FX_BK, ya, 0,
                        full0 + 8 * stage);
            tma_load_3d(smem_u32(sB + stage * B_STAGE), &tmB, p.b_k0 + c * FX_CHUNK + h * FX_BK, yb, 0,
                        full0 + 8 * stage);
            ++issued;
            if (++stage == STAGES) { stage = 0; phase ^= 1; }
          }
        }
      }
      if (!ok) {
        report();
        const long long first = issued > STAGES ? issued - STAGES : 0;
        for (long long i = first; i < issued; ++i)
          mbar_wait_drain(full0 + 8 * (int)(i % STAGES), (uint32_t)((i / STAGES) & 1));
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0, tphase = 0;
      bool ok = true, any = false;
      for (int w = blockIdx.x; w < p.num_work && ok; w += gridDim.x) {
        const Work k = work_item<CHECK>(p, CHECK ? w : w / p.sub);
        if (k.skip) continue;
        for (int c = k.c0; c < k.c1 && ok; ++c) {
          const int ns = chunk_stages(p, c);
          for (int h = 0; h < ns && ok; ++h) {
            if (!mbar_wait(full0 + 8 * stage, phase, abort_flag, p.wait_ns)) { ok = false; break; }
            fence_after();
            const uint64_t da = sdesc(smem_u32(sA + stage * A_STAGE));
            const uint64_t db = sdesc(smem_u32(sB + stage * B_STAGE));
            if constexpr (CHECK) {
              if (h == 0 && c == k.c0) {
                if (!mbar_wait(gfree0, tphase ^ 1, abort_flag, p.wait_ns)) { ok = false; break; }
                fence_after();
              }
#pragma unroll
              for (int kk = 0; kk < FX_BK / 16; ++kk)
                mma_bf16(tbase, da + 2 * kk, db + 2 * kk, idesc_n(64), (c == k.c0 && h == 0 && kk == 0) ? 0u : 1u);
              any = true;
            } else if (h == 0) {
              // first stage of a chunk: lowest group first, each as the fold of the last chunk frees it
#define FX_FIRST(P)                                                                                      \
  if (ok) {                                                                                               \
    if (!mbar_wait(gfree0 + 8 * P, tphase ^ 1, abort_flag, p.wait_ns)) {                                   \
      ok = false;                                                                                          \
    } else {                                                                                               \
      fence_after();                                                                                       \
      mma_plane<S, P>(tbase, da, db, true);                                                                \
      mma_plane<S, P>(tbase, da + 2, db + 2, false);                                                       \
      any = true;                                                                                          \
    }                                                                                                      \
  }
              FX_FIRST(6)
              FX_FIRST(5)
              FX_FIRST(4)
              FX_FIRST(3)
              FX_FIRST(2)
              FX_FIRST(1)
              FX_FIRST(0)
#undef FX_FIRST
              if (!ok) break;
              if constexpr (S > FX_GROUPS) {
                mma_plane<S, 7>(tbase, da, db, false);
                mma_plane<S, 7>(tbase, da + 2, db + 2, false);
              }
            } else {
              mma_kstep<S>(tbase, da, db);
              mma_kstep<S>(tbase, da + 2, db + 2);
            }
            mma_commit(empty0 + 8 * stage);
            if (++stage == STAGES) { stage = 0; phase ^= 1; }
          }
          if (!ok) break;
          if (!CHECK || c + 1 == k.c1) {  // the check sums its whole K range in place
            mma_commit(tfull);
            tphase ^= 1;
          }
        }
      }
      if (!ok) report();
      if (any) {  // every MMA issued above completes before TMEM is released
        mma_commit(drain);
        mbar_wait_drain(drain, 0);
      }
    }
  } else {
    // ---------------- epilogue: warps 2..9; lane quarter = warp % 4, column half by warp pair
    const int q = warp & 3, half = (warp - 2) >> 2;
    // Buffer element (row, c) of a plane at row 8 + (c ^ (row / 4) % 8): both a
    // thread per row (the TMEM layout) and 4 rows x 8 columns per access (64-byte
    // row pieces of global memory) are free of bank conflicts.
    float *tb = epi_buf + (size_t)(warp - 2) * (FX_EPI_BUF / 4);
    const int rl = lane >> 3, cl = lane & 7;
    const uint32_t taddr = tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 32);
    uint32_t tphase = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < p.num_work && ok; w += gridDim.x) {
      const Work k = work_item<CHECK>(p, CHECK ? w : w / p.sub);
      if (k.skip) continue;
      const int row0 = k.tm * FX_BM + q * 32, colh = k.tn * FX_BN + half * 32;
      if constexpr (CHECK) {
        float s[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) s[i] = 0.f;
        if (k.c0 < k.c1) {
          if (!mbar_wait(tfull, tphase, abort_flag, p.wait_ns)) { ok = false; break; }
          tphase ^= 1;
          fence_after();
          tmem_ld32(taddr, s);
          tmem_wait_ld();
          pin32(s);
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(gfree0);
        }
        const int row = row0 + lane;
        const int code_a = row < p.M ? __ldg(p.ra + (size_t)k.b * p.ra_stride + row) : kCodeZero;
        const int code_b = colh + lane < p.N ? __ldg(p.rb + (size_t)k.b * p.rb_stride + colh + lane) : kCodeZero;
        bool bad = false;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int cb = __shfl_sync(0xffffffffu, code_b, i);
          const int col = colh + i;
          if (row < p.M && col < p.N && !(p.lower && col > row) && !k.none) {
            if (code_bad(code_a) || code_bad(cb)) bad = true;
            else if (code_a != kCodeZero && cb != kCodeZero && !(s[i] >= p.theta)) bad = true;
          }
        }
        // one K range that shows every output of the block to be safe is enough
        const bool any = __any_sync(0xffffffffu, bad);
        if (lane == 0 && !any) {
          unsigned char *f = p.flags + (size_t)k.b * p.flag_stride + (size_t)(4 * k.tm + q) * p.flag_ld + 2 * k.tn + half;
          *f = (*f & 1) | 2;
        }
      } else {
        double *base;
        long long ld;
        if (p.partial) {
          base = p.partial + (size_t)k.split * p.M * (size_t)p.N;
          ld = p.N;
        } else {
          base = p.C + (long long)k.b * p.sC;
          ld = p.ldc;
        }
        const bool add = p.accumulate && !p.partial;
        const bool interior =
            row0 + 32 <= p.M && colh + 32 <= p.N && (!p.lower || colh + 31 <= row0);
        const bool live = !p.flags || row0 >= p.M || colh >= p.N ||
                          p.flags[(size_t)k.b * p.flag_stride + (size_t)(4 * k.tm + q) * p.flag_ld + 2 * k.tn + half];
        const int ea = row0 + lane < p.M ? row_exp(p.ra, p.ra_codes, k.b * p.ra_stride + (row0 + lane) * p.ra_mul) -
                                              (p.ra_sub ? __ldg(p.ra_sub + k.b * p.sub_stride + row0 + lane) : 0)
                                        : 0;
        const int ebl = colh + lane < p.N ? row_exp(p.rb, p.rb_codes, k.b * p.rb_stride + colh + lane) : 0;
        if (p.sub == 4 || p.chunks == 1) {
          // 8 columns of each warp's 32 at a time.  With few tiles (sub: the
          // factorisation's chain) every CTA forms the whole tile but folds and
          // writes only one such group; with one chunk the groups take turns.  Folding
          // all 32 columns together needs some 5000 instructions per warp and 60 KB of
          // code, which pays only where a tile's chunks run through it many times.
          // (One chunk, 9.2e3 accumulated tiles of a batch: 38 -> 24 us per tile and SM.)
          const int cg0 = p.sub == 4 ? w & 3 : 0, cg1 = p.sub == 4 ? cg0 + 1 : 4;
          double v[8];
          auto load = [&](int cg) {
            const int col = colh + cg * FX_EPI_COLS + cl;
#pragma unroll
            for (int it = 0; it < 8; ++it) {
              const int row = row0 + 4 * it + rl;
              const bool in = interior || (row < p.M && col < p.N && !(p.lower && col > row));
              v[it] = in ? base[(long long)row * ld + col] : 0.0;
            }
          };
          if (add) load(cg0);
#pragma unroll 1
          for (int cg = cg0; cg < cg1; ++cg) {
            const int col = colh + cg * FX_EPI_COLS + cl;
            const int eb = __shfl_sync(0xffffffffu, ebl, cg * FX_EPI_COLS + cl);
            f2x A[4], B[4], C[4];
            uint32_t off = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) A[i] = B[i] = C[i] = 0ull;
            if (add) {
#pragma unroll
              for (int it = 0; it < 8; ++it) {
                float t0 = 0.f, t1 = 0.f, t2 = 0.f;
                const int sh = eb + __shfl_sync(0xffffffffu, ea, 4 * it + rl);
                if (!f64_to_triple(v[it], sh, t0, t1, t2)) off |= 1u << it;
                const int at = (4 * it + rl) * FX_EPI_COLS + (cl ^ it);
                tb[at] = t0;
                tb[at + 256] = t1;
                tb[at + 512] = t2;
              }
              __syncwarp();
#pragma unroll
              for (int i = 0; i < 8; i += 2) {
                const int a0 = lane * FX_EPI_COLS + (i ^ (lane >> 2)), a1 = lane * FX_EPI_COLS + ((i + 1) ^ (lane >> 2));
                A[i / 2] = pk2(tb[a0], tb[a1]);
                B[i / 2] = pk2(tb[a0 + 256], tb[a1 + 256]);
                C[i / 2] = pk2(tb[a0 + 512], tb[a1 + 512]);
              }
              __syncwarp();
              if (cg + 1 < cg1) load(cg + 1);  // in flight while this group is folded
            }
#pragma unroll 1
            for (int c = k.c0; c < k.c1; ++c) {
              if (cg == cg0) {
                if (!mbar_wait(tfull, tphase, abort_flag, p.wait_ns)) { ok = false; break; }
                tphase ^= 1;
                fence_after();
              }
              float g[FX_GROUPS][8];
#pragma unroll
              for (int grp = 0; grp < FX_GROUPS; ++grp) tmem_ld8(taddr + (uint32_t)(grp * FX_BN + cg * 8), g[grp]);
              tmem_wait_ld();
#pragma unroll
              for (int grp = 0; grp < FX_GROUPS; ++grp) pin8(g[grp]);
              if (cg + 1 == cg1) {
                fence_before();
                __syncwarp();
                if (lane < FX_GROUPS) mbar_arrive(gfree0 + 8 * lane);
              }
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                f2x e, f;
                auto part = [&](int q) { return pk2(g[q][2 * i], g[q][2 * i + 1]); };
                C[i] = NEG ? sub2(C[i], part(6)) : add2(C[i], part(6));
                C[i] = NEG ? sub2(C[i], part(5)) : add2(C[i], part(5));
#pragma unroll
                for (int q = 4; q >= 1; --q) {
                  fold2<NEG>(B[i], part(q), B[i], e);
                  C[i] = add2(C[i], e);
                }
                fold2<NEG>(A[i], part(0), A[i], e);
                two_sum2(B[i], e, B[i], f);
                C[i] = add2(C[i], f);
              }
            }
            if (!ok) break;
            if (!live) continue;
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              const int a0 = lane * FX_EPI_COLS + (i ^ (lane >> 2)), a1 = lane * FX_EPI_COLS + ((i + 1) ^ (lane >> 2));
              upk2(A[i / 2], tb[a0], tb[a1]);
              upk2(B[i / 2], tb[a0 + 256], tb[a1 + 256]);
              upk2(C[i / 2], tb[a0 + 512], tb[a1 + 512]);
            }
            __syncwarp();
#pragma unroll 4
            for (int it = 0; it < 8; ++it) {
              const int row = row0 + 4 * it + rl, at = (4 * it + rl) * FX_EPI_COLS + (cl ^ it);
              const int sh = eb + __shfl_sync(0xffffffffu, ea, 4 * it + rl);
              if (interior || (row < p.M && col < p.N && !(p.lower && col > row))) {
                double *dst = base + (long long)row * ld + col;
                double x = triple_to_f64(tb[at], tb[at + 256], tb[at + 512], sh);
                if (off >> it & 1u) x = *dst + x;
                *dst = x;
              }
            }
            __syncwarp();
          }
          if (!ok) break;
          continue;
        }
        f2x fa[16], fb[16], fc[16];
        uint32_t late = 0;  // values (8 per column group) that do not fit the triple: added in FP64 at the end
        if (add) {
          double v[4][8];  // all loads in flight before the first is used
#pragma unroll
          for (int cg = 0; cg < 4; ++cg)
#pragma unroll
            for (int it = 0; it < 8; ++it) {
              const int row = row0 + 4 * it + rl, col = colh + cg * FX_EPI_COLS + cl;
              const bool in = interior || (row < p.M && col < p.N && !(p.lower && col > row));
              v[cg][it] = in ? base[(long long)row * ld + col] : 0.0;
            }
#pragma unroll
          for (int cg = 0; cg < 4; ++cg) {
            const int eb = __shfl_sync(0xffffffffu, ebl, cg * FX_EPI_COLS + cl);
            uint32_t off = 0;  // which of this thread's eight values do not fit
#pragma unroll
            for (int it = 0; it < 8; ++it) {
              float t0 = 0.f, t1 = 0.f, t2 = 0.f;
              const int sh = eb + __shfl_sync(0xffffffffu, ea, 4 * it + rl);
              if (!f64_to_triple(v[cg][it], sh, t0, t1, t2)) off |= 1u << it;
              const int at = (4 * it + rl) * FX_EPI_COLS + (cl ^ it);
              tb[at] = t0;
              tb[at + 256] = t1;
              tb[at + 512] = t2;
            }
            if (off) late |= off << (8 * cg);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              const int a0 = lane * FX_EPI_COLS + (i ^ (lane >> 2)), a1 = lane * FX_EPI_COLS + ((i + 1) ^ (lane >> 2));
              fa[cg * 4 + i / 2] = pk2(tb[a0], tb[a1]);
              fb[cg * 4 + i / 2] = pk2(tb[a0 + 256], tb[a1 + 256]);
              fc[cg * 4 + i / 2] = pk2(tb[a0 + 512], tb[a1 + 512]);
            }
            __syncwarp();
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) fa[i] = fb[i] = fc[i] = 0ull;
        }
        for (int c = k.c0; c < k.c1; ++c) {
          if (!mbar_wait(tfull, tphase, abort_flag, p.wait_ns)) { ok = false; break; }
          tphase ^= 1;
          fence_after();
          float ga[32], gb[32];
          // group g of this chunk: into C (G7, G8), B with its error into C (G3..G6), or A, error into B (G2)
          auto fold = [&](int g, float(&r)[32]) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const f2x x = pk2(r[2 * i], r[2 * i + 1]);
              if (g >= 5) {
                fc[i] = NEG ? sub2(fc[i], x) : add2(fc[i], x);
              } else if (g >= 1) {
                f2x e;
                fold2<NEG>(fb[i], x, fb[i], e);
                fc[i] = add2(fc[i], e);
              } else {
                f2x e, f;
                fold2<NEG>(fa[i], x, fa[i], e);
                two_sum2(fb[i], e, fb[i], f);
                fc[i] = add2(fc[i], f);
              }
            }
          };
          auto release = [&](int g) {
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(gfree0 + 8 * g);
          };
          tmem_ld32(taddr + 6 * FX_BN, ga);
#define FX_FOLD(G, CUR, NXT)                    \
  tmem_wait_ld();                               \
  pin32(CUR);                                   \
  release(G);                                   \
  if (G > 0) tmem_ld32(taddr + (uint32_t)((G + NG - 1) % NG * FX_BN), NXT); \
  fold(G, CUR);
          FX_FOLD(6, ga, gb)
          FX_FOLD(5, gb, ga)
          FX_FOLD(4, ga, gb)
          FX_FOLD(3, gb, ga)
          FX_FOLD(2, ga, gb)
          FX_FOLD(1, gb, ga)
          FX_FOLD(0, ga, gb)
#undef FX_FOLD
        }
        if (!ok) break;
        if (!live) continue;
#pragma unroll
        for (int cg = 0; cg < 4; ++cg) {
#pragma unroll
          for (int i = 0; i < 8; i += 2) {
            const int a0 = lane * FX_EPI_COLS + (i ^ (lane >> 2)), a1 = lane * FX_EPI_COLS + ((i + 1) ^ (lane >> 2));
            upk2(fa[cg * 4 + i / 2], tb[a0], tb[a1]);
            upk2(fb[cg * 4 + i / 2], tb[a0 + 256], tb[a1 + 256]);
            upk2(fc[cg * 4 + i / 2], tb[a0 + 512], tb[a1 + 512]);
          }
          __syncwarp();
          const int col = colh + cg * FX_EPI_COLS + cl;
          const int eb = __shfl_sync(0xffffffffu, ebl, cg * FX_EPI_COLS + cl);
          // partly rolled: 32 copies of the rounding made the kernel's code so long
          // that a launch of one tile took 34 us, mostly fetching instructions
#pragma unroll 4
          for (int it = 0; it < 8; ++it) {
            const int row = row0 + 4 * it + rl, at = (4 * it + rl) * FX_EPI_COLS + (cl ^ it);
            const int sh = eb + __shfl_sync(0xffffffffu, ea, 4 * it + rl);
            if (interior || (row < p.M && col < p.N && !(p.lower && col > row))) {
              double *dst = base + (long long)row * ld + col;
              double v = triple_to_f64(tb[at], tb[at + 256], tb[at + 512], sh);
              if (late >> (8 * cg + it) & 1u) v = *dst + v;
              *dst = v;
            }
          }
          __syncwarp();
        }
      }
    }
    if (!ok && lane == 0) report();
  }

  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(TCOLS) : "memory");
  }
}

// ------------------------------------------------------------------ splitting
// Operand element (r, k) = src[r rs + k ks], zero outside M x K and, with
// tri = 1 (2), where k < r + tri_off (k > r + tri_off).  Chunk 0 covers k in
// [0, first), chunk c >= 1 covers [first + 128 (c - 1), + 128).  The entry is
// scaled by 2^(kexp[k] kexp_sign - E_r).  Entries above 2^30 after scaling are
// set to 2^30 when sat is 1 (a row of an indefinite matrix: its pivot fails
// either way); otherwise those from 2^100 on become NaN (over_out says so, and by
// how much); NaN stays NaN (codes: both left out, the row is flagged).  Plane p of row r: dst[p plane + (r + row offset) kpad + ..];
// ABS adds plane S with the magnitudes, rounded toward zero to BF16.  One row per
// warp, 8 rows (8 KiB) per CTA, as in ozaki.cu's split.
struct FxOperand {
  const double *src;
  long long rs, ks, src_stride;
  int M, K, row_end, kpad;
  const int *rexp;
  int rexp_mul;          // 0: one exponent for all rows, less rexp_sub[r]
  const int *rexp_sub;
  int *rexp_out;         // non-null (one chunk): rows are scaled by their own largest entry, exponents written here
  int *block_out;        // non-null: largest exponent of all entries, each plus row_exps[r] and, in the rows from
  int block_rows;        // block_rows on, the entry's kexp; less kBlockMargin
  const int *row_exps;
  int *over_out;         // non-null (seven slices, rexp_mul 0): takes *rexp, or where entries of 2^100 and more were met
                         // the common exponent that puts the largest 2^kBlockMargin above the scale
  const int *alt;        // non-null (the same): such an exponent; the launch does nothing unless it is above *rexp, and
                         // splits everything again with it otherwise
  int *counts;           // per row: entries of at least 2^-5 of the row's scale (null: not counted)
  int rexp_stride, tri, tri_off;
  int vec;               // per batch entry of rexp_sub, row_exps and kexp; block_out has one each
  const int *nblk;       // non-null: F64xBatch
  int act, mb, kb, skip_zero;  // skip_zero: chunks of zeros only (tri = 1) are not written
  unsigned short *dst;
  long long plane, dst_stride;
};
struct FxSplit {
  FxOperand op[2];
  int blocks0;           // row blocks of op[0]; the rest of grid.y is op[1]
  int first;
  const int *kexp;
  int codes, kexp_sign, sat;
};
constexpr int kCountExp = -5;
// A block column's common scale lies 2^50 below its largest entry: entries up to
// 2^100 above the scale and chunks down to 2^-70 below it keep all their slices
// in FP32's range, so columns 2^-120 below the largest lose nothing and the
// finished diagonal block may be 2^50 above it.  It is when the equilibrated block's
// inverse stays below some 2^25; above that its split reports the exponent it needs
// (over_out) and the block column is split again with that (alt).
constexpr int kBlockMargin = 50;
constexpr int kNoExp = -100000;  // exponent of nothing but zeros
template <int S, bool ABS>
__global__ void __launch_bounds__(256) f64x_split_kernel(const __grid_constant__ FxSplit p) {
  __shared__ double tile[8][129];
  const bool second = (int)blockIdx.y >= p.blocks0;
  const FxOperand &o = p.op[second ? 1 : 0];
  const int c = blockIdx.x, r0 = ((int)blockIdx.y - (second ? p.blocks0 : 0)) * 8;
  const double *src = o.src + (long long)blockIdx.z * o.src_stride;
  const int kbeg = (c == 0) ? 0 : p.first + (c - 1) * FX_CHUNK;
  if (o.nblk) {
    const int blocks = __ldg(o.nblk + blockIdx.z);
    if (blocks <= o.act || (o.mb >= 0 && r0 >= FX_CHUNK * (blocks - o.mb)) || (o.kb >= 0 && c >= blocks - o.kb) ||
        (o.skip_zero && (c + 1) * FX_CHUNK <= r0))
      return;
  }
  constexpr bool RESCALES = S == kF64xSlices && !ABS;  // has over_out and alt
  if (RESCALES && o.alt && __ldg(o.alt) <= __ldg(o.rexp)) return;
  const size_t vec = (size_t)blockIdx.z * o.vec;
  const int klen = (c == 0) ? min(p.first, o.K) : min(FX_CHUNK, o.K - kbeg);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = r0 + warp;
  auto inside = [&](int row, int kk) {
    const int k = kbeg + kk;
    return row < o.M && kk < klen && !(o.tri == 1 && k < row + o.tri_off) && !(o.tri == 2 && k > row + o.tri_off);
  };
  auto entry = [&](int row, int kk) {
    const int k = kbeg + kk;
    const bool swap = o.tri == 3 && k > row;
    return src[(long long)(swap ? k : row) * o.rs + (long long)(swap ? row : k) * o.ks];
  };
  double val[4];  // row r, K entries 4 lane ..
  if (o.ks == 1 && o.tri != 3) {
    // rows lie along K: a thread's entries are contiguous (two 16-byte loads where
    // the row allows), and no warp waits for another (the splits of a batch of 512
    // 9.3 -> 8.4 ms, the batch 43.1 -> 42.4 ms)
    if (r >= o.row_end) return;
    const double *at = src + (long long)r * o.rs + kbeg + lane * 4;
    if (((uintptr_t)at & 15) == 0 && r < o.M && lane * 4 + 3 < klen) {
      const double2 a = *reinterpret_cast<const double2 *>(at), b = *reinterpret_cast<const double2 *>(at + 2);
      val[0] = a.x;
      val[1] = a.y;
      val[2] = b.x;
      val[3] = b.y;
#pragma unroll
      for (int i = 0; i < 4; ++i) val[i] = inside(r, lane * 4 + i) ? val[i] : 0.0;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) val[i] = inside(r, lane * 4 + i) ? entry(r, lane * 4 + i) : 0.0;
    }
  } else {
    const bool along = o.ks == 1;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int idx = threadIdx.x + 256 * it;
      const int rr = along ? idx >> 7 : idx & 7, kk = along ? idx & 127 : idx >> 3;
      tile[rr][kk] = inside(r0 + rr, kk) ? entry(r0 + rr, kk) : 0.0;
    }
    __syncthreads();
    if (r >= o.row_end) return;  // past the last barrier
#pragma unroll
    for (int i = 0; i < 4; ++i) val[i] = tile[warp][lane * 4 + i];
  }
  int E = 0, common = 0;
  if (o.rexp && r < o.M) {
    E = __ldg(RESCALES && o.alt ? o.alt : o.rexp + (size_t)blockIdx.z * o.rexp_stride + (size_t)r * o.rexp_mul);
    common = E;
    if (p.codes) E = code_exponent(E);
    if (E < kNoExp) E = 0;  // no entry at all
    if (o.rexp_sub) E -= __ldg(o.rexp_sub + vec + r);
  }
  unsigned long long mant[4];
  int ex[4], emax = kNoExp, raw = kNoExp, over = kNoExp;
  uint32_t neg = 0, nan = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(val[i]);
    const int e = (int)((u >> 52) & 0x7FF);
    int kx = 0;
    if (p.kexp) {
      const int k = kbeg + lane * 4 + i;
      kx = (k < o.K) ? p.kexp_sign * __ldg(p.kexp + vec + k) : 0;
    }
    neg |= (uint32_t)(u >> 63) << i;
    mant[i] = (u & ((1ull << 52) - 1)) | (1ull << 52);
    ex[i] = e - 1023 - E + kx;
    if (e == 0 || (e == 2047 && p.codes)) {
      mant[i] = 0;
      ex[i] = kNoExp;
    } else if (e == 2047 || (ex[i] >= 30 && !o.rexp_out)) {
      const bool isnan = e == 2047 && (u << 12) != 0;
      if (RESCALES && e != 2047 && ex[i] >= 100) over = max(over, ex[i]);
      if (isnan || (!p.sat && (e == 2047 || ex[i] >= 100))) nan |= 1u << i;
      if (p.sat || nan >> i & 1u) {
        mant[i] = 1ull << 52;
        ex[i] = 30;
      }
    }
    if (e != 0 && e != 2047) raw = max(raw, e - 1022 + (r < o.block_rows ? 0 : kx));
    emax = max(emax, ex[i]);
  }
  if (o.counts) {
    int n = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) n += ex[i] >= kCountExp ? 1 : 0;
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0 && n > 0) atomicAdd(o.counts + (size_t)blockIdx.z * o.rexp_stride + r, n);
  }
  emax = __reduce_max_sync(0xffffffffu, emax);
  if (RESCALES && o.over_out) {
    over = __reduce_max_sync(0xffffffffu, over);
    if (over > kNoExp) common = (common < kNoExp ? 0 : common) + over + 1 - kBlockMargin;
    if (lane == 0 && r < o.M) atomicMax(o.over_out, common);
  }
  if (o.block_out) {
    raw = __reduce_max_sync(0xffffffffu, raw);
    if (lane == 0 && raw > kNoExp && r < o.M) atomicMax(o.block_out + blockIdx.z, raw + __ldg(o.row_exps + vec + r) - kBlockMargin);
  }
  int shift = 0;  // the row's own exponent, when it is found here
  if (o.rexp_out && r < o.M) {
    shift = emax > kNoExp ? emax + 1 : 0;
    if (lane == 0) o.rexp_out[(size_t)blockIdx.z * o.rexp_stride + r] = shift;
  }
  unsigned short *dst =
      o.dst + (long long)blockIdx.z * o.dst_stride + (long long)r * o.kpad + (long long)c * FX_CHUNK + lane * 4;
  if (ABS) {  // magnitudes, rounded toward zero to BF16
    uint32_t h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      h[i] = (mant[i] != 0 && ex[i] >= -126)
                 ? ((uint32_t)(ex[i] + 127) << 7) | ((uint32_t)(mant[i] >> 45) & 0x7Fu) : 0u;
    *(uint2 *)(dst + S * o.plane) = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
  }
  // X + 128 (1 + 256 + ..) has the balanced digits plus 128 as its lower bytes
  unsigned long long Y[4];
  uint32_t top[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    unsigned long long X = 0;
    const int sh = (emax - ex[i]) - (8 * S - 53);
    if (mant[i] != 0) {
      if (sh <= 0) X = mant[i] << (-sh);
      else if (sh < 64) X = (mant[i] + (1ull << (sh - 1))) >> sh;
    }
    Y[i] = X + (0x8080808080808080ull >> (64 - 8 * (S - 1)));
    top[i] = (uint32_t)(Y[i] >> (8 * (S - 1)));
    if (S == 8 && Y[i] < X) top[i] += 256;  // the sum left 64 bits: leading digit 256
  }
#pragma unroll
  for (int pp = 0; pp < S; ++pp) {
    const int fexp = emax - shift + 1 - 8 * (pp + 1) + 127;
    const uint32_t sb = fexp >= 1 ? (uint32_t)fexp << 23 : 0u;
    uint32_t h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t byte = pp == 0 ? top[i] : (uint32_t)(Y[i] >> (8 * (S - 1 - pp))) & 255u;
      const float d = __fsub_rn(__uint_as_float(0x4B000000u | byte), pp == 0 ? 8388608.0f : 8388736.0f);
      h[i] = __float_as_uint(__fmul_rn(d, __uint_as_float(sb)));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      h[i] ^= (neg >> i & 1u) << 31;
      if (pp == 0 && (nan >> i & 1u)) h[i] = 0x7FC00000u;
    }
    *(uint2 *)(dst + pp * o.plane) = make_uint2((h[0] >> 16) | (h[1] & 0xFFFF0000u), (h[2] >> 16) | (h[3] & 0xFFFF0000u));
  }
}

// Code of every operand row's largest magnitude over k in [0, K): 0 for a row of
// zeros, 2047 with an infinity or a NaN, else the largest biased exponent (a
// denormal counts as 1).  codes is zero on entry; K ranges meet by atomicMax.
struct FxCodes {
  FxOperand op[2];  // rexp unused; counts: the codes
  int blocks0, kper;
};
__global__ void __launch_bounds__(256) row_codes_kernel(const __grid_constant__ FxCodes p) {
  const bool second = (int)blockIdx.x >= p.blocks0;
  const FxOperand &o = p.op[second ? 1 : 0];
  const int blk = (int)blockIdx.x - (second ? p.blocks0 : 0);
  const double *src = o.src + (long long)blockIdx.z * o.src_stride;
  int *codes = o.counts + (size_t)blockIdx.z * o.rexp_stride;
  const int k0 = blockIdx.y * p.kper, k1 = min(o.K, k0 + p.kper);
  auto code = [&](int r, int k) -> int {
    if (o.tri == 1 && k < r + o.tri_off) return 0;
    if (o.tri == 2 && k > r + o.tri_off) return 0;
    const unsigned long long u =
        (unsigned long long)__double_as_longlong(src[(long long)r * o.rs + (long long)k * o.ks]);
    const int e = (int)((u >> 52) & 0x7FF);
    return e == 0 && (u << 1) != 0 ? 1 : e;
  };
  int m = 0;
  if (o.ks == 1) {  // a warp per row
    const int r = blk * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= o.M) return;
#pragma unroll 4
    for (int k = k0 + lane; k < k1; k += 32) m = max(m, code(r, k));
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0 && m > 0) atomicMax(&codes[r], m);
  } else {  // 32 rows x 8 K lanes per CTA
    const int r = blk * 32 + (threadIdx.x & 31), kl = threadIdx.x >> 5;
    if (r >= o.M) return;
#pragma unroll 4
    for (int k = k0 + kl; k < k1; k += 8) m = max(m, code(r, k));
    if (m > 0) atomicMax(&codes[r], m);
  }
}

// Blocks that the row counts alone show to be safe: with cA of a row's and cB of
// a column's K entries at or above 2^-5 of their scales, at least cA + cB - K
// of the K terms are 2^-10 or more; two such terms exceed the 2^-9.5 that a
// checked product needs.  A warp per block row and kCertCols block columns; rows of zeros are safe, bad rows
// (FxCodes) never are.
constexpr int kCertCols = 8;
__global__ void __launch_bounds__(256)
certify_kernel(int M, int N, int K, int rowsA, int rowsB, const int *codes, const int *counts, unsigned char *flags,
               int flag_ld, long long flag_stride) {
  const int lane = threadIdx.x & 31, br = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y;
  if (32 * br >= M) return;
  const int batch = gridDim.y;
  auto low = [&](int base, int r, int n) -> int {
    int v = 1 << 29;
    if (r < n) {
      const int c = __ldg(codes + base + r);
      v = code_bad(c) ? -(1 << 29) : (c == kCodeZero ? 1 << 29 : __ldg(counts + base + r));
    }
    return v;
  };
  const int a = __reduce_min_sync(0xffffffffu, low(b * rowsA, 32 * br + lane, M));
  const int c0 = blockIdx.z * kCertCols, nb = min((N + 31) / 32, c0 + kCertCols);
#pragma unroll 4
  for (int bc = c0; bc < nb; ++bc) {
    const int c = __reduce_min_sync(0xffffffffu, low(batch * rowsA + b * rowsB, 32 * bc + lane, N));
    if (lane == 0 && a > -(1 << 28) && c > -(1 << 28) && (long long)a + c - K >= 2)
      flags[(size_t)b * flag_stride + (size_t)br * flag_ld + bc] = 1;
  }
}

// C = C + sum of partial tiles (or their sum), in order; flagged blocks are left alone.
__global__ void f64x_reduce_kernel(int M, int N, int splits, const double *partial, double *C, long long ldc, int lower,
                                   int accumulate, const unsigned char *flags, int flag_ld) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)M * N) return;
  const int row = (int)(idx / N), col = (int)(idx - (long long)row * N);
  if (lower && col > row) return;
  if (flags && !flags[(size_t)(row / 32) * flag_ld + col / 32]) return;
  double s = 0.0;
  for (int z = 0; z < splits; ++z) s += partial[(size_t)z * M * N + idx];
  double *dst = C + (long long)row * ldc + col;
  *dst = accumulate ? *dst + s : s;
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *q = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &q, 12000, cudaEnableDefault, &r) == cudaSuccess &&
        r == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)q;
  });
  return fn;
}
bool make_map(CUtensorMap *m, const void *base, int kpad, long long rows, int planes, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)kpad, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)kpad * 2, (cuuint64_t)rows * kpad * 2};
  cuuint32_t box[3] = {(cuuint32_t)FX_BK, (cuuint32_t)box_rows, (cuuint32_t)planes};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void *)base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int S, bool NEG, bool CHECK>
cudaError_t launch_product(const CUtensorMap &ma, const CUtensorMap &mb, const FxParams &p, int grid, double flops,
                           double bytes, cudaStream_t s) {
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(f64x_gemm_kernel<S, NEG, CHECK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         fx_smem(S));
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  GPC_LAUNCH(GPC_TRACE_GEMM_MIXED, flops, bytes, s,
             launch_k(f64x_gemm_kernel<S, NEG, CHECK>, grid, FX_THREADS, fx_smem(S), s, ma, mb, p));
  return cudaGetLastError();
}

long long count_tiles(const FxParams &p) {
  if (!p.lower) return (long long)p.tiles_m * p.tiles_n;
  long long t = 0;
  for (int tm = 0; tm < p.tiles_m; ++tm) t += std::min(p.tiles_n, (tm * FX_BM + FX_BM - 1) / FX_BN + 1);
  return t;
}

cudaError_t carveout_max(const void *fn, bool (&done)[64]) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || done[dev]) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

}  // namespace

size_t f64x_slice_bytes(int rows, int kchunks, bool wide) {
  const size_t rp = align_up((size_t)std::max(rows, 1), FX_BM);
  return align_up((size_t)(wide ? kF64xWide : kF64xSlices) * rp * (size_t)kchunks * FX_CHUNK * 2, 1024);
}

cudaError_t f64x_split(const double *src, long long rs, long long ks, int M, int K, int first, const SliceBuf &out,
                       const int *rexp, const int *kexp, int kexp_sign, bool saturate, cudaStream_t s,
                       int chunk_offset, int row_offset, const F64xRow &row) {
  if (M <= 0 || K <= 0) return cudaSuccess;
  const int op_chunks = (K <= first) ? 1 : 1 + (K - first + FX_CHUNK - 1) / FX_CHUNK;
  const int chunks = std::min(op_chunks, out.kpad / FX_CHUNK - chunk_offset);
  if (chunks <= 0 || row_offset < 0 || row_offset + M > out.rows_pad) return cudaErrorInvalidValue;
  static bool carve[2][64] = {};
  const auto fx_split_kernel = row.wide ? f64x_split_kernel<kF64xWide, false> : f64x_split_kernel<kF64xSlices, false>;
  if (cudaError_t e = carveout_max((const void *)fx_split_kernel, carve[row.wide]); e != cudaSuccess) return e;
  FxSplit p = {};
  FxOperand &o = p.op[0];
  o.src = src;
  o.rs = rs;
  o.ks = ks;
  o.M = M;
  o.K = K;
  o.row_end = row_offset > 0 ? M : out.rows_pad;
  o.kpad = out.kpad;
  o.rexp = rexp;
  o.rexp_mul = row.rexp_sub ? 0 : 1;
  o.rexp_sub = row.rexp_sub;
  o.rexp_out = row.rexp_out;
  o.block_out = row.block_out;
  o.block_rows = row.block_rows;
  o.row_exps = row.row_exps;
  o.over_out = row.over_out;
  o.alt = row.alt;
  o.tri = row.tri;
  if (row.rexp_out && chunks != 1) return cudaErrorInvalidValue;
  if (row.block_out)
    if (cudaError_t e = cudaMemsetAsync(row.block_out, 0x80, sizeof(int), s); e != cudaSuccess) return e;
  o.dst = (unsigned short *)out.base + (long long)row_offset * out.kpad + (long long)chunk_offset * FX_CHUNK;
  o.plane = (long long)out.rows_pad * out.kpad;
  p.first = first;
  p.kexp = kexp;
  p.kexp_sign = kexp_sign;
  p.sat = saturate ? 1 : 0;
  p.blocks0 = (o.row_end + 7) / 8;
  dim3 grid((unsigned)chunks, (unsigned)p.blocks0);
  const int S = row.wide ? kF64xWide : kF64xSlices;
  GPC_LAUNCH(GPC_TRACE_SPLIT, 0.0, 8.0 * M * K + 2.0 * S * (double)o.row_end * chunks * FX_CHUNK, s,
             launch_k(fx_split_kernel, grid, 256, 0, s, p));
  return cudaGetLastError();
}

cudaError_t f64x_split_blocks(int nblk, int first, const double *src, long long ld0, long long ld, long long off1,
                              long long stride, void *out, int *exps, cudaStream_t s) {
  constexpr int b = FX_CHUNK;
  const size_t bytes = f64x_slice_bytes(b, 1, true);
  F64xRow row;
  row.wide = true;
  row.rexp_out = exps;
  row.tri = 1;
  if (cudaError_t e = f64x_split(src, 1, ld0, first, first, first, slice_view(out, b, 1), nullptr, nullptr, 0, false, s,
                                 0, 0, row);
      e != cudaSuccess || nblk == 1)
    return e;
  FxSplit p = {};
  FxOperand &o = p.op[0];
  o.src = src + off1;
  o.rs = 1;
  o.ks = ld;
  o.src_stride = stride;
  o.M = o.K = o.row_end = o.kpad = b;
  o.rexp_out = exps + b;
  o.rexp_stride = b;
  o.tri = 1;
  o.dst = (unsigned short *)((char *)out + bytes);
  o.plane = (long long)b * b;
  o.dst_stride = (long long)(bytes / 2);
  p.first = b;
  p.blocks0 = b / 8;
  GPC_LAUNCH(GPC_TRACE_SPLIT, 0.0, (8.0 + 2.0 * kF64xWide) * b * b * (nblk - 1), s,
             launch_k(f64x_split_kernel<kF64xWide, false>, dim3(1, b / 8, (unsigned)(nblk - 1)), 256, 0, s, p));
  return cudaGetLastError();
}

cudaError_t f64x_gemm(const SliceBuf &A, int a_row0, int a_k0, const SliceBuf &B, int b_row0, int b_k0, int M, int N,
                      int chunks, bool lower, const int *ra, const int *rb, double *C, long long ldc, int splits,
                      double *partial, int *err, cudaStream_t s, int max_ctas, int kdepth, int max_items,
                      const int *ra_sub, bool wide) {
  if (M <= 0 || N <= 0 || chunks <= 0) return cudaSuccess;
  if (kdepth <= 0) kdepth = FX_CHUNK;
  if (kdepth > FX_CHUNK || kdepth % FX_BK || (wide && splits > 1)) return cudaErrorInvalidValue;
  CUtensorMap ma, mb;
  const int S = wide ? kF64xWide : kF64xSlices;
  if (!make_map(&ma, A.base, A.kpad, A.rows_pad, S, FX_BM) || !make_map(&mb, B.base, B.kpad, B.rows_pad, S, FX_BN))
    return cudaErrorInvalidValue;
  FxParams p = {};
  p.M = M;
  p.N = N;
  p.chunks = chunks;
  p.qpc = kdepth / FX_BK;
  p.a_row0 = a_row0;
  p.b_row0 = b_row0;
  p.a_k0 = a_k0;
  p.b_k0 = b_k0;
  p.lower = lower ? 1 : 0;
  p.splits = std::max(1, std::min(splits, chunks));
  p.tiles_m = (M + FX_BM - 1) / FX_BM;
  p.tiles_n = (N + FX_BN - 1) / FX_BN;
  p.per_batch = (int)count_tiles(p);
  p.num_work = p.per_batch * p.splits;
  p.accumulate = wide ? 0 : 1;
  p.ra = ra;
  p.ra_mul = ra_sub ? 0 : 1;
  p.ra_sub = ra_sub;
  p.rb = rb;
  p.C = C;
  p.ldc = ldc;
  p.partial = p.splits > 1 ? partial : nullptr;
  p.err = err;
  p.gerr = error_word();
  p.wait_ns = faults().wait_ns;
  p.no_loads = faults().ozaki_no_loads;
  const double mn = !lower ? (double)M * N
                           : (M >= N ? 0.5 * (double)N * (N + 1) + (double)(M - N) * N : 0.5 * (double)M * (M + 1));
  const double flops = 2.0 * mn * (double)chunks * kdepth * (S * (S + 1) / 2);
  const double bytes = 16.0 * mn + (double)(M + N) * chunks * kdepth * 2 * S;
  p.sub = 1;
  if (max_ctas == 0 && 4 * p.num_work <= sm_count()) {
    p.sub = 4;
    p.num_work *= 4;
  }
  int grid = std::min(p.num_work, max_ctas > 0 ? std::min(max_ctas, sm_count()) : sm_count());
  if (max_items > 0) grid = std::max(grid, (p.num_work + max_items - 1) / max_items);
  cudaError_t e = wide ? launch_product<kF64xWide, false, false>(ma, mb, p, grid, flops, bytes, s)
                       : launch_product<kF64xSlices, true, false>(ma, mb, p, grid, flops, bytes, s);
  if (e != cudaSuccess || p.splits == 1) return e;
  const long long total = (long long)M * N;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 8.0 * (p.splits + 2) * mn, s,
             launch_k(f64x_reduce_kernel, (unsigned)((total + 255) / 256), 256, 0, s, M, N, p.splits, (const double *)partial,
                      C, ldc, lower ? 1 : 0, 1, (const unsigned char *)nullptr, 0));
  return cudaGetLastError();
}

// ------------------------------------------------------------------ scales of the factorisation and its adjoint
namespace {

// e_i with K_ii < 4^e_i (|L_ij| <= sqrt(K_ii) < 2^e_i); 0 where K_ii is no
// positive number (the factorisation fails there).  The factor of denormals is normal.
__global__ void diag_exps_kernel(int n, const double *K, long long ldk, int *rexp, const int *nblk, long long stride,
                                 int vec) {
  if (nblk) n = FX_CHUNK * __ldg(nblk + blockIdx.z);
  K += blockIdx.z * stride;
  rexp += blockIdx.z * vec;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned long long u = (unsigned long long)__double_as_longlong(K[(long long)i * ldk + i]);
  const int b = (int)(u >> 52);                              // the sign bit too: negative entries are above 2047
  const int e = b > 0 ? b : 12 - __clzll((long long)u);      // goes on below 1 for denormals
  rexp[i] = (u != 0 && b < 2047) ? (e - 1022 + 1) >> 1 : 0;
}
// rexp[i]: exponent E, 2^E above the largest entry of row i of the lower triangle.  A warp per row.
__global__ void __launch_bounds__(256) lower_row_exps_kernel(int n, const double *L, long long ldl, int *rexp, const int *nblk, long long stride,
                      int vec) {
  if (nblk) n = FX_CHUNK * __ldg(nblk + blockIdx.z);
  L += blockIdx.z * stride;
  rexp += blockIdx.z * vec;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  int m = 0;
#pragma unroll 4
  for (int k = lane; k <= i; k += 32) {
    const int e = (int)((unsigned long long)__double_as_longlong(L[(long long)i * ldl + k]) >> 52) & 0x7FF;
    m = max(m, e == 2047 ? 0 : e);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) rexp[i] = m > 0 ? m - 1022 : 0;
}
// cexp[c]: the same for column c of the rows scaled by 2^-rexp.  32 columns and
// 64 rows per CTA; cexp holds large negative numbers on entry.
__global__ void __launch_bounds__(256)
lower_col_exps_kernel(int n, const double *L, long long ldl, const int *rexp, int *cexp, const int *nblk,
                      long long stride, int vec) {
  if (nblk) n = FX_CHUNK * __ldg(nblk + blockIdx.z);
  L += blockIdx.z * stride;
  rexp += blockIdx.z * vec;
  cexp += blockIdx.z * vec;
  const int c = blockIdx.x * 32 + (threadIdx.x & 31), t0 = blockIdx.y * 64;
  if (c >= n || t0 + 63 < blockIdx.x * 32) return;
  int m = kNoExp;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int t = t0 + (threadIdx.x >> 5) + 8 * q;
    if (t < n && t >= c) {
      const int e = (int)((unsigned long long)__double_as_longlong(L[(long long)t * ldl + c]) >> 52) & 0x7FF;
      if (e != 0 && e != 2047) m = max(m, e - 1022 - __ldg(rexp + t));
    }
  }
  if (m > kNoExp) atomicMax(&cexp[c], m);
}
// *out: 2^(*out + kBlockMargin) above the largest entry of the nb x nb block with row r scaled by 2^rexp[r].
__global__ void __launch_bounds__(256)
block_exp_kernel(int nb, const double *A, long long lda, const int *rexp, int *out) {
  __shared__ int red[8];
  int m = kNoExp;
  for (int idx = threadIdx.x; idx < nb * nb; idx += 256) {
    const int r = idx / nb, c = idx - r * nb;
    const int e = (int)((unsigned long long)__double_as_longlong(A[(long long)r * lda + c]) >> 52) & 0x7FF;
    if (e != 0 && e != 2047) m = max(m, e - 1022 + rexp[r]);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = max(m, red[w]);
    *out = m > kNoExp ? m - kBlockMargin : 0;
  }
}

}  // namespace

cudaError_t f64x_diag_exps(int n, const double *K, long long ldk, int *rexp, cudaStream_t s) {
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 12.0 * n, s,
             launch_k(diag_exps_kernel, (unsigned)((n + 255) / 256), 256, 0, s, n, K, ldk, rexp, (const int *)nullptr, 0ll,
                      0));
  return cudaGetLastError();
}
cudaError_t f64x_lower_exps(int n, const double *L, long long ldl, int *rexp, int *cexp, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(cexp, 0x80, (size_t)n * sizeof(int), s);
  if (e != cudaSuccess) return e;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 4.0 * n * (n + 1.0), s,
             launch_k(lower_row_exps_kernel, (unsigned)((n + 7) / 8), 256, 0, s, n, L, ldl, rexp, (const int *)nullptr, 0ll,
                      0));
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 4.0 * n * (n + 1.0), s,
             launch_k(lower_col_exps_kernel, dim3((unsigned)((n + 31) / 32), (unsigned)((n + 63) / 64)), 256, 0, s, n, L,
                      ldl, (const int *)rexp, cexp, (const int *)nullptr, 0ll, 0));
  return cudaGetLastError();
}
cudaError_t f64x_diag_exps_batch(const F64xBatch &b, int n, const double *K, long long ldk, long long stride, int vec,
                                 int *rexp, cudaStream_t s) {
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 12.0 * n * b.count, s,
             launch_k(diag_exps_kernel, dim3((unsigned)((n + 255) / 256), 1, (unsigned)b.count), 256, 0, s, n, K, ldk,
                      rexp, b.nblk, stride, vec));
  return cudaGetLastError();
}
cudaError_t f64x_lower_exps_batch(const F64xBatch &b, int n, const double *L, long long ldl, long long stride, int vec,
                                  int *rexp, int *cexp, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(cexp, 0x80, (size_t)b.count * vec * sizeof(int), s);
  if (e != cudaSuccess) return e;
  const double bytes = 4.0 * n * (n + 1.0) * b.count;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, bytes, s,
             launch_k(lower_row_exps_kernel, dim3((unsigned)((n + 7) / 8), 1, (unsigned)b.count), 256, 0, s, n, L, ldl,
                      rexp, b.nblk, stride, vec));
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, bytes, s,
             launch_k(lower_col_exps_kernel, dim3((unsigned)((n + 31) / 32), (unsigned)((n + 63) / 64), (unsigned)b.count),
                      256, 0, s, n, L, ldl, (const int *)rexp, cexp, b.nblk, stride, vec));
  return cudaGetLastError();
}

cudaError_t f64x_split_batch(const F64xBatch &b, const F64xBatchSplit &q, cudaStream_t s) {
  if (b.count <= 0 || q.M <= 0 || q.K <= 0) return cudaSuccess;
  if (q.M % FX_CHUNK || q.K % FX_CHUNK || (q.rexp_out && q.K != FX_CHUNK)) return cudaErrorInvalidValue;
  static bool carve[2][64] = {};
  const auto fx_split_kernel = q.wide ? f64x_split_kernel<kF64xWide, false> : f64x_split_kernel<kF64xSlices, false>;
  if (cudaError_t e = carveout_max((const void *)fx_split_kernel, carve[q.wide]); e != cudaSuccess) return e;
  FxSplit p = {};
  FxOperand &o = p.op[0];
  o.src = q.src;
  o.rs = q.rs;
  o.ks = q.ks;
  o.src_stride = q.stride;
  o.M = o.row_end = q.M;
  o.K = q.K;
  o.kpad = q.kpad;
  o.rexp = q.rexp ? q.rexp : q.rexps;
  o.rexp_mul = q.rexp ? 0 : 1;
  o.rexp_sub = q.rexp_sub;
  o.rexp_stride = q.rexp ? 1 : q.vec;
  o.rexp_out = q.rexp_out;
  o.block_out = q.block_out;
  o.block_rows = q.block_out ? FX_CHUNK : 0;
  o.row_exps = q.row_exps;
  o.tri = q.tri;
  o.vec = q.vec;
  o.nblk = b.nblk;
  o.act = b.act;
  o.mb = b.mb;
  o.kb = b.kb;
  o.skip_zero = q.skip_zero ? 1 : 0;
  o.dst = (unsigned short *)q.out + (long long)q.chunk0 * FX_CHUNK;
  o.plane = (long long)b.count * q.rows * q.kpad;
  o.dst_stride = (long long)q.rows * q.kpad;
  p.first = FX_CHUNK;
  p.kexp = q.kexp;
  p.kexp_sign = q.kexp_minus ? -1 : 1;
  p.sat = q.saturate ? 1 : 0;
  p.blocks0 = q.M / 8;
  const int S = q.wide ? kF64xWide : kF64xSlices;
  if (q.block_out)
    if (cudaError_t e = cudaMemsetAsync(q.block_out, 0x80, (size_t)b.count * sizeof(int), s); e != cudaSuccess) return e;
  GPC_LAUNCH(GPC_TRACE_SPLIT, 0.0, (8.0 + 2.0 * S) * q.M * q.K * b.count, s,
             launch_k(fx_split_kernel, dim3((unsigned)(q.K / FX_CHUNK), (unsigned)(q.M / 8), (unsigned)b.count), 256, 0,
                      s, p));
  return cudaGetLastError();
}

cudaError_t f64x_gemm_batch(const F64xBatch &b, const F64xBatchGemm &g, int *err, cudaStream_t s) {
  if (b.count <= 0 || g.M <= 0 || g.N <= 0 || g.chunks <= 0) return cudaSuccess;
  const int S = g.wide ? kF64xWide : kF64xSlices;
  CUtensorMap ma, mb;
  if (!make_map(&ma, g.A, g.a_kpad, b.count * g.a_rows, S, FX_BM) ||
      !make_map(&mb, g.B, g.b_kpad, b.count * g.b_rows, S, FX_BN))
    return cudaErrorInvalidValue;
  FxParams p = {};
  p.M = g.M;
  p.N = g.N;
  p.chunks = g.chunks;
  p.qpc = FX_CHUNK / FX_BK;
  p.a_row0 = g.a_row0;
  p.b_row0 = g.b_row0;
  p.a_k0 = g.a_k0;
  p.b_k0 = g.b_k0;
  p.a_rows = g.a_rows;
  p.b_rows = g.b_rows;
  p.lower = g.lower ? 1 : 0;
  p.splits = 1;
  p.tiles_m = (g.M + FX_BM - 1) / FX_BM;
  p.tiles_n = (g.N + FX_BN - 1) / FX_BN;
  p.per_batch = (int)count_tiles(p);
  p.num_work = p.per_batch * b.count;
  p.accumulate = g.wide ? 0 : 1;
  p.ra = g.ra;
  p.ra_mul = g.ra_sub ? 0 : 1;
  p.ra_stride = g.ra_sub ? 1 : g.vec;
  p.ra_sub = g.ra_sub;
  p.sub_stride = g.vec;
  p.rb = g.rb;
  p.rb_stride = g.vec;
  p.nblk = b.nblk;
  p.act = b.act;
  p.mb = b.mb;
  p.nb = b.nb;
  p.kb = b.kb;
  p.C = g.C;
  p.ldc = g.ldc;
  p.sC = g.sC;
  p.err = err;
  p.gerr = error_word();
  p.wait_ns = faults().wait_ns;
  p.no_loads = faults().ozaki_no_loads;
  p.sub = 1;
  if (4 * p.num_work <= sm_count()) {
    p.sub = 4;
    p.num_work *= 4;
  }
  const int grid = std::min(p.num_work, sm_count());
  const double mn = (g.lower ? 0.5 : 1.0) * g.M * (double)g.N * b.count;
  const double flops = 2.0 * mn * g.chunks * FX_CHUNK * (S * (S + 1) / 2), bytes = 16.0 * mn;
  return g.wide ? launch_product<kF64xWide, false, false>(ma, mb, p, grid, flops, bytes, s)
                : launch_product<kF64xSlices, true, false>(ma, mb, p, grid, flops, bytes, s);
}
cudaError_t f64x_block_exp(int nb, const double *A, long long lda, const int *rexp, int *out, cudaStream_t s) {
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 8.0 * nb * nb, s, launch_k(block_exp_kernel, 1, 256, 0, s, nb, A, lda, rexp, out));
  return cudaGetLastError();
}

// ------------------------------------------------------------------ general products
namespace {

constexpr int GX_S = kF64xWide;        // slices of a checked product
constexpr int GX_PLANES = GX_S + 1;    // and the plane of leading magnitudes
constexpr size_t kGxMinScratch = size_t(8) << 20;

// Partial tiles of a split K range: at most one 128 x 64 tile of FP64 per SM.
size_t gx_partial_bytes() { return (size_t)sm_count() * FX_BM * FX_BN * sizeof(double); }

struct Panels {
  int mp, np, kp;  // rows of op(A), columns of op(B), K entries per pass (kp: a multiple of 128)
};
size_t panel_bytes(int mp, int np, int kp, int batch) {
  const size_t rows = (align_up((size_t)mp, 128) + align_up((size_t)np, 128)) * (size_t)batch;
  const size_t flags = (size_t)batch * (align_up((size_t)mp, 128) / 32) * (align_up((size_t)np, 128) / 32);
  return align_up(2 * rows * sizeof(int) + flags, 1024) +
         align_up(rows * (size_t)kp * 2 * GX_PLANES, 1024) + gx_partial_bytes() + 2048;
}
// The largest K range per pass that fits, shrinking the panels of M and N when
// less than 512 would (a pass reads and writes its outputs once).
bool choose_panels(const Gemm &g, size_t bytes, Panels &out) {
  const int kall = (g.K + 127) / 128 * 128;
  int mp = g.M, np = g.N;
  for (;;) {
    int kp = kall;
    while (kp > 128 && panel_bytes(mp, np, kp, g.batch) > bytes) kp = (kp / 2 + 127) / 128 * 128;
    // one grid row per 8 operand rows of the split, 65535 at most, however large the workspace
    const bool fits = panel_bytes(mp, np, kp, g.batch) <= bytes &&
                      align_up((size_t)mp, 128) + align_up((size_t)np, 128) <= 8 * 65535;
    if (fits && kp >= std::min(kall, 512)) {
      out = {mp, np, kp};
      return true;
    }
    if (g.batch > 1) return false;
    if (mp <= 512 && np <= 512) {
      if (fits) out = {mp, np, kp};
      return fits;
    }
    if (g.uplo != UPLO_FULL) mp = np = (mp / 2 + 127) / 128 * 128;
    else if (mp >= np) mp = (mp / 2 + 127) / 128 * 128;
    else np = (np / 2 + 127) / 128 * 128;
  }
}

cudaError_t one_panel(const Gemm &g, const Panels &pn, int mo, int no, int ko, char *ws, char *ws_end, cudaStream_t s) {
  const int M = std::min(pn.mp, g.M - mo), N = std::min(pn.np, g.N - no), K = std::min(pn.kp, g.K - ko);
  const int mpad = (int)align_up((size_t)M, 128), npad = (int)align_up((size_t)N, 128);
  const int kpad = (K + 127) / 128 * 128;
  const size_t rows = (size_t)g.batch * (mpad + npad);
  int *codes = (int *)ws, *counts = codes + rows;
  unsigned char *flags = (unsigned char *)(counts + rows);
  const size_t fbytes = (size_t)g.batch * (mpad / 32) * (npad / 32);
  unsigned short *sa = (unsigned short *)(ws + align_up(2 * rows * sizeof(int) + fbytes, 1024));
  unsigned short *sb = sa + (size_t)GX_PLANES * g.batch * mpad * kpad;
  double *partial = (double *)((char *)sa + align_up((size_t)GX_PLANES * rows * kpad * 2, 1024));
  int *cA = codes, *cB = codes + (size_t)g.batch * mpad;
  cudaError_t e = cudaMemsetAsync(ws, 0, 2 * rows * sizeof(int) + fbytes, s);
  if (e != cudaSuccess) return e;
  const double *A = g.A + (g.transA ? (long long)ko * g.lda + mo : (long long)mo * g.lda + ko);
  const double *B = g.B + (g.transB ? (long long)no * g.ldb + ko : (long long)ko * g.ldb + no);
  FxSplit sp = {};
  auto operand = [&](FxOperand &o, const double *src, bool kmajor, long long ld, long long stride, int n, int pad,
                     int tri, int tri_off, int *code, unsigned short *dst) {
    o.src = src;
    o.rs = kmajor ? ld : 1;
    o.ks = kmajor ? 1 : ld;
    o.src_stride = stride;
    o.M = n;
    o.K = K;
    o.row_end = pad;
    o.kpad = kpad;
    o.rexp = code;
    o.rexp_mul = 1;
    o.rexp_stride = pad;
    o.tri = tri;  // element (r, k) is zero for k + ko < r + panel offset (1) or > (2)
    o.tri_off = tri_off;
    o.dst = dst;
    o.plane = (long long)g.batch * pad * kpad;
    o.dst_stride = (long long)pad * kpad;
  };
  operand(sp.op[0], A, !g.transA, g.lda, g.sA, M, mpad, g.kskip == KSKIP_ROWS ? 1 : (g.kskip == KSKIP_ROWS_END ? 2 : 0),
          mo - ko, cA, sa);
  operand(sp.op[1], B, g.transB, g.ldb, g.sB, N, npad, g.kskip == KSKIP_COLS ? 1 : (g.kskip == KSKIP_COLS_END ? 2 : 0),
          no - ko, cB, sb);
  FxCodes cd = {};
  auto code_blocks = [](const FxOperand &o) { return o.ks == 1 ? (o.M + 7) / 8 : (o.M + 31) / 32; };
  const int cblocks = code_blocks(sp.op[0]) + code_blocks(sp.op[1]);
  for (int i = 0; i < 2; ++i) {
    cd.op[i] = sp.op[i];
    cd.op[i].counts = i ? cB : cA;
    sp.op[i].counts = counts + (i ? (size_t)g.batch * mpad : 0);
  }
  cd.blocks0 = code_blocks(sp.op[0]);
  // up to 64 CTAs per SM, each over at least 256 of K: short chains of loads
  const int kparts = std::max(1, std::min((K + 255) / 256, 64 * sm_count() / std::max(1, cblocks * g.batch)));
  cd.kper = (K + kparts - 1) / kparts;
  GPC_LAUNCH(GPC_TRACE_SPLIT, 0.0, 8.0 * g.batch * ((double)M + N) * K, s,
             row_codes_kernel<<<dim3((unsigned)cblocks, (unsigned)kparts, (unsigned)g.batch), 256, 0, s>>>(cd));
  sp.first = FX_CHUNK;
  sp.codes = 1;
  sp.blocks0 = mpad / 8;
  GPC_LAUNCH(GPC_TRACE_SPLIT, 0.0, g.batch * (8.0 * ((double)M + N) * K + 2.0 * GX_PLANES * (double)(mpad + npad) * kpad),
             s,
             f64x_split_kernel<GX_S, true><<<dim3((unsigned)(kpad / FX_CHUNK), (unsigned)((mpad + npad) / 8),
                                                  (unsigned)g.batch), 256, 0, s>>>(sp));
  const long long rowsA = (long long)g.batch * mpad, rowsB = (long long)g.batch * npad;
  CUtensorMap ma, mb, ma1, mb1;
  if (!make_map(&ma, sa, kpad, rowsA, GX_S, FX_BM) || !make_map(&mb, sb, kpad, rowsB, GX_S, FX_BN) ||
      !make_map(&ma1, sa + (size_t)GX_S * rowsA * kpad, kpad, rowsA, 1, FX_BM) ||
      !make_map(&mb1, sb + (size_t)GX_S * rowsB * kpad, kpad, rowsB, 1, FX_BN))
    return cudaErrorInvalidValue;
  FxParams p = {};
  p.M = M;
  p.N = N;
  p.chunks = kpad / FX_CHUNK;
  p.qpc = FX_CHUNK / FX_BK;
  p.kstages = (K + FX_BK - 1) / FX_BK;
  p.lower = g.uplo == UPLO_LOWER && mo == no ? 1 : 0;
  p.kskip = g.kskip;
  p.ksh_m = mo - ko;
  p.ksh_n = no - ko;
  p.tiles_m = (M + FX_BM - 1) / FX_BM;
  p.tiles_n = (N + FX_BN - 1) / FX_BN;
  p.per_batch = (int)count_tiles(p);
  // fewer tiles than SMs: split K, at least four chunks per range
  p.splits = 1;
  if (g.batch == 1 && p.per_batch < sm_count())
    p.splits = std::max(1, std::min(sm_count() / p.per_batch, p.chunks / 4));
  if ((size_t)p.splits * M * N * sizeof(double) > gx_partial_bytes()) p.splits = 1;
  p.num_work = p.per_batch * g.batch * p.splits;
  p.a_rows = mpad;
  p.b_rows = npad;
  p.accumulate = (ko > 0 || g.beta != 0.0) ? 1 : 0;
  p.ra = cA;
  p.rb = cB;
  p.ra_mul = 1;
  p.ra_codes = p.rb_codes = 1;
  p.ra_stride = mpad;
  p.rb_stride = npad;
  p.C = g.C + (long long)mo * g.ldc + no;
  p.ldc = g.ldc;
  p.sC = g.sC;
  p.flags = flags;
  p.flag_ld = npad / 32;
  p.flag_stride = (long long)(mpad / 32) * (npad / 32);
  p.theta = kF64xTheta;
  p.gerr = error_word();
  p.wait_ns = faults().wait_ns;
  p.no_loads = faults().ozaki_no_loads;
  GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 0.0, s,
             certify_kernel<<<dim3((unsigned)(mpad / 256 + 1), (unsigned)g.batch, (unsigned)((npad / 32 + kCertCols - 1) / kCertCols)),
                              256, 0, s>>>(
                 M, N, K, mpad, npad, codes, counts, flags, p.flag_ld, p.flag_stride));
  const int grid = std::min(p.num_work, sm_count());
  const double mnk = (double)g.batch * M * N * K;
  e = launch_product<1, false, true>(ma1, mb1, p, grid, 2.0 * mnk, 0.0, s);
  if (e != cudaSuccess) return e;
  p.partial = p.splits > 1 ? partial : nullptr;
  p.sub = 1;
  if (4 * p.num_work <= sm_count()) {
    p.sub = 4;
    p.num_work *= 4;
  }
  const int pgrid = std::min(p.num_work, sm_count());
  e = g.alpha < 0.0 ? launch_product<GX_S, true, false>(ma, mb, p, pgrid, 72.0 * mnk, 0.0, s)
                    : launch_product<GX_S, false, false>(ma, mb, p, pgrid, 72.0 * mnk, 0.0, s);
  if (e != cudaSuccess) return e;
  if (p.splits > 1) {
    const long long total = (long long)M * N;
    GPC_LAUNCH(GPC_TRACE_ELEM, 0.0, 8.0 * (p.splits + 2) * (double)total, s,
               f64x_reduce_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(
                   M, N, p.splits, partial, p.C, p.ldc, p.lower, p.accumulate, flags, p.flag_ld));
  }
  // the blocks the check left out, in FP64 (the slices' memory is free again: its split-K scratch)
  Gemm r = g;
  r.M = M;
  r.N = N;
  r.K = K;
  r.A = A;
  r.B = B;
  r.C = p.C;
  r.beta = p.accumulate ? 1.0 : 0.0;
  r.uplo = p.lower ? UPLO_LOWER : UPLO_FULL;
  r.flags = flags;
  r.flag_ld = p.flag_ld;
  r.flag_stride = p.flag_stride;
  r.ksh_m = p.ksh_m;
  r.ksh_n = p.ksh_n;
  return gemm_f64(r, (char *)sa + gemm_f64_scratch_bytes() <= ws_end ? (double *)sa : nullptr, s);
}

}  // namespace

size_t f64x_scratch_bytes(int M, int N, int K, int batch) {
  if (M <= 0 || N <= 0 || K <= 0) return 0;
  // the whole K range where that takes at most 256 MB, else up to 4096 of it
  const int kall = (K + 127) / 128 * 128;
  const size_t whole = panel_bytes(M, N, kall, std::max(batch, 1)) + 1024;
  const size_t part = panel_bytes(M, N, std::min(kall, 4096), std::max(batch, 1)) + 1024;
  return std::min(std::min(whole, std::max(part, size_t(256) << 20)), kF64xScratchCap);
}

// A checked product is seven launches, about 60 us end to end at the smallest
// sizes; the FP64 kernel with split K takes 28 us at 256 x 256 x 128 (padded to
// its 64-wide tiles 8e6), 87 us at 512 x 512 x 96 (2.5e7; 68 us here) and 166 us
// at 1024 x 1024 x 64 (6.7e7; 62 us here).
bool f64x_worth(const Gemm &g) {
  auto pad = [](int v) { return (double)((v + 63) / 64 * 64); };
  return g.M >= 8 && g.N >= 8 && g.K >= 16 && g.batch * pad(g.M) * pad(g.N) * g.K >= 3e7;
}

cudaError_t gemm_f64x(const Gemm &g, void *ws, size_t ws_bytes, cudaStream_t s) {
  Panels pn;
  const bool simple = (g.alpha == 1.0 || g.alpha == -1.0) && (g.beta == 0.0 || g.beta == 1.0) &&
                      g.uplo != UPLO_LOWER_MIRROR;
  if (!ws || !simple || !f64x_worth(g) || ws_bytes < kGxMinScratch || !choose_panels(g, ws_bytes - 1024, pn))
    return gemm_f64(g, g.batch == 1 && ws_bytes >= gemm_f64_scratch_bytes() ? (double *)ws : nullptr, s);
  char *base = (char *)align_up((size_t)ws, 1024);
  for (int mo = 0; mo < g.M; mo += pn.mp)
    for (int no = 0; no < g.N; no += pn.np) {
      if (g.uplo == UPLO_LOWER && no > mo) continue;
      for (int ko = 0; ko < g.K; ko += pn.kp)
        if (cudaError_t e = one_panel(g, pn, mo, no, ko, base, (char *)ws + ws_bytes, s); e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

}  // namespace gpc
