// Fused GLM log likelihoods with their gradients (Section 3.4).
//
// For observations (x_i, y_i), i < n, the linear predictor is
// eta_i = alpha + x_i . beta; each family gives lp_i and d_i = d lp_i / d eta_i:
//   normal-identity  lp_i = -((y_i - eta_i)/sigma)^2/2 - log sigma - log(2 pi)/2,  d_i = (y_i - eta_i)/sigma^2
//   Bernoulli-logit  lp_i = y_i eta_i - log(1 + e^eta_i),                          d_i = y_i - 1/(1 + e^-eta_i)
//   Poisson-log      lp_i = y_i eta_i - e^eta_i - lgamma(y_i + 1),                  d_i = y_i - e^eta_i
//   negative-binomial-log (mu_i = e^eta_i, dispersion phi = sigma)
//                    lp_i = lgamma(y_i + phi) - lgamma(y_i + 1) - lgamma(phi)
//                           + phi (log phi - log(mu_i + phi)) + y_i (eta_i - log(mu_i + phi)),
//                    d_i = y_i - (y_i + phi) mu_i / (mu_i + phi)
//   ordinal-logit    (C ordered classes, cut points c_0 < .. < c_{C-2}, no intercept)
//                    lp_i = log(s(eta_i - c_{y_i - 1}) - s(eta_i - c_{y_i})), s(t) = 1/(1 + e^-t),
//                    the missing ends reading s = 1 (y_i = 0) and s = 0 (y_i = C - 1)
// and the outputs are lp = sum lp_i, dalpha = sum d_i, dbeta = X^T d and, for
// the normal family, dsigma = sum ((y_i - eta_i)^2/sigma^3 - 1/sigma); for the
// negative binomial dsigma = d lp / d phi = sum (psi(y_i + phi) - psi(phi) +
// log phi - log(mu_i + phi) + 1 - (y_i + phi)/(mu_i + phi)); for the ordinal
// family dcuts_m = d lp / d c_m.
//
// As in the paper each likelihood is one kernel that produces the value and
// the analytic gradient together; here the GEMV for dbeta is fused in as well,
// so X (the only large operand) crosses HBM once.  A CTA walks blocks of R
// rows: its warps first form eta_i for the block (four rows per warp, lanes
// strided over the columns, a fixed-order shuffle reduction), then one thread
// per row evaluates the family's terms, then every thread adds d_i x_ij for
// the columns it owns (j = thread, thread + 256, ...) over the block's rows,
// re-reading the block from L1/L2.  FP64 work (two multiply-adds per element
// of X) rather than HBM bounds this on GB300, so every FP64 instruction
// carries 32 active lanes: the per-row exp/log1p run one row per thread, not
// on one lane of a warp.  The column sums stay in
// shared memory for the CTA's whole share of rows and go out once as one
// partial row; a second kernel adds the partial rows in CTA order.  Every sum
// has a fixed order, so results are bitwise reproducible.
#include "common.cuh"

#include <algorithm>

namespace gpc {
namespace {

constexpr int GT = 256;  // threads per CTA
constexpr int kMaxRowsPerBlock = 64;
constexpr int kFamilyOrdinal = 100;  // internal family id of the ordinal-logit GLM
constexpr int kMaxCuts = GPC_GLM_MAX_CLASSES - 1;
constexpr int kScalars = 3 + kMaxCuts;  // per-CTA partial scalars: lp, dalpha, dsigma, dcuts

struct GlmParams {
  int family, k, R, ncut;
  long long n, ldx;
  const double *X, *y, *beta, *cuts;
  double alpha, inv_sigma, log_norm;  // log_norm = log(sigma) + log(2 pi)/2
  double phi, log_phi, lgamma_phi;    // negative binomial
  double *part, *part_s;
};

// Digamma psi(x), x > 0: the recurrence psi(x) = psi(x + 1) - 1/x (Abramowitz
// and Stegun 6.3.5) until x >= 10, then the asymptotic expansion (A&S 6.3.18)
//   psi(x) = ln x - 1/(2x) - sum_{k=1..7} B_2k / (2k x^2k) + O(x^-16),
// with B_2 .. B_14 = 1/6, -1/30, 1/42, -1/30, 5/66, -691/2730, 7/6; the first
// omitted term is below 5e-17 at x = 10.
__device__ double digamma_dev(double x) {
  double acc = 0.0;
  while (x < 10.0) {
    acc -= 1.0 / x;
    x += 1.0;
  }
  const double r = 1.0 / (x * x);
  double t = 1.0 / 12.0;  // B_14 / 14
  t = fma(t, r, -691.0 / 32760.0);
  t = fma(t, r, 1.0 / 132.0);
  t = fma(t, r, -1.0 / 240.0);
  t = fma(t, r, 1.0 / 252.0);
  t = fma(t, r, -1.0 / 120.0);
  t = fma(t, r, 1.0 / 12.0);
  return acc + log(x) - 0.5 / x - t * r;
}

// log(y!) for y = 0 .. 127, correctly rounded: counts in earnest are small
// integers, and lgamma is some hundred FP64 instructions, the longest chain of a
// row's terms.
__constant__ double kLogFactorial[128] = {
    0.0, 0.0, 0x1.62e42fefa39efp-1, 0x1.cab0bfa2a2002p+0, 0x1.96ca77c922cf9p+1, 0x1.326643c4479c9p+2,
    0x1.a51273acf01cap+2, 0x1.10ce1f32dcc30p+3, 0x1.5358e82fcb70dp+3, 0x1.99a8921a7f7cfp+3, 0x1.e357590954d15p+3, 0x1.180973f3a8d74p+4,
    0x1.3fcba16d50143p+4, 0x1.68d5a9c3b32cep+4, 0x1.930f3df162a42p+4, 0x1.be636a63fd346p+4, 0x1.eabff061f1a84p+4, 0x1.0c0a63f2f353ap+5,
    0x1.2329df2d5ee52p+5, 0x1.3ab8153363985p+5, 0x1.52af57aed77bep+5, 0x1.6b0a8643472a9p+5, 0x1.83c4faba84f06p+5, 0x1.9cda78b856a45p+5,
    0x1.b6472034e8d14p+5, 0x1.d007622cd65e7p+5, 0x1.ea17f717c6794p+5, 0x1.023aeb67e4fefp+6, 0x1.0f8f18d330240p+6, 0x1.1d07353917231p+6,
    0x1.2aa208b59d0e5p+6, 0x1.385e6fd9e5a40p+6, 0x1.463b59b942084p+6, 0x1.5437c633ace4ap+6, 0x1.6252c474896bap+6, 0x1.708b719e11658p+6,
    0x1.7ee0f79b26758p+6, 0x1.8d528c1243d96p+6, 0x1.9bdf6f75257a3p+6, 0x1.aa86ec2969812p+6, 0x1.b94855c702ba2p+6, 0x1.c8230869ca105p+6,
    0x1.d7166813e12eep+6, 0x1.e621e01eeba4fp+6, 0x1.f544e2ba69cf1p+6, 0x1.023f743addd9fp+7, 0x1.09e7b7ea41ea9p+7, 0x1.119afe762626bp+7,
    0x1.19590c853a559p+7, 0x1.2121a930c6ec3p+7, 0x1.28f49ddeb1f31p+7, 0x1.30d1b61e86335p+7, 0x1.38b8bf8931ddbp+7, 0x1.40a989a33a6cdp+7,
    0x1.48a3e5c12af19p+7, 0x1.50a7a6ee08711p+7, 0x1.58b4a1d39da73p+7, 0x1.60caaca474746p+7, 0x1.68e99f0757979p+7, 0x1.711152043b2c4p+7,
    0x1.79419ff26dc59p+7, 0x1.817a6467f6fb9p+7, 0x1.89bb7c2a0aea1p+7, 0x1.9204c51e7c761p+7, 0x1.9a561e3e1a4bdp+7, 0x1.a2af6787e4609p+7,
    0x1.ab1081f509726p+7, 0x1.b3794f6d9d7afp+7, 0x1.bbe9b2bdfb621p+7, 0x1.c4618f8cc56f7p+7, 0x1.cce0ca5179100p+7, 0x1.d567484b8b7b6p+7,
    0x1.ddf4ef7a05a70p+7, 0x1.e689a69396befp+7, 0x1.ef2554ff15148p+7, 0x1.f7c7e2cc66183p+7, 0x1.00389c56e3462p+8, 0x1.04909ff8b652bp+8,
    0x1.08ebf13dbf263p+8, 0x1.0d4a85602b129p+8, 0x1.11ac51df8932ap+8, 0x1.16114c7e34736p+8, 0x1.1a796b3ede1acp+8, 0x1.1ee4a46236d3ep+8,
    0x1.2352ee64b46d5p+8, 0x1.27c43ffc72962p+8, 0x1.2c3890172d057p+8, 0x1.30afd5d851956p+8, 0x1.352a089728f1bp+8, 0x1.39a71fdd14947p+8,
    0x1.3e271363e0df7p+8, 0x1.42a9db142a36ap+8, 0x1.472f6f03d410cp+8, 0x1.4bb7c77491066p+8, 0x1.5042dcd27af64p+8, 0x1.54d0a7b2ba658p+8,
    0x1.596120d23c4ecp+8, 0x1.5df4411475a1cp+8, 0x1.628a018233bedp+8, 0x1.67225b4879462p+8, 0x1.6bbd47b7669b6p+8, 0x1.705ac0412d89fp+8,
    0x1.74fabe790f7bep+8, 0x1.799d3c1265c0ep+8, 0x1.7e4232dfb367dp+8, 0x1.82e99cd1c0368p+8, 0x1.879373f6bc4fep+8, 0x1.8c3fb2796c21cp+8,
    0x1.90ee52a05c35fp+8, 0x1.959f4ecd1c8b3p+8, 0x1.9a52a17b831ccp+8, 0x1.9f084540f545ep+8, 0x1.a3c034cbb7b2cp+8, 0x1.a87a6ae24493ap+8,
    0x1.ad36e262a7cc0p+8, 0x1.b1f59641e0db5p+8, 0x1.b6b6818b4a3ebp+8, 0x1.bb799f600610ap+8, 0x1.c03eeaf66facdp+8, 0x1.c5065f9992226p+8,
    0x1.c9cff8a8a340dp+8, 0x1.ce9bb196830eap+8, 0x1.d36985e93f7b8p+8, 0x1.d83971399c213p+8, 0x1.dd0b6f329dea4p+8, 0x1.e1df7b911a74cp+8,
    0x1.e6b592234b0c9p+8, 0x1.eb8daec863182p+8};
__device__ __forceinline__ double log_factorial(double y) {
  const int i = (int)y;
  if (y >= 0.0 && y < 128.0 && (double)i == y) return kLogFactorial[i];
  return lgamma(y + 1.0);
}

// cut: the ordinal family's contributions to its cut-point derivatives
// (index lo gets -du, lo + 1 gets -dv; lo = -2 when there are none).
__device__ __forceinline__ void glm_row(const GlmParams &p, double eta, double y, double &lp, double &d,
                                        double &ds, int &lo, double &du, double &dv, double psi_phi) {
  lo = -2;
  du = dv = 0.0;
  if (p.family == GPC_GLM_NORMAL_ID) {
    const double r = y - eta, z = r * p.inv_sigma;
    lp = -0.5 * z * z - p.log_norm;
    d = z * p.inv_sigma;
    ds = (z * z - 1.0) * p.inv_sigma;
  } else if (p.family == GPC_GLM_BERNOULLI_LOGIT) {
    const double e = exp(-fabs(eta));  // log(1 + e^eta) = max(eta, 0) + log1p(e^-|eta|)
    lp = y * eta - (fmax(eta, 0.0) + log1p(e));
    d = y - (eta >= 0.0 ? 1.0 / (1.0 + e) : e / (1.0 + e));
    ds = 0.0;
  } else if (p.family == GPC_GLM_POISSON_LOG) {
    const double mu = exp(eta);
    lp = y * eta - mu - log_factorial(y);
    d = y - mu;
    ds = 0.0;
  } else if (p.family == GPC_GLM_NEG_BINOMIAL_LOG) {
    const double phi = p.phi, mu = exp(eta), ypp = y + phi, mpp = mu + phi, lmp = log(mpp);
    lp = lgamma(ypp) - log_factorial(y) - p.lgamma_phi + phi * (p.log_phi - lmp) + y * (eta - lmp);
    d = y - ypp * mu / mpp;
    ds = digamma_dev(ypp) - psi_phi + p.log_phi - lmp + 1.0 - ypp / mpp;
  } else {  // ordinal logit: y in {0 .. ncut}
    const int C = p.ncut + 1, yi = (int)y;
    ds = 0.0;
    if (!(y >= 0.0) || yi >= C || (double)yi != y) {  // outside the support: NaN, nothing indexed
      lp = __longlong_as_double(0x7ff8000000000000ll);
      d = 0.0;
      return;
    }
    const double su = yi > 0 ? 1.0 / (1.0 + exp(-(eta - p.cuts[yi - 1]))) : 1.0;
    const double sv = yi < C - 1 ? 1.0 / (1.0 + exp(-(eta - p.cuts[yi]))) : 0.0;
    const double P = su - sv;
    lp = log(P);
    du = yi > 0 ? su * (1.0 - su) / P : 0.0;
    dv = yi < C - 1 ? -sv * (1.0 - sv) / P : 0.0;
    d = du + dv;
    lo = yi - 1;
  }
}

__global__ void __launch_bounds__(GT) glm_kernel(GlmParams p) {
  extern __shared__ double sm[];
  double *acc = sm;                      // k column sums; thread t owns j = t, t + GT, ...
  double *bs = sm + p.k;                 // beta
  double *eta_s = bs + p.k;              // eta of the current block's rows
  double *dblk = eta_s + kMaxRowsPerBlock;  // d_i of the current block's rows
  double *cut_s = dblk + kMaxRowsPerBlock;  // ordinal: per-thread cut sums, kMaxRowsPerBlock x kMaxCuts
  __shared__ double red[3][GT / 32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  for (int j = t; j < p.k; j += GT) {
    acc[j] = 0.0;
    bs[j] = p.beta[j];
  }
  if (p.family == kFamilyOrdinal)
    for (int q = t; q < kMaxRowsPerBlock * kMaxCuts; q += GT) cut_s[q] = 0.0;
  const double psi_phi = p.family == GPC_GLM_NEG_BINOMIAL_LOG ? digamma_dev(p.phi) : 0.0;
  __syncthreads();
  double slp = 0.0, sda = 0.0, sds = 0.0;  // per thread (threads below R)
  const long long nblk = (p.n + p.R - 1) / p.R;
  for (long long b = blockIdx.x; b < nblk; b += gridDim.x) {
    const long long i0 = b * p.R;
    const int rows = (int)min((long long)p.R, p.n - i0);
    // eta for four rows per warp: four independent FMA chains per lane, then a
    // transposed butterfly that leaves row 2 bit4 + bit3 of the lane index in
    // every lane (6 adds for the four rows).  Missing rows of a short last
    // group re-read the group's first row and are not stored.
    for (int g = warp; 4 * g < rows; g += GT / 32) {
      const int r0 = 4 * g, nr = min(4, rows - r0);
      const double *x0 = p.X + (i0 + r0) * p.ldx;
      const double *x1 = nr > 1 ? x0 + p.ldx : x0;
      const double *x2 = nr > 2 ? x0 + 2 * p.ldx : x0;
      const double *x3 = nr > 3 ? x0 + 3 * p.ldx : x0;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll 2
      for (int j = lane; j < p.k; j += 32) {
        const double bj = bs[j];
        s0 = fma(x0[j], bj, s0);
        s1 = fma(x1[j], bj, s1);
        s2 = fma(x2[j], bj, s2);
        s3 = fma(x3[j], bj, s3);
      }
      const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
      double k0 = h16 ? s2 : s0, k1 = h16 ? s3 : s1;
      k0 += __shfl_xor_sync(0xffffffffu, h16 ? s0 : s2, 16);
      k1 += __shfl_xor_sync(0xffffffffu, h16 ? s1 : s3, 16);
      double v = h8 ? k1 : k0;
      v += __shfl_xor_sync(0xffffffffu, h8 ? k0 : k1, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      const int row = ((lane >> 4) << 1) | ((lane >> 3) & 1);
      if ((lane & 7) == 0 && row < nr) eta_s[r0 + row] = v + p.alpha;
    }
    __syncthreads();
    // the family's terms, one row per thread
    if (t < rows) {
      double lp, d, ds, du, dv;
      int lo;
      glm_row(p, eta_s[t], p.y[i0 + t], lp, d, ds, lo, du, dv, psi_phi);
      dblk[t] = d;
      slp += lp;
      sda += d;
      sds += ds;
      if (lo >= 0) cut_s[t * kMaxCuts + lo] -= du;
      if (lo >= -1 && lo + 1 < p.ncut) cut_s[t * kMaxCuts + lo + 1] -= dv;
    }
    __syncthreads();
    // dbeta: column-owned sums over the block's rows (two chains), X from L1/L2
    for (int j = t; j < p.k; j += GT) {
      const double *xc = p.X + i0 * p.ldx + j;
      double a0 = 0.0, a1 = 0.0;
      int r = 0;
      for (; r + 1 < rows; r += 2) {
        a0 = fma(xc[(long long)r * p.ldx], dblk[r], a0);
        a1 = fma(xc[(long long)(r + 1) * p.ldx], dblk[r + 1], a1);
      }
      if (r < rows) a0 = fma(xc[(long long)r * p.ldx], dblk[r], a0);
      acc[j] += a0 + a1;
    }
    __syncthreads();
  }
  for (int j = t; j < p.k; j += GT) p.part[(long long)blockIdx.x * p.k + j] = acc[j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    slp += __shfl_down_sync(0xffffffffu, slp, o);
    sda += __shfl_down_sync(0xffffffffu, sda, o);
    sds += __shfl_down_sync(0xffffffffu, sds, o);
  }
  if (lane == 0) {
    red[0][warp] = slp;
    red[1][warp] = sda;
    red[2][warp] = sds;
  }
  __syncthreads();
  if (t < 3) {
    double v = 0.0;
    for (int w = 0; w < GT / 32; ++w) v += red[t][w];
    p.part_s[(long long)kScalars * blockIdx.x + t] = v;
  } else if (t < 3 + p.ncut) {  // ordinal: this CTA's cut sums, rows' threads in order
    const int m = t - 3;
    double v = 0.0;
    for (int r = 0; r < kMaxRowsPerBlock; ++r) v += cut_s[r * kMaxCuts + m];
    p.part_s[(long long)kScalars * blockIdx.x + t] = v;
  }
}

// The same likelihood for k <= kNarrow covariates.  There the wide kernel's
// lane-per-column passes waste the FP64 pipe (an instruction costs it the same
// whatever its active lanes): a row's eta took 6 reduction adds beside k / 32
// multiply-adds per lane, and the gradient pass had ceil(k / 32) of 8 warps at
// work.  Here a block of R rows is staged in shared memory (odd row stride), one
// thread forms a row's eta and terms by itself, and the gradient pass deals the
// rows over all warps, lanes = columns (several rows per warp when k <= 16),
// with the column sums in registers for the CTA's whole share of rows.
// Measured (call, before and after): Bernoulli-logit 200 000 x 40 208 -> 101 us,
// 200 000 x 64 180 -> 118, 500 000 x 2 293 -> 134; normal 300 000 x 10 183 -> 55;
// negative binomial 50 000 x 30 184 -> 89; at 65 covariates the wide kernel takes 157.
constexpr int kNarrow = 64;
__global__ void __launch_bounds__(GT) glm_narrow_kernel(GlmParams p) {
  extern __shared__ double sm[];
  const int k = p.k, kp = k | 1, R = p.R;
  double *xs = sm;                // R x kp
  double *bs = xs + (size_t)R * kp;  // beta
  double *dblk = bs + kNarrow;    // d_i of the block's rows
  double *accs = dblk + GT;       // column sums of the warps, 8 x 32
  double *cut_s = accs + (GT / 32) * 32;  // ordinal: per-thread cut sums
  __shared__ double red[3][GT / 32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  for (int j = t; j < k; j += GT) bs[j] = p.beta[j];
  if (p.family == kFamilyOrdinal)
    for (int q = t; q < R * kMaxCuts; q += GT) cut_s[q] = 0.0;
  const double psi_phi = p.family == GPC_GLM_NEG_BINOMIAL_LOG ? digamma_dev(p.phi) : 0.0;
  // gradient pass: lane = (row of a group of subs, column of a chunk of kc <= 32)
  int kc = 1;
  while (kc < 32 && kc < k) kc *= 2;
  const int chunks = k > 32 ? 2 : 1, subs = 32 / kc;
  const int col = (lane & (kc - 1)) + 32 * (chunks == 2 ? (warp & 1) : 0), sub = lane / kc;
  const int first = (chunks == 2 ? warp >> 1 : warp) * subs + sub, step = (GT / 32 / chunks) * subs;
  double g0 = 0.0, g1 = 0.0;
  double slp = 0.0, sda = 0.0, sds = 0.0;
  const long long nblk = (p.n + R - 1) / R;
  for (long long b = blockIdx.x; b < nblk; b += gridDim.x) {
    const long long i0 = b * R;
    const int rows = (int)min((long long)R, p.n - i0);
    const double yi = t < rows ? p.y[i0 + t] : 0.0;
    __syncthreads();  // the previous block's gradient pass is done
    const double *src = p.X + i0 * p.ldx;
    if (k > 0) {
      const unsigned total = (unsigned)rows * (unsigned)k;
#pragma unroll 8
      for (unsigned idx = t; idx < total; idx += GT) {
        const unsigned r = idx / (unsigned)k, c = idx - r * (unsigned)k;
        xs[r * kp + c] = src[(long long)r * p.ldx + c];
      }
    }
    __syncthreads();
    if (t < rows) {
      const double *x = xs + t * kp;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      int j = 0;
      for (; j + 3 < k; j += 4) {
        s0 = fma(x[j], bs[j], s0);
        s1 = fma(x[j + 1], bs[j + 1], s1);
        s2 = fma(x[j + 2], bs[j + 2], s2);
        s3 = fma(x[j + 3], bs[j + 3], s3);
      }
      for (; j < k; ++j) s0 = fma(x[j], bs[j], s0);
      double lp, d, ds, du, dv;
      int lo;
      glm_row(p, ((s0 + s1) + (s2 + s3)) + p.alpha, yi, lp, d, ds, lo, du, dv, psi_phi);
      dblk[t] = d;
      slp += lp;
      sda += d;
      sds += ds;
      if (lo >= 0) cut_s[t * kMaxCuts + lo] -= du;
      if (lo >= -1 && lo + 1 < p.ncut) cut_s[t * kMaxCuts + lo + 1] -= dv;
    }
    __syncthreads();
    if (col < k) {
      int r = first;
      for (; r + step < rows; r += 2 * step) {
        g0 = fma(xs[r * kp + col], dblk[r], g0);
        g1 = fma(xs[(r + step) * kp + col], dblk[r + step], g1);
      }
      if (r < rows) g0 = fma(xs[r * kp + col], dblk[r], g0);
    }
  }
  accs[t] = g0 + g1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    slp += __shfl_down_sync(0xffffffffu, slp, o);
    sda += __shfl_down_sync(0xffffffffu, sda, o);
    sds += __shfl_down_sync(0xffffffffu, sds, o);
  }
  if (lane == 0) {
    red[0][warp] = slp;
    red[1][warp] = sda;
    red[2][warp] = sds;
  }
  __syncthreads();
  if (t < k) {  // this column's sums: warps of its chunk, then rows of the group, in order
    double v = 0.0;
    for (int w = chunks == 2 ? t >> 5 : 0; w < GT / 32; w += chunks)
      for (int q = 0; q < subs; ++q) v += accs[32 * w + q * kc + (t & 31)];
    p.part[(long long)blockIdx.x * k + t] = v;
  }
  if (t >= 64 && t < 67) {
    double v = 0.0;
    for (int w = 0; w < GT / 32; ++w) v += red[t - 64][w];
    p.part_s[(long long)kScalars * blockIdx.x + t - 64] = v;
  } else if (t >= 67 && t < 67 + p.ncut) {
    double v = 0.0;
    for (int r = 0; r < R; ++r) v += cut_s[r * kMaxCuts + t - 67];
    p.part_s[(long long)kScalars * blockIdx.x + t - 64] = v;
  }
}

// dbeta_j = sum over CTAs of the partial rows, and the scalars (lp, dalpha,
// dsigma, then the ordinal family's ncut cut derivatives).  32 outputs per CTA,
// the partial rows dealt over 8 warps with four sums each (a chain of hundreds
// of dependent FP64 additions per output took 28 to 78 us), added in fixed order.
__global__ void __launch_bounds__(GT)
glm_reduce_kernel(int k, int ctas, int ncut, const double *part, const double *part_s, double *dbeta, double *lp,
                  double *dalpha, double *dsigma, double *dcuts) {
  __shared__ double sums[GT / 32][33];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, j = blockIdx.x * 32 + lane, outs = k + 3 + ncut;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (j < outs) {
    const double *src = j < k ? part + j : part_s + (j - k);
    const long long ld = j < k ? k : kScalars;
    int c = w;
    for (; c + 24 < ctas; c += 32) {
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += src[(long long)(c + 8 * u) * ld];
    }
    for (int u = 0; c < ctas; c += 8, ++u) s[u & 3] += src[(long long)c * ld];
  }
  sums[w][lane] = (s[0] + s[1]) + (s[2] + s[3]);
  __syncthreads();
  if (w == 0 && j < outs) {
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < GT / 32; ++q) v += sums[q][lane];
    const int q = j - k;
    double *dst = j < k ? dbeta + j : (q == 0 ? lp : (q == 1 ? dalpha : (q == 2 ? dsigma : dcuts + (q - 3))));
    if (j < k || dst) *dst = v;
  }
}

int rows_per_block(int k) {
  const int r = 16384 / std::max(k, 1);  // about 128 KiB of X per block, re-read from L1/L2
  return std::max(8, std::min(kMaxRowsPerBlock, r / 8 * 8));
}

// Rows per block of the narrow kernel: one per thread where the staged block
// stays within 64 KB (three CTAs per SM), fewer (a warp's worth at least) where
// the whole input would not give every SM two blocks.
int narrow_rows(long long n, int k) {
  int r = GT;
  while (r > 64 && (size_t)r * (k | 1) * sizeof(double) > 64 * 1024) r /= 2;
  while (r > 32 && n < 2LL * sm_count() * r) r /= 2;
  return r;
}
size_t narrow_smem_bytes(int R, int k, bool ordinal) {
  return ((size_t)R * (k | 1) + kNarrow + GT + (GT / 32) * 32 + (ordinal ? (size_t)R * kMaxCuts : 0)) * sizeof(double);
}

size_t smem_bytes(int k) {
  return (2 * (size_t)k + 2 * kMaxRowsPerBlock + (size_t)kMaxRowsPerBlock * kMaxCuts) * sizeof(double);
}

int max_ctas(int k) {
  const size_t per = smem_bytes(k) + 1024;
  const int by_smem = (int)std::max<size_t>(1, (size_t)(228 * 1024) / per);
  return sm_count() * std::max(1, std::min(4, by_smem));
}

}  // namespace

size_t glm_workspace_bytes(int k) {
  const size_t ctas = (size_t)max_ctas(k);
  return align_up(ctas * (size_t)std::max(k, 1) * sizeof(double), 256) +
         align_up(ctas * kScalars * sizeof(double), 256);
}

namespace {

cudaError_t glm_launch(GlmParams &p, long long n, int k, double *lp, double *dalpha, double *dbeta, double *dsigma,
                       double *dcuts, void *ws, cudaStream_t s) {
  p.n = n;
  p.k = k;
  const bool narrow = k <= kNarrow;
  p.R = narrow ? narrow_rows(n, k) : rows_per_block(k);
  const long long nblk = std::max<long long>(1, (n + p.R - 1) / p.R);
  const int ctas = (int)std::min<long long>(nblk, max_ctas(k));
  char *w = (char *)ws;
  p.part = (double *)w;
  p.part_s = (double *)(w + align_up((size_t)max_ctas(k) * (size_t)std::max(k, 1) * sizeof(double), 256));
  const size_t smem = narrow ? narrow_smem_bytes(p.R, k, p.family == kFamilyOrdinal) : smem_bytes(k);
  if (smem > 48 * 1024) {
    static bool done[2][64] = {};
    cudaError_t e = allow_all_smem(narrow ? (const void *)glm_narrow_kernel : (const void *)glm_kernel, done[narrow]);
    if (e != cudaSuccess) return e;
  }
  const double bytes = 8.0 * ((double)n * k + 2.0 * n + k);
  if (narrow)
    GPC_LAUNCH(GPC_TRACE_GLM, 4.0 * (double)n * k, bytes, s, glm_narrow_kernel<<<ctas, GT, smem, s>>>(p));
  else
    GPC_LAUNCH(GPC_TRACE_GLM, 4.0 * (double)n * k, bytes, s, glm_kernel<<<ctas, GT, smem, s>>>(p));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int outs = k + 3 + p.ncut;
  GPC_LAUNCH(GPC_TRACE_ELEM, (double)ctas * outs, 8.0 * (double)ctas * outs, s,
             glm_reduce_kernel<<<(outs + 31) / 32, GT, 0, s>>>(k, ctas, p.ncut, p.part, p.part_s, dbeta, lp,
                                                                   dalpha, dsigma, dcuts));
  return cudaGetLastError();
}

GlmParams base_params(int family, long long ldx, const double *X, const double *y, const double *beta) {
  GlmParams p{};
  p.family = family;
  p.ldx = ldx;
  p.X = X;
  p.y = y;
  p.beta = beta;
  p.cuts = nullptr;
  p.ncut = 0;
  p.inv_sigma = 1.0;
  p.log_norm = 0.0;
  return p;
}

}  // namespace

cudaError_t glm(int family, long long n, int k, const double *X, long long ldx, const double *y, double alpha,
                const double *beta, double sigma, double *lp, double *dalpha, double *dbeta, double *dsigma,
                void *ws, cudaStream_t s) {
  GlmParams p = base_params(family, ldx, X, y, beta);
  p.alpha = alpha;
  if (family == GPC_GLM_NORMAL_ID) {
    p.inv_sigma = 1.0 / sigma;
    p.log_norm = log(sigma) + 0.91893853320467274178;
  } else if (family == GPC_GLM_NEG_BINOMIAL_LOG) {
    p.phi = sigma;
    p.log_phi = log(sigma);
    p.lgamma_phi = lgamma(sigma);
  }
  return glm_launch(p, n, k, lp, dalpha, dbeta, dsigma, nullptr, ws, s);
}

cudaError_t glm_ordinal(long long n, int k, int C, const double *X, long long ldx, const double *y,
                        const double *beta, const double *cuts, double *lp, double *dbeta, double *dcuts, void *ws,
                        cudaStream_t s) {
  GlmParams p = base_params(kFamilyOrdinal, ldx, X, y, beta);
  p.alpha = 0.0;  // the cut points take the intercept's place
  p.cuts = cuts;
  p.ncut = C - 1;
  return glm_launch(p, n, k, lp, nullptr, dbeta, nullptr, dcuts, ws, s);
}

}  // namespace gpc
