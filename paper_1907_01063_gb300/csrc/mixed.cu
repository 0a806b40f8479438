// Mixed-precision blocked Cholesky and blocked adjoint (precision GPC_MIXED).
//
// Same block algorithms as chol.cu (Section 3.3), with the O(n^3) products
// moved to split-BF16 tensor-core products (ozaki.cu).  The FP64 path runs the
// same code on FP64 storage with the FP64-accurate products of f64x.cu (f64).
//   forward: the trailing update A22 -= L21 L21^T;
//   adjoint: Bbar -= Cbar R, Dbar -= Cbar^T C and Rbar -= [Dbar; Cbar]^T [R; B].
// The diagonal-block factors, their inverses, the factorisation's panel solves and
// the Dbar symbolic step stay FP64; the adjoint's panels Cbar D^-1 are FP64 solves on
// the mixed path and products with the inverses at FP64 accuracy (f64x.cu) on the
// FP64 path.  Matrices that the split products update (the
// trailing part of L, the not-yet-final part of Lbar) are held in
// double-float storage (FP32 hi + lo in each 8-byte element); each block
// column is read as FP64 when it becomes current (the diagonal factor and the
// panel solves convert it as they load it), so every output is FP64 at the
// end.  The sweeps move by the 128-wide chunk of the split products so chunk
// boundaries line up with the blocks; within a block column the FP64 steps
// work on 64-wide halves (the blocked algorithm with b = 64 for its FP64
// steps, the updates of two consecutive 64-steps merged into one K = 128
// product), which halves the FP64 work of the panel solves and quarters that
// of the diagonal factors -- the FP64 pipe, not the tensor cores, bounds the
// critical path on this part.
#include "common.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <vector>

namespace gpc {
namespace {

constexpr int MB = 128;  // block size of the mixed path (== slice chunk)
constexpr int MH = 64;   // panel sub-block of the factorisation's FP64 steps
constexpr size_t kPartialCap = size_t(40) << 20;

#define TRY(x)                        \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

struct MixWs {
  double *inv, *m, *t, *scratch;          // FP64 pieces (scratch doubles as the split-K partials)
  void *sc, *sdc, *lt;                    // slices: panel rows, block-column columns, L^T
  void *grp, *tmp;                        // factorisation: two group buffers, per-step temporaries
  void *sx, *si;                          // adjoint, eight slices: panel rows, diagonal-block inverses
  int *rexp, *cexp, *xexp, *iexp, *bexp;  // scale exponents: rows of L, its columns, panel rows, inverses, block column
  int *oexp;                              // per block column: bexp, or what its finished block needs
};
constexpr int kMaxDefer = 8;
// Block columns per deferred update.  The knob belongs to the mixed path: the FP64
// path's workspace, and whether a call fits into one that was made before, must not
// change with it.  Six is the tuner's choice at n = 16384.
constexpr int kF64Defer = 6;
int defer_depth(bool f64) { return f64 ? kF64Defer : std::max(1, std::min(tuning().mixed_defer, kMaxDefer)); }

size_t b2() { return align_up((size_t)MB * MB * sizeof(double), 256); }

// Auxiliary stream and events of one factorisation or adjoint.  A call leases a
// set for as long as it enqueues: two host threads that shared one would record
// each other's events between a record and its wait, and the background products
// would start before their operands are written.  Sets stay with the caller's
// stream that used them last, so that calls on different streams do not queue up
// behind each other on a shared one, and one that a graph capture still holds goes
// to callers in that capture only (any other call's work would be captured too).
struct Aux {
  cudaStream_t st = nullptr;
  cudaEvent_t ev_split = nullptr, ev_rest = nullptr, ev_fork = nullptr;
  cudaStream_t last = nullptr;  // the caller's stream of the last lease (compared only)
  bool leased = false;
};
constexpr size_t kAuxKept = 8;  // sets kept per device; more exist only while that many calls enqueue at once
std::mutex g_aux_mu;
std::vector<Aux *> g_aux[64];

cudaError_t aux_create(Aux &a) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // creation is no part of any capture
  const bool swapped = cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess;
  cudaError_t e = cudaStreamCreateWithFlags(&a.st, cudaStreamNonBlocking);
  for (cudaEvent_t *ev : {&a.ev_split, &a.ev_rest, &a.ev_fork})
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
  if (swapped) cudaThreadExchangeStreamCaptureMode(&mode);
  return e;
}
void aux_destroy(Aux *a) {
  for (cudaEvent_t ev : {a->ev_split, a->ev_rest, a->ev_fork})
    if (ev) cudaEventDestroy(ev);
  if (a->st) cudaStreamDestroy(a->st);  // work in flight completes
  delete a;
}
// 0: not capturing; otherwise the capture's id (all ones: an invalidated one).
unsigned long long capture_id(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(s, &st, &id) != cudaSuccess) {
    cudaGetLastError();  // the legacy stream beside a capture: the launches that follow report it
    return 0;
  }
  return st == cudaStreamCaptureStatusNone ? 0 : (st == cudaStreamCaptureStatusActive ? id : ~0ull);
}

class AuxLease {
 public:
  explicit AuxLease(cudaStream_t s) : s_(s) {}
  AuxLease(const AuxLease &) = delete;
  AuxLease &operator=(const AuxLease &) = delete;
  cudaError_t take(Aux **out) {
    cudaError_t e = cudaGetDevice(&dev_);
    if (e != cudaSuccess) return e;
    if (dev_ < 0 || dev_ >= 64) return cudaErrorInvalidDevice;
    const unsigned long long want = capture_id(s_);
    std::lock_guard<std::mutex> g(g_aux_mu);
    std::vector<Aux *> &pool = g_aux[dev_];
    Aux *other = nullptr;
    for (Aux *a : pool) {
      if (a->leased) continue;
      const unsigned long long held = capture_id(a->st);
      if (held != 0 && held != want) continue;
      if (a->last == s_) {
        aux_ = a;
        break;
      }
      if (!other) other = a;  // the one returned longest ago: returns go to the back
    }
    if (!aux_ && pool.size() >= kAuxKept) aux_ = other;
    if (!aux_) {
      Aux *a = new (std::nothrow) Aux;
      if (!a) return cudaErrorMemoryAllocation;
      if ((e = aux_create(*a)) != cudaSuccess) {
        aux_destroy(a);
        return e;
      }
      try {
        pool.push_back(a);
      } catch (...) {
        aux_destroy(a);
        return cudaErrorMemoryAllocation;
      }
      aux_ = a;
    }
    aux_->leased = true;
    *out = aux_;
    return cudaSuccess;
  }
  void joined() { joined_ = true; }
  // Returned once the join is enqueued (after an error: joined here, so that the
  // caller's stream still ends after everything that uses its buffers).
  ~AuxLease() {
    if (!aux_) return;
    if (!joined_ && cudaEventRecord(aux_->ev_rest, aux_->st) == cudaSuccess) cudaStreamWaitEvent(s_, aux_->ev_rest, 0);
    std::lock_guard<std::mutex> g(g_aux_mu);
    std::vector<Aux *> &pool = g_aux[dev_];
    pool.erase(std::find(pool.begin(), pool.end(), aux_));
    if (pool.size() >= kAuxKept && capture_id(aux_->st) == 0) {
      aux_destroy(aux_);
      return;
    }
    aux_->leased = false;
    aux_->last = s_;
    pool.push_back(aux_);  // no allocation: one was just erased
  }

 private:
  cudaStream_t s_;
  int dev_ = 0;
  Aux *aux_ = nullptr;
  bool joined_ = false;
};
size_t scratch_bytes() { return std::max(gemm_f64_scratch_bytes(), kPartialCap); }
int nchunks(int n) { return std::max(1, (n + MB - 1) / MB); }

// Slices per operand: five on the mixed path (ozaki.cu), seven on the FP64 path (f64x.cu).
size_t sbytes(int rows, int kchunks, bool f64) {
  return f64 ? f64x_slice_bytes(rows, kchunks) : slice_bytes(rows, kchunks);
}
// Panel rows of the adjoint; the mixed path's solved half panel has a buffer of its own.
size_t sc_bytes(int n, bool f64) { return (f64 ? 1 : 2) * sbytes(n, 1, f64); }
size_t exps_bytes(int n) { return align_up((size_t)n * sizeof(int), 256); }

MixWs carve(void *ws, int n, bool adjoint, bool f64) {
  char *p = (char *)ws;
  MixWs w{};
  w.inv = (double *)p; p += (size_t)nchunks(n) * b2();  // every diagonal-block inverse
  w.m = (double *)p; p += b2();
  w.t = (double *)p; p += b2();
  w.scratch = (double *)p; p += scratch_bytes();
  w.sc = p; p += sc_bytes(n, f64);
  if (adjoint) {
    w.sdc = p; p += sbytes(MB, nchunks(n), f64);
    w.lt = p; p += sbytes(n, nchunks(n), f64);
    if (f64) {
      w.sx = p; p += f64x_slice_bytes(n, 1, true);
      w.si = p; p += (size_t)nchunks(n) * f64x_slice_bytes(MB, 1, true);
    }
  } else {
    w.grp = p; p += 2 * sbytes(n, defer_depth(f64), f64);
    w.tmp = p; p += sbytes(n, 1, f64);
  }
  if (!f64) return w;
  w.rexp = (int *)p; p += exps_bytes(n);
  w.cexp = (int *)p; p += exps_bytes(n);
  w.xexp = (int *)p; p += exps_bytes(n);
  w.iexp = (int *)p; p += exps_bytes(nchunks(n) * MB);
  w.bexp = (int *)p; p += 256;
  w.oexp = (int *)p;
  return w;
}

}  // namespace

size_t mixed_workspace_bytes(int n, bool f64) {
  n = std::max(n, 1);
  size_t common = ((size_t)nchunks(n) + 2) * b2() + scratch_bytes() + sc_bytes(n, f64) + 1024;
  size_t adj = sbytes(MB, nchunks(n), f64) + sbytes(n, nchunks(n), f64);
  const size_t fwd = 2 * sbytes(n, defer_depth(f64), f64) + sbytes(n, 1, f64);
  if (f64) {
    common += 3 * exps_bytes(n) + exps_bytes(nchunks(n) * MB) + 256 + exps_bytes(nchunks(n));
    adj += f64x_slice_bytes(n, 1, true) + (size_t)nchunks(n) * f64x_slice_bytes(MB, 1, true);
  }
  return common + std::max(adj, fwd);
}

// Factorisation with deferred trailing updates.  Block columns (128 wide)
// form groups of D = tuning().mixed_defer; the slices of a group's panels
// collect in one buffer (chunk t = the group's t-th block column, rows
// relative to the group's first column), and the group's update of the
// columns to its right is applied as products with K = 128 D:
//   * next-column update, after every block column (caller's stream): the
//     next block column minus the products of all of the group's block
//     columns so far (K = 128 (t + 1));
//   * after the group's last block column, on the auxiliary stream: the
//     strip (the next group's other block columns) and then the rest (every
//     column right of the next group), both with K = 128 D; the rest is cut
//     into D - 1 column slabs released one after each of the next group's
//     next-column updates.
// The background products leave tuning().mixed_free_sms SMs to the caller's
// stream, where the FP64 chain of the next group runs meanwhile (its panel
// solves also fit beside a product CTA on every SM: they use the FP64 pipes,
// the products the tensor cores).  The caller's stream waits for the strip
// before the first next-column update of the following group and for the
// rest before that group's last one -- the first writes into each update's
// region -- and group buffers alternate, so a split never overwrites slices
// still being read.  D = 1 is the one-block lookahead (rest of every step in
// the background).
//
// f64 (precision GPC_FP64): the same schedule with the products of f64x.cu on
// FP64 storage.  Row i of L is scaled by 2^-e_i, e_i from K's diagonal
// (|L_ij| <= sqrt(K_ii)); the slices' error is then relative to
// sqrt(K_ii K_jj), the form of the FP64 factorisation's own error bound.
cudaError_t chol_mixed(int n, double *L, long long ldl, void *ws, int *info, cudaStream_t s, bool f64) {
  MixWs w = carve(ws, n, false, f64);
  if (f64) TRY(f64x_diag_exps(n, L, ldl, w.rexp, s));
  const bool df = !f64;  // the matrices the products update are in double-float storage
  // slices of M rows of L, the first at global row `row`, K columns
  auto split = [&](const double *src, int M, int K, const SliceBuf &out, int row, int chunk = 0, int roff = 0) {
    return f64 ? f64x_split(src, ldl, 1, M, K, K, out, w.rexp + row, nullptr, 0, true, s, chunk, roff)
               : split_operand(src, ldl, 1, M, K, K, out, s, chunk, roff);
  };
  // C -= A B^T; C's first row and column are global rows gi and gj of L
  auto product = [&](const SliceBuf &A, int ar, const SliceBuf &B, int br, int M, int N, int chunks, bool lower,
                     double *C, int gi, int gj, cudaStream_t st, int ctas, int kdepth, int items) {
    int *e = info ? info + 1 : nullptr;
    return f64 ? f64x_gemm(A, ar, 0, B, br, 0, M, N, chunks, lower, w.rexp + gi, w.rexp + gj, C, ldl, 1, nullptr, e,
                           st, ctas, kdepth, items)
               : ozaki_gemm(A, ar, 0, B, br, 0, M, N, chunks, lower, -1.0f, (float2 *)C, ldl, 1, nullptr, e, st, ctas,
                            kdepth, items);
  };
  AuxLease lease(s);
  Aux *aux = nullptr;
  TRY(lease.take(&aux));
  const int D = defer_depth(f64);
  const int nbc = nchunks(n);
  const int bg_ctas = std::max(1, sm_count() - std::max(0, std::min(tuning().mixed_free_sms, sm_count() / 2)));
  const int bg_items = std::max(0, tuning().mixed_cta_items);
  // the caller's stream carries the critical chain: its launches go first
  PriorityScope chain(tuning().mixed_priority ? greatest_priority() : 0);
  bool strip_pending = false, rest_pending = false;
  // The previous group's rest, cut into column slabs of about equal work: slab
  // i is released (by an event) after the i-th next-column update of the
  // current group, so the background work interleaves with the chain the way
  // a one-block lookahead does while every slab keeps K = 128 D.
  struct Slabs {
    SliceBuf G;
    int p0 = 0, chunks = 0, next = 0, count = 0;
    int cut[kMaxDefer + 1] = {};
  } slabs;
  auto launch_slab = [&]() -> cudaError_t {
    const int c0 = slabs.cut[slabs.next], c1 = slabs.cut[slabs.next + 1];
    ++slabs.next;
    cudaError_t e = cudaEventRecord(aux->ev_fork, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(aux->st, aux->ev_fork, 0);
    PriorityScope background(0);
    if (e == cudaSuccess && c1 > c0)
      e = product(slabs.G, c0 - slabs.p0, slabs.G, c0 - slabs.p0, n - c0, c1 - c0, slabs.chunks, true,
                  L + (long long)c0 * ldl + c0, c0, c0, aux->st, bg_ctas, 0, bg_items);
    if (e == cudaSuccess && slabs.next == slabs.count) e = cudaEventRecord(aux->ev_rest, aux->st);
    return e;
  };
  for (int bc = 0; bc < nbc; ++bc) {
    const int g = bc / D, t = bc - g * D;
    const int p0 = g * D * MB, p1 = std::min(n, p0 + D * MB);
    const int k0 = bc * MB, nb = std::min(MB, n - k0), m = n - k0 - nb;
    double *A11 = L + (long long)k0 * ldl + k0;
    SliceBuf G = slice_view((char *)w.grp + (size_t)(g & 1) * sbytes(n, D, f64), n - p0, D);
    // ---- FP64 steps of this block column (its updates are all applied)
    if (nb > MH) {
      // Two 64-wide steps: factor and solve the left half, update the right
      // half of the block column with it (split-BF16, K = 64), then factor and
      // solve the right half.  The diagonal block's share (both halves'
      // factors and the 64 x 64 update between them, a chain of small
      // launches) runs first; the panel rows below follow.
      const int hb = nb - MH;
      double *Aba = A11 + (long long)MH * ldl;  // right half's rows, left half's columns
      double *Ab = Aba + MH;                    // right half's diagonal block
      const size_t sb_small = sbytes(MH, 1, f64);
      SliceBuf Sba = slice_view((char *)w.tmp + sbytes(n, 1, f64) - sb_small, hb, 1);
      TRY(potrf_diag(MH, A11, ldl, info, k0, s, df));
      TRY(trsm_rows(hb, MH, Aba, ldl, A11, ldl, 0, s, df));
      TRY(split(Aba, hb, MH, Sba, k0 + MH));
      TRY(product(Sba, 0, Sba, 0, hb, hb, 1, true, Ab, k0 + MH, k0 + MH, s, 0, MH, 0));
      TRY(potrf_diag(hb, Ab, ldl, info, k0 + MH, s, df));
      if (m > 0) {
        double *Ca = A11 + (long long)nb * ldl;  // panel rows below the diagonal block, left half
        TRY(trsm_rows(m, MH, Ca, ldl, A11, ldl, 0, s, df));
        SliceBuf Sc = slice_view(w.tmp, m, 1);
        TRY(split(Ca, m, MH, Sc, k0 + nb));
        TRY(product(Sc, 0, Sba, 0, m, hb, 1, false, Ca + MH, k0 + nb, k0 + MH, s, 0, MH, 0));
        TRY(trsm_rows(m, hb, Ca + MH, ldl, Ab, ldl, 0, s, df));
      }
    } else {
      TRY(potrf_diag(nb, A11, ldl, info, k0, s, df));
      if (m > 0) TRY(trsm_rows(m, nb, A11 + (long long)nb * ldl, ldl, A11, ldl, 0, s, df));  // L21 = A21 L11^{-T}
    }
    if (m <= 0) continue;
    // ---- this block column's slices: chunk t of the group buffer, rows from k0 + nb
    const int r0 = k0 + nb - p0;  // first panel row, relative to the group
    TRY(split(A11 + (long long)nb * ldl, m, nb, G, k0 + nb, t, r0));
    // ---- next block column minus all of the group's block columns so far
    const int nb2 = std::min(MB, m);
    const bool last_in_group = (k0 + nb == p1);
    if (t == 0 && strip_pending) {  // the strip of the previous group writes this group's other columns
      TRY(cudaStreamWaitEvent(s, aux->ev_split, 0));
      strip_pending = false;
    }
    if (last_in_group && rest_pending) {  // the previous group's rest writes the next group's columns
      while (slabs.next < slabs.count) TRY(launch_slab());
      TRY(cudaStreamWaitEvent(s, aux->ev_rest, 0));
      rest_pending = false;
    }
    TRY(product(G, r0, G, r0, m, nb2, t + 1, true, A11 + (long long)nb * ldl + nb, k0 + nb, k0 + nb, s, 0, 0, 0));
    if (rest_pending && slabs.next < slabs.count) TRY(launch_slab());
    if (!last_in_group || m <= nb2) continue;
    // ---- the group's deferred update of the columns right of the next block column
    const int q1 = p1 + nb2;                   // strip: [q1, p2) of the next group
    const int p2 = std::min(n, p1 + D * MB);   // the next group's end
    const int chunks = t + 1;
    TRY(cudaEventRecord(aux->ev_fork, s));
    TRY(cudaStreamWaitEvent(aux->st, aux->ev_fork, 0));
    PriorityScope background(0);
    if (p2 > q1) {
      TRY(product(G, q1 - p0, G, q1 - p0, n - q1, p2 - q1, chunks, true, L + (long long)q1 * ldl + q1, q1, q1,
                  aux->st, bg_ctas, 0, bg_items));
      TRY(cudaEventRecord(aux->ev_split, aux->st));
      strip_pending = true;
    }
    if (n > p2) {
      slabs.G = G;
      slabs.p0 = p0;
      slabs.chunks = chunks;
      slabs.next = 0;
      // D - 1 slabs (one per next-column update before the next group's
      // last), cut where the remaining lower area falls by equal shares
      const int count = std::max(1, D - 1), width = n - p2;
      slabs.count = count;
      slabs.cut[0] = p2;
      for (int i = 1; i < count; ++i) {
        const double f = 1.0 - std::sqrt(1.0 - (double)i / count);
        const int c = p2 + (int)(f * width) / MB * MB;
        slabs.cut[i] = std::min(n, std::max(slabs.cut[i - 1], c));
      }
      slabs.cut[count] = n;
      rest_pending = true;
      if (D == 1) TRY(launch_slab());  // one-block lookahead: the rest goes at once
    }
  }
  while (rest_pending && slabs.next < slabs.count) TRY(launch_slab());
  if (strip_pending) TRY(cudaStreamWaitEvent(s, aux->ev_split, 0));
  if (rest_pending) TRY(cudaStreamWaitEvent(s, aux->ev_rest, 0));
  lease.joined();
  // every diagonal-block inverse, for the solves that follow the factorisation
  return f64 ? trtri_batched(n, L, ldl, std::min(MB, n), MB, w.inv, s)
             : trtri_sweep(n, L, ldl, std::min(MB, n), MB, w.inv, s);
}

// f64 (precision GPC_FP64): the same sweep with the products of f64x.cu on FP64
// storage.  The rows of L are equilibrated by powers of two first, L' = S^-1 L
// with S = diag(2^s_t), 2^s_t above row t's largest entry: every product sums
// over rows t of L (or columns t of the adjoint), L's entries entering with
// 2^-s_t and the adjoint's with 2^s_t, so a diagonal scaling of K changes no
// rounding.  Operand rows are then scaled by their largest entry: columns of
// L' (cexp), panel rows of the adjoint (xexp, found by the split itself) and, for
// its columns c, the block column's largest entry in equilibrated units less s_c
// (bexp; each chunk of 128 keeps its own exponent, so this one only has to keep
// FP32's range).  The finished diagonal block D^-T sym(tril(D^T Dbar)) D^-1 may grow
// past that range, by the square of the equilibrated block's inverse: its split then
// reports the exponent it needs (oexp) and the block column is split again, in a
// launch that otherwise ends at once.
cudaError_t chol_adjoint_mixed(int n, const double *L, long long ldl, double *A, long long lda, void *ws,
                               int *err, cudaStream_t s, bool f64) {
  MixWs w = carve(ws, n, true, f64);
  const int nblk = nchunks(n);
  const int first = n - (nblk - 1) * MB;  // rows in the top-left block
  // L^T slices: operand row t = column t of L, K = rows of L, chunked like the sweep's blocks.
  SliceBuf LT = slice_view(w.lt, n, nblk);
  if (f64) {
    TRY(f64x_lower_exps(n, L, ldl, w.rexp, w.cexp, s));
    TRY(cudaMemsetAsync(w.oexp, 0x80, exps_bytes(nblk), s));
    TRY(f64x_split(L, 1, ldl, n, n, first, LT, w.cexp, w.rexp, -1, false, s, 0, 0, F64xRow{nullptr, nullptr, nullptr, 0, 1, nullptr}));
  } else {
    TRY(split_operand(L, 1, ldl, n, n, first, LT, s));
  }
  if (f64) {  // the inverses, independent of the sweep
    TRY(trtri_batched(n, L, ldl, first, MB, w.inv, s));
    TRY(f64x_split_blocks(nblk, first, w.inv, first, MB, (long long)MB * MB, (long long)MB * MB, w.si, w.iexp, s));
  } else {
    TRY(trtri_sweep(n, L, ldl, first, MB, w.inv, s));
  }
  AuxLease lease(s);
  Aux *aux = nullptr;
  TRY(lease.take(&aux));
  // Within a step the Bbar update (rows below, columns left: the largest
  // product) runs on the auxiliary stream on all but tuning().mixed_adj_free_sms
  // SMs (16 by default; 8 to 32 differ by less than 2%) while the caller's stream
  // takes the rest of the Dbar chain (three small FP64 products) on the others; Rbar follows the chain
  // and takes SMs as the Bbar update frees them, and the next step's Cbar,
  // which both updates write, waits for both.
  const int side = std::min(tuning().mixed_adj_free_sms, sm_count() / 2);
  for (int ib = nblk - 1; ib >= 0; --ib) {
    const int j = (ib == 0) ? 0 : first + (ib - 1) * MB;
    const int k = first + ib * MB;
    const int nb = k - j, m = n - k;
    const int chunks = nblk - ib;  // K chunks of the block column, rows j..n
    const double *D = L + (long long)j * ldl + j;
    double *Dbar = A + (long long)j * lda + j;
    const double *dinv = w.inv + (size_t)ib * MB * MB;
    SliceBuf SDC = slice_view(w.sdc, nb, chunks);
    bool bbar_pending = false;
    if (m > 0) {
      double *Cbar = A + (long long)k * lda + j;
      if (f64) {
        // Cbar <- Cbar D^{-1} as one product with the block's inverse on eight slices
        // (with seven the adjoint's error grows to twice that of a substitution;
        // with eight it is about half).  Over the sweep at n = 16384 the split takes
        // 16 us and the product 37 us a step; two 64-wide substitutions, FP64 work of
        // m 128^2 / 2 multiply-adds, 52 us each in mid-sweep, and a split and a product
        // between them.
        SliceBuf SX = slice_view(w.sx, m, 1);
        TRY(f64x_split(Cbar, lda, 1, m, nb, nb, SX, nullptr, nullptr, 0, false, s, 0, 0,
                       F64xRow{w.xexp, nullptr, nullptr, 0, 0, nullptr, true}));
        TRY(f64x_gemm(SX, 0, 0, slice_view((char *)w.si + (size_t)ib * f64x_slice_bytes(MB, 1, true), MB, 1), 0, 0, m, nb,
                      1, false, w.xexp, w.iexp + (size_t)ib * MB, Cbar, lda, 1, nullptr, err, s, 0, 0, 0, nullptr, true));
      } else if (nb > MH) {
        // Cbar <- Cbar D^{-1} as two 64-wide steps, right half first: with
        // D = [Da 0; Dba Db], Xb = Cb Db^{-1}, then Ca -= Xb Dba (split-BF16,
        // K = nb - 64) and Xa = Ca Da^{-1}.  The FP64 solves halve.  (The product with
        // the inverse above is faster here too, 142 -> 128 ms a step at n = 16384,
        // but the gradient moved by its own error with it: see
        // potrf_lookahead_kernel.)
        const int hb = nb - MH;
        double *Cb = Cbar + MH;
        const double *Dba = D + (long long)MH * ldl;
        TRY(trsm_rows(m, hb, Cb, lda, Dba + MH, ldl, 1, s, true));
        SliceBuf SX = slice_view((char *)w.sc + sbytes(n, 1, false), m, 1);
        SliceBuf SD = slice_view(w.sdc, MH, 1);
        TRY(split_operand(Cb, lda, 1, m, hb, hb, SX, s));
        TRY(split_operand(Dba, 1, ldl, MH, hb, hb, SD, s));  // row c, K index t: Dba[t][c]
        TRY(ozaki_gemm(SX, 0, 0, SD, 0, 0, m, MH, 1, false, -1.0f, (float2 *)Cbar, lda, 1, nullptr, err, s, 0,
                       (hb + 31) / 32 * 32));
        TRY(trsm_rows(m, MH, Cbar, lda, D, ldl, 1, s, true));
      } else {
        TRY(trsm_rows(m, nb, Cbar, lda, D, ldl, 1, s, true));  // Cbar <- Cbar D^{-1} (FP64)
      }
      // Dbar -= Cbar^T C on slices (mixed: Dbar still in double-float storage):
      // the columns of Cbar (K = rows k..n) fill chunks 1.. of the block
      // column's slices; C^T is rows j..k of the L^T slices.
      SliceBuf SC = slice_view(w.sc, f64 ? m + nb : m, 1);
      if (f64) {
        // panel rows of the block column with their exponents, and bexp in
        // equilibrated units: Kbar' = S Kbar S for Cbar, Lbar' = S Lbar for Dbar's
        // rows, which only count here
        TRY(f64x_split(Dbar, lda, 1, m + nb, nb, nb, SC, nullptr, w.rexp + j, 1, false, s, 0, 0,
                       F64xRow{w.xexp, w.bexp, w.rexp + j, nb, 0, nullptr}));
        TRY(f64x_split(Cbar, 1, lda, nb, m, MB, SDC, w.bexp, w.rexp + k, 1, false, s, 1, 0,
                       F64xRow{nullptr, nullptr, nullptr, 0, 0, w.rexp + j}));
      } else {
        TRY(split_operand(Cbar, 1, lda, nb, m, MB, SDC, s, 1));
      }
      const int dch = chunks - 1;
      int dsplits = std::max(1, std::min(dch, (2 * sm_count() + 1) / 2));
      while (dsplits > 1 && ozaki_partial_bytes(nb, nb, dsplits) > kPartialCap) --dsplits;
      if (f64)
        TRY(f64x_gemm(SDC, 0, MB, LT, j, (ib + 1) * MB, nb, nb, dch, true, w.bexp, w.cexp + j, Dbar, lda, dsplits,
                      w.scratch, err, s, 0, 0, 0, w.rexp + j));
      else
        TRY(ozaki_gemm(SDC, 0, MB, LT, j, (ib + 1) * MB, nb, nb, dch, true, -1.0f, (float2 *)Dbar, lda, dsplits,
                       (float2 *)w.scratch, err, s));
      if (j > 0) {  // Bbar -= Cbar R on slices
        if (!f64) TRY(split_operand(Cbar, lda, 1, m, nb, nb, SC, s));
        TRY(cudaEventRecord(aux->ev_split, s));
        TRY(cudaStreamWaitEvent(aux->st, aux->ev_split, 0));
        if (f64)
          TRY(f64x_gemm(SC, nb, 0, LT, 0, ib * MB, m, j, 1, false, w.xexp + nb, w.cexp, A + (long long)k * lda, lda, 1,
                        nullptr, err, aux->st, sm_count() - side));
        else
          TRY(ozaki_gemm(SC, 0, 0, LT, 0, ib * MB, m, j, 1, false, -1.0f, (float2 *)(A + (long long)k * lda),
                         lda, 1, nullptr, err, aux->st, sm_count() - side));
        TRY(cudaEventRecord(aux->ev_rest, aux->st));
        bbar_pending = true;
      }
    } else if (f64) {
      TRY(f64x_block_exp(nb, Dbar, lda, w.rexp + j, w.bexp, s));
    }
    if (!f64) TRY(from_df_rect(nb, nb, Dbar, lda, s));
    {
      Gemm p;  // M = sym(tril(D^T Dbar))
      p.M = nb; p.N = nb; p.K = nb;
      p.A = D; p.lda = ldl; p.transA = true;
      p.B = Dbar; p.ldb = lda;
      p.C = w.m; p.ldc = nb;
      p.uplo = UPLO_LOWER_MIRROR;
      p.kskip = KSKIP_ROWS;  // D^T upper triangular
      p.algo_flops = (double)nb * nb * nb / 3.0;
      TRY(gemm_f64(p, w.scratch, s));
      Gemm t;  // T = M D^{-1}
      t.M = nb; t.N = nb; t.K = nb;
      t.A = w.m; t.lda = nb;
      t.B = dinv; t.ldb = nb;
      t.C = w.t; t.ldc = nb;
      t.kskip = KSKIP_COLS;  // D^{-1} lower triangular
      t.algo_flops = (double)nb * nb * (nb + 1);
      TRY(gemm_f64(t, w.scratch, s));
      Gemm d;  // Dbar = D^{-T} T, symmetric
      d.M = nb; d.N = nb; d.K = nb;
      d.A = dinv; d.lda = nb; d.transA = true;
      d.B = w.t; d.ldb = nb;
      d.C = Dbar; d.ldc = lda;
      d.uplo = UPLO_LOWER_MIRROR;
      d.kskip = KSKIP_ROWS;  // D^{-T} upper triangular
      d.algo_flops = (double)nb * nb * nb / 3.0 * 2.0;
      TRY(gemm_f64(d, w.scratch, s));
    }
    if (j > 0) {  // Rbar -= [Dbar; Cbar]^T [R; B] on slices (Rbar in double-float storage)
      if (f64) {  // chunk 0: the finished Dbar
        F64xRow row;
        row.rexp_sub = w.rexp + j;
        row.over_out = w.oexp + ib;
        TRY(f64x_split(Dbar, 1, lda, nb, nb, nb, SDC, w.bexp, w.rexp + j, 1, false, s, 0, 0, row));
        row.over_out = nullptr;
        row.alt = w.oexp + ib;
        TRY(f64x_split(Dbar, 1, lda, nb, m + nb, nb, SDC, w.bexp, w.rexp + j, 1, false, s, 0, 0, row));
      } else {
        TRY(split_operand(Dbar, 1, lda, nb, nb, nb, SDC, s, 0));
      }
      const int tiles = (j + 63) / 64;
      int splits = std::max(1, std::min(chunks, (2 * sm_count() + tiles - 1) / tiles));
      while (splits > 1 && ozaki_partial_bytes(nb, j, splits) > kPartialCap) --splits;
      if (f64)
        TRY(f64x_gemm(SDC, 0, 0, LT, 0, ib * MB, nb, j, chunks, false, w.oexp + ib, w.cexp, A + (long long)j * lda, lda,
                      splits, w.scratch, err, s, 0, 0, 0, w.rexp + j));
      else
        TRY(ozaki_gemm(SDC, 0, 0, LT, 0, ib * MB, nb, j, chunks, false, -1.0f, (float2 *)(A + (long long)j * lda),
                       lda, splits, (float2 *)w.scratch, err, s));
    }
    TRY(phi_block(nb, Dbar, lda, s));
    if (bbar_pending) {
      TRY(cudaStreamWaitEvent(s, aux->ev_rest, 0));
      bbar_pending = false;
    }
  }
  lease.joined();
  return cudaSuccess;
}

}  // namespace gpc
