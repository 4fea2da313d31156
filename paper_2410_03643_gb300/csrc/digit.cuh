// Digit passes: a transform along one grid axis (the DST-I S, or the Toeplitz product mu_a T_0) as a
// dense product on the tensor cores, exact to FP64 rounding.  GB300 issues two FP64 FMAs per SM and
// cycle, 1/61 of its FP32 rate, so an FP64 FFT pass is bound by that pipe; a tensor-core product of
// FP16 digits is not.
//
// Every line is scaled by a power of two to a fixed-point integer, X = sum_i x_i 2^(54 - 9i) with seven
// balanced digits |x_i| <= 256; the operator's entries likewise, A = sum_i a_i 2^(54 - 9i), |a_0| <= 128,
// tabulated at set-up.  Digits are FP16 operands of tcgen05.mma with FP32 accumulators in TMEM.  The
// products of one weight, D_d = sum_{i + j = d} sum_k a_i[r,k] x_j[k] over 128 entries k, are integers below
// 2^24 (a row's lower digits average 128: 2^22 per product), so the FP32 sums of the leading weights are exact;
// d = 0..6 are formed, 28 products, and combined in 64-bit integers.  What is dropped is 2^-61 of a line's
// largest entry times the operator's largest; the roundings left are those of the tabulated entries, of the
// integer sum and of the conversion to double.  On random and on smooth lines of 3 to 511 points the
// result is as near the exact product as an FP64 FFT's or nearer (two digits less would not be: the Toeplitz
// product of a smooth line cancels to 10^-3 of its terms).
//
// Both operators commute with the reflection j -> N - j of a line (N = n + 1, up to the parity of the
// sine mode), so for n >= 255 a line is folded into its sums s_j = x_j + x_{N-j} (with x_{N/2}) and
// differences d_j = x_j - x_{N-j}, and each half is a product of size N/2: half the work.  Shorter
// lines are not folded; 128 / N of them are stacked into one column of 128 entries and the operator is
// block diagonal.  Each stacked line has its own scale: with one for the whole column a line 2^30 smaller
// than another of its column has an error of 2e-8, and a finite line beside a non-finite one is NaN.
//
// Tile of a block: 128 operator rows of one half (all of it for n <= 255) times 32 columns (the real and
// imaginary parts of 16 lines).
#pragma once
#include <cstdint>
#include "internal.cuh"
#include "passes.cuh"

namespace rfnse {

constexpr int kDigits = 7;        // digits of an entry = accumulators (weights) per output
// result = sum_d D_d 2^(shift - 9d) in 64 bits: |D_0| < 2^17 for the Toeplitz rows (sum |c_k| = 2 c_0), and
// < 2^23 for the sine rows of two 128-entry blocks
constexpr int kDigShiftT = 45, kDigShiftS = 40;
constexpr int kDigits32 = 3;      // of the FP32 passes (digit32.cu)
constexpr int kDigExpBits = 61;   // operator entry = integer * 2^exp, |integer| <= 2^61
constexpr int kDigCols = 32;      // columns of a tile: 16 lines, real and imaginary part
constexpr int kDigLines = 16;
constexpr int kDigChunkK = 32;    // operator entries along K per chunk: 128 rows x 32 x 2 B = 8 KB
constexpr int kDigChunkBytes = 128 * kDigChunkK * 2;
constexpr int kDigStages = 5;     // chunks in flight

// Geometry of an axis of n points: K/128 per half, halves, lines stacked in one column.  1023 and 2047 points have none:
// a tile of 128 rows and 32 columns holds kb x 7 weights x 32 columns of TMEM, 448 of its 512 columns for 511 points
// and 896 for 1023 (a narrower tile, or rows of sums over fewer entries, has not been built).
struct DigitShape {
  int kb, halves, stack;
};
inline bool digit_shape(int n, DigitShape* s) {
  const int N = n + 1;
  if (N <= 128) *s = {1, 1, 128 / N};
  else if (N == 256) *s = {1, 2, 1};
  else if (N == 512) *s = {2, 2, 1};
  else return false;
  return true;
}
// bytes of an operator's digit table: halves x row blocks x digits x K/32 chunks
inline size_t digit_table_bytes(const DigitShape& s, int digits = kDigits) {
  return (size_t)s.halves * s.kb * digits * (s.kb * 128 / kDigChunkK) * kDigChunkBytes;
}

// The operator tables of one axis (set-up): S and mu_a T_0, each value = integer * 2^exp.
// entry = 0: the DST-I, 1: the Toeplitz operator (coefficients c scaled by mu)
// digits = kDigits: the FP64 passes' table; kDigits32: the FP32 passes'
void launch_setup_digits(const double* c, int n, double mu, int toeplitz, int exp, bool xax, int digits, void* table,
                         cudaStream_t s);
// exponent e with every |entry| <= 2^(e + 61)
int digit_exp_dst(int n);
int digit_exp_toeplitz(double alpha, double mu);

// Whether a context has digit tables at all, whether the FP64 passes of an axis run as digit passes (by default;
// the tuner may choose the line pass), and one digit pass: all storage FP64, FLAGS as for the line passes with one transform ([F_INSCALE |] F_DST, F_DST | F_LAM =
// S x / (omega + i Lambda), F_DST | F_DSCALE, F_TOEP_X, F_TOEP_ACC [| F_DOT0]); half: the first step's mu_a / 2.
bool digit_context(const rfnse_ctx* c);
bool digit_possible(const rfnse_ctx* c, int axis);
template <int FLAGS>
cudaError_t run_digit(rfnse_ctx* c, PassParams p, int axis, int half, cudaStream_t s);

// The FP32 passes of the mixed form: whether an axis has them, and one pass with the given storage types (input
// in FP32).
bool digit32_possible(const rfnse_ctx* c, int axis);
template <typename TOUT, typename TACCI, typename TACCO, int FLAGS>
cudaError_t run_digit32(rfnse_ctx* c, PassParams p, int axis, int half, cudaStream_t s);

// The passes that have a digit form: a sine transform or a Toeplitz product, and not the fused pass of 1-D
// grids (one launch there, three as digit passes); FP64 throughout, or FP32 with the storage types of the
// mixed form's Arnoldi step.
template <typename R, typename TIN, typename TOUT, typename TACCI, typename TACCO, int FLAGS>
constexpr bool digit_form() {
  if ((FLAGS & F_CIRC) || (!(FLAGS & F_DST) && (FLAGS & F_DSCALE)) || ((FLAGS & F_LAM) && (FLAGS & F_DSCALE)))
    return false;
  constexpr bool in16 = sizeof(TIN) == 16, out16 = sizeof(TOUT) == 16, ai16 = sizeof(TACCI) == 16,
                 ao16 = sizeof(TACCO) == 16;
  if (sizeof(R) == 8) return in16 && out16 && ai16 && ao16;
  if (out16 || in16) return false;
  if (FLAGS & F_DSCALE) return (FLAGS & F_TOEP_X) && !(FLAGS & F_DOT0) && ai16 && !ao16;
  if (FLAGS & F_DST) return ai16 && ao16;
  return (FLAGS & F_TOEP_ACC) && !ai16 && (ao16 || !(FLAGS & F_DOT0));
}

template <typename R, typename TIN, typename TOUT, typename TACCI, typename TACCO, int FLAGS>
cudaError_t run_digit_any(rfnse_ctx* c, const PassParams& p, int axis, int half, cudaStream_t s) {
  if constexpr (sizeof(R) == 8) return run_digit<FLAGS>(c, p, axis, half, s);
  else return run_digit32<TOUT, TACCI, TACCO, FLAGS>(c, p, axis, half, s);
}

// CUDA events around the launches of a profiled pass (rfnse_profile): the stop event, null when the pass
// is not of the profiled kind.
template <int KIND>
cudaError_t prof_start(rfnse_ctx* c, cudaStream_t s, cudaEvent_t* stop) {
  *stop = nullptr;
  if (c->prof_kind == 0 || (c->prof_kind | F_INSCALE | F_DOT0) != (KIND | F_INSCALE | F_DOT0)) return cudaSuccess;
  while (c->prof_used + 2 > c->prof_events.size()) {
    cudaEvent_t ev;
    const cudaError_t e = cudaEventCreate(&ev);
    if (e != cudaSuccess) return e;
    c->prof_events.push_back(ev);
  }
  *stop = c->prof_events[c->prof_used + 1];
  const cudaError_t e = cudaEventRecord(c->prof_events[c->prof_used], s);
  c->prof_used += 2;
  return e;
}

// One pass as digit passes: one transform per launch, so DST-Lambda-DST goes through the work vector zb
// (free until the pass that writes z) and the fused sub-solve and product through z itself.
// KIND: the kernel class under which rfnse_profile times it.
template <typename R, typename TIN, typename TOUT, typename TACCI, typename TACCO, int FLAGS,
          int KIND = FLAGS | (sizeof(R) == 4 ? 256 : 0)>
cudaError_t launch_digit_form(rfnse_ctx* c, const PassParams& p, int axis, int half, cudaStream_t s) {
  cudaEvent_t stop;
  cudaError_t e = prof_start<KIND>(c, s, &stop);
  if (e != cudaSuccess) return e;
  {
    NvtxRange range("rfnse pass");
    if constexpr ((FLAGS & F_LAM) != 0) {
      PassParams q = p;
      q.out = c->zb;
      e = run_digit_any<R, TIN, TOUT, TACCI, TACCO, F_DST | F_LAM>(c, q, axis, half, s);
      q.in = c->zb;
      q.out = p.out;
      if (e == cudaSuccess) e = run_digit_any<R, TOUT, TOUT, TACCI, TACCO, F_DST>(c, q, axis, half, s);
    } else if constexpr ((FLAGS & F_DSCALE) != 0) {
      e = run_digit_any<R, TIN, TOUT, TACCI, TACCO, F_DST | F_DSCALE>(c, p, axis, half, s);
      if constexpr ((FLAGS & F_TOEP_X) != 0) {
        PassParams q = p;
        q.in = p.out;
        q.in_dyn_z = (p.gdyn && p.zbase) ? 1 : 0;
        if (e == cudaSuccess) e = run_digit_any<R, TOUT, TOUT, TACCI, TACCO, F_TOEP_X>(c, q, axis, half, s);
      }
    } else {
      e = run_digit_any<R, TIN, TOUT, TACCI, TACCO, FLAGS>(c, p, axis, half, s);
    }
  }
  if (stop) {
    cudaEventRecord(stop, s);
    double fl, by;
    pass_work<R, TIN, TOUT, TACCI, TACCO, FLAGS>(p, fl, by);
    c->prof_flops += fl;
    c->prof_bytes += by;
  }
  cudaStreamCaptureStatus cap_st = cudaStreamCaptureStatusNone;
  if (e == cudaSuccess && c->debug && cudaStreamIsCapturing(s, &cap_st) == cudaSuccess &&
      cap_st == cudaStreamCaptureStatusNone) {
    char what[96];
    std::snprintf(what, sizeof what, "digit line pass (flags %d, %s, axis stride %lld)", FLAGS,
                  sizeof(R) == 4 ? "FP32" : "FP64", p.stride);
    const void* outs[3] = {(FLAGS & (F_DST | F_DSCALE)) ? p.out : nullptr,
                           (FLAGS & (F_TOEP_X | F_TOEP_ACC)) ? p.acc_out : nullptr,
                           (FLAGS & F_INSCALE) ? (const void*)p.copy_out : nullptr};
    const int elems[3] = {(int)sizeof(TOUT), (int)sizeof(TACCO), 16};
    if (p.gdyn) outs[0] = outs[2] = nullptr;  // device-resolved operands: not known on the host
    return debug_after_pass(c, s, what, outs, elems, 3, c->N);
  }
  return e;
}

// Geometry of an FP64 line pass without tuning: the default tile, halved while that leaves fewer than two
// blocks per SM.  A block's FFTs are bound by its SM's FP64 pipe (2 operations per cycle: eight lines of 64 points
// took 9 us), so on a small grid every line goes to an SM of its own.
template <int FLAGS>
PassGeom fp64_pass_geometry(const PassParams& p) {
  PassGeom g = default_pass_geometry<FLAGS>(p, false);
  auto blocks = [&](int B) {
    return p.stride == 1 ? (p.nlines + B - 1) / B : ((p.stride + B - 1) / B) * (p.nlines / p.stride);
  };
  while (g.B > 1 && blocks(g.B) < 2 * 152) g.B >>= 1;
  return g;
}

// One pass of the solver along `axis`: the digit form where the context has its tables (or where the tuner found
// it fastest), the line pass otherwise.  To the tuner the digit form is one more geometry (variant 2).
template <typename R, typename TIN, typename TOUT, typename TACCI, typename TACCO, int FLAGS>
cudaError_t solver_pass(rfnse_ctx* c, const PassParams& p, int axis, int half, cudaStream_t s) {
  constexpr bool form = digit_form<R, TIN, TOUT, TACCI, TACCO, FLAGS>();
  const bool possible = form && (sizeof(R) == 8 ? digit_possible(c, axis) : digit32_possible(c, axis));
  if (c->param_rec || (sizeof(R) == 4 && !possible)) {
    return launch_pass<R, TIN, TOUT, TACCI, TACCO, FLAGS>(c, p, s);
  } else {
    auto launch = [c, p, axis, half, s](const PassGeom& g) {
      if constexpr (form) {
        if (g.variant == 2) return launch_digit_form<R, TIN, TOUT, TACCI, TACCO, FLAGS>(c, p, axis, half, s);
      }
      return launch_pass_geom<R, TIN, TOUT, TACCI, TACCO, FLAGS>(c, p, s, g);
    };
    PassGeom g = possible ? PassGeom{1, 1, 2} : fp64_pass_geometry<FLAGS>(p);
    if (c->tune_rec || !c->tune.empty()) {
      const unsigned long long key = pass_key<R, TIN, TOUT, TACCI, TACCO, FLAGS>(c, p);
      if (c->tune_rec) {  // rfnse_autotune is recording the solver's pass configurations
        bool seen = false;
        for (const TuneRecord& r : *c->tune_rec) seen = seen || r.key == key;
        if (!seen) {
          TuneRecord r;
          r.key = key;
          r.dflt = g;
          r.cands = pass_candidates<FLAGS>(p, sizeof(R) == 4 && fixed_fft_length(p.log2L), sizeof(cv<R>));
          r.launch = launch;
          c->tune_rec->push_back(std::move(r));
        }
      } else {
        const auto it = c->tune.find(key);
        if (it != c->tune.end()) {
          g = it->second;
          c->tuned_launches += 1;
        }
      }
    }
    return launch(g);
  }
}

}  // namespace rfnse
