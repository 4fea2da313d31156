// The FP64 digit-pass kernel and its launches (see digit.cuh).
#include <cuda_fp16.h>
#include <cmath>
#include "digit.cuh"
#include "tc05.cuh"

namespace rfnse {

namespace {

struct DigitArgs {
  const unsigned char* table;  // operator digits (k_digit_table)
  int oexp;                    // operator entry = integer * 2^oexp
  int log2N, stack;            // log2(n + 1), lines stacked in one column
  int ca_code, cb_code;        // ca, cb as in the double-float passes (-1: any value)
  double lam_scale;            // 1 / dst_scale: lamfac holds i dst_scale / (omega + i Lambda)
  int give_up;                 // the chunk whose request gives up untried (rfnse_test_give_up; none if negative)
  int *err, *loop_err;         // set when a wait gives up: for the host, and for the loop conditions on the device
};

// Shared memory: barriers and line exponents (of every line stacked in a column), the vector's digits, the chunk
// ring.  The digits are one K-major operand of 224 columns, digit j of column n at 32 j + n, because D_i .. D_6 are
// neighbours in TMEM: for one operator digit a_i a single MMA of N = 32 (7 - i) columns forms its products with x_0 ..
// x_{6-i}.  (An MMA costs 44 + N/2 cycles with A in shared memory, measured for N = 16..128: seven MMAs of
// 32..224 columns per 16 entries take 751 cycles, 28 of 32 columns 1680.)  Core matrices lie 128 B (next
// 8 columns) and 3616 B (next 8 entries) apart, so that both the threads of a strided pass (neighbouring
// columns) and of an x pass (neighbouring entries, real and imaginary column) store without bank conflicts.
constexpr int kSbo = 128, kLbo = kDigits * (kDigCols / 8) * kSbo + 32;
constexpr int kDigitPitch = (kDigCols / 8) * kSbo;  // bytes from a digit to the next
constexpr int kCtrl = 128 + 32 * kDigLines * 4;  // up to 32 lines are stacked in each of the 16 columns
static_assert(kCtrl % 128 == 0, "alignment");
constexpr int kRowPitch = kDigLines * 16 + 16;  // staged results: a row's 16 lines, 16 B each
template <int KB> constexpr int digit_bytes() { return (16 * KB * kLbo + 127) & ~127; }
template <int KB> constexpr int digit_smem() { return kCtrl + digit_bytes<KB>() + kDigStages * kDigChunkBytes; }

// x as a fixed-point integer on the scale of exponent emax: |X| < 2^61, x = X 2^(emax - 1083), by 32-bit
// shifts (what lies below 2^-61 of the scale is cut off).  All integer: an FP64 operation takes half a cycle of
// an SM, an integer one 1/64.
__device__ __forceinline__ long long to_fixed(uint32_t hi, uint32_t lo, int emax) {
  const int e = (int)((hi >> 20) & 0x7ff);
  const uint32_t mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const int sh = emax - max(e, 1);
  const uint32_t H = __funnelshift_l(lo, mh, 8), L = lo << 8;
  const uint32_t l = __funnelshift_rc(__funnelshift_rc(L, H, sh), 0u, max(sh - 32, 0));
  const uint32_t u = __funnelshift_rc(H, 0u, sh);
  const long long X = (long long)(((unsigned long long)u << 32) | l);
  return (int)hi < 0 ? -X : X;
}

// v 2^ex rounded to nearest (truncated below the normal range, infinity above it)
__device__ __forceinline__ double from_fixed(long long v, int ex) {
  const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  if (m == 0) return 0.0;
  const int lz = __clzll((long long)m);
  const unsigned long long t = m << lz;
  const unsigned long long r = (t >> 11) + ((t >> 10) & 1);  // 2^52 .. 2^53
  const int E = ex + 63 - lz + 1023;
  unsigned long long b = E <= 0 ? (E < -60 ? 0ull : r >> (1 - E))
                         : E >= 2047 ? 0x7ff0000000000000ull
                                     : ((unsigned long long)(E - 1) << 52) + r;
  b |= (unsigned long long)v & 0x8000000000000000ull;
  return __longlong_as_double((long long)b);
}

__device__ __forceinline__ uint32_t half2_sub(uint32_t a, uint32_t b) {
  const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// The seven digits of two fixed-point values, packed as FP16 pairs: digit i of Y (biased so that every
// field is unsigned) is put below the exponent of 1024, whose ulp is one unit, and the offset subtracted.
__device__ __forceinline__ void digits2(long long y0, long long y1, uint32_t (&d)[kDigits]) {
  constexpr long long bias = 0x4020100804020100ll;  // 256 (1 + 2^9 + ... + 2^54)
  const unsigned long long a = (unsigned long long)(y0 + bias), b = (unsigned long long)(y1 + bias);
#pragma unroll
  for (int i = 0; i < kDigits; ++i) {
    const uint32_t fa = (uint32_t)(a >> (54 - 9 * i)), fb = (uint32_t)(b >> (54 - 9 * i));
    const uint32_t f = __byte_perm(fa, fb, 0x5410) & (i == 0 ? 0x03ff03ffu : 0x01ff01ffu);
    d[i] = half2_sub(f | 0x64006400u, 0x65006500u);
  }
}

__device__ __forceinline__ double2 coef_times(int code, double2 c, double2 v) {
  switch (code) {
    case 0: return make_double2(0.0, 0.0);
    case 1: return v;
    case 2: return make_double2(-v.x, -v.y);
    case 3: return make_double2(-v.y, v.x);
    case 4: return make_double2(v.y, -v.x);
    default: return cmul(c, v);
  }
}

// KB: K / 128 of a half; FOLD: sums and differences (two halves), else stacked whole lines.
// 255^3, S 2000 -> 415 us, T 3870 -> 480 us (the FP64 FFT passes before, these now); 511^2, S 47 -> 24 us, T 87 -> 27.
// An exponent for each stacked line (one for their column would not do: digit.cuh) takes 127 x 255 x 63 runs from 14.13 to 14.35 ms.
// Nothing is saturated (255 x 255 x 63, S: ALU pipe 49%, tensor 24%, L2 17% of peak; T also FP64 23%): two blocks
// per SM, all that TMEM holds, take turns at the integer work of the digits (4000 cycles of a tile of 16 lines
// and one half), the products (6400), the sums (2100) and the results (3000, T 7600 with the exchange of the halves).
// 512 threads of one part each against 256 of both: 415 against 438 us.  Folding in FP64 instead of integers: 494.
template <int FLAGS, int KB, bool FOLD>
__global__ void __launch_bounds__(512 * KB, KB == 1 ? 2 : 1) k_digit(const PassParams p, const DigitArgs a) {
  constexpr bool TOEP = (FLAGS & (F_TOEP_X | F_TOEP_ACC)) != 0;
  constexpr bool PAIR = FOLD && TOEP;  // both halves of a result are needed: a cluster of two blocks
  constexpr int NT = 512 * KB;
  constexpr int NK = 128 * KB / kDigChunkK;  // chunks per operator digit
  constexpr int NC = kDigits * NK;
  constexpr uint32_t COLS = KB == 1 ? 256 : 512;
  if (p.skip && *p.skip) return;  // uniform over the launch
  extern __shared__ __align__(128) unsigned char sm[];
  unsigned char* dig = sm + kCtrl;
  const uint32_t s0 = tc::smem_addr(sm), sdig = s0 + kCtrl;
  const uint32_t sring = sdig + digit_bytes<KB>();
  const uint32_t b_full = s0, b_empty = s0 + 8 * kDigStages, b_done = s0 + 16 * kDigStages;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sm + 96);
  volatile int* s_fail = reinterpret_cast<volatile int*>(sm + 100);
  unsigned* smax = reinterpret_cast<unsigned*>(sm + 128);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  int h = 0, mb = 0;
  long long tile = blockIdx.x;
  if (FOLD) {
    h = (int)(tile & 1);
    tile >>= 1;
    if (KB == 2) {
      mb = (int)(tile & 1);
      tile >>= 1;
    }
  }
  const unsigned char* tab = a.table + ((size_t)h * KB + mb) * NC * kDigChunkBytes;

  if (warp == 0) {
    if (lane == 0) {
      for (int i = 0; i < kDigStages; ++i) {
        tc::mbar_init(b_full + 8 * i, 1);
        tc::mbar_init(b_empty + 8 * i, 1);
      }
      tc::mbar_init(b_done, 1);
      tc::mbar_init_fence();
      *s_fail = 0;
    }
    for (int i = lane; i < kDigLines * a.stack; i += 32) smax[i] = 0;
    __syncwarp();
    tc::tmem_alloc(tc::smem_addr(s_tmem), COLS);
    tc::fence_before();
  }
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *s_tmem;
  auto load_chunk = [&](int c) {
    const int st = c % kDigStages;
    tc::mbar_expect_tx(b_full + 8 * st, kDigChunkBytes);
    tc::bulk_load(sring + st * kDigChunkBytes, tab + (size_t)c * kDigChunkBytes, kDigChunkBytes, b_full + 8 * st);
  };
  if (tid == 32)
    for (int c = 0; c < kDigStages; ++c) load_chunk(c);

  // ---- this thread's eight entries (and their mirror images) of one column: the real or the imaginary
  // part of a line, neighbouring lanes of a warp, so that a warp reads 256 consecutive bytes -------------
  const bool xax = p.stride == 1;
  const int n = p.n;
  const int part = tid & 1, t16 = (tid >> 1) & 15;
  const int l = xax ? ((tid >> 5) & 15) : t16;
  const int kg = xax ? ((tid >> 9) * 16 + t16) : (tid >> 5);
  auto slot_pos = [&](int i) { return xax ? (kg >> 4) * 128 + i * 16 + t16 : kg * 8 + i; };
  const long long hi = xax ? 0 : tile / p.tiles_inner;
  const long long line0 = xax ? tile * (kDigLines * a.stack) : (tile - hi * p.tiles_inner) * (kDigLines * a.stack);
  const long long nline = xax ? p.nlines : p.stride;       // lines that line0 + ... runs over
  const long long base0 = xax ? 0 : hi * p.stride * n;
  const long long lstep = xax ? n : 1, estep = xax ? 1 : p.stride;

  double va[8];
  [[maybe_unused]] double vb[8];
  const bool mid = FOLD && 2 * slot_pos(7) == n - 1;  // the thread's last entry is the middle of the line
  {
    const double2* in = reinterpret_cast<const double2*>(p.in);
    double2* cpy = p.copy_out;
    double sc = 1.0;
    if constexpr ((FLAGS & F_INSCALE) != 0) {
      if (p.gdyn) {
        in = p.gdyn->src;
        sc = p.gdyn->src_scale;
        cpy = p.vbase + (long long)p.gdyn->j * p.ldv;
      } else {
        sc = *p.in_scale;
      }
    }
    if constexpr (FOLD) {
      const bool ok = line0 + l < nline;
      const long long g0 = base0 + (line0 + l) * lstep, g1 = g0 + (long long)(n - 1 - slot_pos(0)) * estep;
      const long long step = (xax ? 16 : 1) * estep;
      const long long g = g0 + slot_pos(0) * estep;
      const double* s = reinterpret_cast<const double*>(in + g) + part;
      const double* t = reinterpret_cast<const double*>(in + g1) + part;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        va[i] = ok ? s[2 * i * step] : 0.0;
        vb[i] = ok && !(i == 7 && mid) ? t[-2 * i * step] : 0.0;
      }
      if constexpr ((FLAGS & F_INSCALE) != 0) {
        double* d = reinterpret_cast<double*>(cpy + g) + part;
        double* f = reinterpret_cast<double*>(cpy + g1) + part;
        const bool wr = ok && h == 0 && mb == 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          va[i] *= sc;
          vb[i] *= sc;
          if (wr) d[2 * i * step] = va[i];
          if (wr && !(i == 7 && mid)) f[-2 * i * step] = vb[i];
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int q = slot_pos(i);
        const int sl = q >> a.log2N, pos = q - (sl << a.log2N);
        const long long ln = line0 + sl * kDigLines + l;
        const long long g = base0 + ln * lstep + pos * estep;
        const bool ok = ln < nline && pos < n;
        va[i] = ok ? reinterpret_cast<const double*>(in + g)[part] : 0.0;
        if constexpr ((FLAGS & F_INSCALE) != 0) {
          va[i] *= sc;
          if (ok) reinterpret_cast<double*>(cpy + g)[part] = va[i];
        }
      }
    }
  }
  // the largest exponent of each line: an exponent per stacked line (the operator is block diagonal, so the lines of
  // a column need no common scale, and a tiny line beside a large or non-finite one keeps its digits)
  if constexpr (FOLD) {
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      m = max(m, max((unsigned)__double2hiint(va[i]) & 0x7fffffffu, (unsigned)__double2hiint(vb[i]) & 0x7fffffffu));
    if (xax) {
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) atomicMax(&smax[l], m);
    } else {
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      if (part == 0) atomicMax(&smax[l], m);
    }
  } else {
    const int width = min(32, 2 << a.log2N);  // along x: neighbouring lanes that hold entries of one stacked line
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      m = max(m, (unsigned)__double2hiint(va[i]) & 0x7fffffffu);
      const int sl = slot_pos(i) >> a.log2N;
      if (i < 7 && slot_pos(i + 1) >> a.log2N == sl) continue;  // uniform over the warp
      if (xax) {
        if (width == 32) m = __reduce_max_sync(0xffffffffu, m);
        else
          for (int o = 1; o < width; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((lane & (width - 1)) == 0) atomicMax(&smax[sl * kDigLines + l], m);
      } else {
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
        if (part == 0) atomicMax(&smax[sl * kDigLines + l], m);
      }
      m = 0;
    }
  }
  __syncthreads();
  {
    [[maybe_unused]] const int emax_l = max((int)(smax[l] >> 20), 1);
    auto exponent = [&](int i) {
      if constexpr (FOLD) return emax_l;
      else return max((int)(smax[(slot_pos(i) >> a.log2N) * kDigLines + l] >> 20), 1);
    };
    const int col = 2 * l + part;
    unsigned char* dst = dig + kg * kLbo + (col >> 3) * kSbo + (col & 7) * 16;
    uint32_t w[kDigits][4];
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      long long y[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int emax = exponent(i + k);
        y[k] = to_fixed((uint32_t)__double2hiint(va[i + k]), (uint32_t)__double2loint(va[i + k]), emax);
        if constexpr (FOLD) {  // + or - the mirror image; the middle belongs to the sums alone
          y[k] += to_fixed((uint32_t)__double2hiint(vb[i + k]) ^ ((uint32_t)h << 31),
                           (uint32_t)__double2loint(vb[i + k]), emax);
          if (i + k == 7 && h == 1 && mid) y[k] = 0;
        }
      }
      uint32_t d[kDigits];
      digits2(y[0], y[1], d);
#pragma unroll
      for (int j = 0; j < kDigits; ++j) w[j][i >> 1] = d[j];
    }
#pragma unroll
    for (int j = 0; j < kDigits; ++j)
      *reinterpret_cast<uint4*>(dst + j * kDigitPitch) = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
  }
  tc::fence_async_smem();
  __syncthreads();

  // ---- products: one warp issues the MMAs (all its values warp-uniform: an MMA issued from a divergent
  // branch costs 125 cycles or more of issue), another refills the chunk ring --------------------------
  int chunks = kDigStages;  // warp 1: chunks requested so far; warp 0: chunks multiplied
  const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
  if (uwarp == 0) {
    tc::fence_after();
    const bool one = tc::elect_one();
    const uint32_t ud = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t da0 = tc::smem_desc(__shfl_sync(0xffffffffu, sring, 0), 2048, 128);
    const uint64_t db0 = tc::smem_desc(__shfl_sync(0xffffffffu, sdig, 0), kLbo, kSbo);
    bool ok = true;
    int st = 0, ph = 0;
    for (int i = 0; i < kDigits && ok; ++i) {
      const uint32_t id = tc::idesc_f16(128, kDigCols * (kDigits - i));
      for (int kc = 0; kc < NK; ++kc) {
        ok = tc::mbar_wait(b_full + 8 * st, ph, s_fail);
        if (!ok) {
          chunks = i * NK + kc;
          break;
        }
        const uint32_t kb = KB == 1 ? 0 : (uint32_t)kc / (128 / kDigChunkK);
        const uint32_t d = ud + (kb * kDigits + i) * kDigCols;
        const bool first = i == 0 && kc % (128 / kDigChunkK) == 0;
#pragma unroll
        for (int ks = 0; ks < kDigChunkK / 16; ++ks) {
          const uint64_t da = da0 + (uint32_t)((st * kDigChunkBytes + ks * 4096) >> 4);
          const uint64_t db = db0 + (uint32_t)(((kc * (kDigChunkK / 16) + ks) * 2 * kLbo) >> 4);
          if (one) tc::mma_f16(d, da, db, id, !(first && ks == 0));
        }
        if (one) tc::mma_commit(b_empty + 8 * st);
        if (++st == kDigStages) {
          st = 0;
          ph ^= 1;
        }
      }
    }
    if (one) tc::mma_commit(b_done);
    if (ok) chunks = NC;
    __syncwarp();
    if (!__all_sync(0xffffffffu, ok)) {  // the issuing lane's count is the one to go by
      chunks = __shfl_sync(0xffffffffu, chunks, __ffs(__ballot_sync(0xffffffffu, one)) - 1);
      *s_fail = 1;
    }
  } else if (uwarp == 1) {
    bool ok = true;
    for (int c = kDigStages; c < NC; ++c) {
      ok = c != a.give_up && tc::mbar_wait(b_empty + 8 * (c % kDigStages), ((c / kDigStages) & 1) ^ 1, s_fail);
      if (!ok) break;
      if (lane == 0) load_chunk(c);
      chunks = c + 1;
    }
    __syncwarp();
    if (!__all_sync(0xffffffffu, ok)) {
      chunks = __shfl_sync(0xffffffffu, chunks, 0);
      *s_fail = 1;
    }
  }
  __syncwarp();
  if (uwarp == 0 && !tc::mbar_wait(b_done, 0) && lane == 0) *s_fail = 1;
  __syncthreads();  // the other warps sleep here rather than poll
  tc::fence_after();
  if (*s_fail) {  // uniform: a wait gave up.  Wait for the products and copies in flight (they write TMEM and this
                  // block's barriers and shared memory), free TMEM and leave
    if (uwarp == 0) {
      for (int c = max(chunks - kDigStages, 0); c < chunks; ++c)
        tc::mbar_wait(b_empty + 8 * (c % kDigStages), (c / kDigStages) & 1);
      tc::mbar_wait(b_done, 0);
    } else if (uwarp == 1) {
      for (int c = chunks - kDigStages; c < chunks; ++c)
        tc::mbar_wait(b_full + 8 * (c % kDigStages), (c / kDigStages) & 1);
      if (lane == 0) {
        *(volatile int*)a.err = 1;
        *(volatile int*)a.loop_err = 1;
      }
    }
    __syncthreads();
    if (warp == 0) tc::tmem_free(tmem, COLS);
    if constexpr (PAIR) {
      tc::cluster_sync();
      tc::cluster_sync();
    }
    return;
  }

  // ---- accumulators -> 64-bit integers, staged by row (over the digits, which the MMAs have read) --------
  {
    constexpr int CW = kDigCols / (4 * KB);  // columns of this warp
    constexpr int SH = TOEP ? kDigShiftT : kDigShiftS;
    const int row = 32 * (warp & 3) + lane;
#pragma unroll
    for (int c0 = (warp >> 2) * CW, b = 0; b < CW / 4; ++b, c0 += 4) {
      const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
      long long v[4];
#pragma unroll
      for (int kb = 0; kb < KB; ++kb) {
        float D[kDigits][4];
#pragma unroll
        for (int d = 0; d < kDigits; ++d) tc::tmem_ld(ta + (kb * kDigits + d) * kDigCols, D[d]);
        tc::tmem_ld_wait(D);
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // sum_d D_d 2^(SH - 9d)
          const long long up = (long long)__float2int_rn(D[0][i]) * 262144 +
                               ((long long)__float2int_rn(D[1][i]) * 512 + __float2int_rn(D[2][i]));
          const long long mid = (long long)__float2int_rn(D[3][i]) * 512 + __float2int_rn(D[4][i]);
          const int low = __float2int_rn(fmaf(D[6][i], 0x1p-9f, D[5][i]) * (TOEP ? 1.0f : 0x1p-5f));
          const long long s = (up << (SH - 18)) + (mid << (SH - 36)) + low;
          v[i] = kb ? v[i] + s : s;
        }
      }
      unsigned char* dst = dig + row * kRowPitch + (c0 >> 1) * 16;
#pragma unroll
      for (int i = 0; i < 4; i += 2)
        *reinterpret_cast<longlong2*>(dst + (i >> 1) * 16) = make_longlong2(v[i], v[i + 1]);
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_free(tmem, COLS);
  }
  if constexpr (PAIR) tc::cluster_sync();

  // ---- results: convert and apply the pass's pointwise work, in grid order -------------------------------
  [[maybe_unused]] double dot = 0.0, nrm = 0.0;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  struct Operands {
    double2 u, z, acc;
    double D;
  };
  [[maybe_unused]] double2* zout = reinterpret_cast<double2*>(p.out);
  auto fetch = [&](long long g, bool ok) {
    Operands o;
    o.u = o.z = o.acc = make_double2(0.0, 0.0);
    o.D = 0.0;
    if (!ok) return o;
    if constexpr ((FLAGS & F_LAM) != 0) o.u = reinterpret_cast<const double2*>(p.lamfac)[g];
    if constexpr ((FLAGS & F_DSCALE) != 0) {
      o.u = reinterpret_cast<const double2*>(p.dfac)[g];
      if (p.z_add) o.acc = zout[g];
    }
    if constexpr (TOEP) {
      if (p.acc_in) o.acc = reinterpret_cast<const double2*>(p.acc_in)[g];
      if constexpr ((FLAGS & F_TOEP_X) != 0) {
        o.z = reinterpret_cast<const double2*>(p.in)[g];
        if (p.Dr) o.D = reinterpret_cast<const double*>(p.Dr)[g];
      }
      if constexpr ((FLAGS & F_DOT0) != 0) o.u = p.dot_v0[g];
    }
    return o;
  };
  auto emit = [&](long long g, long long re, long long im, int ln, const Operands& o) {  // ln: its place in smax
    const int emax = (int)(smax[ln] >> 20);
    const int ex = max(emax, 1) - 975 - (TOEP ? kDigShiftT : kDigShiftS) + a.oexp;
    double2 y = make_double2(from_fixed(re, ex), from_fixed(im, ex));
    if (emax == 2047) y = make_double2(nan, nan);  // an infinity or NaN on the line
    if constexpr ((FLAGS & F_DST) != 0 && (FLAGS & F_DSCALE) == 0) {
      if constexpr ((FLAGS & F_LAM) != 0) {
        y = cmul(y, o.u);
        y = make_double2(y.y * a.lam_scale, -y.x * a.lam_scale);
      }
      reinterpret_cast<double2*>(p.out)[g] = y;
    }
    if constexpr ((FLAGS & F_DSCALE) != 0) {
      y = cmul(y, o.u);
      zout[g] = p.z_add ? cadd(o.acc, y) : y;
    }
    if constexpr (TOEP) {
      double2 acc = o.acc;
      if constexpr ((FLAGS & F_TOEP_X) != 0) {
        if (p.Dr) {
          y.x = fma(-o.D, o.z.x, y.x);
          y.y = fma(-o.D, o.z.y, y.y);
        }
        if (a.ca_code != 0) acc = cadd(acc, coef_times(a.ca_code, p.ca, o.z));
      }
      acc = cadd(acc, coef_times(a.cb_code, p.cb, y));
      reinterpret_cast<double2*>(p.acc_out)[g] = acc;
      if constexpr ((FLAGS & F_DOT0) != 0) {
        dot = fma(o.u.x, acc.x, dot);
        dot = fma(o.u.y, acc.y, dot);
      }
      if (p.nrm_part) {
        nrm = fma(acc.x, acc.x, nrm);
        nrm = fma(acc.y, acc.y, nrm);
      }
    }
  };
  if constexpr (PAIR) {  // y_j = e_j + o_j, y_{N-j} = e_j - o_j; this block finishes eight of the lines
    constexpr int ITEMS = 128 * 8 / NT;
    int r = xax ? (tid & 127) : (tid >> 3), ln = 8 * h + (xax ? (tid >> 7) : (tid & 7));
    long long g = base0 + (line0 + ln) * lstep + (mb * 128 + r) * estep;
    long long g2 = base0 + (line0 + ln) * lstep + (n - 1 - mb * 128 - r) * estep;
    const long long dg = xax ? (NT / 128) * lstep : (NT / 8) * estep;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const bool ok = line0 + ln < nline, two = 2 * (mb * 128 + r) != n - 1;
      const Operands o1 = fetch(g, ok), o2 = fetch(g2, ok && two);
      const uint32_t at = sdig + r * kRowPitch + ln * 16;
      long long er, ei, dr, di;
      tc::ld_cluster(at, 0, er, ei);
      tc::ld_cluster(at, 1, dr, di);
      if (ok) emit(g, er + dr, ei + di, ln, o1);
      if (ok && two) emit(g2, er - dr, ei - di, ln, o2);
      g += dg;
      g2 += xax ? dg : -dg;
      if (xax) ln += NT / 128;
      else r += NT / 8;
    }
    tc::cluster_sync();
  } else {
    constexpr int ITEMS = 128 * kDigLines / NT;
    int r = xax ? (tid & 127) : (tid >> 4), ln = xax ? (tid >> 7) : (tid & 15);
    long long g = base0 + (line0 + ln) * lstep + (long long)(2 * (mb * 128 + r) + h) * estep;  // FOLD
    const long long dg = xax ? (NT / 128) * lstep : 2 * (NT / 16) * estep;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      int pos = 2 * (mb * 128 + r) + h, sl = 0;
      long long line = line0 + ln;
      if constexpr (!FOLD) {
        sl = r >> a.log2N;
        pos = r - (sl << a.log2N);
        line += sl * kDigLines;
        g = base0 + line * lstep + pos * estep;
      }
      const bool ok = line < nline && pos < n;
      const Operands o = fetch(g, ok);
      const longlong2 v = *reinterpret_cast<const longlong2*>(dig + r * kRowPitch + ln * 16);
      if (ok) emit(g, v.x, v.y, sl * kDigLines + ln, o);
      g += dg;
      if (xax) ln += NT / 128;
      else r += NT / 16;
    }
  }
  if constexpr ((FLAGS & F_DOT0) != 0) block_sum_store(dot, p.dot_part + blockIdx.x);
  if constexpr (TOEP)
    if (p.nrm_part) block_sum_store(nrm, p.nrm_part + blockIdx.x);
}

int coef_code(double2 c) {
  if (c.x == 0.0 && c.y == 0.0) return 0;
  if (c.x == 1.0 && c.y == 0.0) return 1;
  if (c.x == -1.0 && c.y == 0.0) return 2;
  if (c.x == 0.0 && c.y == 1.0) return 3;
  if (c.x == 0.0 && c.y == -1.0) return 4;
  return -1;
}

template <int FLAGS, int KB, bool FOLD>
cudaError_t launch_digit(const PassParams& p, const DigitArgs& a, unsigned grid, cudaStream_t s) {
  auto kern = k_digit<FLAGS, KB, FOLD>;
  constexpr int smem = digit_smem<KB>();
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(512 * KB);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (FOLD && (FLAGS & (F_TOEP_X | F_TOEP_ACC))) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, p, a);
}

}  // namespace

bool digit_possible(const rfnse_ctx* c, int axis) { return c->digS[axis] != nullptr; }

// FP64 form: a tile takes 8 us whatever its size, and the fused FFT passes are two launches each here, while an
// FP64 FFT pass costs in proportion to the points.  A time step of the FP64 form (4 Arnoldi steps) with digit /
// FFT passes: 127^2 0.52 / 0.40 ms, 255 x 127 0.55 / 0.43, 15 x 63 x 63 0.686 / 0.679, 255^2 0.58 / 0.60,
// 511 x 255 0.72 / 1.04, 511^2 0.92 / 2.04, 127 x 63 x 127 1.80 / 7.01: they meet at 60000 points.
// Mixed form: the residual products have double-float passes to beat: 255^3 y, z 860 and x 973 us against 480-540 and
// 620-630 here, 511^2 33 against 27, but a batch of 16 grids of 127..511 points per axis took 24.9 ms with those and 25.9
// with these (a block here fills half an SM, so the instances' streams overlap less), hence from 2^20 points on.  The FP32
// passes follow the same line; on smaller grids they have not been measured (digit32.cu takes axes of up to 255 points).
bool digit_context(const rfnse_ctx* c) { return c->d > 1 && c->N >= (c->p.precision == 1 ? 1 << 20 : 60000); }

template <int FLAGS>
cudaError_t run_digit(rfnse_ctx* c, PassParams p, int axis, int half, cudaStream_t s) {
  constexpr bool TOEP = (FLAGS & (F_TOEP_X | F_TOEP_ACC)) != 0;
  DigitShape sh;
  if (!digit_possible(c, axis) || !digit_shape(p.n, &sh)) return cudaErrorInvalidValue;
  DigitArgs a{};
  a.table = static_cast<const unsigned char*>(TOEP ? c->digT[axis] : c->digS[axis]);
  a.oexp = TOEP ? c->digT_exp[axis] - (half ? 1 : 0) : digit_exp_dst(p.n);
  a.log2N = p.log2L - 1;
  a.stack = sh.stack;
  a.ca_code = coef_code(p.ca);
  a.cb_code = coef_code(p.cb);
  a.lam_scale = 1.0 / p.dst_scale;
  a.give_up = c->give_up_at < 0 ? -1 : kDigStages + c->give_up_at;
  a.err = &c->peek[2].err;  // pinned
  a.loop_err = &c->gs->err;
  const long long per = (long long)kDigLines * sh.stack;
  long long tiles;
  if (p.stride == 1) {
    p.tiles_inner = 1;
    tiles = (p.nlines + per - 1) / per;
  } else {
    p.tiles_inner = (p.stride + per - 1) / per;
    tiles = p.tiles_inner * (p.nlines / p.stride);
  }
  const long long grid = tiles * sh.halves * sh.kb;
  if (grid <= 0) return cudaSuccess;
  if constexpr ((FLAGS & F_DOT0) != 0) {  // too many partials for the Arnoldi kernel to sum: plain pass
    if (grid > kDot0MaxBlocks) {
      c->dot0_blocks = 0;
      return run_digit<(FLAGS & ~F_DOT0)>(c, p, axis, half, s);
    }
    c->dot0_blocks = (int)grid;
  }
  if (p.nrm_part) {
    if (grid > kNormPartMax) p.nrm_part = nullptr;
    c->nrm_df_blocks = p.nrm_part ? (int)grid : 0;
  }
  if (sh.halves == 1) return launch_digit<FLAGS, 1, false>(p, a, (unsigned)grid, s);
  if (sh.kb == 1) return launch_digit<FLAGS, 1, true>(p, a, (unsigned)grid, s);
  return launch_digit<FLAGS, 2, true>(p, a, (unsigned)grid, s);
}

#define RFNSE_DIGIT(F) template cudaError_t run_digit<F>(rfnse_ctx*, PassParams, int, int, cudaStream_t);
RFNSE_DIGIT(F_INSCALE | F_DST)
RFNSE_DIGIT(F_DST)
RFNSE_DIGIT(F_DST | F_LAM)
RFNSE_DIGIT(F_DST | F_DSCALE)
RFNSE_DIGIT(F_TOEP_X)
RFNSE_DIGIT(F_TOEP_ACC)
RFNSE_DIGIT(F_TOEP_ACC | F_DOT0)

}  // namespace rfnse
