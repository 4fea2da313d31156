// FP32 digit passes: the mixed form's transforms of large grids on the tensor cores (see digit.cuh for the
// folding, the stacking and the operator tables).
//
// An entry of a line, scaled by a power of two to |t| <= 256, is x_0 + 2^-11 x_1 + 2^-22 x_2 with x_0 the
// nearest integer and x_1, x_2 the FP16 roundings of what is left, all of an FP32 value's bits; the operator's
// entries likewise.  D_0 = sum a_0 x_0 is an integer below 2^24, exact in FP32; D_1 and D_2 (the products of
// weight 2^-11 and 2^-22) are accumulated in FP32, whose rounding is 2^-11 of D_0's scale down.  So a pass
// rounds like one FP32 operation per result, where an FP32 FFT rounds in every stage.
//
// Bound: an FP32 FFT pass of 255^3 points issues 230 instructions per point (132 us for S, 230 us for T, at
// 57-79% of the issue slots).  A first digit form, one tile of 16 lines per block and the operator (192 KB)
// streamed through shared memory for every tile, was bound by that stream at 60 B per cycle and SM (157 and
// 249 us).  So a block stays on its SM, keeps the operator in TMEM (five of its six digit blocks, the sixth in
// shared memory) and runs its tiles through two roles at once: two groups of warps read lines, split them into
// digits and issue the products (alternate tiles), one group drains the accumulators and does the pointwise work,
// which bounds the passes now.  255^3, us (bytes over time in TB/s) before and after: S 125 -> 72 (3.7), S / (w + i
// Lambda) and S together 230 -> 191, S with the sub-solve and T_x 300 -> 217, T 227 -> 114 (3.5), T with the
// first Gram-Schmidt dot product 203 (3.9).  The pass that also scales and stores the FP64 basis vector stays an
// FFT pass: it is bound by the FP64 products of that (148 us against 156).
#include <cuda_fp16.h>
#include <cmath>
#include "digit.cuh"
#include "tc05.cuh"

namespace rfnse {

namespace {

struct Digit32Args {
  const unsigned char* table;
  int oexp;          // operator entry = (a_0 + 2^-11 a_1 + 2^-22 a_2) 2^oexp
  int log2N, stack;  // log2(n + 1), lines stacked in one column
  long long tiles;   // of 16 lines (columns)
  float lam_scale;   // 1 / dst_scale: lamfac holds i dst_scale / (omega + i Lambda)
  int give_up;       // the block's tile whose results are given up untried (rfnse_test_give_up; none if negative)
  int *err, *loop_err;  // set when a wait gives up: for the host, and for the loop conditions on the device
};

// Warps 0-7 and 8-15 split even and odd tiles of the block, 16-23 finish them; 24 warps leave 80 registers each.
constexpr int kGroup = 256;           // threads of a group
constexpr int kNt = 3 * kGroup;
// The digits of a half are one K-major operand of 96 columns (digit j of column n at 32 j + n: see digit.cu),
// core matrices 144 B (next 8 columns) and 1744 B (next 8 entries) apart: neighbouring lines' and neighbouring
// entries' 16-byte stores both spread over the banks.
constexpr int kSbo = 144, kLbo = kDigits32 * (kDigCols / 8) * kSbo + 16;
constexpr int kHalfBytes = 16 * kLbo;
constexpr int kBufBytes = 2 * kHalfBytes;
constexpr int kPitch = kDigLines * 8 + 8;  // staged results: a position's 16 lines, 8 B each
constexpr int kCtrl = 2048;                // barriers, line exponents and result scales of eight tiles
constexpr int kOperBytes = 128 * 128 * 2;  // one digit block of the operator
// the results of a sine pass are staged half by half, the second 64 B further on (neighbouring positions'
// banks), those of a Toeplitz pass by position
constexpr int kStage = kCtrl + 2 * kBufBytes, kOperS = (kStage + 256 * kPitch + 64 + 127) & ~127;
constexpr int kSmem = kOperS + kOperBytes;
static_assert(kStage % 16 == 0 && kOperS % 128 == 0, "alignment");
// unfolded passes keep their whole operator in TMEM; its place holds the maxima and scales of up to 32 stacked lines
// per column, for eight tiles
constexpr int kStackMax = 32;
static_assert(2 * 8 * kStackMax * kDigLines * 4 <= kOperBytes, "room for the stacked lines' scales");

__device__ __forceinline__ void group_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kGroup) : "memory"); }

// FP32 -> FP64, exact, by integer operations and one FP32 product: a subnormal is scaled to the normal range first, and
// the exponent's offset makes up for it.  (A conversion instruction for the subnormals alone, as df_f2d has, made a
// 255^3 mixed run take 52.7 ms, this one 49.3; with subnormals set to zero by comparisons and branches it was 50.1.)
__device__ __forceinline__ double widen(float v) {
  const uint32_t m = __float_as_uint(v) & 0x7fffffffu;
  const bool small = m < 0x00800000u;
  const uint32_t b = __float_as_uint(v * (small ? 0x1p64f : 1.0f)), t = b & 0x7fffffffu;
  const uint32_t offset = small ? (m ? 0x34000000u : 0u) : m >= 0x7f800000u ? 0x70000000u : 0x38000000u;
  return __hiloint2double((int)(((t >> 3) + offset) | (b & 0x80000000u)), (int)(t << 29));
}
__device__ __forceinline__ void put_c(double2* p, float2 v) { *p = make_double2(widen(v.x), widen(v.y)); }
__device__ __forceinline__ void put_c(float2* p, float2 v) { *p = v; }

__device__ __forceinline__ uint32_t pack(float a, float b) {
  const __half2 r = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ float2 unpack(uint32_t v) { return __half22float2(*reinterpret_cast<const __half2*>(&v)); }

// The digits of two scaled values (|t| <= 256) as FP16 pairs.
__device__ __forceinline__ void split2(float a, float b, uint32_t (&d)[kDigits32]) {
  constexpr float kMagic = 12582912.0f;  // 1.5 2^23: adding it rounds to an integer
  const float a0 = __fsub_rn(__fadd_rn(a, kMagic), kMagic), b0 = __fsub_rn(__fadd_rn(b, kMagic), kMagic);
  const float ra = a - a0, rb = b - b0;
  d[0] = pack(a0, b0);
  d[1] = pack(ra * 0x1p11f, rb * 0x1p11f);
  const float2 u = unpack(d[1]);
  d[2] = pack(fmaf(u.x, -0x1p-11f, ra) * 0x1p22f, fmaf(u.y, -0x1p-11f, rb) * 0x1p22f);
}

template <typename TOUT, typename TACCI, typename TACCO, int FLAGS, bool FOLD>
__global__ void __launch_bounds__(kNt, 1) k_digit32(const PassParams p, const Digit32Args a) {
  constexpr bool TOEP = (FLAGS & (F_TOEP_X | F_TOEP_ACC)) != 0;
  constexpr int HALVES = FOLD ? 2 : 1;
  constexpr uint32_t kACol = FOLD ? 192 : 128;  // TMEM: accumulators below, operator digits (64 columns each) from here
  if (p.skip && *p.skip) return;                // uniform over the launch
  extern __shared__ __align__(128) unsigned char sm[];
  const uint32_t s0 = tc::smem_addr(sm), sdig = s0 + kCtrl;
  const uint32_t b_empty = s0, b_dfull = s0 + 16, b_dfree = s0 + 24;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sm + 48);
  volatile int* s_fail = reinterpret_cast<volatile int*>(sm + 52);
  int* s_tiles = reinterpret_cast<int*>(sm + 56);  // [2]: tiles whose products each group issued
  // of eight tiles: each line's largest magnitude, and the scales of its results; [8][SL], one entry per stacked line
  // (the operator is block diagonal, so the lines of a column need no common scale)
  constexpr int SL = FOLD ? kDigLines : kStackMax * kDigLines;
  unsigned* smax = reinterpret_cast<unsigned*>(sm + (FOLD ? 64 : kOperS));
  float* sout = reinterpret_cast<float*>(sm + (FOLD ? 576 : kOperS + 8 * SL * 4));
  unsigned char* stage = sm + kStage;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int uwarp = __shfl_sync(0xffffffffu, warp, 0);

  // ---- set-up: barriers, TMEM, the operator's digits ---------------------------------------------------------
  if (uwarp == 16) {
    if (lane == 0) {
      for (int i = 0; i < 2; ++i) {
        tc::mbar_init(b_empty + 8 * i, 1);
        tc::mbar_init(b_dfree + 8 * i, kGroup / 32);
      }
      tc::mbar_init(b_dfull, 1);
      tc::mbar_init_fence();
      *s_fail = 0;
    }
    __syncwarp();
    tc::tmem_alloc(tc::smem_addr(s_tmem), 512);
    tc::fence_before();
  }
  for (int i = tid; i < 8 * SL; i += kNt) smax[i] = 0;
  if (FOLD) {  // digit 2 of the differences' half: K-major core matrices in shared memory
    const uint4* src = reinterpret_cast<const uint4*>(a.table + (size_t)5 * kOperBytes);
    for (int i = tid; i < kOperBytes / 16; i += kNt) {
      const int r = i >> 4, kq = i & 15;
      *reinterpret_cast<uint4*>(sm + kOperS + kq * 2048 + (r >> 3) * 128 + (r & 7) * 16) = __ldg(src + i);
    }
    tc::fence_async_smem();
  }
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *s_tmem;
  if (uwarp < 4) {
    const uint4* src = reinterpret_cast<const uint4*>(a.table) + (32 * warp + lane) * 16;
    for (int b = 0; b < (FOLD ? 5 : 3); ++b)
      for (int q = 0; q < 4; ++q) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldg(src + (size_t)b * (kOperBytes / 16) + q * 4 + k);
        tc::tmem_st16(tmem + ((uint32_t)(32 * warp) << 16) + kACol + b * 64 + q * 16, v);
      }
    tc::tmem_st_wait();
    tc::fence_before();
  }
  __syncthreads();
  tc::fence_after();

  // A wait that gives up sets s_fail, and every later one returns at once: the roles run through their tiles without
  // further products or results, and the block ends, once the products in flight are done, reporting the failure.
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (!*s_fail && !tc::mbar_wait(bar, parity, s_fail)) *s_fail = 1;
  };
  auto failed = [&]() { return __shfl_sync(0xffffffffu, *s_fail, 0) != 0; };  // the same in the whole warp
  const bool xax = p.stride == 1;
  const int n = p.n;
  const long long nline = xax ? p.nlines : p.stride;
  const long long lstep = xax ? n : 1, estep = xax ? 1 : p.stride;
  auto tile_base = [&](long long tile, long long& base0, long long& line0) {
    const long long hi = xax ? 0 : tile / p.tiles_inner;
    line0 = (xax ? tile : tile - hi * p.tiles_inner) * (kDigLines * a.stack);
    base0 = xax ? 0 : hi * p.stride * n;
  };
  const float2* in = reinterpret_cast<const float2*>(p.in);
  if (p.gdyn && p.in_dyn_z) in = reinterpret_cast<const float2*>(p.zbase) + (long long)p.gdyn->j * p.ldv;
  [[maybe_unused]] double dot = 0.0;

  if (uwarp < 16) {
    // ---- lines -> digits: eight entries of one line and their mirror images per thread ----------------------
    const int grp = uwarp >> 3, t = tid & (kGroup - 1);
    const int l = xax ? (t >> 4) : (t & 15), kg = xax ? (t & 15) : (t >> 4);
    auto slot_pos = [&](int i) { return xax ? i * 16 + kg : kg * 8 + i; };
    const bool mid = FOLD && 2 * slot_pos(7) == n - 1;  // the thread's last entry is the middle of the line
    unsigned char* dst0 = sm + kCtrl + grp * kBufBytes + kg * kLbo + ((2 * l) >> 3) * kSbo + ((2 * l) & 7) * 16;
    const float2 zero = make_float2(0.0f, 0.0f);
    [[maybe_unused]] int issued = 0;  // tiles whose products this group has issued (its first warp)
    for (int k = grp; (long long)k * gridDim.x + blockIdx.x < a.tiles; k += 2) {
      long long base0, line0;
      tile_base((long long)k * gridDim.x + blockIdx.x, base0, line0);
      float2 va[8];
      [[maybe_unused]] float2 vb[8];
      if constexpr (FOLD) {
        const bool ok = line0 + l < nline;
        const long long g0 = base0 + (line0 + l) * lstep;
        const long long step = (xax ? 16 : 1) * estep;
        const long long ga = g0 + slot_pos(0) * estep, gb = g0 + (long long)(n - 1 - slot_pos(0)) * estep;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          va[i] = ok ? __ldg(in + ga + i * step) : zero;
          vb[i] = ok && !(i == 7 && mid) ? __ldg(in + gb - i * step) : zero;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int q = slot_pos(i);
          const int sl = q >> a.log2N, pos = q - (sl << a.log2N);
          const long long ln = line0 + sl * kDigLines + l;
          const long long g = base0 + ln * lstep + pos * estep;
          va[i] = ln < nline && pos < n ? __ldg(in + g) : zero;
        }
      }
      // the largest magnitude of each line
      unsigned* tmax = smax + (k & 7) * SL + l;
      if constexpr (FOLD) {
        unsigned m = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          m = max(m, max(__float_as_uint(va[i].x) & 0x7fffffffu, __float_as_uint(va[i].y) & 0x7fffffffu));
          m = max(m, max(__float_as_uint(vb[i].x) & 0x7fffffffu, __float_as_uint(vb[i].y) & 0x7fffffffu));
        }
        m = max(m, __shfl_xor_sync(0xffffffffu, m, xax ? 8 : 16));
        if (xax) {
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 4));
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
        }
        if (xax ? (lane & 15) == 0 : lane < 16) atomicMax(tmax, m);
      } else {
        const int width = min(16, 1 << a.log2N);  // along x: neighbouring lanes that hold entries of one stacked line
        unsigned m = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          m = max(m, max(__float_as_uint(va[i].x) & 0x7fffffffu, __float_as_uint(va[i].y) & 0x7fffffffu));
          const int sl = slot_pos(i) >> a.log2N;
          if (i < 7 && slot_pos(i + 1) >> a.log2N == sl) continue;  // uniform over the warp
          if (xax) {
            for (int o = 1; o < width; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            if ((lane & (width - 1)) == 0) atomicMax(tmax + sl * kDigLines, m);
          } else if (a.log2N >= 4) {  // both halves of the warp are on this stacked line
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
            if (lane < 16) atomicMax(tmax + sl * kDigLines, m);
          } else {
            atomicMax(tmax + sl * kDigLines, m);
          }
          m = 0;
        }
      }
      group_sync(1 + grp);
      // the products of this buffer's last tile (k - 2) are done; so is everything that used tile k - 4's
      // exponents, whose place tile k + 4 takes
      if (k >= 2) wait(b_empty + 8 * grp, ((k >> 1) & 1) ^ 1);
      for (int i = t; i < kDigLines * a.stack; i += kGroup) smax[((k + 4) & 7) * SL + i] = 0;
      // scale: sums of two entries below 2^(eb - 125) become at most 256; a line with an infinity or NaN is NaN (folded:
      // through its digits; else through its results' scale, its digits zero, so that its column's other lines stay
      // as they are)
      auto line_scale = [&](unsigned mx, bool first, int sl) {
        const int se = min(133 - max((int)(mx >> 23), 1), 126);
        const bool bad = mx >= 0x7f800000u;
        if (first) sout[(k & 7) * SL + sl * kDigLines + l] = !FOLD && bad ? __uint_as_float(0x7fc00000u) : ldexpf(1.0f, a.oexp - se);
        return FOLD && bad ? __uint_as_float(0x7fc00000u) : __uint_as_float((unsigned)(se + 127) << 23);
      };
      [[maybe_unused]] float f = 0.0f;
      if constexpr (FOLD) {
        f = line_scale(*tmax, kg == 0, 0);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int q = slot_pos(i), sl = q >> a.log2N;
          const unsigned mx = tmax[sl * kDigLines];
          const float fi = line_scale(mx, q == sl << a.log2N, sl);
          va[i] = mx >= 0x7f800000u ? zero : make_float2(va[i].x * fi, va[i].y * fi);
        }
      }
#pragma unroll
      for (int h = 0; h < HALVES; ++h)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t w[kDigits32][4];
#pragma unroll
          for (int i = 0; i < 8; i += 2) {
            float y[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              y[q] = c ? va[i + q].y : va[i + q].x;
              if constexpr (FOLD) {
                const float u = c ? vb[i + q].y : vb[i + q].x;
                y[q] = h == 0 ? y[q] + u : y[q] - u;
                if (i + q == 7 && h == 1 && mid) y[q] = 0.0f;
              }
            }
            uint32_t d[kDigits32];
            if constexpr (FOLD) split2(y[0] * f, y[1] * f, d);
            else split2(y[0], y[1], d);
#pragma unroll
            for (int j = 0; j < kDigits32; ++j) w[j][i >> 1] = d[j];
          }
#pragma unroll
          for (int j = 0; j < kDigits32; ++j)
            *reinterpret_cast<uint4*>(dst0 + h * kHalfBytes + j * (kDigCols / 8) * kSbo + c * 16) =
                make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
        }
      tc::fence_async_smem();
      group_sync(1 + grp);
      if ((uwarp & 7) == 0) {
        // products: per 16 entries three MMAs of a half, a_i times x_0 .. x_{2-i} into D_i .. D_2
        // the accumulators of tile k - 1 (the other group's) have been drained; a barrier per group, so that its
        // phase is known: this group's last products, of tile k - 2, waited for tile k - 3
        if (k >= 1) wait(b_dfree + 8 * (grp ^ 1), ((k - 1) >> 1) & 1);
        tc::fence_after();
        __syncwarp();
        const bool live = !failed();
        const bool one = tc::elect_one() && live;
        const uint32_t ud = __shfl_sync(0xffffffffu, tmem, 0);
        const uint64_t db0 = tc::smem_desc(__shfl_sync(0xffffffffu, sdig + grp * kBufBytes, 0), kLbo, kSbo);
        const uint64_t da0 = tc::smem_desc(__shfl_sync(0xffffffffu, s0 + kOperS, 0), 2048, 128);
#pragma unroll
        for (int h = 0; h < HALVES; ++h)
#pragma unroll
          for (int i = 0; i < kDigits32; ++i) {
            const uint32_t id = tc::idesc_f16(128, kDigCols * (kDigits32 - i));
            const uint32_t d = ud + (h * kDigits32 + i) * kDigCols;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const uint64_t db = db0 + (uint32_t)((h * kHalfBytes + ks * 2 * kLbo) >> 4);
              const bool acc = !(i == 0 && ks == 0);
              if (h * kDigits32 + i < 5) {
                if (one) tc::mma_f16_ts(d, ud + kACol + (h * kDigits32 + i) * 64 + ks * 8, db, id, acc);
              } else {
                if (one) tc::mma_f16(d, da0 + (uint32_t)((ks * 4096) >> 4), db, id, acc);
              }
            }
          }
        if (one) tc::mma_commit(b_empty + 8 * grp);
        if (one) tc::mma_commit(b_dfull);
        issued += live;
        __syncwarp();
      }
    }
    if ((uwarp & 7) == 0) {  // nothing of this block's is in flight when it ends
      if (issued) tc::mbar_wait(b_empty + 8 * grp, (issued - 1) & 1);
      if (lane == 0) s_tiles[grp] = issued;
    }
  } else {
    // ---- accumulators -> results, staged by position, then the pass's pointwise work in grid order ---------------
    const int t = tid - 2 * kGroup, wq = uwarp & 3, cg = (uwarp - 16) >> 2;
    [[maybe_unused]] TOUT* out = reinterpret_cast<TOUT*>(p.out);
    if constexpr ((FLAGS & F_DSCALE) != 0) {
      if (p.gdyn && p.zbase) out = reinterpret_cast<TOUT*>(p.zbase) + (long long)p.gdyn->j * p.ldv;
    }
    constexpr int ROWS = FOLD ? 256 : 128;
    constexpr int ITEMS = ROWS * kDigLines / kGroup;
    constexpr int B = (FLAGS & F_DOT0) ? 4 : 8;  // items of a thread handled at a time
    const int r0 = xax ? (t & (ROWS - 1)) : (t >> 4), ln0 = xax ? t / ROWS : (t & 15);
    for (int k = 0; (long long)k * gridDim.x + blockIdx.x < a.tiles; ++k) {
      long long base0, line0;
      tile_base((long long)k * gridDim.x + blockIdx.x, base0, line0);
      const long long ga = base0 + (line0 + ln0) * lstep + r0 * estep;
      const long long dg = xax ? (kGroup / ROWS) * lstep : (kGroup / 16) * estep;
      auto element = [&](int it, int& at, long long& g) -> bool {  // item it: where it is staged, its grid index
        const int r = xax ? r0 : r0 + it * (kGroup / 16), ln = xax ? ln0 + it * (kGroup / ROWS) : ln0;
        int pos = r;
        long long line = line0 + ln;
        g = ga + it * dg;
        if constexpr (!FOLD) {
          const int sl = r >> a.log2N;
          pos = r - (sl << a.log2N);
          line += sl * kDigLines;
          g = base0 + line * lstep + pos * estep;
        }
        at = FOLD && !TOEP ? (r >> 1) * kPitch + (r & 1) * (128 * kPitch + 64) + ln * 8 : r * kPitch + ln * 8;
        return line < nline && pos < n;
      };
      [[maybe_unused]] float2 op[B];  // lamfac, dfac, z or the FP32 accumulator
      [[maybe_unused]] float Dv[B];
      [[maybe_unused]] double2 v0[B];
      auto fetch = [&](int it0) {
#pragma unroll
        for (int q = 0; q < B; ++q) {
          int at;
          long long g;
          const bool ok = element(it0 + q, at, g);
          op[q] = make_float2(0.0f, 0.0f);
          Dv[q] = 0.0f;
          if constexpr ((FLAGS & F_LAM) != 0) {
            if (ok) op[q] = __ldg(reinterpret_cast<const float2*>(p.lamfac) + g);
          }
          if constexpr ((FLAGS & F_DSCALE) != 0) {
            if (ok) op[q] = __ldg(reinterpret_cast<const float2*>(p.dfac) + g);
          }
          if constexpr ((FLAGS & F_TOEP_X) != 0) {
            if (ok) op[q] = __ldg(in + g);
            if (ok && p.Dr) Dv[q] = __ldg(reinterpret_cast<const float*>(p.Dr) + g);
          }
          if constexpr ((FLAGS & F_TOEP_ACC) != 0) {
            if (ok) op[q] = reinterpret_cast<const float2*>(p.acc_in)[g];
          }
          if constexpr ((FLAGS & F_DOT0) != 0) v0[q] = ok ? __ldg(p.dot_v0 + g) : make_double2(0.0, 0.0);
        }
      };
      fetch(0);  // the first eight items' operands arrive while the products run
      if (k == a.give_up) *s_fail = 1;
      wait(b_dfull, k & 1);
      tc::fence_after();
      __syncwarp();
      const bool live = !failed();
      if (k) group_sync(3);  // the staged results of the tile before have been read
      if (live) {
        const int row = 32 * wq + lane;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c0 = cg * 16 + b * 4;
          const uint32_t ta = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)c0;
          float D[HALVES * kDigits32][4], v[HALVES][4];
#pragma unroll
          for (int d = 0; d < HALVES * kDigits32; ++d) tc::tmem_ld(ta + d * kDigCols, D[d]);
          tc::tmem_ld_wait(D);
#pragma unroll
          for (int h = 0; h < HALVES; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              v[h][i] = fmaf(fmaf(D[3 * h + 2][i], 0x1p-11f, D[3 * h + 1][i]), 0x1p-11f, D[3 * h][i]);
#pragma unroll
          for (int i = 0; i < 4; i += 2) {
            const int ln = (c0 + i) >> 1;
            const float f = sout[(k & 7) * SL + (FOLD ? 0 : (row >> a.log2N) * kDigLines) + ln];
            unsigned char* st = stage + ln * 8;
            if constexpr (FOLD && TOEP) {  // y_j = e_j + o_j, y_{N-j} = e_j - o_j
              *reinterpret_cast<float2*>(st + row * kPitch) =
                  make_float2((v[0][i] + v[HALVES - 1][i]) * f, (v[0][i + 1] + v[HALVES - 1][i + 1]) * f);
              if (2 * row != n - 1)
                *reinterpret_cast<float2*>(st + (n - 1 - row) * kPitch) =
                    make_float2((v[0][i] - v[HALVES - 1][i]) * f, (v[0][i + 1] - v[HALVES - 1][i + 1]) * f);
            } else {
#pragma unroll
              for (int h = 0; h < HALVES; ++h)
                *reinterpret_cast<float2*>(st + row * kPitch + h * (128 * kPitch + 64)) =
                    make_float2(v[h][i] * f, v[h][i + 1] * f);
            }
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(b_dfree + 8 * (k & 1));
      }
      group_sync(3);
      if (!live) continue;
#pragma unroll
      for (int it0 = 0; it0 < ITEMS; it0 += B) {
        if (it0) fetch(it0);
#pragma unroll
        for (int q = 0; q < B; ++q) {
          int at;
          long long g;
          if (!element(it0 + q, at, g)) continue;
          float2 y = *reinterpret_cast<const float2*>(stage + at);
          if constexpr ((FLAGS & F_LAM) != 0) {
            y = cmul(y, op[q]);
            y = make_float2(y.y * a.lam_scale, -y.x * a.lam_scale);
          }
          if constexpr ((FLAGS & F_DSCALE) != 0) y = cmul(y, op[q]);
          if constexpr ((FLAGS & F_DST) != 0) put_c(out + g, y);
          if constexpr (TOEP) {
            float2 acc = op[q];
            if constexpr ((FLAGS & F_TOEP_X) != 0) {
              y = csub(y, cscale(op[q], Dv[q]));
              acc = cmul(p.ca_f, op[q]);
              if (p.acc_in) acc = cadd(acc, to_c<float>(reinterpret_cast<const TACCI*>(p.acc_in)[g]));
            }
            acc = cadd(acc, cmul(p.cb_f, y));
            put_c(reinterpret_cast<TACCO*>(p.acc_out) + g, acc);
            if constexpr ((FLAGS & F_DOT0) != 0) {
              dot = fma(v0[q].x, widen(acc.x), dot);
              dot = fma(v0[q].y, widen(acc.y), dot);
            }
          }
        }
      }
    }
  }
  __syncthreads();
  if (uwarp == 16) {
    const int tiles = s_tiles[0] + s_tiles[1];  // products are issued tile after tile, each when the one before is drained
    if (tiles) tc::mbar_wait(b_dfull, (tiles - 1) & 1);
    tc::fence_after();
    tc::tmem_free(tmem, 512);
    if (lane == 0 && *s_fail) {
      *(volatile int*)a.err = 1;
      *(volatile int*)a.loop_err = 1;
    }
  }
  if constexpr ((FLAGS & F_DOT0) != 0) block_sum_store(dot, p.dot_part + blockIdx.x);
}

template <typename TOUT, typename TACCI, typename TACCO, int FLAGS, bool FOLD>
cudaError_t launch32(const PassParams& p, const Digit32Args& a, unsigned grid, cudaStream_t s) {
  auto kern = k_digit32<TOUT, TACCI, TACCO, FLAGS, FOLD>;
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (attr != cudaSuccess) return attr;
  count_launch();
  kern<<<grid, kNt, kSmem, s>>>(p, a);
  return cudaGetLastError();
}

}  // namespace

bool digit32_possible(const rfnse_ctx* c, int axis) { return c->digS32[axis] != nullptr; }

template <typename TOUT, typename TACCI, typename TACCO, int FLAGS>
cudaError_t run_digit32(rfnse_ctx* c, PassParams p, int axis, int half, cudaStream_t s) {
  constexpr bool TOEP = (FLAGS & (F_TOEP_X | F_TOEP_ACC)) != 0;
  DigitShape sh;
  if (!digit32_possible(c, axis) || !digit_shape(p.n, &sh) || sh.kb != 1) return cudaErrorInvalidValue;
  Digit32Args a{};
  a.table = static_cast<const unsigned char*>(TOEP ? c->digT32[axis] : c->digS32[axis]);
  a.oexp = (TOEP ? c->digT_exp[axis] - (half ? 1 : 0) : digit_exp_dst(p.n)) + kDigExpBits - 8;
  a.log2N = p.log2L - 1;
  a.stack = sh.stack;
  a.lam_scale = (float)(1.0 / p.dst_scale);
  a.give_up = c->give_up_at;
  a.err = &c->peek[2].err;  // pinned
  a.loop_err = &c->gs->err;
  p.ca_f = make_float2((float)p.ca.x, (float)p.ca.y);
  p.cb_f = make_float2((float)p.cb.x, (float)p.cb.y);
  const long long per = (long long)kDigLines * sh.stack;
  long long grid;
  if (p.stride == 1) {
    p.tiles_inner = 1;
    grid = (p.nlines + per - 1) / per;
  } else {
    p.tiles_inner = (p.stride + per - 1) / per;
    grid = p.tiles_inner * (p.nlines / p.stride);
  }
  if (grid <= 0) return cudaSuccess;
  a.tiles = grid;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (grid > sms) grid = sms;  // one block per SM, each over its share of the tiles
  if (FLAGS & F_DOT0) c->dot0_blocks = (int)grid;
  if (sh.halves == 2) return launch32<TOUT, TACCI, TACCO, FLAGS, true>(p, a, (unsigned)grid, s);
  return launch32<TOUT, TACCI, TACCO, FLAGS, false>(p, a, (unsigned)grid, s);
}

#define RFNSE_DIGIT32(TO, TAI, TAO, F) \
  template cudaError_t run_digit32<TO, TAI, TAO, F>(rfnse_ctx*, PassParams, int, int, cudaStream_t);
RFNSE_DIGIT32(float2, double2, double2, F_DST)
RFNSE_DIGIT32(float2, double2, double2, F_DST | F_LAM)
RFNSE_DIGIT32(float2, double2, float2, F_DST | F_DSCALE)
RFNSE_DIGIT32(float2, double2, float2, F_TOEP_X)
RFNSE_DIGIT32(float2, float2, float2, F_TOEP_ACC)
RFNSE_DIGIT32(float2, float2, double2, F_TOEP_ACC)
RFNSE_DIGIT32(float2, float2, double2, F_TOEP_ACC | F_DOT0)

}  // namespace rfnse
