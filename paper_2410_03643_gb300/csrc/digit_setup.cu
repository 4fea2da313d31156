// Operator tables of the digit passes (digit.cuh): the folded (or stacked) DST-I and Toeplitz matrices of
// an axis, split into balanced base-512 digits and stored chunk by chunk as the shared-memory image that
// the kernel copies.
#include <cuda_fp16.h>
#include <cmath>
#include "digit.cuh"

namespace rfnse {

// Column slot kap (0..128 kb - 1) -> position along the column.  Along x the kernel's threads read
// entries 16 apart (16 threads per line, so that a warp reads consecutive points); along a strided axis
// eight consecutive ones.
__host__ __device__ inline int digit_slot_pos(int kap, bool xax) {
  if (!xax) return kap;
  const int b = kap & ~127, t = kap & 127;
  return b + (t & 7) * 16 + (t >> 3);
}

__global__ void k_digit_table(const double* __restrict__ c, int n, double mu, int toeplitz, int exp, int xax,
                              int kb, int halves, int digits, __half* __restrict__ table) {
  const int K = 128 * kb, N = n + 1;
  const long long total = (long long)halves * K * K;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int kap = (int)(t % K);
    const int row = (int)((t / K) % K);
    const int h = (int)(t / ((long long)K * K));
    const int q = digit_slot_pos(kap, xax != 0);  // position of the column entry
    // the entry as f g (1, or e of rounding error in g): its product is kept to twice FP64 precision
    double f = 0.0, g = 0.0, e = 0.0, fe = 0.0;
    const double root = sqrt(2.0 / N);
    const double root_e = fma(-root, root, 2.0 / N) / (2.0 * root);
    if (halves == 1) {  // stacked lines: block diagonal
      const int jr = row % N + 1, jc = q % N + 1;
      if (row / N == q / N && jr <= n && jc <= n) {
        f = toeplitz ? mu : root;
        fe = toeplitz ? 0.0 : root_e;
        g = toeplitz ? c[jr > jc ? jr - jc : jc - jr] : sinpi((double)((jr * jc) % (2 * N)) / (double)N);
      }
    } else if (toeplitz) {  // even part (h = 0) acts on the sums, odd part on the differences
      const int j = row + 1, i = q + 1;  // 1..N/2
      const double near = c[j > i ? j - i : i - j];
      if (i == N / 2) {
        f = h == 0 ? mu : 0.0;
        g = near;
      } else {
        const double far = h == 0 ? c[N - i - j] : -c[N - i - j];  // |j - (N - i)|, j <= N/2 < N - i
        f = 0.5 * mu;
        g = near + far;
        const double b = g - near;
        e = (near - (g - b)) + (far - b);
      }
    } else {  // odd modes k = 2 row + 1 from the sums, even modes k = 2 row + 2 from the differences
      const int k = 2 * row + 1 + h, i = q + 1;
      if (!(h == 1 && (k > n || i == N / 2))) {
        f = root;
        fe = root_e;
        g = sinpi((double)((long long)k * i % (2 * N)) / (double)N);
      }
    }
    const double a = f * g, ae = fma(f, g, -a) + f * e + fe * g;
    const int nk = K / kDigChunkK;
    const int chunk = kap / kDigChunkK, kin = kap % kDigChunkK, mb = row >> 7, r = row & 127;
    // K-major core matrices: 8 rows x 8 entries, rows of 16 B; 16 row groups, then the next 8 entries
    const size_t off = (size_t)(kin >> 3) * 1024 + (size_t)(r >> 3) * 64 + (size_t)(r & 7) * 8 + (kin & 7);
    auto put = [&](int i, __half d) {
      const size_t ch = (((size_t)h * kb + mb) * digits + i) * nk + chunk;
      table[ch * (kDigChunkBytes / 2) + off] = d;
    };
    if (digits == kDigits32) {  // nearest integer (at most 256), then FP16 remainders, row by row
      auto put32 = [&](int i, __half d) { table[(((size_t)h * digits + i) * 128 + row) * 128 + kap] = d; };
      const double s = ldexp(a, 8 - kDigExpBits - exp);
      const double d0 = rint(s), r1 = (s - d0) * 2048.0;
      const __half d1 = __double2half(r1);
      put32(0, __double2half(d0));
      put32(1, d1);
      put32(2, __double2half((r1 - (double)__half2float(d1)) * 2048.0));
      continue;
    }
    long long v = llrint(ldexp(a, -exp)) + llrint(ldexp(ae, -exp));
    long long bias = 0;
    for (int i = 0; i < kDigits; ++i) bias += 256LL << (9 * i);
    v += bias;
    for (int i = 0; i < kDigits; ++i) {
      const long long u = v >> (9 * (kDigits - 1 - i));
      const int dg = (int)(i == 0 ? u : (u & 511)) - 256;
      put(i, __int2half_rn(dg));
    }
  }
}

void launch_setup_digits(const double* c, int n, double mu, int toeplitz, int exp, bool xax, int digits, void* table,
                         cudaStream_t s) {
  DigitShape sh;
  if (!digit_shape(n, &sh)) return;
  const long long total = (long long)sh.halves * 128 * sh.kb * 128 * sh.kb;
  count_launch();
  k_digit_table<<<(unsigned)((total + 127) / 128), 128, 0, s>>>(c, n, mu, toeplitz, exp, xax ? 1 : 0, sh.kb,
                                                               sh.halves, digits, reinterpret_cast<__half*>(table));
}

// |entry| <= sqrt(2/N), N a power of two: sqrt(2/N) <= 2^ceil((1 - log2 N)/2)
int digit_exp_dst(int n) {
  int l = 0;
  while ((1 << l) < n + 1) ++l;
  const int e = -((l - 1) / 2);  // ceil((1 - l) / 2)
  return e - kDigExpBits;
}

// |entry| <= mu c_0, c_0 = Gamma(alpha + 1) / Gamma(alpha/2 + 1)^2 (every |c_k| <= c_0)
int digit_exp_toeplitz(double alpha, double mu) {
  const double g = std::tgamma(alpha / 2 + 1);
  int e = 0;
  std::frexp(mu * std::tgamma(alpha + 1) / (g * g) * (1.0 + 1e-9), &e);
  return e - kDigExpBits;
}

}  // namespace rfnse
