// green_mma.cu -- the contraction of gf1, G[r][e] = sum_n mom[r][n] W[e][n]
// (complex, FP64 in and out), on the tensor cores.
//
// FP64 units give two multiply-adds a clock and SM, the tensor cores a thousand.
// (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 95 (2012): a matrix product as products of
// exact slices.)  Each operand row is scaled by a power of two and written as a 64-bit fixed-point number,
// eight signed base-256 digits (-128 .. 128) of bf16: x = 2^k sum_i d_i 2^(-7-8i).
// Digits multiply exactly, a K-block of 128 terms adds them exactly in FP32 (of the
// digit pairs (i, j) with the same i + j = d at most 8: 8 * 128 * 2^14 = 2^24), and
// the sums of K-blocks are kept in 64-bit integers: d = 0 .. 3 in one, d = 4 .. 7 in
// another.  What is left out, and all that rounds before the last conversion to FP64, are
// digits beyond the eighth and the pairs with i + j > 7, both of 2^-64 of the largest
// entry of the rows, where an FP64 sum rounds by 2^-54 of the sum so far at every term.
//
// The complex sum is a real one of twice the length: moments (re, im, re, im, ..)
// against two rows an energy, (w.re, -w.im, ..) and (w.im, w.re, ..).
//
// A CTA owns 64 x 64 (rows x 2 energies); eight warps of 32 x 16 keep the eight diagonals d of
// 16 outputs in registers (128) and their integers in shared memory (64 KB).  Digit planes
// come in by cp.async, two stages of 32 terms (64 KB each); the planes of a k-step of 16 are
// read once for its 36 digit pairs.
//
// Bound: the rate of mma.sync, one m16n8k16 in ten cycles of a scheduler (370 TFLOP/s of digit
// products); shared memory is read at a quarter of its rate.
// FP64 kernel (green.cu) -> this one: 16 x 256 rows, 1024 energies, M = 1024: 27.5 -> 3.3 ms;
// 512 x 1 rows, 400 energies: 24.4 -> 0.42 ms; 4 x 64 rows, 128 energies: 1.12 -> 0.41 ms; 1 x 1,
// 200 energies, M = 512: 0.53 -> 0.14 ms.  Largest and mean square error of an output against
// 128-bit sums, relative, 4 x 64 rows, M = 1024: 7.5e-14 and 2.2e-15 -> 3.3e-16 and 4.8e-17.
// Seven digits (28 pairs) take 2.7 ms in place of 3.3, but round like the FP64 kernel.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"

namespace cbdg {
namespace {

constexpr int kDigits = 8;
constexpr int kTile = 64, kStageK = 32, kStages = 2, kFlushK = 128;
constexpr int kPlane = kTile * kStageK * 2;           // bytes of one digit of a tile's stage
constexpr int kStageBytes = 2 * kDigits * kPlane;     // A, then B
constexpr int kContractSmem = kStages * kStageBytes + kTile * kTile * 16;
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;

__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7fffffffffffffffull;
}
// k with |x| < 2^k for every entry of a row, from the largest entry's bits (0 for a row of zeros or
// subnormal numbers); a row that is not finite gets the scale NaN.
__device__ __forceinline__ int row_exponent(unsigned long long bits) {
  const int e = static_cast<int>(bits >> 52);
  return e == 0 || bits >= kInfBits ? 0 : e - 1022;
}
__device__ __forceinline__ double row_scale(unsigned long long bits) {
  return bits >= kInfBits ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(1.0, row_exponent(bits));
}
// The digits of x 2^-k, most significant first.
__device__ __forceinline__ void digits_of(double x, int k, int (&d)[kDigits]) {
  long long v = __double2ll_rn(scalbn(x, 63 - k));
#pragma unroll
  for (int i = kDigits - 1; i > 0; --i) {
    d[i] = static_cast<int>(static_cast<signed char>(v & 0xff));
    v = (v - d[i]) >> 8;
  }
  d[0] = static_cast<int>(v);
}
__device__ __forceinline__ unsigned digit_pair(int lo, int hi) {
  const __nv_bfloat162 p(__int2bfloat16_rn(lo), __int2bfloat16_rn(hi));
  return *reinterpret_cast<const unsigned *>(&p);
}

// Digits of the moments of rows row0 .. row0 + rows - 1 (row = start site * n_t + target):
// planes[i][row - row0][kp], terms 2 n (re) and 2 n + 1 (im).  A block takes 32 rows: first
// their largest entries, then tiles of 32 moments, turned in shared memory.
__global__ void __launch_bounds__(256) moment_digits_kernel(long long row0, int rows, int n_t, int M, int kp,
                                                            size_t plane, const double2 *mom, unsigned *planes,
                                                            double *scale) {
  __shared__ double2 tile[32][33];
  __shared__ unsigned long long peak[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r0 = blockIdx.x * 32;
  auto column = [&](int r) {  // first moment of local row r
    const long long g = row0 + min(r, rows - 1);
    return mom + (g / n_t) * M * n_t + g % n_t;
  };
  const double2 *mine = column(r0 + lane);
  unsigned long long big = 0;
  for (int n = w; n < M; n += 8) {
    const double2 z = mine[static_cast<size_t>(n) * n_t];
    big = max(big, max(abs_bits(z.x), abs_bits(z.y)));
  }
  peak[w][lane] = big;
  __syncthreads();
  if (w == 0) {
    for (int j = 1; j < 8; ++j) big = max(big, peak[j][lane]);
    peak[0][lane] = big;
    if (r0 + lane < rows) scale[r0 + lane] = row_scale(big);
  }
  __syncthreads();
  for (int n0 = 0; n0 < kp / 2; n0 += 32) {
    for (int j = w; j < 32; j += 8)
      tile[j][lane] = n0 + j < M ? mine[static_cast<size_t>(n0 + j) * n_t] : make_double2(0.0, 0.0);
    __syncthreads();
    for (int j = w; j < 32; j += 8) {
      if (r0 + j >= rows) continue;
      const int k = row_exponent(peak[0][j]);
      const double2 z = tile[lane][j];
      int a[kDigits], b[kDigits];
      digits_of(z.x, k, a);
      digits_of(z.y, k, b);
#pragma unroll
      for (int i = 0; i < kDigits; ++i)
        planes[(i * plane + static_cast<size_t>(r0 + j) * kp) / 2 + n0 + lane] = digit_pair(a[i], b[i]);
    }
    __syncthreads();
  }
}

// Digits of the weights of energies e0 + blockIdx.x: rows 2 e (w.re, -w.im, ..) and 2 e + 1 (w.im, w.re, ..).
__global__ void __launch_bounds__(256) weight_digits_kernel(int e0, int M, int kp, size_t plane, const double2 *W,
                                                            unsigned *planes, double *scale) {
  __shared__ unsigned long long peak[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x;
  const double2 *row = W + static_cast<size_t>(e0 + e) * M;
  unsigned long long big = 0;
  for (int n = threadIdx.x; n < M; n += blockDim.x) {
    const double2 z = row[n];
    big = max(big, max(abs_bits(z.x), abs_bits(z.y)));
  }
  for (int o = 16; o > 0; o >>= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
  if (lane == 0) peak[w] = big;
  __syncthreads();
  for (int j = 0; j < 8; ++j) big = max(big, peak[j]);
  if (threadIdx.x == 0) scale[e] = row_scale(big);
  const int k = row_exponent(big);
  for (int n = threadIdx.x; n < kp / 2; n += blockDim.x) {
    const double2 z = n < M ? row[n] : make_double2(0.0, 0.0);
    int a[kDigits], b[kDigits];
    digits_of(z.x, k, a);
    digits_of(z.y, k, b);
#pragma unroll
    for (int i = 0; i < kDigits; ++i) {
      unsigned *p = planes + (i * plane + static_cast<size_t>(2 * e) * kp) / 2 + n;
      p[0] = digit_pair(a[i], -b[i]);
      p[kp / 2] = digit_pair(b[i], a[i]);
    }
  }
}

__device__ __forceinline__ unsigned smem_at(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldmatrix4(unsigned a, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// D[row][e] (row stride ld) of rows x n_e from the digit planes; tiles of energies run fastest, so the
// CTAs that share a tile of moments run together.
__global__ void __launch_bounds__(256, 1) digits_contract_kernel(int rows, int n_e, int kp, const unsigned char *pa,
                                                                 size_t plane_a, const double *scale_a,
                                                                 const unsigned char *pb, size_t plane_b,
                                                                 const double *scale_b, double2 *D, size_t ld) {
  extern __shared__ __align__(128) unsigned char raw[];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int wm = (w >> 2) * 32, wn = (w & 3) * 16;
  const int tiles_n = (2 * n_e + kTile - 1) / kTile;
  const int m0 = blockIdx.x / tiles_n * kTile, n0 = blockIdx.x % tiles_n * kTile;
  const unsigned smem = smem_at(raw);
  // this thread's 16 bytes of every digit's tile (rows past the end repeat the last one)
  const int r = t >> 2, ch = t & 3;
  const unsigned char *ga = pa + (static_cast<size_t>(min(m0 + r, rows - 1)) * kp + ch * 8) * 2;
  const unsigned char *gb = pb + (static_cast<size_t>(min(n0 + r, 2 * n_e - 1)) * kp + ch * 8) * 2;
  const unsigned to = r * 64 + ((ch ^ ((r >> 1) & 3)) << 4);
  const int steps = kp / kStageK;
  auto fetch = [&](int s) {
    if (s < steps) {
      const unsigned base = smem + (s % kStages) * kStageBytes + to;
      const size_t k = static_cast<size_t>(s) * kStageK * 2;
#pragma unroll
      for (int i = 0; i < kDigits; ++i) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(base + i * kPlane),
                     "l"(ga + i * plane_a * 2 + k));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(base + (kDigits + i) * kPlane),
                     "l"(gb + i * plane_b * 2 + k));
      }
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  float acc[kDigits][2][2][4];
  // (head, tail) of output q of this thread: the sums over K-blocks of d = 0 .. 3, in units of 2^-38, and of
  // d = 4 .. 7, in units of 2^-70
  longlong2 *sums = reinterpret_cast<longlong2 *>(raw + kStages * kStageBytes) + t;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        sums[((a * 2 + b) * 4 + c) * 256] = longlong2{0, 0};
#pragma unroll
        for (int d = 0; d < kDigits; ++d) acc[d][a][b][c] = 0.f;
      }
  // fragment addresses in a stage (row, 16-byte chunk swizzled with the row)
  const int ra = wm + (lane & 15), rb = wn + (lane & 7) + ((lane >> 4) << 3);
  const int ca = lane >> 4, cb = (lane >> 3) & 1;
  const unsigned fa = ra * 64, fb = rb * 64, xa = (ra >> 1) & 3, xb = (rb >> 1) & 3;
  for (int s = 0; s < kStages - 1; ++s) fetch(s);
  for (int s = 0; s < steps; ++s) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kStages - 2));
    __syncthreads();
    fetch(s + kStages - 1);
    const unsigned base = smem + (s % kStages) * kStageBytes;
#pragma unroll
    for (int kk = 0; kk < kStageK / 16; ++kk) {
      unsigned b[kDigits][4];
#pragma unroll
      for (int j = 0; j < kDigits; ++j)
        ldmatrix4(base + (kDigits + j) * kPlane + fb + (((kk * 2 + cb) ^ xb) << 4), b[j]);
#pragma unroll
      for (int i = 0; i < kDigits; ++i) {
        unsigned a[2][4];
#pragma unroll
        for (int m = 0; m < 2; ++m)  // (16 rows on, the swizzle is the same)
          ldmatrix4(base + i * kPlane + fa + m * 16 * 64 + (((kk * 2 + ca) ^ xa) << 4), a[m]);
#pragma unroll
        for (int j = 0; j < kDigits - i; ++j)
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n) mma_bf16(acc[i + j][m][n], a[m], b[j][2 * n], b[j][2 * n + 1]);
      }
    }
    if ((s + 1) % (kFlushK / kStageK) == 0) {
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            auto whole = [&](int d) { return static_cast<long long>(__float2int_rn(acc[d][m][n][c])); };
            longlong2 &q = sums[((m * 2 + n) * 4 + c) * 256];
            longlong2 v = q;
            v.x += (whole(0) << 24) + (whole(1) << 16) + (whole(2) << 8) + whole(3);
            v.y += (whole(4) << 24) + (whole(5) << 16) + (whole(6) << 8) + whole(7);
            q = v;
#pragma unroll
            for (int d = 0; d < kDigits; ++d) acc[d][m][n][c] = 0.f;
          }
    }
  }
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = m0 + wm + m * 16 + h * 8 + (lane >> 2);
      if (row >= rows) continue;
      const double sr = scale_a[row];
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const int e = (n0 + wn + n * 8) / 2 + (lane & 3);
        if (e >= n_e) continue;
        const double sc = sr * scale_b[e];
        auto value = [&](int c) {
          const longlong2 v = sums[((m * 2 + n) * 4 + c) * 256];
          return sc * fma(static_cast<double>(v.y), 0x1p-70, static_cast<double>(v.x) * 0x1p-38);
        };
        D[static_cast<size_t>(row) * ld + e] = make_double2(value(2 * h), value(2 * h + 1));
      }
    }
}

// Bytes of the planes of the moments, and of the weights, at a time: half a gigabyte together, but never
// fewer than one tile of 64 rows each (smaller pieces would leave a CTA's tile empty and form the digits of
// the moments again for each of them), so more above M = 131,072, up to 2 GB each at M = 2^20.
constexpr size_t kPlaneBudget = size_t{256} << 20;

struct Chunks {
  int kp, rows, energies;  // terms (padded), rows and energies at a time
  size_t a_bytes, b_bytes, scale_a, scale_b;
};
Chunks chunks_of(long long rows, int M, int n_E) {
  Chunks c;
  c.kp = (2 * M + kFlushK - 1) / kFlushK * kFlushK;
  const size_t row_bytes = static_cast<size_t>(c.kp) * 2 * kDigits;
  const long long fit = std::max<long long>(1, static_cast<long long>(kPlaneBudget / row_bytes) / kTile) * kTile;
  c.rows = static_cast<int>(std::min(rows, fit));
  c.energies = static_cast<int>(std::min<long long>(n_E, fit / 2));
  auto r256 = [](size_t b) { return (b + 255) & ~static_cast<size_t>(255); };
  c.a_bytes = r256(c.rows * row_bytes);
  c.b_bytes = r256(2 * static_cast<size_t>(c.energies) * row_bytes);
  c.scale_a = r256(static_cast<size_t>(c.rows) * 8);
  c.scale_b = r256(static_cast<size_t>(c.energies) * 8);
  return c;
}

}  // namespace

// From M = 64 on (64 x 64 outputs: 75 -> 43 us; at M = 32 the FP64 kernel's 39 us stand against
// 42), to the length at which the 64-bit sums may still hold every digit at its largest; not where the
// digits of the weights outweigh a short sum over few rows (3 rows, 66,000 energies, M = 64: 480 us, 541 here).
bool green_mma_wanted(long long rows, int M, int n_E) {
  return rows > 0 && n_E > 0 && M >= 64 && M <= (1 << 20) && (M >= 128 || rows >= 16 || n_E <= 16384);
}

size_t green_mma_scratch(long long rows, int M, int n_E) {
  const Chunks c = chunks_of(rows, M, n_E);
  return c.a_bytes + c.b_bytes + c.scale_a + c.scale_b;
}

cudaError_t launch_green_mma(int n_sites, int n_t, int M, int n_E, const double2 *mom, const double2 *W, double2 *G,
                             void *scratch, int *launches, cudaStream_t s) {
  const long long all = static_cast<long long>(n_sites) * n_t;
  const Chunks c = chunks_of(all, M, n_E);
  unsigned char *pa = static_cast<unsigned char *>(scratch), *pb = pa + c.a_bytes;
  double *sa = reinterpret_cast<double *>(pb + c.b_bytes);
  double *sb = reinterpret_cast<double *>(pb + c.b_bytes + c.scale_a);
  cudaError_t err = cudaFuncSetAttribute(digits_contract_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kContractSmem);
  if (err != cudaSuccess) return err;
  *launches = 0;
  for (int e0 = 0; e0 < n_E; e0 += c.energies) {
    const int ne = std::min(c.energies, n_E - e0);
    const size_t plane_b = static_cast<size_t>(2 * ne) * c.kp;
    weight_digits_kernel<<<ne, 256, 0, s>>>(e0, M, c.kp, plane_b, W, reinterpret_cast<unsigned *>(pb), sb);
    *launches += 1;
    for (long long r0 = 0; r0 < all; r0 += c.rows) {
      const int rows = static_cast<int>(std::min<long long>(c.rows, all - r0));
      const size_t plane_a = static_cast<size_t>(rows) * c.kp;
      moment_digits_kernel<<<(rows + 31) / 32, 256, 0, s>>>(r0, rows, n_t, M, c.kp, plane_a, mom,
                                                            reinterpret_cast<unsigned *>(pa), sa);
      const unsigned tiles = static_cast<unsigned>((rows + kTile - 1) / kTile) * ((2 * ne + kTile - 1) / kTile);
      digits_contract_kernel<<<tiles, 256, kContractSmem, s>>>(rows, ne, c.kp, pa, plane_a, sa, pb, plane_b,
                                                                       sb, G + r0 * n_E + e0, n_E);
      *launches += 2;
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
  }
  return cudaSuccess;
}

}  // namespace cbdg
