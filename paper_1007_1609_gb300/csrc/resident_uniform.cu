// resident_uniform.cu -- the FP64 recursion of a real on-site lattice with one hopping,
// a column in the shared memory of one CTA (see resident.cu).
//
// FP64 units bound it, two operations a clock and SM, so it is laid out for few of
// them.  With one hopping t the four neighbours enter by their sum, three
// additions, and the sum of the left and the upper neighbour of (x, y) is that of the
// right and the lower one of (x - 1, y + 1): a thread that walks (x, y), (x - 1, y + 1), ..
// forms one new pair sum a site, two additions in place of three: 16 operations a site
// with the six of the column sums, where a fused multiply-add for each neighbour makes
// 18.  An open side gets one more column (row) of zeros, so that every walk is periodic.
// The walks of the (Lx + 1) x (Ly + 1) torus are gcd(Lx', Ly') cycles; a thread
// takes consecutive sites of the cycles laid end to end.
//
// Sites are (u, v) pairs: 48 bytes with j_{n-1}, j_n, e and Delta, so lattices of more than
// 4,000 sites fit (resident.cu stores the four hoppings: 96 bytes, 48 x 48).
//
// Bound: the FP64 units, busy 96 % of the time with the operations above (61 x 45, M = 512, 2,745
// columns: 10 warps x 149 operations x 16 cycles a step and column = 60.2 ms of 62.5; the last of its
// 19 rounds fills nine SMs).  The streamed kernel, 20.7 operations a site and two
// launches a step: 75.5 ms.
#include <algorithm>

#include "internal.h"

namespace cbdg {
namespace {

constexpr int kMaxThreads = 384, kMaxWarps = kMaxThreads / 32;
constexpr int kCheckEvery = 16;  // as resident.cu

struct UniformArgs {
  const double *j0, *j1;  // [ncols][2 N], from init_real at slab width 1
  const double *params;   // [N][kParamStride]
  const double *C, *mu1, *scal;
  const double2 *dA;
  double *acc_n;
  double2 *acc_d;
  double *mu_ee;
  double2 *mu_eh;
  int mom_stride;
  unsigned int *flags;
  double tol, hop;
  int Lx, Ly, X, Y, M, steps, len;  // X, Y: with the zeros beside open sides; len: sites of a thread
};

template <bool LINEAR>
__global__ void __launch_bounds__(kMaxThreads) resident_uniform_kernel(UniformArgs a) {
  const int Lx = a.Lx, Ly = a.Ly, X = a.X, Y = a.Y, XY = X * Y, M = a.M;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2 *prev = reinterpret_cast<double2 *>(smem_raw);  // j_{n-1} -> j_{n+1}, [Y][X]
  double2 *cur = prev + XY;                               // j_n
  double2 *par = cur + XY;                                // (e, Delta)
  double *wt = reinterpret_cast<double *>(par + XY);      // [M] -2 C
  double *wred = wt + M;                                  // [2][3][kMaxWarps]

  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
  const int col = blockIdx.x;
  {
    const double *g0 = a.j0 + static_cast<size_t>(col) * 2 * Lx * Ly, *g1 = a.j1 + static_cast<size_t>(col) * 2 * Lx * Ly;
    for (int k = t; k < XY; k += blockDim.x) {
      const int x = k % X, y = k / X;
      double2 p = make_double2(0.0, 0.0), q = p, r = p;
      if (x < Lx && y < Ly) {
        const int e = 2 * Lx * y + x;
        p = make_double2(g0[e], g0[e + Lx]);
        q = make_double2(g1[e], g1[e + Lx]);
        const double *g = a.params + static_cast<size_t>(y * Lx + x) * kParamStride;
        r = make_double2(g[0], g[1]);
      }
      prev[k] = p;
      cur[k] = q;
      par[k] = r;
    }
    for (int k = t; k < M; k += blockDim.x) wt[k] = -2.0 * a.C[k];
  }
  const double th = 2.0 / a.scal[kScalA] * a.hop;
  // this thread's sites k0 .. k0 + len - 1 of the cycles: site i of cycle c is (c - i mod X, i mod Y)
  const int g = a.len, k0 = t * g, k1 = min(k0 + g, XY);
  int cycle_len = X, gc = Y;
  while (gc) {  // gcd(X, Y)
    const int r = cycle_len % gc;
    cycle_len = gc;
    gc = r;
  }
  cycle_len = XY / cycle_len;
  const int c0 = k0 / cycle_len, i0 = k0 % cycle_len;
  const int xs = ((c0 - i0) % X + X) % X, ys = i0 % Y;

  const bool folder = t == 0;
  double an = 0.0, m1 = 0.0;
  double2 ad = make_double2(0.0, 0.0), da = ad;
  if (folder) {
    an = a.acc_n[col];
    ad = a.acc_d[col];
    m1 = a.mu1[col];
    da = a.dA[col];
  }
  bool bad = false;
  double ln = 0.0, ld = 0.0;  // linear fold: this thread's share of acc_n and Re acc_d
  __syncthreads();

  for (int n = 1; n <= a.steps; ++n) {
    double pa = 0.0, pb = 0.0, pc = 0.0;
    int x = xs, y = ys, c = c0, left_in_cycle = cycle_len - i0;
    double qu = 0.0, qv = 0.0;  // right + lower neighbour of the site
    bool fresh = true;
    for (int k = k0; k < k1; ++k) {
      const int row = y * X, up = y + 1 == Y ? 0 : row + X, xl = x == 0 ? X - 1 : x - 1, at = row + x;
      const double2 z = cur[at], zl = cur[row + xl], zu = cur[up + x], o = prev[at], p = par[at];
      if (fresh) {
        const double2 zr = cur[row + (x + 1 == X ? 0 : x + 1)], zd = cur[(y == 0 ? XY - X : row - X) + x];
        qu = zr.x + zd.x;
        qv = zr.y + zd.y;
        fresh = false;
      }
      const double lu = zl.x + zu.x, lv = zl.y + zu.y;
      const double su = qu + lu, sv = qv + lv;
      const double un = fma(-th, su, fma(p.x, z.x, fma(p.y, z.y, -o.x)));
      const double vn = fma(th, sv, fma(p.y, z.x, fma(-p.x, z.y, -o.y)));
      if (x < Lx && y < Ly) prev[at] = make_double2(un, vn);
      pa = fma(z.x, z.x, fma(z.y, z.y, pa));  // (z is zero beside open sides)
      pb = fma(un, z.x, fma(vn, z.y, pb));
      pc = fma(un, z.y, fma(-vn, z.x, pc));
      qu = lu;
      qv = lv;
      x = xl;
      y = y + 1 == Y ? 0 : y + 1;
      if (--left_in_cycle == 0) {
        left_in_cycle = cycle_len;
        x = ++c;
        y = 0;
        fresh = true;
      }
    }
    const int m0 = 2 * n, mo = 2 * n + 1;
    if (LINEAR) {
      if (m0 < M) ln = fma(wt[m0], pa, ln);
      if (mo < M) {
        ln = fma(wt[mo], pb, ln);
        ld = fma((n & 1) ? -wt[mo] : wt[mo], pc, ld);
      }
    }
    const bool reduce = !LINEAR || n % kCheckEvery == 0 || n == a.steps;
    double *wr = wred + (n & 1) * 3 * kMaxWarps;
    if (reduce) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        pa += __shfl_xor_sync(0xffffffffu, pa, o);
        pb += __shfl_xor_sync(0xffffffffu, pb, o);
        if (!LINEAR) pc += __shfl_xor_sync(0xffffffffu, pc, o);
      }
      if (lane == 0) {
        wr[warp] = pa;
        wr[kMaxWarps + warp] = pb;
        wr[2 * kMaxWarps + warp] = pc;
      }
    }
    __syncthreads();  // j_{n+1} complete; this step's warp sums visible
    if (folder && reduce) {
      double A = 0.0, B = 0.0, Cc = 0.0;
      for (int w = 0; w < nw; ++w) {
        A += wr[w];
        B += wr[kMaxWarps + w];
        Cc += wr[2 * kMaxWarps + w];
      }
      const double e0 = 2.0 * A - 1.0, e1 = 2.0 * B - m1;
      const double sgn = (n & 1) ? 1.0 : -1.0;  // (-1)^(n+1)
      const double2 h1 = make_double2(2.0 * sgn * Cc - da.x, -da.y);
      if (m0 < M) {
        if (!LINEAR) an += 0.5 * wt[m0] * e0;
        bad |= fabs(e0) > 1.0 + a.tol;
        if (a.mu_ee) a.mu_ee[static_cast<size_t>(col) * M + m0] = e0;
        if (a.mu_eh) a.mu_eh[(static_cast<size_t>(col) * M + m0) * a.mom_stride] = make_double2(0.0, 0.0);
      }
      if (mo < M) {
        if (!LINEAR) {
          an += 0.5 * wt[mo] * e1;
          ad.x -= 0.5 * wt[mo] * h1.x;
          ad.y += 0.5 * wt[mo] * h1.y;
        }
        bad |= fabs(e1) > 1.0 + a.tol;
        if (a.mu_ee) a.mu_ee[static_cast<size_t>(col) * M + mo] = e1;
        if (a.mu_eh) a.mu_eh[(static_cast<size_t>(col) * M + mo) * a.mom_stride] = h1;
      }
      if (!(fabs(e0) < 1e300) || !(fabs(e1) < 1e300)) bad = true;  // NaN / inf
    }
    double2 *tmp = prev;
    prev = cur;
    cur = tmp;
  }
  if (LINEAR) {
    __syncthreads();  // the last check's sums have been read before wred is reused
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ln += __shfl_xor_sync(0xffffffffu, ln, o);
      ld += __shfl_xor_sync(0xffffffffu, ld, o);
    }
    if (lane == 0) {
      wred[warp] = ln;
      wred[kMaxWarps + warp] = ld;
    }
    __syncthreads();
    if (folder) {  // the constant terms as in resident.cu
      double sn = 0.0, sd = 0.0, even = 0.0, odd = 0.0;
      for (int w = 0; w < nw; ++w) {
        sn += wred[w];
        sd += wred[kMaxWarps + w];
      }
      for (int n = 1; n <= a.steps; ++n) {
        if (2 * n < M) even -= 0.5 * wt[2 * n];
        if (2 * n + 1 < M) odd -= 0.5 * wt[2 * n + 1];
      }
      an += sn + even + m1 * odd;
      ad.x += sd - da.x * odd;
      ad.y += da.y * odd;
    }
  }
  if (folder) {
    a.acc_n[col] = an;
    a.acc_d[col] = ad;
    if (bad) atomicOr(a.flags, kFlagSpectrum);
  }
}

size_t uniform_smem(int XY, int M) { return static_cast<size_t>(XY) * 48 + static_cast<size_t>(M) * 8 + 6 * kMaxWarps * 8; }

constexpr size_t kMaxSmem = 227 * 1024 - 1024;

// Warp operations of a step: each costs 16 cycles of the SM's FP64 units.
double warp_ops(int XY, int threads) {
  const int len = (XY + threads - 1) / threads;
  return threads / 32 * (16.0 * len + 5.0);
}
// A CTA alone on its SM wants eight warps and a multiple of the four schedulers (61 x 45, M = 512:
// 128 threads 74.0 ms, 160: 66.3, 256: 65.3, 288: 65.6, 320: 62.5, 384: 67.0; 64 x 64, M = 256: 70.9, -,
// 61.2, 72.0, 66.2, 67.1; 512 threads: 64.1 and 64.7); among several the fewest operations win (32 x 32: 4.16 with 128, 4.40 with 256).
int best_threads(int XY, int M, int ncols) {
  const bool alone = uniform_smem(XY, M) > kMaxSmem / 2 || ncols <= 152;
  int best = 0;
  double cost = 0.0;
  for (int th = alone ? 256 : 128; th <= kMaxThreads; th += 32) {
    const int nw = th / 32;
    const double c = warp_ops(XY, th) * (alone ? 1.0 + 0.25 * ((nw + 3) / 4 * 4.0 / nw - 1.0) : 1.0);
    if (best == 0 || c < cost) {
      best = th;
      cost = c;
    }
  }
  return best;
}

}  // namespace

// Always faster than the streamed kernels, which take 15 us a step at least and 20.7 operations a
// site (61 x 45, M = 256: one column 4.2 -> 2.1 ms, 300: 5.8 -> 4.1; all of 56 x 56: 48.6 -> 41.7;
// 60 x 60: 56.6 -> 50.7).  Lattices of 64 x 64 and more stay with the streamed kernels, as the
// header says of CBDG_OPT_RESIDENT, though those that fit would be faster here (64 x 64, M = 256: 77.3 -> 61.2
// ms): their pass has a tile to choose.  Against the general kernel in shared memory (18 operations, no zeros beside the
// lattice; W_general its slab width) by the operations of an SM: 16 x 16 stays there (0.54 ms, 0.62
// here), 32 x 32 periodic does not (4.94 -> 4.16), nor 40 x 40 (12.2 -> 11.6).
bool plan_resident_uniform(int Lx, int Ly, int px, int py, int ncols, int M, int W_general) {
  const int XY = (Lx + !px) * (Ly + !py);
  if (ncols < 1 || Lx * Ly >= 4096 || uniform_smem(XY, M) > kMaxSmem) return false;
  if (!W_general) return true;
  if (ncols <= 152) return false;  // a CTA an SM: 40 x 40, 20 columns: 1.40 ms, 1.44 here
  const int W = W_general;
  const double here = (ncols + 151) / 152 * warp_ops(XY, best_threads(XY, M, ncols));
  const double there = ((ncols + W - 1) / W + 151) / 152 * (18.0 * Lx * Ly * W / 32 + 24.0 * std::min(W, 2));
  return here < 0.95 * there;
}

cudaError_t launch_resident_uniform(int Lx, int Ly, int px, int py, int ncols, int M, int steps, double hop,
                                    const void *j0, const void *j1, const void *params, const double *scal,
                                    const double *C, const double *mu1, const double2 *dA, double *acc_n, double2 *acc_d,
                                    double *mu_ee, double2 *mu_eh, int mom_stride, unsigned int *flags, double tol,
                                    cudaStream_t s) {
  const int X = Lx + !px, Y = Ly + !py, threads = best_threads(X * Y, M, ncols);
  const UniformArgs a{static_cast<const double *>(j0), static_cast<const double *>(j1), static_cast<const double *>(params),
                      C, mu1, scal, dA, acc_n, acc_d, mu_ee, mu_eh, mom_stride, flags, tol, hop,
                      Lx, Ly, X, Y, M, steps, (X * Y + threads - 1) / threads};
  auto k = !mu_ee && !mu_eh ? resident_uniform_kernel<true> : resident_uniform_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kMaxSmem));
  if (e != cudaSuccess) return e;
  k<<<ncols, threads, uniform_smem(X * Y, M), s>>>(a);
  return cudaGetLastError();
}

}  // namespace cbdg
