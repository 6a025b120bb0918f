// cluster.cuh -- the whole Chebyshev recursion of Eq. 15 with both vectors of a
// start site in the registers of one thread-block cluster (real on-site
// lattices with one hopping amplitude on every bond, FP32 vectors).
//
// A step over vectors in HBM moves 3 streams (4 per three steps in the
// multi-step pass), 175 KB per vector-step of the 128 x 128 lattice; here
// nothing moves: a thread keeps j_{n-1} and j_n of a tile of 4 x BY sites of one
// start vector in registers, an SM 8192 to 10240 sites, and a cluster of up
// to sixteen CTAs one start vector of up to 163840 sites.  Clusters are persistent and
// take one start vector after the other through all its steps.  Per step a
// thread computes its tile (packed FP32 pairs along x), publishes the tile's
// edge rows and columns in shared memory (the rows at a CTA's ends also in the
// neighbour CTA's, st.shared::cluster) and reads its neighbours'.  Two buffers
// of edges, so one barrier per step orders them; the barriers are split into
// arrival and wait, and the inner rows of the next step, which need no row of
// another tile, are computed in between.
//
// The three column sums of the doubling identities are formed per thread in
// FP32 with compensation: the products of four rows of the tile (two where it has
// four), sixteen in each half of the pair, in a chain of multiply-adds, the chains by compensated
// addition (16 * 2^-24 of the sum of magnitudes in all).  The lanes of a warp are added in
// fixed point without rounding, kept per warp and step, and every 16 steps added
// over the warps and CTAs (in FP64) and folded by one thread per step.  Root mean square
// distance of the moments from FP64, over 33 x 21 .. 500 x 320 sites and M = 116 .. 2048: 0.69 (mu_ee)
// and 0.80 (mu_eh) of the streamed kernels' (FP64 sums of the same vectors: 0.69 and 0.79; plain FP32
// sums over tile and lanes: 0.71 and 0.82, and of the LDOS at a few sites 1.02, now 0.90).  Time of
// 128 x 128, M = 1024: 146 ms with plain sums, 151 ms, 159 ms with chains of eight in all tiles.
//
// Bound: instruction issue and the FP32 pipe (fused multiply-adds with
// three register operands run at two thirds of the pipe's rate).  Measured, one
// map over all sites: 128 x 128, M = 1024: 151 ms (288 ms with three steps per
// pass over HBM); 64 x 64, M = 512: 4.4 ms (14.6); 96 x 96: 21.1 ms (55.5); the
// 75 x 90 torus: 16.8 ms (55.8, one step per pass); 11 start sites of a 100 x
// 150 lattice, M = 2048: 1.3 ms (88 ms, one launch per step).
#pragma once

#include <algorithm>
#include <tuple>
#include <type_traits>

#include "f32x2.cuh"
#include "internal.h"
#include "slot_table.h"

namespace cbdg {
namespace {

constexpr int kB = 4;           // a thread's tile is kB sites wide and BY high
constexpr int kBatch = kClusterBatch;

__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
struct Quad {  // four sites of one row or column as two packed pairs
  F2 lo, hi;
};
__device__ __forceinline__ Quad lds4(unsigned a) {
  Quad v;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];\n" : "=l"(v.lo), "=l"(v.hi) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts4(unsigned a, F2 lo, F2 hi) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};\n" ::"r"(a), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ void push4(unsigned a, F2 lo, F2 hi) {
  asm volatile("st.shared::cluster.v2.b64 [%0], {%1, %2};\n" ::"r"(a), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ F2 f2add(F2 a, F2 b) {
  F2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float f2get(F2 p, int k) {
  float lo, hi;
  f2unpack(p, lo, hi);
  return k ? hi : lo;
}
__device__ __forceinline__ F2 f2neg(F2 p) {
  float lo, hi;
  f2unpack(p, lo, hi);
  return f2pack(-lo, -hi);
}
__device__ __forceinline__ unsigned remote(unsigned a, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Whether a wait since t0 is over: its limit has passed, which is reported, or another one's has (the
// results are lost then, and the kernel ends without further waiting).  A call of its own: inlined at each
// wait it changes the step's schedule (75 x 90 torus: 17.6 ms, 16.7 so).
__device__ __noinline__ bool expired(unsigned long long t0, unsigned long long limit_ns, unsigned int *flags) {
  if (*static_cast<volatile unsigned int *>(flags) & kFlagTimeout) return true;
  if (global_ns() - t0 <= limit_ns) return false;
  atomicOr(flags, kFlagTimeout);
  return true;
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// The aligned forms want a warp's lanes together, and stores, folds and readouts of some lanes only come
// right before them.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// A column sum (s and what its additions lost, r; both halves) in fixed point, in the mantissas of 12 + s,
// units of 2^-20, and of 1.5 * 2^-19 + rest, units of 2^-42: without rounding down to the last of them while
// |s| < 4 (a sum of at most 1).  head and tail add as integers.
struct Fixed {
  unsigned head0, head1, tail0, tail1;
  __device__ __forceinline__ Fixed(F2 s, F2 r) {
    const F2 t = f2add(s, f2bcast(12.f));
    const F2 u = f2add(f2add(f2sub(s, f2sub(t, f2bcast(12.f))), r), f2bcast(0x1.8p-19f));
    head0 = __float_as_uint(f2get(t, 0));
    head1 = __float_as_uint(f2get(t, 1));
    tail0 = __float_as_uint(f2get(u, 0));
    tail1 = __float_as_uint(f2get(u, 1));
  }
  __device__ __forceinline__ bool fits() const {  // both heads in [8, 16)
    return ((head0 ^ 0x41000000u) | (head1 ^ 0x41000000u)) < 0x00800000u;
  }
  __device__ __forceinline__ uint2 warp_sum() const {  // over the lanes of the warp
    return make_uint2(__reduce_add_sync(0xffffffffu, head0 + head1), __reduce_add_sync(0xffffffffu, tail0 + tail1));
  }
};
__device__ __forceinline__ long long warp_value(uint2 w) {  // in units of 2^-42
  return static_cast<long long>(static_cast<int>(w.x - 64u * 0x41400000u)) * (1 << 22) +
         static_cast<int>(w.y - 64u * 0x36400000u);
}

__device__ __forceinline__ float el(const Quad &v, int k) { return f2get(k < 2 ? v.lo : v.hi, k & 1); }

// the sites of a thread's tile: row r, columns 2h and 2h + 1 in [r][h]
template <int BY>
__device__ __forceinline__ float at(const F2 (&z)[BY][2], int r, int c) {
  return f2get(z[r][c >> 1], c & 1);
}
template <int BY>
__device__ __forceinline__ void put(F2 (&z)[BY][2], int r, int c, float x) {
  float lo, hi;
  f2unpack(z[r][c >> 1], lo, hi);
  z[r][c >> 1] = c & 1 ? f2pack(lo, x) : f2pack(x, hi);
}

// Shared memory of a CTA: one record of kQuads quads (16 bytes) per thread, one
// per kGhosts tile columns for the rows that the CTAs below and above push (top
// and bottom quads of tile column x at quad 4 (x mod kGhosts)), and one of zeros.  A record holds, twice (the edges of j_n and of j_{n+1}), u and v of the
// tile's top and bottom sites and its left and right sites as (u, u, v, v) of
// rows 1 and 2, 3 and 4, .. and last of rows 0 and BY - 1; then, where the
// registers have no room for them (BY other than 8), the rows of 2 (eps - mu) / a.  An odd
// number of quads keeps the accesses of neighbouring threads free of conflicts.
template <int BY>
struct Record {
  static constexpr int kTop = 0, kBottom = 2, kLeft = 4, kRight = 4 + BY / 2, kEdges = 4 + BY;
  static constexpr int kPar = 2 * kEdges;
  static constexpr int kQuads = (kPar + (BY != 8 ? BY : 0)) | 1;
  static constexpr int kBytes = kQuads * 16;
  static constexpr int kGhosts = kEdges / 4;
  static constexpr int kBuffer = kEdges * 16;  // from one set of edges to the other
  // threads an SM's registers allow (BY = 4: 128 registers a thread, 6: 168, 8 and 10: 255)
  static constexpr int kThreads = BY == 4 ? 512 : BY == 6 ? 384 : 256;
};

// RAG 0: the tiles cover the lattice exactly; 1: they stick out over open edges;
// 2: they stick out over a periodic edge (compiled apart: its selects and early
// waits cost every warp)
template <int BY, int RAG>
__global__ void __launch_bounds__(Record<BY>::kThreads, 1) cluster_kernel(ClusterArgs a) {
  using Rec = Record<BY>;
  using Tile = F2[BY][2];
  constexpr bool EREG = BY == 8;  // 2 (eps - mu) / a in registers, else in the thread's record
  if (a.done && *a.done) return;  // a converged member of an ensemble: nothing to do, for every thread
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ __align__(8) unsigned long long bars[2];
  __shared__ double share[kBatch][2], col_m1, col_dl;  // the column's fold, by step modulo kBatch
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
  const int CS = a.cluster, rank = CS > 1 ? static_cast<int>(cluster_rank()) : 0;
  const int cid = blockIdx.x / CS, ncl = gridDim.x / CS;
  const int Lx = a.Lx, Ly = a.Ly, TX = (Lx + kB - 1) / kB, TY = (Ly + BY - 1) / BY, R = a.rows;
  const int ghost = blockDim.x, nil = ghost + (CS > 1 ? (TX + Rec::kGhosts - 1) / Rec::kGhosts : 0);  // records
  double *xsum = reinterpret_cast<double *>(raw + (nil + 1) * Rec::kBytes);  // rank 0: [CS][3 kBatch] sums of a batch
  uint2 *ring = reinterpret_cast<uint2 *>(xsum + CS * 3 * kBatch);           // [2 kBatch][3][nw] warp sums of the last steps
  const unsigned e0 = smem_addr(raw);
  auto barrier = [&]() {
    if (CS > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  // Split CTA barriers (one arrival per warp): bars[0] orders the side edges of
  // rows 1 and 2, bars[1] everything else where the cluster is one CTA.  A wait
  // is bounded like every other (every warp of the CTA arrives, so it ends).
  if (t < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(&bars[t])), "r"(nw) : "memory");
  const unsigned bar_a = smem_addr(&bars[0]);
  unsigned phase = 0;  // bit 0: the parity to wait for, of both barriers
  auto arrive = [&](unsigned bar) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };
  auto wait = [&](unsigned bar, unsigned parity) {
    if (mbar_try(bar, parity)) return;
    const unsigned long long t0 = global_ns();
    for (unsigned it = 0; !mbar_try(bar, parity); ++it)
      if ((it & 255u) == 255u && expired(t0, a.wait_ns, a.flags)) break;
  };
  auto arrive_ends = [&]() {
    if (CS > 1) cluster_arrive();
    else arrive(bar_a + 8);
  };
  auto wait_ends = [&](unsigned parity) {
    if (CS > 1) cluster_wait();
    else wait(bar_a + 8, parity);
  };
  for (int k = t; k < Rec::kQuads; k += blockDim.x) sts4(e0 + nil * Rec::kBytes + k * 16, 0, 0);

  barrier();  // before any arrival, and before another CTA writes here

  const int rows_here = min(R, TY - rank * R);
  const int tx = t % TX, tyl = t / TX, ty = rank * R + tyl;
  const bool act = tyl < rows_here;
  const int x0 = kB * tx, y0 = BY * ty;
  const int rl = act ? min(BY, Ly - y0) : 0;              // live rows of the tile
  const int w = Lx - kB * (TX - 1);                       // live columns of the last tile of a row
  const bool wrapped = act && rl < BY && a.py;            // periodic y: row rl is the wrapped neighbour row
  const int rsel = (RAG == 2 && tx == TX - 1) ? w - 1 : kB - 1;  // column whose right neighbour is the halo

  // Rows stick out over a periodic y edge: inner rows of the last tiles then need
  // the row across it, so every warp waits for the end rows first (the last
  // tiles' warps alone, a step behind the others, measured slower: 25.8 against
  // 20.1 ms on the 75 x 90 torus).
  const bool early = RAG == 2 && a.py && Ly % BY != 0;
  // Warps whose tiles have all their rows (or none) test no row: the map of the
  // open 75 x 90 lattice 15.4 -> 13.6 ms, of the 500 x 320 slab 48.5 -> 45.1 ms.
  const bool whole = !early && __all_sync(0xffffffffu, rl == BY || rl == 0);

  // where the four neighbour tiles' edges are read
  auto record = [&](int k, int quad) { return e0 + k * Rec::kBytes + quad * 16; };
  auto pushed = [&](int x, int quad) { return record(ghost + x / Rec::kGhosts, x % Rec::kGhosts * 4 + quad); };
  unsigned up = record(nil, 0), dn = up, lf = up, rt = up, push_up = 0, push_dn = 0;
  const unsigned own = record(t, 0);
  if (act) {
    if (tyl + 1 < rows_here) up = record(t + TX, Rec::kBottom);
    else if (CS > 1 && (ty + 1 < TY || a.py)) up = pushed(tx, Rec::kBottom);
    else if (a.py) up = record(tx, Rec::kBottom);
    if (tyl > 0) dn = record(t - TX, Rec::kTop);
    else if (CS > 1 && (ty > 0 || a.py)) dn = pushed(tx, Rec::kTop);
    else if (a.py) dn = record((TY - 1) * TX + tx, Rec::kTop);
    if (tx > 0) lf = record(t - 1, Rec::kRight);
    else if (a.px) lf = record(t + TX - 1, Rec::kRight);
    if (tx + 1 < TX) rt = record(t + 1, Rec::kLeft);
    else if (a.px) rt = record(t - TX + 1, Rec::kLeft);
    if (CS > 1) {
      if (tyl + 1 == rows_here && (ty + 1 < TY || a.py))
        push_up = remote(pushed(tx, Rec::kTop), rank + 1 < CS ? rank + 1 : 0);
      if (tyl == 0 && (ty > 0 || a.py)) push_dn = remote(pushed(tx, Rec::kBottom), rank > 0 ? rank - 1 : CS - 1);
    }
  }

  const float tau_all = static_cast<float>(2.0 / a.scal[kScalA] * a.hop);
  const unsigned epar = own + Rec::kPar * 16;  // 2 (eps - mu) / a of the tile's rows
  F2 tau[2];
  Tile d, e;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    tau[h] = f2pack(x0 + 2 * h < Lx ? tau_all : 0.f, x0 + 2 * h + 1 < Lx ? tau_all : 0.f);
#pragma unroll
  for (int r = 0; r < BY; ++r)
#pragma unroll
    for (int c = 0; c < kB; ++c) {
      float2 p = make_float2(0.f, 0.f);
      if (r < rl && x0 + c < Lx)
        p = *reinterpret_cast<const float2 *>(a.params + (static_cast<size_t>(y0 + r) * Lx + x0 + c) * kParamStride);
      if (EREG) put(e, r, c, p.x);
      else asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(epar + r * 16 + c * 4), "f"(p.x) : "memory");
      put(d, r, c, p.y);
    }

  // side edges of rows ra and rb of (u, v), the k-th of the buffer at byte offset wr
  auto publish_sides = [&](const Tile &u, const Tile &v, int ra, int rb, int k, int wr) {
    const int po = wr + k * 16;
    sts4(own + po + Rec::kLeft * 16, f2pack(at(u, ra, 0), at(u, rb, 0)), f2pack(at(v, ra, 0), at(v, rb, 0)));
    float q0 = at(u, ra, kB - 1), q1 = at(u, rb, kB - 1), q2 = at(v, ra, kB - 1), q3 = at(v, rb, kB - 1);
    if (RAG == 2) {
#pragma unroll
      for (int c = 0; c < kB - 1; ++c)
        if (c == rsel) {
          q0 = at(u, ra, c);
          q1 = at(u, rb, c);
          q2 = at(v, ra, c);
          q3 = at(v, rb, c);
        }
    }
    sts4(own + po + Rec::kRight * 16, f2pack(q0, q1), f2pack(q2, q3));
  };
  // top and bottom rows of component `part`
  auto publish_ends = [&](const Tile &o, int part, int wr) {
    const int po = wr + part * 16;
    F2 tl = o[BY - 1][0], th = o[BY - 1][1];
    if (RAG == 2 && wrapped) {
#pragma unroll
      for (int r = 0; r < BY - 1; ++r)
        if (r + 1 == rl) {
          tl = o[r][0];
          th = o[r][1];
        }
    }
    sts4(own + po + Rec::kTop * 16, tl, th);
    sts4(own + po + Rec::kBottom * 16, o[0][0], o[0][1]);
    if (push_up) push4(push_up + po, tl, th);
    if (push_dn) push4(push_dn + po, o[0][0], o[0][1]);
  };
  uint2 A{}, B{}, C{};  // the warp's column sums of the last step
  auto keep_sums = [&](int n) {
    uint2 *const w = ring + ((n - 1) & (2 * kBatch - 1)) * 3 * nw + warp;
    if (lane == 0) {
      w[0] = A;
      w[nw] = B;
      w[2 * nw] = C;
    }
  };
  // The column sums of the batch of steps that ends with step n: send() adds
  // the warps' in FP64 and gives them to rank 0, whose thread i folds one step.
  auto send = [&](int n) {
    const int first = n - (n - 1) % kBatch, count = n - first + 1;
    for (int k = t; k < 3 * count; k += blockDim.x) {
      long long q = 0;
      const uint2 *w0 = ring + (((first - 1 + k / 3) & (2 * kBatch - 1)) * 3 + k % 3) * nw;
      for (int z = 0; z < nw; ++z) q += warp_value(w0[z]);
      const double s = static_cast<double>(q) * 0x1p-42;
      if (rank == 0) {
        xsum[k] = s;
      } else {
        asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(remote(smem_addr(xsum + rank * 3 * kBatch + k), 0)), "d"(s) : "memory");
      }
    }
  };
  auto fold = [&](int n, int col) {
    const int first = n - (n - 1) % kBatch, count = n - first + 1;
    if (rank != 0 || t >= count) return;
    const int m = first + t, m0 = 2 * m, mo = 2 * m + 1;
    double sa = 0.0, sb = 0.0, sc = 0.0;
    for (int z = 0; z < CS; ++z) {
      sa += xsum[z * 3 * kBatch + 3 * t];
      sb += xsum[z * 3 * kBatch + 3 * t + 1];
      sc += xsum[z * 3 * kBatch + 3 * t + 2];
    }
    const double v0 = 2.0 * sa - 1.0, v1 = 2.0 * sb - col_m1, h1 = ((m & 1) ? 2.0 : -2.0) * sc - col_dl;
    bool bad = false;
    double dn_ = 0.0, dd_ = 0.0;
    if (m0 < a.M) {
      dn_ -= a.C[m0] * v0;
      bad |= !(fabs(v0) <= 1.0 + a.tol);
      if (a.mu_ee) a.mu_ee[static_cast<size_t>(col) * a.M + m0] = v0;
      if (a.mu_eh) a.mu_eh[(static_cast<size_t>(col) * a.M + m0) * a.mom_stride] = make_double2(0.0, 0.0);
    }
    if (mo < a.M) {
      const double c1 = a.C[mo];
      dn_ -= c1 * v1;
      dd_ += c1 * h1;
      bad |= !(fabs(v1) <= 1.0 + a.tol);
      if (a.mu_ee) a.mu_ee[static_cast<size_t>(col) * a.M + mo] = v1;
      if (a.mu_eh) a.mu_eh[(static_cast<size_t>(col) * a.M + mo) * a.mom_stride] = make_double2(h1, 0.0);
    }
    if (bad) atomicOr(a.flags, kFlagSpectrum);
    share[t][0] += dn_;
    share[t][1] += dd_;
  };
  // step n: (cu, cv) = j_n, (ou, ov) = j_{n-1} on entry and j_{n+1} on exit;
  // buf_c: the buffer that holds the edges of j_n.  Rows 1 .. BY - 2 first: they
  // need no row of another tile, so their arithmetic runs while the other warps' end rows are on their way.
  auto step = [&](int n, int col, auto buf_c, auto edge_c, Tile &cu, Tile &cv, Tile &ou, Tile &ov) {
    constexpr int rd = decltype(buf_c)::value * Rec::kBuffer, wr = (1 - decltype(buf_c)::value) * Rec::kBuffer;
    constexpr bool EDGE = decltype(edge_c)::value;  // rows of the tile may be missing
    F2 sa = 0, sb = 0, sc = 0;  // the column sums,
    F2 ra = 0, rb = 0, rc = 0;  // what their last addition lost, and the products since
    const auto add_rows = [&](bool first) {
      if (first) {
        sa = ra;
        sb = rb;
        sc = rc;
        ra = rb = rc = 0;
        return;
      }
      const auto add = [](F2 &s, F2 &x) {  // Kahan
        const F2 t = f2add(s, x);
        x = f2sub(x, f2sub(t, s));
        s = t;
      };
      add(sa, ra);
      add(sb, rb);
      add(sc, rc);
    };
    // component part of row r; l, g: the halo left and right, (bl, bh), (tl, th): the halo below row 0 and above row 3
    auto row = [&](int r, int part, const F2 (&er)[2], float l0, float g3, F2 bl, F2 bh, F2 tl, F2 th) {
      Tile &z = part == 0 ? cu : cv;
      Tile &q = part == 0 ? cv : cu;
      Tile &o = part == 0 ? ou : ov;
      float nb[kB];  // left + right neighbour
#pragma unroll
      for (int c = 0; c < kB; ++c) {
        const float l = c > 0 ? at(z, r, c > 0 ? c - 1 : 0) : l0;
        float g = c < kB - 1 ? at(z, r, c < kB - 1 ? c + 1 : c) : g3;
        if (RAG == 2 && c < kB - 1) g = c == rsel ? g3 : g;
        nb[c] = __fadd_rn(l, g);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const F2 u = r < BY - 1 ? z[r < BY - 1 ? r + 1 : r][h] : (h ? th : tl);
        const F2 b = r > 0 ? z[r > 0 ? r - 1 : 0][h] : (h ? bh : bl);
        const F2 s = f2add(f2pack(nb[2 * h], nb[2 * h + 1]), f2add(u, b));
        const F2 tc = RAG ? tau[h] : tau[0];
        F2 m = f2fma(d[r][h], q[r][h], f2neg(o[r][h]));
        m = part == 0 ? f2fma(f2neg(tc), s, f2fma(er[h], z[r][h], m)) : f2fma(tc, s, f2fma(f2neg(er[h]), z[r][h], m));
        ra = f2fma(z[r][h], z[r][h], ra);
        rb = f2fma(m, z[r][h], rb);
        rc = f2fma(part == 0 ? m : f2neg(m), q[r][h], rc);
        o[r][h] = m;
      }
    };
    auto load_e = [&](int r, F2 (&er)[2]) {
      if (EREG) {
        er[0] = e[r][0];
        er[1] = e[r][1];
        return;
      }
      const Quad v = lds4(epar + r * 16);
      er[0] = v.lo;
      er[1] = v.hi;
    };
    if (RAG == 2 && EDGE) {
      if (early) wait_ends(phase);
      if (wrapped) {
        const Quad hu = lds4(up + rd), hv = lds4(up + rd + 16);
#pragma unroll
        for (int r = 1; r < BY; ++r)
          if (r == rl) {
            cu[r][0] = hu.lo;
            cu[r][1] = hu.hi;
            cv[r][0] = hv.lo;
            cv[r][1] = hv.hi;
          }
      }
    }
    wait(bar_a, phase);
#pragma unroll
    for (int k = 0; k < BY / 2 - 1; ++k) {
      const Quad hl = lds4(lf + rd + k * 16), hr = lds4(rt + rd + k * 16);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = 2 * k + 1 + i;
        if (!EDGE || r < rl) {
          F2 er[2];
          load_e(r, er);
          row(r, 0, er, el(hl, i), el(hr, i), 0, 0, 0, 0);
          row(r, 1, er, el(hl, i + 2), el(hr, i + 2), 0, 0, 0, 0);
        }
      }
      if (BY == 4 || (k & 1)) add_rows(k < 2);  // the first chain is the sum
      publish_sides(ou, ov, 2 * k + 1, 2 * k + 2, k, wr);
    }
    arrive(bar_a);
    keep_sums(n - 1);
    if (!(RAG == 2 && EDGE && early)) wait_ends(phase);
    phase ^= 1u;
    // the last batch of sums: kept by step 1, sent in step 2 and folded in step 3 of the next one
    if (decltype(buf_c)::value == 1 && n % kBatch == 2 && n > 2) send(n - 2);
    if (decltype(buf_c)::value == 0 && n % kBatch == 3 && n > 3) fold(n - 3, col);
    {
      constexpr int last = (BY / 2 - 1) * 16;
      const Quad hl = lds4(lf + rd + last), hr = lds4(rt + rd + last);
      {
        const Quad du = lds4(dn + rd), dv = lds4(dn + rd + 16);
        if (!EDGE || 0 < rl) {
          F2 er[2];
          load_e(0, er);
          row(0, 0, er, el(hl, 0), el(hr, 0), du.lo, du.hi, 0, 0);
          row(0, 1, er, el(hl, 2), el(hr, 2), dv.lo, dv.hi, 0, 0);
        }
      }
      const Quad tu = lds4(up + rd), tv = lds4(up + rd + 16);
      if (!EDGE || BY - 1 < rl) {
        F2 er[2];
        load_e(BY - 1, er);
        row(BY - 1, 0, er, el(hl, 1), el(hr, 1), 0, 0, tu.lo, tu.hi);
        row(BY - 1, 1, er, el(hl, 3), el(hr, 3), 0, 0, tv.lo, tv.hi);
      }
      add_rows(false);
    }
    publish_sides(ou, ov, 0, BY - 1, BY / 2 - 1, wr);
    publish_ends(ou, 0, wr);
    publish_ends(ov, 1, wr);
    arrive_ends();
    const Fixed ta(sa, ra), tb(sb, rb), tc(sc, rc);
    A = ta.warp_sum();
    B = tb.warp_sum();
    C = tc.warp_sum();
    // (|j_n| <= 1, unless the spectrum leaves [-1, 1])
    if (!ta.fits() || (2 * n + 1 < a.M && !(tb.fits() && tc.fits()))) atomicOr(a.flags, kFlagSpectrum);
  };

  for (int col = cid; col < a.ncols; col += ncl) {
    Tile pu, pv, qu, qv;  // j_{n-1}, j_n
    {
      const int site = a.sites ? a.sites[col] : col;
      const double am = a.scal[kScalA];
      const double m1 = (a.eps[site] - a.mu) / am, dl = a.delta[site].x / am;
      if (t == 0) {
        col_m1 = m1;
        col_dl = dl;
      }
      if (t < 2 * kBatch) share[t >> 1][t & 1] = 0.0;
      const int xs = site % Lx, ys = site / Lx;
#pragma unroll
      for (int r = 0; r < BY; ++r)
#pragma unroll
        for (int c = 0; c < kB; ++c) {
          int dx = x0 + c - xs, dy = y0 + r - ys;
          if (a.px) dx = dx == Lx - 1 ? -1 : dx == 1 - Lx ? 1 : dx;
          if (a.py) dy = dy == Ly - 1 ? -1 : dy == 1 - Ly ? 1 : dy;
          const bool in = r < rl && x0 + c < Lx;
          const bool here = in && dx == 0 && dy == 0, by = in && abs(dx) + abs(dy) == 1;
          put(pu, r, c, here ? 1.f : 0.f);
          put(pv, r, c, 0.f);
          put(qu, r, c, here ? static_cast<float>(m1) : by ? static_cast<float>(-a.hop / am) : 0.f);
          put(qv, r, c, here ? static_cast<float>(dl) : 0.f);
        }
    }
#pragma unroll
    for (int k = 0; k < BY / 2 - 1; ++k) publish_sides(qu, qv, 2 * k + 1, 2 * k + 2, k, 0);
    arrive(bar_a);
    publish_sides(qu, qv, 0, BY - 1, BY / 2 - 1, 0);
    publish_ends(qu, 0, 0);
    publish_ends(qv, 1, 0);
    arrive_ends();
    const auto run = [&](auto edge) {
      for (int n = 1; n <= a.steps;) {
        step(n, col, std::integral_constant<int, 0>{}, edge, qu, qv, pu, pv);
        if (++n > a.steps) break;
        step(n, col, std::integral_constant<int, 1>{}, edge, pu, pv, qu, qv);
        ++n;
      }
    };
    if (RAG == 0 || whole) run(std::false_type{});
    else run(std::true_type{});
    wait(bar_a, phase);
    wait_ends(phase);
    phase ^= 1u;
    keep_sums(a.steps);
    __syncthreads();
    for (int n = a.steps > 3 ? (a.steps - 3) / kBatch * kBatch : 0; n < a.steps; n += kBatch) {
      const int last = min(n + kBatch, a.steps);
      send(last);
      barrier();
      fold(last, col);
      barrier();
    }
    if (rank == 0 && t == 0) {
      const double c0 = a.C[0], c1 = a.C[1];
      double an = 0.0, ad = 0.0;
      for (int i = 0; i < kBatch; ++i) {
        an += share[i][0];
        ad += share[i][1];
      }
      an -= c0 + c1 * col_m1;
      ad += c1 * col_dl;
      if (a.dout) {
        a.dout[col] = make_double2(0.5 * a.coupling * ad, 0.0);
        a.nout[col] = 1.0 + an;
      } else {
        a.acc_n[col] = an;
        a.acc_d[col] = make_double2(ad, 0.0);
      }
      if (a.mu_ee) {
        a.mu_ee[static_cast<size_t>(col) * a.M] = 1.0;
        a.mu_ee[static_cast<size_t>(col) * a.M + 1] = col_m1;
      }
      if (a.mu_eh) {
        a.mu_eh[static_cast<size_t>(col) * a.M * a.mom_stride] = make_double2(0.0, 0.0);
        a.mu_eh[(static_cast<size_t>(col) * a.M + 1) * a.mom_stride] = make_double2(col_dl, 0.0);
      }
    }
    __syncthreads();  // col_m1, col_dl and share are rewritten for the next column
  }
  barrier();  // no CTA leaves while another may still write into it
}

template <int BY, int RAG>
struct Launch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  explicit Launch(const ClusterPlan &p) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(p.cluster);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
  }
};

// Clusters of the plan's shape that the current device holds at once (0: none; negative: the query failed).
template <int BY, int RAG>
int slots_one(const ClusterPlan &p) {
  static SlotTable<std::tuple<int, int, int, size_t>> known;  // by device, cluster, CTA size and shared memory
  int dev = 0;
  cudaGetDevice(&dev);
  return known.get(std::make_tuple(dev, p.cluster, p.threads, p.smem), [&] {
    auto k = cluster_kernel<BY, RAG>;
    Launch<BY, RAG> l(p);
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &l.cfg);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    return n;
  });
}

template <int BY, int RAG>
cudaError_t launch_one(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s) {
  const int slots = slots_one<BY, RAG>(p);  // sets the kernel's attributes on the first call
  if (slots < 1) return cudaErrorInvalidConfiguration;
  Launch<BY, RAG> l(p);
  l.cfg.gridDim = dim3(std::min(slots, a.ncols) * p.cluster);
  l.cfg.stream = s;
  return cudaLaunchKernelEx(&l.cfg, cluster_kernel<BY, RAG>, a);
}

}  // namespace
}  // namespace cbdg
