// adjoint_cluster.cuh -- the adjoint of adjoint.cu with every vector in the
// registers of one thread-block cluster (real on-site lattices with one hopping,
// FP32 vectors; a periodic side a multiple of 4).
//
// A cluster takes one start site at a time through the forward recursion and
// back.  The forward pass leaves every j_n in a scratch of the cluster (32 floats a thread
// and step, written past the caches' working set), the way back fetches them again, each
// thread what it wrote itself: j_{m-2} is on its way while step m forms lam_{m-1} = y_{m-1} +
// 2 H~ lam_m - lam_{m+1} and the gradient sums, which need lam_m and j_{m-1} at a site and at
// its right and upper neighbours.  (Running the recursion backwards between pairs kept every
// 8 steps takes a quarter of the scratch and adds the rounding of the reversed steps: table below.)
//
// The layout is cluster.cuh's with tiles of 4 x 4: a thread holds the four
// vectors (128 registers) and 64 gradient sums of its sites.  The products of a step are
// added first, then to FP32 sums over kFlush steps of one column, those to compensated
// pairs (an FP32 head and the exact rounding errors) in a scratch of the CTA, and the final
// kernel adds the pairs over the clusters in FP64.
//
// Distance of the gradient from FP64, root mean square relative to the streamed adjoint's
// (columns added with compensation, steps in FP64), geometric mean over 24 gradients of 16^2 .. 64^2 sites,
// M = 77 .. 512, in eps, t and Delta, and the time of 64 x 64, M = 512:
//   reversed between pairs every 8 steps, products added one by one:  0.97 1.05 0.93   35.2 ms
//   the same, every sum in FP64:                                      0.92 0.96 0.89
//   stored vectors, products of a step first (this):                  0.91 0.93 0.84   36.5 ms
//   with kFlush 32 or 16 in place of 64:                              0.92 0.94 0.84   3 and 8 ms more
//   stored vectors, every sum in FP64:                                0.86 0.86 0.79
//
// Bound: the FP32 pipe and instruction issue, 24 multiply-adds per site and step
// on the way back and 12 on the way there, beside 69 GB written and as much read (64 x 64, M = 512).
// That call took 101 ms with one launch per step (forward, recomputation and reverse three
// steps per pass, sums in launches of their own).
#pragma once

#include "cluster.cuh"

namespace cbdg {
namespace {

constexpr int kAhead = 4;    // steps that a vector is asked for ahead of its loads
constexpr int kFlush = 64;   // steps between two moves of the sums to the scratch
// A thread's record in shared memory, in quads: twice (double buffer) the edges
// of j and of lam (Record<4>'s eight quads each), then its rows of 2 (eps - mu) / a
// and of 2 Delta / a; odd, as in Record.
constexpr int kAdjField = 8, kAdjBuffer = 16, kAdjPar = 32, kAdjQuads = 41, kAdjGhosts = 2;

using Tile4 = F2[4][2];

// o = 2 H~ z - o of component PART (0 electron, 1 hole) in row r; q: the other component
template <int PART>
__device__ __forceinline__ void stencil_row(const Tile4 &z, const Tile4 &q, Tile4 &o, int r, const F2 (&er)[2],
                                            const F2 (&dr)[2], const F2 (&tau)[2], float l0, float g3, F2 bl, F2 bh,
                                            F2 tl, F2 th) {
  float nb[4];
#pragma unroll
  for (int c = 0; c < 4; ++c)
    nb[c] = __fadd_rn(c > 0 ? at(z, r, c > 0 ? c - 1 : 0) : l0, c < 3 ? at(z, r, c < 3 ? c + 1 : c) : g3);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const F2 u = r < 3 ? z[r < 3 ? r + 1 : r][h] : (h ? th : tl);
    const F2 b = r > 0 ? z[r > 0 ? r - 1 : 0][h] : (h ? bh : bl);
    const F2 s = f2add(f2pack(nb[2 * h], nb[2 * h + 1]), f2add(u, b));
    const F2 m = f2fma(dr[h], q[r][h], f2neg(o[r][h]));
    o[r][h] = PART == 0 ? f2fma(f2neg(tau[h]), s, f2fma(er[h], z[r][h], m))
                        : f2fma(tau[h], s, f2fma(f2neg(er[h]), z[r][h], m));
  }
}

// Sums of row r: g_eps += lu ju - lv jv, g_delta += lu jv + lv ju, and over the bond
// to the right (gx) and upper (gy) neighbour (primed) lv jv' + lv' jv - lu ju' - lu' ju.
struct GradSums {
  Tile4 e, d, y;
  float x[4][4];
};
__device__ __forceinline__ void grad_row(GradSums &g, int r, const Tile4 &lu, const Tile4 &lv, const Tile4 &ju,
                                         const Tile4 &jv, float rlu, float rlv, float rju, float rjv,
                                         const Quad &tlu, const Quad &tlv, const Quad &tju, const Quad &tjv) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const F2 a = lu[r][h], b = lv[r][h], c = ju[r][h], e = jv[r][h];
    g.e[r][h] = f2add(g.e[r][h], f2fma(a, c, f2fma(f2neg(b), e, 0)));
    g.d[r][h] = f2add(g.d[r][h], f2fma(a, e, f2fma(b, c, 0)));
    const F2 a1 = r < 3 ? lu[r < 3 ? r + 1 : r][h] : (h ? tlu.hi : tlu.lo);
    const F2 b1 = r < 3 ? lv[r < 3 ? r + 1 : r][h] : (h ? tlv.hi : tlv.lo);
    const F2 c1 = r < 3 ? ju[r < 3 ? r + 1 : r][h] : (h ? tju.hi : tju.lo);
    const F2 e1 = r < 3 ? jv[r < 3 ? r + 1 : r][h] : (h ? tjv.hi : tjv.lo);
    g.y[r][h] = f2add(g.y[r][h], f2fma(f2neg(a), c1, f2fma(f2neg(a1), c, f2fma(b, e1, f2fma(b1, e, 0)))));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float a = at(lu, r, k), b = at(lv, r, k), c = at(ju, r, k), e = at(jv, r, k);
    const float a1 = k < 3 ? at(lu, r, k < 3 ? k + 1 : k) : rlu, b1 = k < 3 ? at(lv, r, k < 3 ? k + 1 : k) : rlv;
    const float c1 = k < 3 ? at(ju, r, k < 3 ? k + 1 : k) : rju, e1 = k < 3 ? at(jv, r, k < 3 ? k + 1 : k) : rjv;
    g.x[r][k] = __fadd_rn(g.x[r][k], __fmaf_rn(-a, c1, __fmaf_rn(-a1, c, __fmaf_rn(b, e1, __fmul_rn(b1, e)))));
  }
}

// RAG 1: the tiles stick out over open edges (rows and columns of zeros)
template <int RAG>
__global__ void __launch_bounds__(256, 1) adjoint_cluster_kernel(AdjointClusterArgs a) {
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ __align__(8) unsigned long long bars[2];
  const int t = threadIdx.x, lane = t & 31, nw = blockDim.x >> 5;
  const int CS = a.cluster, rank = CS > 1 ? static_cast<int>(cluster_rank()) : 0;
  const int cid = blockIdx.x / CS, ncl = gridDim.x / CS;
  const int Lx = a.Lx, Ly = a.Ly, TX = (Lx + 3) / 4, TY = (Ly + 3) / 4, R = a.rows;
  const int ghost = blockDim.x, nil = ghost + (CS > 1 ? (TX + kAdjGhosts - 1) / kAdjGhosts : 0);
  double *tab = reinterpret_cast<double *>(raw + (nil + 1) * kAdjQuads * 16);  // [M] this column's source values
  const unsigned e0 = smem_addr(raw);
  auto barrier = [&]() {
    if (CS > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  // the split barriers of cluster.cuh
  if (t < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(&bars[t])), "r"(nw) : "memory");
  const unsigned bar_a = smem_addr(&bars[0]);
  unsigned phase = 0;
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
  for (int k = t; k < kAdjQuads; k += blockDim.x) sts4(e0 + nil * kAdjQuads * 16 + k * 16, 0, 0);
  barrier();  // before any arrival, and before another CTA writes here

  const int rows_here = min(R, TY - rank * R);
  const int tx = t % TX, tyl = t / TX, ty = rank * R + tyl;
  const bool act = tyl < rows_here;
  const int x0 = 4 * tx, y0 = 4 * ty;
  const int rl = act ? min(4, Ly - y0) : 0;  // live rows of the tile
  auto record = [&](int k, int quad) { return e0 + (k * kAdjQuads + quad) * 16; };
  auto pushed = [&](int x, int quad) { return record(ghost + x / kAdjGhosts, x % kAdjGhosts * 4 + quad); };
  using Rec = Record<4>;
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
  F2 tau[2];
  {
    const float t2 = static_cast<float>(2.0 / a.scal[kScalA] * a.hop);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      tau[h] = f2pack(!RAG || x0 + 2 * h < Lx ? t2 : 0.f, !RAG || x0 + 2 * h + 1 < Lx ? t2 : 0.f);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float2 p = make_float2(0.f, 0.f);
        if (r < rl && x0 + c < Lx)
          p = *reinterpret_cast<const float2 *>(a.params + (static_cast<size_t>(y0 + r) * Lx + x0 + c) * kParamStride);
        asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(own + (kAdjPar + r) * 16 + c * 4), "f"(p.x) : "memory");
        asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(own + (kAdjPar + 4 + r) * 16 + c * 4), "f"(p.y) : "memory");
      }
  }
  auto params = [&](int r, F2 (&er)[2], F2 (&dr)[2]) {
    const Quad v = lds4(own + (kAdjPar + r) * 16), w = lds4(own + (kAdjPar + 4 + r) * 16);
    er[0] = v.lo;
    er[1] = v.hi;
    dr[0] = w.lo;
    dr[1] = w.hi;
  };
  // side edges of rows ra and rb (the k-th) and end rows of field f, at byte offset wr
  auto publish_sides = [&](const Tile4 &u, const Tile4 &v, int ra, int rb, int k, int f, int wr) {
    const int po = wr + (f * kAdjField + k) * 16;
    sts4(own + po + Rec::kLeft * 16, f2pack(at(u, ra, 0), at(u, rb, 0)), f2pack(at(v, ra, 0), at(v, rb, 0)));
    sts4(own + po + Rec::kRight * 16, f2pack(at(u, ra, 3), at(u, rb, 3)), f2pack(at(v, ra, 3), at(v, rb, 3)));
  };
  auto publish_ends = [&](const Tile4 &u, const Tile4 &v, int f, int wr) {
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      const Tile4 &o = part ? v : u;
      const int po = wr + (f * kAdjField + part) * 16;
      sts4(own + po + Rec::kTop * 16, o[3][0], o[3][1]);
      sts4(own + po + Rec::kBottom * 16, o[0][0], o[0][1]);
      if (push_up) push4(push_up + po, o[3][0], o[3][1]);
      if (push_dn) push4(push_dn + po, o[0][0], o[0][1]);
    }
  };
  auto live = [&](int r) { return !RAG || r < rl; };
  float4 *const ck = a.ck + static_cast<size_t>(blockIdx.x) * (a.M - 1) * 8 * blockDim.x + t;
  float2 *const acc = a.acc + static_cast<size_t>(blockIdx.x) * 64 * blockDim.x + t;

  // forward: (cu, cv) = j_n, (ou, ov) = j_{n-1} -> j_{n+1}
  auto forward = [&](auto buf_c, Tile4 &cu, Tile4 &cv, Tile4 &ou, Tile4 &ov) {
    constexpr int rd = decltype(buf_c)::value * kAdjBuffer * 16, wr = (1 - decltype(buf_c)::value) * kAdjBuffer * 16;
    F2 er[2], dr[2];
    wait(bar_a, phase);
    {
      const Quad hl = lds4(lf + rd), hr = lds4(rt + rd);
#pragma unroll
      for (int r = 1; r < 3; ++r)
        if (live(r)) {
          params(r, er, dr);
          stencil_row<0>(cu, cv, ou, r, er, dr, tau, el(hl, r - 1), el(hr, r - 1), 0, 0, 0, 0);
          stencil_row<1>(cv, cu, ov, r, er, dr, tau, el(hl, r + 1), el(hr, r + 1), 0, 0, 0, 0);
        }
    }
    publish_sides(ou, ov, 1, 2, 0, 0, wr);
    arrive(bar_a);
    wait_ends(phase);
    phase ^= 1u;
    {
      const Quad hl = lds4(lf + rd + 16), hr = lds4(rt + rd + 16);
      if (live(0)) {
        const Quad bu = lds4(dn + rd), bv = lds4(dn + rd + 16);
        params(0, er, dr);
        stencil_row<0>(cu, cv, ou, 0, er, dr, tau, el(hl, 0), el(hr, 0), bu.lo, bu.hi, 0, 0);
        stencil_row<1>(cv, cu, ov, 0, er, dr, tau, el(hl, 2), el(hr, 2), bv.lo, bv.hi, 0, 0);
      }
      if (live(3)) {
        const Quad tu = lds4(up + rd), tv = lds4(up + rd + 16);
        params(3, er, dr);
        stencil_row<0>(cu, cv, ou, 3, er, dr, tau, el(hl, 1), el(hr, 1), 0, 0, tu.lo, tu.hi);
        stencil_row<1>(cv, cu, ov, 3, er, dr, tau, el(hl, 3), el(hr, 3), 0, 0, tv.lo, tv.hi);
      }
    }
    publish_sides(ou, ov, 0, 3, 1, 0, wr);
    publish_ends(ou, ov, 0, wr);
    arrive_ends();
  };
  // j_n to and from the cluster's scratch; a thread reads what it wrote itself
  auto keep = [&](int n, const Tile4 &u, const Tile4 &v) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      __stcs(ck + (static_cast<size_t>(n) * 8 + r) * blockDim.x, make_float4(at(u, r, 0), at(u, r, 1), at(u, r, 2), at(u, r, 3)));
      __stcs(ck + (static_cast<size_t>(n) * 8 + 4 + r) * blockDim.x, make_float4(at(v, r, 0), at(v, r, 1), at(v, r, 2), at(v, r, 3)));
    }
  };
  // (volatile: at the head of the step among its reads of shared memory, not where the result is used: 37.2 ->
  // 36.4 ms)
  auto load_row = [](const float4 *p, F2 (&z)[2]) {
    asm volatile("ld.global.cs.v2.b64 {%0, %1}, [%2];\n" : "=l"(z[0]), "=l"(z[1]) : "l"(p) : "memory");
  };
  // j_n of a warp, 32 lines, into L2: a line a lane (64 x 64, M = 512: 36.4 -> 36.0 ms)
  auto prefetch = [&](int n) {
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(ck + (static_cast<size_t>(n) * 8 + (lane >> 2)) * blockDim.x - lane + (lane & 3) * 8));
  };
  auto fetch = [&](int n, Tile4 &u, Tile4 &v) {
#pragma unroll
    for (int r : {1, 2, 0, 3}) {
      load_row(ck + (static_cast<size_t>(n) * 8 + r) * blockDim.x, u[r]);
      load_row(ck + (static_cast<size_t>(n) * 8 + 4 + r) * blockDim.x, v[r]);
    }
  };

  for (int col = cid; col < a.ncols; col += ncl) {
    const int site = a.sites[col];
    const int xs = site % Lx, ys = site / Lx;
    const bool owner = act && xs / 4 == tx && ys / 4 == ty;  // holds the start site, at (sr, sc) of its tile
    const int sr = ys % 4, sc = xs % 4;
    {
      const double wv = (a.w ? a.w[site] : 1.0) * (a.u ? a.u[site] : 1.0);
      const double *src = a.tab + static_cast<size_t>(a.stride) * col;
      for (int m = t; m < a.M; m += blockDim.x) tab[m] = wv * (a.scale * src[m]);
    }
    // lam_m's source, in double and rounded once, on rows r and r2 of the owner's tile
    auto add_source = [&](int m, int r, int r2, Tile4 &z) {
      if (!owner || (sr != r && sr != r2)) return;
      float v = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        v = sr == r && sc == c ? at(z, r, c) : v;
        v = sr == r2 && sc == c ? at(z, r2, c) : v;
      }
      v = static_cast<float>(static_cast<double>(v) + tab[m]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        put(z, r, c, sr == r && sc == c ? v : at(z, r, c));
        put(z, r2, c, sr == r2 && sc == c ? v : at(z, r2, c));
      }
    };
    Tile4 pu, pv, qu, qv;  // j_{n-1}, j_n, later j_{m-1}, j_{m-2}
    {
      const double am = a.scal[kScalA];
      const float m1 = static_cast<float>((a.eps[site] - a.mu) / am), dl = static_cast<float>(a.delta[site].x / am);
      const float tn = static_cast<float>(-a.hop / am);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          int dx = x0 + c - xs, dy = y0 + r - ys;
          if (a.px) dx = dx == Lx - 1 ? -1 : dx == 1 - Lx ? 1 : dx;
          if (a.py) dy = dy == Ly - 1 ? -1 : dy == 1 - Ly ? 1 : dy;
          const bool in = r < rl && x0 + c < Lx;
          const bool here = in && dx == 0 && dy == 0, by = in && abs(dx) + abs(dy) == 1;
          put(pu, r, c, here ? 1.f : 0.f);
          put(pv, r, c, 0.f);
          put(qu, r, c, here ? m1 : by ? tn : 0.f);
          put(qv, r, c, here ? dl : 0.f);
        }
    }
    publish_sides(qu, qv, 1, 2, 0, 0, 0);
    arrive(bar_a);
    publish_sides(qu, qv, 0, 3, 1, 0, 0);
    publish_ends(qu, qv, 0, 0);
    arrive_ends();
    keep(0, pu, pv);
    if (a.M > 2) keep(1, qu, qv);
    // up to j_{M-2}, the last one that the sums read
    for (int n = 1; n <= a.M - 3;) {
      forward(std::integral_constant<int, 0>{}, qu, qv, pu, pv);
      keep(++n, pu, pv);
      if (n > a.M - 3) break;
      forward(std::integral_constant<int, 1>{}, pu, pv, qu, qv);
      keep(++n, qu, qv);
    }
    if (a.M & 1) {  // (p) = j_{M-2}
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          pu[r][h] = qu[r][h];
          pv[r][h] = qv[r][h];
        }
    }
    wait(bar_a, phase);
    wait_ends(phase);
    phase ^= 1u;
    __syncthreads();  // tab
    // back: (p) = j_{m-1}, (l) = lam_m, (k) = lam_{m+1}, m = M - 1
    Tile4 lu, lv, ku, kv;
    GradSums g;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        lu[r][h] = lv[r][h] = ku[r][h] = kv[r][h] = 0;
        g.e[r][h] = g.d[r][h] = g.y[r][h] = 0;
        g.x[r][2 * h] = g.x[r][2 * h + 1] = 0.f;
      }
    add_source(a.M - 1, 1, 2, a.part ? lv : lu);
    add_source(a.M - 1, 0, 3, a.part ? lv : lu);
    publish_sides(pu, pv, 1, 2, 0, 0, 0);
    publish_sides(lu, lv, 1, 2, 0, 1, 0);
    arrive(bar_a);
    publish_sides(pu, pv, 0, 3, 1, 0, 0);
    publish_sides(lu, lv, 0, 3, 1, 1, 0);
    publish_ends(pu, pv, 0, 0);
    publish_ends(lu, lv, 1, 0);
    arrive_ends();
    // step m: sums of lam_m and (j) = j_{m-1}; (o) = j_{m-2}, (w) = lam_{m+1} -> lam_{m-1} (m > 1)
    auto back = [&](int m, auto buf_c, Tile4 &ju, Tile4 &jv, Tile4 &ou, Tile4 &ov, Tile4 &zu, Tile4 &zv, Tile4 &wu,
                    Tile4 &wv) {
      constexpr int rd = decltype(buf_c)::value * kAdjBuffer * 16, wr = (1 - decltype(buf_c)::value) * kAdjBuffer * 16;
      constexpr int fl = kAdjField * 16;  // lam's edges
      const Quad none{0, 0};
      F2 er[2], dr[2];
      if (m >= 2) fetch(m - 2, ou, ov);  // on its way during the step
      if (m >= 2 + kAhead) prefetch(m - 2 - kAhead);
      wait(bar_a, phase);
      {
        const Quad hr = lds4(rt + rd), ll = lds4(lf + rd + fl), lr = lds4(rt + rd + fl);
#pragma unroll
        for (int r = 1; r < 3; ++r)
          if (live(r)) {
            grad_row(g, r, zu, zv, ju, jv, el(lr, r - 1), el(lr, r + 1), el(hr, r - 1), el(hr, r + 1), none, none, none,
                     none);
            params(r, er, dr);
            stencil_row<0>(zu, zv, wu, r, er, dr, tau, el(ll, r - 1), el(lr, r - 1), 0, 0, 0, 0);
            stencil_row<1>(zv, zu, wv, r, er, dr, tau, el(ll, r + 1), el(lr, r + 1), 0, 0, 0, 0);
          }
      }
      add_source(m - 1, 1, 2, a.part ? wv : wu);
      publish_sides(ou, ov, 1, 2, 0, 0, wr);
      publish_sides(wu, wv, 1, 2, 0, 1, wr);
      arrive(bar_a);
      wait_ends(phase);
      phase ^= 1u;
      {
        const Quad hr = lds4(rt + rd + 16), ll = lds4(lf + rd + fl + 16), lr = lds4(rt + rd + fl + 16);
        if (live(0)) {
          grad_row(g, 0, zu, zv, ju, jv, el(lr, 0), el(lr, 2), el(hr, 0), el(hr, 2), none, none, none, none);
          params(0, er, dr);
          const Quad cu = lds4(dn + rd + fl), cv = lds4(dn + rd + fl + 16);
          stencil_row<0>(zu, zv, wu, 0, er, dr, tau, el(ll, 0), el(lr, 0), cu.lo, cu.hi, 0, 0);
          stencil_row<1>(zv, zu, wv, 0, er, dr, tau, el(ll, 2), el(lr, 2), cv.lo, cv.hi, 0, 0);
        }
        if (live(3)) {
          const Quad tu = lds4(up + rd), tv = lds4(up + rd + 16), su = lds4(up + rd + fl), sv = lds4(up + rd + fl + 16);
          grad_row(g, 3, zu, zv, ju, jv, el(lr, 1), el(lr, 3), el(hr, 1), el(hr, 3), su, sv, tu, tv);
          params(3, er, dr);
          stencil_row<0>(zu, zv, wu, 3, er, dr, tau, el(ll, 1), el(lr, 1), 0, 0, su.lo, su.hi);
          stencil_row<1>(zv, zu, wv, 3, er, dr, tau, el(ll, 3), el(lr, 3), 0, 0, sv.lo, sv.hi);
        }
      }
      add_source(m - 1, 0, 3, a.part ? wv : wu);
      publish_sides(ou, ov, 0, 3, 1, 0, wr);
      publish_sides(wu, wv, 0, 3, 1, 1, wr);
      publish_ends(ou, ov, 0, wr);
      publish_ends(wu, wv, 1, wr);
      arrive_ends();
      // the sums leave every kFlush steps, before the last step and after it: f_m
      // = 2, and 1 for m = 1
      if (m % kFlush == 2 || m == 1) {
        const float f = m == 1 ? 1.f : 2.f;
        auto add = [&](int i, float x) {
          float2 s = acc[static_cast<size_t>(i) * blockDim.x];
          x *= f;
          const float hi = __fadd_rn(s.x, x), bb = __fsub_rn(hi, s.x);
          s.y = __fadd_rn(s.y, __fadd_rn(__fsub_rn(s.x, __fsub_rn(hi, bb)), __fsub_rn(x, bb)));
          s.x = hi;
          acc[static_cast<size_t>(i) * blockDim.x] = s;
        };
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            add(r * 4 + c, at(g.e, r, c));
            add(16 + r * 4 + c, at(g.d, r, c));
            add(32 + r * 4 + c, g.x[r][c]);
            add(48 + r * 4 + c, at(g.y, r, c));
            g.x[r][c] = 0.f;
          }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int h = 0; h < 2; ++h) g.e[r][h] = g.d[r][h] = g.y[r][h] = 0;
      }
    };
    for (int m = a.M - 1; m >= 1;) {
      back(m, std::integral_constant<int, 0>{}, pu, pv, qu, qv, lu, lv, ku, kv);
      if (--m < 1) break;
      back(m, std::integral_constant<int, 1>{}, qu, qv, pu, pv, ku, kv, lu, lv);
      --m;
    }
    wait(bar_a, phase);
    wait_ends(phase);
    phase ^= 1u;
  }
  barrier();  // no CTA leaves while another may still write into it
}

template <int RAG>
int adjoint_slots_one(const ClusterPlan &p) {
  auto k = adjoint_cluster_kernel<RAG>;
  Launch<4, RAG> l(p);
  int n = 0;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &l.cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return n;
}

template <int RAG>
cudaError_t adjoint_launch_one(const AdjointClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  Launch<4, RAG> l(p);
  l.cfg.gridDim = dim3(clusters * p.cluster);
  l.cfg.stream = s;
  return cudaLaunchKernelEx(&l.cfg, adjoint_cluster_kernel<RAG>, a);
}

}  // namespace
}  // namespace cbdg
