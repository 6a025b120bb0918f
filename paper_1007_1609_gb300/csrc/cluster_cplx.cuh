// cluster_cplx.cuh -- the direct recursion of Eq. 15 for general lattices
// (complex hoppings, next-nearest neighbours, on-site or bond pairing; complex64
// vectors) with both vectors of two start sites in the registers of one
// thread-block cluster.
//
// As in cluster.cuh a cluster takes its start sites through all steps and
// nothing but the moments asked for leaves the chip.  A thread holds a tile of 4 x 2
// sites of one start vector (64 registers), the two halves of a CTA the two start
// vectors of a pair of columns.  An element is a packed pair (re, im), and a
// coefficient c acts by A += (c.re, c.re) z, S += (c.im, c.im) z as in
// cplx_stencil.cuh.  Every site of j_n is published in shared memory (u and v in
// one 16-byte quad), so a thread reads the ring around its tile and a readout any
// site; the coefficients stay in shared memory (forward hoppings and bonds, four
// quads a site, the backward ones read at the neighbours) and serve both halves.
// Shared memory holds about 1500 sites an SM.  One barrier a step; what is read of
// j_n is loaded before it and folded in FP64 behind it.
//
// Bound: shared memory.  A tile takes 68 quads a step (52 of coefficients, 16 of the
// ring) with eight hoppings and bond pairing, 272 wavefronts of its warp: at 64 x 64
// (four CTAs, eight warps an SM) 2,500 of a step's 3,560 cycles, the packed
// multiply-adds 1,600; the rest is the chain load - multiply-add - store - barrier,
// which two warps a scheduler do not hide.  A store holds back the loads after it, so
// CTAs of up to 256 threads, which may use 255 registers each, publish a tile when all of
// it is formed (currents below: 63.8 -> 54.0 ms); wider ones spill that way and
// publish each column of sites (33.4 ms for the vortex lattice when two are held).
// Both start vectors in one thread read the coefficients once for two (50 quads a
// vector) but leave one warp a scheduler: 75.3 ms for the currents.
// Streamed kernel -> this one: d-wave vortex lattices, 96 x 96, 512 start sites,
// M = 1024: 59.8 -> 32.4 ms; bond currents of 64 x 64, M = 512: 75.1 -> 52.5 ms;
// Green's functions of 128 x 128, 16 x 256 sites, M = 1024: 17.0 -> 9.8 ms (3.4 of them the
// contraction with the energies).  The sums are those of the streamed kernels in
// their order: the same moments bit for bit.  (Starting from e u - u_old instead of
// u_old takes six registers fewer a site and 6 % less time, but rounds differently:
// 7.7e-7 from 64 bits instead of 7.1e-7 for the Green's functions.)
#pragma once

#include "cluster.cuh"

namespace cbdg {
namespace {

constexpr int kCx = 4, kCy = 2;               // sites of a tile
constexpr int kCols = 2;                      // start vectors of a cluster at a time
constexpr int kCxSet = kCx * kCy * kCols;     // quads of one set of published sites
constexpr int kCxRec = 2 * kCxSet + 1;        // quads of a tile's record (two sets; odd, as in Record)
constexpr int kCxChunk = 32;                  // coefficients C_m staged at a time
constexpr int kCxNarrow = 256;                // threads up to which a CTA may use 255 registers each
constexpr int kCxPlaces = 512;                // targets (of all start vectors) whose place is kept

// As expired() of cluster.cuh, inline and without its look at the flags (the caller keeps that it gave up;
// bond currents of 64 x 64: 54.3 -> 52.5 ms).
__device__ __forceinline__ bool expired_here(unsigned long long t0, unsigned long long limit_ns, unsigned int *flags) {
  if (global_ns() - t0 <= limit_ns) return false;
  atomicOr(flags, kFlagTimeout);
  return true;
}
__device__ __forceinline__ F2 pairs(float x) { return f2pack(x, x); }

// Coefficients of a site as read: a complex value in each half of a quad.
struct Coef {
  float r0, i0, r1, i1;
};
__device__ __forceinline__ Coef ldc(unsigned a) {
  Coef v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.r0), "=f"(v.i0), "=f"(v.r1), "=f"(v.i1) : "r"(a));
  return v;
}

// Running sums of a site's update, those of cplx_stencil.cuh's packed form in its order (the
// streamed kernels' moments bit for bit):
//   u' = P_u - N_u, N_u = u_old + sum t_d z_d.u;  v' = P_v - (e v + v_old).
struct Update {
  F2 pua, pus, nua, nus, pva, pvs;
  __device__ __forceinline__ Update(bool bond, const Coef &s, const Quad &z, F2 u_old) {  // s: e, Delta
    pua = f2fma(pairs(s.r0), z.lo, 0);
    pus = pva = pvs = nus = 0;
    nua = u_old;
    if (!bond) {
      const F2 r = pairs(s.r1), i = pairs(s.i1);
      pua = f2fma(r, z.hi, pua);
      pus = f2fma(i, z.hi, 0);
      pva = f2fma(r, z.lo, 0);
      pvs = f2fma(i, z.lo, 0);
    }
  }
  // hopping t to a neighbour z: u' -= t z.u, v' += conj(t) z.v
  __device__ __forceinline__ void hop(float re, float im, const Quad &z) {
    const F2 r = pairs(re), i = pairs(im);
    nua = f2fma(r, z.lo, nua);
    nus = f2fma(i, z.lo, nus);
    pva = f2fma(r, z.hi, pva);
    pvs = f2fma(i, z.hi, pvs);
  }
  // pairing b with a neighbour z: u' += b z.v, v' += conj(b) z.u
  __device__ __forceinline__ void pair(float re, float im, const Quad &z) {
    const F2 r = pairs(re), i = pairs(im);
    pua = f2fma(r, z.hi, pua);
    pus = f2fma(i, z.hi, pus);
    pva = f2fma(r, z.lo, pva);
    pvs = f2fma(i, z.lo, pvs);
  }
  __device__ __forceinline__ void finish(float e, const Quad &z, F2 &u, F2 &v) const {
    float ax, ay, sx, sy;
    f2unpack(f2sub(pua, nua), ax, ay);
    f2unpack(f2sub(pus, nus), sx, sy);
    u = f2pack(__fsub_rn(ax, sy), __fadd_rn(ay, sx));
    f2unpack(f2sub(pva, f2fma(pairs(e), z.hi, v)), ax, ay);
    f2unpack(pvs, sx, sy);
    v = f2pack(__fadd_rn(ax, sy), __fsub_rn(ay, sx));
  }
};

template <bool NNN, bool BOND, bool WIDE, bool RAG>
__global__ void __launch_bounds__(WIDE ? 384 : kCxNarrow, 1) cluster_cplx_kernel(CplxClusterArgs a) {
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ __align__(8) unsigned long long bar_mem;
  __shared__ double ctab[2][kCxChunk];     // C_m of the current and the next chunk of moments
  __shared__ double sums[kCols * 8][4];    // sum_m C_m (<e_t|j_m>, <h_t|j_m>) of the first 8 targets
  __shared__ unsigned places[kCxPlaces];   // where the targets' quads lie (0: not in this CTA)
  const int t = threadIdx.x, lane = t & 31, nw = blockDim.x >> 5;
  const int CS = a.cluster, rank = CS > 1 ? static_cast<int>(cluster_rank()) : 0;
  const int cid = blockIdx.x / CS, ncl = gridDim.x / CS;
  const int Lx = a.Lx, Ly = a.Ly, TX = (Lx + kCx - 1) / kCx, TY = (Ly + kCy - 1) / kCy, R = a.rows;
  const int ghost = TX * R, nil = ghost + (CS > 1 ? TX : 0);
  const unsigned e0 = smem_addr(raw), poff = (nil + 1) * kCxRec * 16;  // from a tile's sites to its coefficients
  const unsigned bar = smem_addr(&bar_mem);
  if (t == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(nw) : "memory");
  unsigned phase = 0;
  auto arrive = [&]() {
    if (CS > 1) {
      cluster_arrive();
    } else {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    }
  };
  auto wait = [&]() {
    if (CS > 1) {
      cluster_wait();
    } else if (phase < 2u && !mbar_try(bar, phase)) {
      const unsigned long long t0 = global_ns();
      for (unsigned it = 0; !mbar_try(bar, phase); ++it)
        if ((it & 255u) == 255u && expired_here(t0, a.wait_ns, a.flags)) {
          phase |= 2u;  // no further waits
          break;
        }
    }
    phase ^= 1u;
  };
  auto record = [&](int j) { return e0 + j * kCxRec * 16; };
  for (int j = t; j < (nil + 1) * kCxRec * 2; j += blockDim.x) sts4(e0 + j * 16, 0, 0);
  __syncthreads();

  const int rows_here = min(R, TY - rank * R);
  // half k of the threads takes start vector k, one tile a thread; the bases below are those of its quads
  const int half = blockDim.x >> 1, k = t >= half ? 1 : 0, tt = t - k * half;
  const int tx = tt % TX, tyl = tt / TX, ty = rank * R + tyl;
  const bool act = tyl < rows_here;
  const int x0 = kCx * tx, y0 = kCy * ty;
  // the eight tiles around (a tile outside the lattice: zeros)
  auto tile = [&](int dx, int dy) {
    int x = tx + dx, y = tyl + dy;
    if (x < 0 || x >= TX) {
      if (!a.px) return record(nil) + k * 16;
      x = x < 0 ? TX - 1 : 0;
    }
    if (y >= 0 && y < rows_here) return record(y * TX + x) + k * 16;
    const int gy = ty + dy;
    if ((gy < 0 || gy >= TY) && !a.py) return record(nil) + k * 16;
    return (CS > 1 ? record(ghost + x) : record((gy < 0 ? TY - 1 : 0) * TX + x)) + k * 16;
  };
  const unsigned own = (act ? record(tt) : record(nil)) + k * 16;
  // Periodic sides that the tiles do not divide (RAG): the last tiles have rx columns or one row.  What
  // lies beyond it takes the place of the missing one: rt's column 0 of column rx, up's row 0 of row 1.
  // Seen from the first tiles, the last ones' column rx - 1 (row 0) is the neighbour: the addresses of lf,
  // ul and dl (dn, dl and dr) move by back_x (back_y) sites.
  const int rx = Lx - kCx * (TX - 1);
  const int rsel = RAG && a.px && tx == TX - 1 ? rx : kCx;
  const bool end_y = RAG && a.py && (Ly & 1) && act && ty == TY - 1;
  const int back_x = RAG && a.px && tx == 0 ? rx - kCx : 0;
  const int back_y = RAG && a.py && (Ly & 1) && CS == 1 && ty == 0 ? -kCx : 0;
  const unsigned lf = act ? tile(-1, 0) : own, rt = act ? tile(1, 0) : own, up = act ? tile(0, 1) : own;
  const unsigned dn = act ? tile(0, -1) : own, ul = act ? tile(-1, 1) : own, ur = act ? tile(1, 1) : own;
  const unsigned dl = act ? tile(-1, -1) : own, dr = act ? tile(1, -1) : own;
  // a CTA's lowest row of sites goes to the CTA below (its ghosts' row 0), the highest above (row 1)
  unsigned push_up = 0, push_dn = 0;
  if (act && CS > 1) {
    if (tyl + 1 == rows_here && (ty + 1 < TY || a.py)) push_up = remote(record(ghost + tx) + k * 16, rank + 1 < CS ? rank + 1 : 0);
    if (tyl == 0 && (ty > 0 || a.py)) push_dn = remote(record(ghost + tx) + k * 16, rank > 0 ? rank - 1 : CS - 1);
  }
  // coefficients of the tile's sites: quads (t_+x, t_+y), (t_+x+y, t_-x+y), (B_+x, B_+y), (e, Delta)
  auto load_coef = [&](unsigned rec, int gx, int gy, int r, int skip = 0) {
    for (int c = 0; c < kCx; ++c) {
      const int x = gx + c, y = gy + r - skip;
      if (x >= Lx || y >= Ly) continue;
      auto field = [&](int k) {
        return *reinterpret_cast<const float2 *>(a.params + ((static_cast<size_t>(y) * kCplxFields + k) * Lx + x) * 2);
      };
      const unsigned q = rec + poff + (r * kCx + c) * 64;
      const int first[4] = {kCpHop, kCpHop + 2, kCpBond, kCpE};
      for (int k = 0; k < 4; ++k) {
        const float2 p = field(first[k]), s = field(first[k] + 1);
        sts4(q + k * 16, f2pack(p.x, p.y), f2pack(s.x, s.y));
      }
    }
  };
  if (act) load_coef(record(tt), x0, y0, k);
  if (CS > 1 && t < TX) {  // of the row below this CTA's
    const int gy = rank * R - 1;
    // (the last row of tiles may have one row of sites: it takes the place of the second)
    if (gy >= 0 || a.py) load_coef(record(ghost + t), kCx * t, kCy * (gy < 0 ? TY - 1 : gy), 1, RAG && gy < 0 ? Ly & 1 : 0);
  }
  if (CS > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }

  const unsigned coff = poff - k * 16;
  F2 pu[kCy][kCx], pv[kCy][kCx], qu[kCy][kCx], qv[kCy][kCx];  // j_{n-1}, j_n
  auto publish = [&](int r, int c, F2 u, F2 v, int wr) {
    const int at_ = wr + (r * kCx + c) * kCols * 16;
    sts4(own + at_, u, v);
    if (RAG && end_y) {
      if (r == 0 && push_up) push4(push_up + at_ + kCx * kCols * 16, u, v);
    } else if (r == 1 && push_up) {
      push4(push_up + at_, u, v);
    }
    if (r == 0 && push_dn) push4(push_dn + at_, u, v);
  };
  // (o) = 2 H~ (z) - (o), published as it is formed; both rows of a column of sites at once
  auto step = [&](auto buf_c, F2 (&zu)[kCy][kCx], F2 (&zv)[kCy][kCx], F2 (&ou)[kCy][kCx], F2 (&ov)[kCy][kCx]) {
    constexpr int rd = decltype(buf_c)::value * kCxSet * 16, wr = (1 - decltype(buf_c)::value) * kCxSet * 16;
    if (!act) return;
    auto far = [&](unsigned rec, int r, int c) { return lds4(rec + rd + (r * kCx + c) * kCols * 16); };
    auto coef = [&](unsigned rec, int r, int c, int q) { return ldc(rec + coff + (r * kCx + c) * 64 + q * 16); };
    // (the same in tiles seen across a ragged edge)
    const unsigned lv = lf + back_x * kCols * 16, lc = lf + back_x * 64, ulv = ul + back_x * kCols * 16;
    const unsigned dnv = dn + back_y * kCols * 16, dnc = dn + back_y * 64, drv = dr + back_y * kCols * 16, drc = dr + back_y * 64;
    const unsigned dlv = dl + (back_x + back_y) * kCols * 16, dlc = dl + (back_x + back_y) * 64;
    // columns x - 1 and x of the rows below (d) and above (p) the tile, and of the tile's own rows 0 and 1
    Quad d0{}, p0{}, l0 = far(lv, 0, kCx - 1), l1 = far(lv, 1, kCx - 1);
    if (NNN) {
      d0 = far(dlv, 1, kCx - 1);
      p0 = far(ulv, 0, kCx - 1);
    }
    Quad d1 = far(dnv, 1, 0), p1 = far(up, 0, 0);
    // column x - 1's forward x hopping and bond of rows 0 and 1; the diagonal hoppings of the
    // row below and of row 0 at x - 1 and x
    Coef tl0 = coef(lc, 0, kCx - 1, 0), tl1 = coef(lc, 1, kCx - 1, 0), bl0{}, bl1{}, gd0{}, gd1{}, go0{}, go1{};
    if (BOND) {
      bl0 = coef(lc, 0, kCx - 1, 2);
      bl1 = coef(lc, 1, kCx - 1, 2);
    }
    if (NNN) {
      gd0 = coef(dlc, 1, kCx - 1, 1);
      gd1 = coef(dnc, 1, 0, 1);
      go0 = coef(lc, 0, kCx - 1, 1);
      go1 = coef(own, 0, 0, 1);
    }
#pragma unroll
    for (int c = 0; c < kCx; ++c) {
      const int cn = c < kCx - 1 ? c + 1 : c;
      const bool last = c == kCx - 1;
      const bool wrap = RAG && !last && c + 1 == rsel;  // column x + 1 is rt's first
      const Quad m0{zu[0][c], zv[0][c]}, m1{zu[1][c], zv[1][c]};
      Quad r0{zu[0][cn], zv[0][cn]}, r1{zu[1][cn], zv[1][cn]}, d2{}, p2{};  // column x + 1
      if (last) {
        r0 = far(rt, 0, 0);
        r1 = far(rt, 1, 0);
        if (NNN) {
          d2 = far(drv, 1, 0);
          p2 = far(ur, 0, 0);
        }
      } else {
        d2 = far(wrap ? drv - cn * kCols * 16 : dnv, 1, cn);
        p2 = far(wrap ? ur - cn * kCols * 16 : up, 0, cn);
        if (wrap) {
          r0 = far(rt, 0, 0);
          r1 = far(rt, 1, 0);
        }
      }
      // row 0's neighbours above: row 1, or what lies beyond a last row
      const Quad a0 = RAG && end_y ? p0 : l1, a1 = RAG && end_y ? p1 : m1, a2 = RAG && end_y ? p2 : r1;
      {  // row 0
        const Coef on = coef(own, 0, c, 3), tf = coef(own, 0, c, 0), td = coef(dnc, 1, c, 0);
        Update w(BOND, on, m0, ou[0][c]);
        Coef bf{}, bd{};
        if (BOND) {
          bf = coef(own, 0, c, 2);
          bd = coef(dnc, 1, c, 2);
        }
        w.hop(tf.r0, tf.i0, r0);
        if (BOND) w.pair(bf.r0, bf.i0, r0);
        w.hop(tl0.r0, -tl0.i0, l0);
        if (BOND) w.pair(bl0.r0, bl0.i0, l0);
        w.hop(tf.r1, tf.i1, a1);
        if (BOND) w.pair(bf.r1, bf.i1, a1);
        w.hop(td.r1, -td.i1, d1);
        if (BOND) w.pair(bd.r1, bd.i1, d1);
        if (NNN) {
          // (t_+x+y, t_-x+y) of the site; backward, the lower left site's t_+x+y and the lower right's t_-x+y
          const Coef gd2 = last ? coef(drc, 1, 0, 1) : coef(wrap ? drc - cn * 64 : dnc, 1, cn, 1);
          w.hop(go1.r0, go1.i0, a2);
          w.hop(gd0.r0, -gd0.i0, d0);
          w.hop(gd2.r1, -gd2.i1, d2);
          w.hop(go1.r1, go1.i1, a0);
          gd0 = gd1;
          gd1 = gd2;
        }
        w.finish(on.r0, m0, ou[0][c], ov[0][c]);
        tl0 = tf;
        bl0 = bf;
      }
      {  // row 1; tl0 and bl0 are now those of row 0 at x
        const Coef on = coef(own, 1, c, 3), tf = coef(own, 1, c, 0);
        Update w(BOND, on, m1, ou[1][c]);
        Coef bf{};
        if (BOND) bf = coef(own, 1, c, 2);
        w.hop(tf.r0, tf.i0, r1);
        if (BOND) w.pair(bf.r0, bf.i0, r1);
        w.hop(tl1.r0, -tl1.i0, l1);
        if (BOND) w.pair(bl1.r0, bl1.i0, l1);
        w.hop(tf.r1, tf.i1, p1);
        if (BOND) w.pair(bf.r1, bf.i1, p1);
        w.hop(tl0.r1, -tl0.i1, m0);
        if (BOND) w.pair(bl0.r1, bl0.i1, m0);
        if (NNN) {
          const Coef gp = coef(own, 1, c, 1), go2 = last ? coef(rt, 0, 0, 1) : coef(wrap ? rt - cn * 64 : own, 0, cn, 1);
          w.hop(gp.r0, gp.i0, p2);
          w.hop(go0.r0, -go0.i0, l0);
          w.hop(go2.r1, -go2.i1, r0);
          w.hop(gp.r1, gp.i1, p0);
          go0 = go1;
          go1 = go2;
        }
        w.finish(on.r0, m1, ou[1][c], ov[1][c]);
        tl1 = tf;
        bl1 = bf;
      }
      l0 = m0;
      l1 = m1;
      d0 = d1;
      p0 = p1;
      d1 = d2;
      p1 = p2;
      if (WIDE) {
        publish(0, c, ou[0][c], ov[0][c], wr);
        publish(1, c, ou[1][c], ov[1][c], wr);
      }
    }
    if (!WIDE) {
#pragma unroll
      for (int r = 0; r < kCy; ++r)
#pragma unroll
        for (int c = 0; c < kCx; ++c) publish(r, c, ou[r][c], ov[r][c], wr);
    }
  };

  const float bound = static_cast<float>(1.0 + a.tol);
  for (int col0 = cid * kCols; col0 < a.ncols; col0 += ncl * kCols) {
    // ---- readout of j_m: target k of column col0 + q (thread q n_t + k, + blockDim, ..)
    auto target_of = [&](int q, int k) {
      const int site = a.sites[min(col0 + q, a.ncols - 1)];
      if (a.targets) return a.targets[k];
      if (a.mode == kReadBonds) return k == 0 ? site : neighbour_site(Lx, Ly, a.px, a.py, site, k - 1);
      return neighbour_site(Lx, Ly, a.px, a.py, site, k);
    };
    // the first target of this thread, where its quad lies in set 0 (0: not in this CTA)
    const int n_all = kCols * a.n_t;
    auto place = [&](int idx) -> unsigned {
      const int q = idx / a.n_t, s = target_of(q, idx % a.n_t);
      if (s < 0) return 0u;
      const int x = s % Lx, y = s / Lx, row = y / kCy - rank * R;
      if (row < 0 || row >= rows_here) return 0u;
      return record(row * TX + x / kCx) + ((y % kCy * kCx + x % kCx) * kCols + q) * 16;
    };
    const unsigned mine = t < n_all ? place(t) : 0u;
    for (int idx = t + blockDim.x; idx < min(n_all, kCxPlaces); idx += blockDim.x) places[idx] = place(idx);
    if (t < kCols * 8)
      for (int i = 0; i < 4; ++i) sums[t][i] = 0.0;
    if (t < kCxChunk) ctab[0][t] = t < a.M ? a.C[t] : 0.0;
    auto deliver = [&](int m, int idx, const Quad &z) {
      const int q = idx / a.n_t, k = idx % a.n_t, col = col0 + q;
      float er, ei, hr, hi;
      f2unpack(z.lo, er, ei);
      f2unpack(z.hi, hr, hi);
      if (a.n_t <= 8) {
        const double c = ctab[(m / kCxChunk) & 1][m % kCxChunk];
        double *s = sums[q * 8 + k];
        s[0] = fma(c, static_cast<double>(er), s[0]);
        s[1] = fma(c, static_cast<double>(ei), s[1]);
        s[2] = fma(c, static_cast<double>(hr), s[2]);
        s[3] = fma(c, static_cast<double>(hi), s[3]);
      }
      if (col >= a.ncols) return;
      const size_t o = (static_cast<size_t>(col) * a.M + m) * (a.mode == kReadBonds ? 5 : a.n_t) + k;
      if (a.mode == kReadBonds) {
        if (k == 0 && a.a_re) a.a_re[static_cast<size_t>(col) * a.M + m] = er;
        if (k == 0 && !(fabsf(er) <= bound)) atomicOr(a.flags, kFlagSpectrum);
        if (a.a_h) a.a_h[o] = make_double2(hr, hi);
      } else {
        if (a.a_e) a.a_e[o] = make_double2(er, ei);
        if (a.a_h) a.a_h[o] = make_double2(hr, hi);
        const float e2 = er * er + ei * ei, h2 = hr * hr + hi * hi;
        if (!(e2 <= bound * bound) || (a.a_h && !(h2 <= bound * bound))) atomicOr(a.flags, kFlagSpectrum);
      }
    };
    // the quads of j_m are read before the threads meet and delivered after that (`now`), but for
    // those of targets beyond one a thread
    auto readout = [&](int m, int set, auto now) {
      const Quad z = mine ? lds4(mine + set * kCxSet * 16) : Quad{0, 0};
      for (int idx = t + blockDim.x; idx < n_all; idx += blockDim.x) {
        const unsigned p = idx < kCxPlaces ? places[idx] : place(idx);  // this thread's own entry
        if (p) deliver(m, idx, lds4(p + set * kCxSet * 16));
      }
      // (every thread has delivered the chunk before)
      if (m % kCxChunk == 8 && t < kCxChunk) {
        const int next = m - 8 + kCxChunk + t;
        ctab[(m / kCxChunk + 1) & 1][t] = next < a.M ? a.C[next] : 0.0;
      }
      now();
      if (mine) deliver(m, t, z);
    };
    // targets across an open edge read zero: the moments of one CTA's threads
    if (rank == 0 && !a.targets && (a.a_e || a.a_h))
      for (int idx = t; idx < n_all; idx += blockDim.x) {
        const int q = idx / a.n_t, k = idx % a.n_t, col = col0 + q;
        if (col >= a.ncols || target_of(q, k) >= 0) continue;
        for (int m = 0; m < a.M; ++m) {
          const size_t o = (static_cast<size_t>(col) * a.M + m) * (a.mode == kReadBonds ? 5 : a.n_t) + k;
          if (a.a_e) a.a_e[o] = make_double2(0.0, 0.0);
          if (a.a_h) a.a_h[o] = make_double2(0.0, 0.0);
        }
      }
    // ---- j_0 = e_i and j_1 = H~ e_i
    const double am = a.scal[kScalA];
    const int start_site = a.sites[min(col0 + k, a.ncols - 1)];
    const int xs = start_site % Lx, ys = start_site / Lx;
#pragma unroll
    for (int r = 0; r < kCy; ++r)
#pragma unroll
      for (int c = 0; c < kCx; ++c) {
        int dx = x0 + c - xs, dy = y0 + r - ys;
        if (a.px) dx = dx == Lx - 1 ? -1 : dx == 1 - Lx ? 1 : dx;
        if (a.py) dy = dy == Ly - 1 ? -1 : dy == 1 - Ly ? 1 : dy;
        float one = 0.f, ur_ = 0.f, ui = 0.f, vr = 0.f, vi = 0.f;
        if (act && x0 + c < Lx && y0 + r < Ly && abs(dx) <= 1 && abs(dy) <= 1) {
          double2 eu = make_double2(0.0, 0.0), ev = eu;
          if (dx == 0 && dy == 0) {
            one = 1.f;
            eu.x = a.eps[start_site] - a.mu;
            if (!BOND) ev = make_double2(a.delta[start_site].x, -a.delta[start_site].y);
          } else {
            // direction of this site from the start site
            const int d = dy == 0 ? (dx > 0 ? 0 : 1) : dx == 0 ? (dy > 0 ? 2 : 3) : dx == dy ? (dx > 0 ? 4 : 5) : (dx > 0 ? 6 : 7);
            if (d < a.n_dirs) {
              const double2 h = a.hop[static_cast<size_t>(start_site) * a.n_dirs + d];
              eu = make_double2(-h.x, h.y);
              if (BOND && d < 4) {
                const double2 b = a.delta[static_cast<size_t>(start_site) * 4 + d];
                ev = make_double2(b.x, -b.y);
              }
            }
          }
          ur_ = static_cast<float>(eu.x / am);
          ui = static_cast<float>(eu.y / am);
          vr = static_cast<float>(ev.x / am);
          vi = static_cast<float>(ev.y / am);
        }
        pu[r][c] = f2pack(one, 0.f);
        pv[r][c] = 0;
        qu[r][c] = f2pack(ur_, ui);
        qv[r][c] = f2pack(vr, vi);
        if (act) sts4(own + (kCxSet + (r * kCx + c) * kCols) * 16, pu[r][c], pv[r][c]);
      }
    __syncthreads();
    readout(0, 1, [] {});  // j_0 from the second set
    if (act) {
#pragma unroll
      for (int r = 0; r < kCy; ++r)
#pragma unroll
        for (int c = 0; c < kCx; ++c) publish(r, c, qu[r][c], qv[r][c], 0);
    }
    arrive();
    // step n reads j_n in set (n - 1) & 1
    int n = 1;
    for (; n <= a.M - 2;) {
      wait();
      step(std::integral_constant<int, 0>{}, qu, qv, pu, pv);
      readout(n, 0, arrive);
      if (++n > a.M - 2) break;
      wait();
      step(std::integral_constant<int, 1>{}, pu, pv, qu, qv);
      readout(n, 1, arrive);
      ++n;
    }
    wait();
    readout(n, (n - 1) & 1, [] {});  // n = M - 1
    // ---- the folds
    if (mine && t < n_all && a.n_t <= 8) {
      const int q = t / a.n_t, k = t % a.n_t, col = col0 + q;
      const double *s = sums[q * 8 + k];
      if (col < a.ncols) {
        if (a.mode == kReadBonds) {
          if (k == 0 && a.acc_n) a.acc_n[col] -= s[0];
          if (k > 0 && a.acc) {
            double2 &o = a.acc[static_cast<size_t>(col) * 4 + k - 1];
            o.x += s[2];
            o.y -= s[3];
          }
        } else if (a.acc) {
          double2 &o = a.acc[static_cast<size_t>(col) * a.n_t + k];
          o.x += s[0];
          o.y += s[1];
        }
      }
    }
    __syncwarp();
    if (CS > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  }
}

template <bool NNN, bool BOND>
auto cplx_kernel_of(const ClusterPlan &p) {  // p.rag bit 2: ragged periodic sides
  if (p.rag & 4) return p.threads > kCxNarrow ? cluster_cplx_kernel<NNN, BOND, true, true> : cluster_cplx_kernel<NNN, BOND, false, true>;
  return p.threads > kCxNarrow ? cluster_cplx_kernel<NNN, BOND, true, false> : cluster_cplx_kernel<NNN, BOND, false, false>;
}

template <bool NNN, bool BOND>
int cplx_slots_one(const ClusterPlan &p) {
  auto k = cplx_kernel_of<NNN, BOND>(p);
  Launch<4, 0> l(p);
  int n = 0;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kCplxClusterSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &l.cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return n;
}

template <bool NNN, bool BOND>
cudaError_t cplx_launch_one(const CplxClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  Launch<4, 0> l(p);
  l.cfg.gridDim = dim3(clusters * p.cluster);
  l.cfg.stream = s;
  auto k = cplx_kernel_of<NNN, BOND>(p);
  return cudaLaunchKernelEx(&l.cfg, k, a);
}

}  // namespace
}  // namespace cbdg
