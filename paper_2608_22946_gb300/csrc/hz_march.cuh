// Forward 27-point IOFD stencil in single precision, all levels, for sm_103a.
//
// Operator (Sec. 2.2, Eq. iofd-shell-form and Eq. pml-second-difference): with
// c, e, k the centre, the four face neighbours and the four corners of a
// column in one z-plane, and m, o, n the planes below, at and above the row,
//   (H x) = C_0 c_o + C_1 (e_o + c_m + c_n) + C_2 (k_o + e_m + e_n) + C_3 (k_m + k_n)
// where no axis is stretched.  A stretched axis j adds
//   eps+_j (T_j(+1) - T_j(0)) + eps-_j (T_j(-1) - T_j(0)),
//   eps+-_j = -ell^-2 (abar_j - 1 +- achk_j),
// T_j(t) the transverse-weighted sum (alpha_4, alpha_5 / 4, (1 - alpha_4 -
// alpha_5) / 4) of the plane at offset t along j.
//
// What bounds it: issue slots.  The algorithm needs 20 B of HBM traffic and about
// 60 instructions per node; a kernel of 160 instructions per node (the
// accumulation form of hz_fwd.cuh in single precision, which this replaces) ran at
// a third of the HBM rate however many warps were resident.  So:
//  - a thread owns 2 x 2 adjacent columns (2 x 1 with two right-hand sides) and
//    marches in z; the four rows it needs of a plane come as 128-bit shared-memory
//    loads, the in-plane sums are shared between its columns and run as packed
//    two-float adds (re, im);
//  - the gather form keeps (c, e, k) of one plane and what the plane before adds to
//    the next row, so a row's weights are needed in one place, its completion;
//  - the weights of A are cubics on parts of a segment (16 multiply-adds fewer loads
//    and steps than the quintics on whole ones); kappa's segment comes from a
//    round-to-nearest add instead of conversions, and the local coordinate is
//    measured in segments so that one subtraction gives it;
//  - the core's planes come by TMA, issued by one thread (below);
//  - the PML-free core, the PML frame around it and the z-PML slabs are block
//    ranges of ONE launch, each with its own compact body: no second stream, and
//    the costly PML rows fill the SMs from the start;
//  - blocks of 128 threads, three per SM (four with two right-hand sides): at 128
//    registers the PML bodies spill, and every spill is a stall on a thrashed L1
//    (289^3 A_h 147 us at four blocks, 138 at three).
// Measured, in a CUDA graph, accumulation form / this (us): 289^3 A_h 194 / 135,
// residual 278 / 182, J_2 290 / 224; its 2h level (145^3) A 36.5 / 26.7, B 36.4 / 27.6,
// residual 58 / 46, J_2 50.2 / 43.3; 225^3 x 16 right-hand sides A_h 1191 / 972.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "hz_fwd.cuh"

namespace hz {
namespace march {

constexpr int NT = 128;

// Tile of NPX TXT x NPY TYT columns, NPX x NPY columns per thread, and its plane
// with a one-node halo.
template <int TXT_, int NPX_, int NPY_>
struct Tile {
  static constexpr int TXT = TXT_, NPX = NPX_, NPY = NPY_, TYT = NT / TXT_;
  static constexpr int W = NPX_ * TXT_, H = NPY_ * TYT;
  static constexpr int PW = W + 2, PLN = (PW * (H + 2) + 1) & ~1;
  static constexpr int NSLOT = (PLN + NT - 1) / NT;
};
template <int NPY>
using CoreT = Tile<32, 2, NPY>;  // 64 x 8 or 64 x 4

// Coefficient tables of a level (single precision), NS = nseg + 1 segments, the
// last one the clamp eta >= 0.4, in the local coordinate u = eta / ds - segment:
//   Q: shell weights of Q_h, cubics, [segment][power][4]
//   F: alpha_4 - 3/4, alpha_5 - 1/4 and the mass weights M_0..M_3, cubics,
//      [segment][power][6].  The offsets keep the two alphas small, and the stiffness
//      weights that B forms from them (6 alpha_4 most of all) accurate: random fields,
//      interior rows, 5.4e-8 of the norm against 7.2e-8 with the alphas themselves.
//   S: C_0..C_3 of A (stiffness and mass weights combined), as the interpolating
//      cubics of nsub equal parts of each segment (u in parts), [part][power][4]; the
//      clamp is the last part.  After them alpha_4, alpha_5 in the same parts,
//      [power][2].  nsub is the smallest that reproduces the quintics, which C is
//      exactly, to kSubTol of the row's largest weight: 4 with the shipped table
//      (4e-10; 2 leave 7e-9), more with a coarser one, up to kMaxParts parts in all.
// B evaluates L - (1 + i sigma) kappa^2 M from F.  Taking C from S there (5.4e-8 too)
// costs a fifth of the 2h level's time, 41.7 -> 49.9 us for J_2 on 145^3: two more
// 128-bit table loads per node, and 65 parts where F has 17 rows.
constexpr int kMtQ = 16, kMtF = 24, kMtS = 24, kMaxParts = 512;
constexpr double kSubTol = 6e-9;
constexpr double kA4Off = 0.75, kA5Off = 0.25;  // offsets of table F
__host__ __device__ constexpr int mt_off_F(int ns) { return kMtQ * ns; }
__host__ __device__ constexpr int mt_off_S(int ns) { return (kMtQ + kMtF) * ns; }
__host__ __device__ constexpr int mt_size(int ns) { return mt_off_S(ns) + kMtS * (kMaxParts + 1); }
// The table of an operator kind (A: S, B: F, Q): its place, and floats per row.
template <int OPK>
__host__ __device__ constexpr int tab_off(int ns) {
  return OPK == OPK_A ? mt_off_S(ns) : OPK == OPK_B ? mt_off_F(ns) : 0;
}
template <int OPK>
constexpr int kTabRow = OPK == OPK_A ? kMtS : OPK == OPK_B ? kMtF : kMtQ;

template <int MODE, class TL, int RB>
struct Smem {
  // the Jacobi map reads 1/diag of the previous plane and transforms the next
  // one in place, so its ring keeps one more plane than it prefetches
  static constexpr int NSTG = MODE == M_J2 ? 5 : 6;
  static constexpr int PREF = MODE == M_J2 ? 3 : 5;
  static constexpr size_t a16(size_t x) { return (x + 15) & ~(size_t)15; }
  static constexpr size_t o_d = a16((size_t)NSTG * RB * TL::PLN * 8);
  static constexpr size_t o_red = a16(o_d + (MODE == M_J2 ? (size_t)NSTG * TL::PLN * 8 : 0));
  static constexpr size_t o_tab = o_red + 32 * sizeof(double);  // sized at the launch
};

// Blocks of a launch, in this order: the z-PML slabs (whole x-y range, general
// rows), the PML frame of the z-range between them, its PML-free core.  The
// costlier blocks start first; tiles of one z-block are neighbours.
struct Plan {
  int zs0 = 0, zc0 = 0, zc1 = 0, zs1 = 0;  // rows: slab [zs0, zc0), core [zc0, zc1), slab [zc1, zs1)
  int zb = 4, zbf = 4;                     // planes per block of the core; of slabs and frame
  int SW = 0, SH = 0, nlo = 0, nsl = 0;    // slab tiles, z-blocks of the lower slab, slab blocks
  TileMap fm;                              // frame tiles (count per z-block), core bounds px0..py1
  int nfr = 0;                             // slab and frame blocks
  int RW = 0, RH = 0;                      // core tiles
  int items = 0;                           // all blocks of one right-hand side (group)
  bool rows = false;                       // core planes come by TMA (odd nx, ny; halo inside the grid)
};

// ----------------------------------------------------------------------------
// device helpers
// ----------------------------------------------------------------------------
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ void rfma(float2& s, float w, float2 v) {
  s.x = fmaf(w, v.x, s.x);
  s.y = fmaf(w, v.y, s.y);
}
__device__ __forceinline__ void cfma2(float2& s, float2 w, float2 v) {
  s.x = fmaf(w.x, v.x, s.x);
  s.x = fmaf(-w.y, v.y, s.x);
  s.y = fmaf(w.x, v.y, s.y);
  s.y = fmaf(w.y, v.x, s.y);
}
__device__ __forceinline__ void cp8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem));
}
__device__ __forceinline__ float2 ldf2(const cx<float>* p) { return *reinterpret_cast<const float2*>(p); }

// Segment of kappa and local coordinate: round(t - 1/2) of t = eta / ds through
// the 1.5 * 2^23 addition, saturated to [0, nseg].  At a segment boundary either
// neighbour may be taken (the functions are continuous there).
struct SegK {
  float s1, sc, off, hi;  // t = kappa s1; (t - 1/2) / nseg = kappa sc + off; hi = nseg
};
__device__ __forceinline__ int seg_u(const SegK& K, float kap, float& u) {
  constexpr float kMagic = 12582912.f;
  const float t = kap * K.s1;
  const float m = __saturatef(fmaf(kap, K.sc, K.off));
  const float r = fmaf(m, K.hi, kMagic);
  u = t - (r - kMagic);
  return __float_as_int(r) - 0x4B400000;
}

// State of one column between planes: the sums c, e, k (and the PML
// corrections A, B) of the last plane o, and of the plane m before it either
// the sums themselves (z-PML blocks need them one by one) or what they add to
// the row of plane o: p1 = e_o + c_m, p2 = k_o + e_m, p3 = k_m; BA = B_o + A_m,
// Bm = B_m.
struct Sums {
  float2 c, e, k;
};
template <bool CORR>
struct Column {
  float2 c, e, k, p1, p2, p3;
};
template <>
struct Column<true> {
  float2 c, e, k, p1, p2, p3, A, B, BA, Bm;
};

// Takes in the sums n (A, B: nA, nB) of the next plane and returns H x of the
// row of plane o.
template <int OPK, bool CORR, bool ZP>
__device__ __forceinline__ float2 row_value(const float* w, float k2, float inv_l2, float sigma, Column<CORR>& s,
                                            const Sums& n, float2 nA, float2 nB, bool zp, float2 ezp, float2 ezm,
                                            float a4, float a5) {
  float2 N1, N2;
  if constexpr (ZP) {
    N1 = add2(add2(s.e, s.p1), n.c);
    N2 = add2(add2(s.k, s.p2), n.e);
  } else {
    N1 = add2(s.p1, n.c);
    N2 = add2(s.p2, n.e);
  }
  const float2 N3 = add2(s.p3, n.k);
  // Terms are added smallest first (corners inwards, PML corrections before the faces):
  // only the last addition then rounds at the size of the centre's term.
  float2 h = make_float2(w[3] * N3.x, w[3] * N3.y);
  rfma(h, w[2], N2);
  // (B scales its rows by ell^-2 at the end: its corrections wait in a sum of their own)
  [[maybe_unused]] float2 cor = make_float2(0.f, 0.f);
  if constexpr (CORR) {
    const float q5 = 0.25f * a5, qb = fmaf(-0.25f, a4 + a5, 0.25f);
    float2& t0 = OPK == OPK_B ? cor : h;
    rfma(t0, qb, add2(s.Bm, nB));
    rfma(t0, q5, add2(s.BA, nA));
    rfma(t0, a4, s.A);
    s.BA = add2(nB, s.A);
    s.Bm = s.B;
    s.A = nA;
    s.B = nB;
    if constexpr (ZP) {
      if (zp) {  // eps+ T(n - o) + eps- T(m - o), T the transverse-weighted sum
        float2 t = make_float2(0.f, 0.f);
        rfma(t, qb, sub2(n.k, s.k));
        rfma(t, q5, sub2(n.e, s.e));
        rfma(t, a4, sub2(n.c, s.c));
        cfma2(t0, ezp, t);
        t = make_float2(0.f, 0.f);
        rfma(t, qb, sub2(s.p3, s.k));
        rfma(t, q5, sub2(s.p2, s.e));
        rfma(t, a4, sub2(s.p1, s.c));
        cfma2(t0, ezm, t);
      }
    }
  }
  rfma(h, w[1], N1);
  rfma(h, w[0], s.c);
  if constexpr (OPK == OPK_B) {
    // w[4..7]: mass weights; H = ell^-2 (L - (1 + i sigma) kappa^2 M)
    float2 q = make_float2(w[7] * N3.x, w[7] * N3.y);
    rfma(q, w[6], N2);
    rfma(q, w[5], N1);
    rfma(q, w[4], s.c);
    const float k2s = sigma * k2;
    const float hx = fmaf(k2s, q.y, fmaf(-k2, q.x, h.x)), hy = fmaf(-k2s, q.x, fmaf(-k2, q.y, h.y));
    h.x = CORR ? fmaf(inv_l2, hx, cor.x) : inv_l2 * hx;
    h.y = CORR ? fmaf(inv_l2, hy, cor.y) : inv_l2 * hy;
  }
  if constexpr (ZP) {
    s.p1 = s.c;
    s.p2 = s.e;
  } else {
    s.p1 = add2(n.e, s.c);
    s.p2 = add2(n.k, s.e);
  }
  s.p3 = s.k;
  s.c = n.c;
  s.e = n.e;
  s.k = n.k;
  return h;
}

__device__ __forceinline__ float4 lds128(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ float2 lds64(unsigned a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ float lds32(unsigned a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
// Rows of the launch's table, without the clamp, and its segments.
template <int OPK>
__device__ __forceinline__ int tab_rows(const StencilCall<float>& a) {
  return a.tab.nseg * (OPK == OPK_A ? a.lv.nsub : 1);
}
template <int OPK>
__device__ __forceinline__ SegK tab_seg(const StencilCall<float>& a) {
  SegK K;
  K.s1 = a.tab.inv_ds * (float)kInv2Pi * (OPK == OPK_A ? (float)a.lv.nsub : 1.f);
  K.hi = (float)tab_rows<OPK>(a);
  K.sc = K.s1 / K.hi;
  K.off = -0.5f / K.hi;
  return K;
}
template <int OPK>
__device__ __forceinline__ void load_table(const StencilCall<float>& a, unsigned char* dst) {
  const float4* g = reinterpret_cast<const float4*>(a.lv.mtab + tab_off<OPK>(a.tab.nseg + 1));
  float4* t = reinterpret_cast<float4*>(dst);
  for (int i = threadIdx.x; i < kTabRow<OPK> / 4 * (tab_rows<OPK>(a) + 1); i += NT) t[i] = g[i];
}
// Weights of a row: 4 of A or Q, 4 stiffness and 4 mass weights of B; with T also
// alpha_4 and alpha_5.
template <int OPK, bool T = false>
__device__ __forceinline__ void row_weights(const SegK& K, unsigned tab, float kap, float* w, float* a45 = nullptr) {
  float u;
  const unsigned t = tab + 4u * kTabRow<OPK> * (unsigned)seg_u(K, kap, u);
  if constexpr (OPK != OPK_B) {
    const float4 c3 = lds128(t + 48), c2 = lds128(t + 32), c1 = lds128(t + 16), c0 = lds128(t);
    w[0] = fmaf(fmaf(fmaf(c3.x, u, c2.x), u, c1.x), u, c0.x);
    w[1] = fmaf(fmaf(fmaf(c3.y, u, c2.y), u, c1.y), u, c0.y);
    w[2] = fmaf(fmaf(fmaf(c3.z, u, c2.z), u, c1.z), u, c0.z);
    w[3] = fmaf(fmaf(fmaf(c3.w, u, c2.w), u, c1.w), u, c0.w);
    if constexpr (T) {
      const float4 lo = lds128(t + 64), hi = lds128(t + 80);
      a45[0] = fmaf(fmaf(fmaf(hi.z, u, hi.x), u, lo.z), u, lo.x);
      a45[1] = fmaf(fmaf(fmaf(hi.w, u, hi.y), u, lo.w), u, lo.y);
    }
  } else {
    float c[24], f[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const float4 v = lds128(t + 16 * i);
      c[4 * i] = v.x;
      c[4 * i + 1] = v.y;
      c[4 * i + 2] = v.z;
      c[4 * i + 3] = v.w;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) f[i] = fmaf(fmaf(fmaf(c[18 + i], u, c[12 + i]), u, c[6 + i]), u, c[i]);
    // 6 a4, a5 - a4, (1 - a4) / 2 - a5, 3 (a4 + a5 - 1) / 4 of a4 = f0 + 3/4, a5 = f1 + 1/4
    w[0] = fmaf(6.f, f[0], 4.5f);
    w[1] = (f[1] - f[0]) - 0.5f;
    w[2] = fmaf(-0.5f, f[0], -0.125f) - f[1];
    w[3] = 0.75f * (f[0] + f[1]);
#pragma unroll
    for (int q = 0; q < 4; ++q) w[4 + q] = f[2 + q];
    if constexpr (T) {
      a45[0] = f[0] + (float)kA4Off;
      a45[1] = f[1] + (float)kA5Off;
    }
  }
}

// The two-sweep Jacobi map of a row: with y1 = omega D^-1 g and c = y1 / omega,
// y1 + omega D^-1 (g - H y1) = omega (2 c - omega D^-1 H c); d = 1/diag, h = H c.
// Rounding c to single precision is what rounding g once would do to the result.
// Reading g again for the residual itself takes that out (289^3 9.5e-8 -> 9.05e-8 of
// the norm) and costs 14 % (226 -> 258 us): the planes hold c by then.
__device__ __forceinline__ float2 jacobi2(float om, float2 d, float2 c, float2 h) {
  const float tx = d.x * h.x - d.y * h.y, ty = d.x * h.y + d.y * h.x;
  return make_float2(om * fmaf(-om, tx, c.x + c.x), om * fmaf(-om, ty, c.y + c.y));
}

// Sum of nrm2 over the launch's blocks for each right-hand side of this block:
// partial sums in block order, combined by the last block to arrive.
template <int RB>
__device__ __forceinline__ void reduce_norm(const StencilCall<float>& a, double* sRed, const float* nrm2, int rhs0,
                                            unsigned bid, unsigned nblk) {
  if (!a.red.out) return;
  const int tid = threadIdx.x;
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    const unsigned rr = (unsigned)(rhs0 + r);
    const double s = block_sum((double)nrm2[r], sRed, tid, NT);
    if (tid == 0) a.red.partial[(size_t)rr * nblk + bid] = s;
    if (last_block_arrive(a.red.count + rr, nblk, tid)) {
      double t = 0.0;
      for (unsigned b = tid; b < nblk; b += NT) t += __ldcg(a.red.partial + (size_t)rr * nblk + b);
      t = block_sum(t, sRed, tid, NT);
      if (tid == 0) {
        a.red.out[rr] = t;
        if (a.red.root) a.red.root[rr] = sqrt(t);
        if (a.red.inv_root) a.red.inv_root[rr] = t > 1e-300 ? 1.0 / sqrt(t) : 0.0;
        a.red.count[rr] = 0;
      }
    }
  }
}

// ----------------------------------------------------------------------------
// one block: tile (x0, y0) writing columns up to (rx1, ry1), z-block bz,
// right-hand sides rhs0 .. rhs0 + RB - 1
// ----------------------------------------------------------------------------
template <int MODE, int OPK, class TL, int RB>
__device__ __forceinline__ void tile_body(const StencilCall<float>& a, unsigned char* smem, int zb0, int zb1, int x0,
                                          int y0, int rx1, int ry1, int rhs0, unsigned bid, unsigned nblk) {
  using SM = Smem<MODE, TL, RB>;
  constexpr int NSTG = SM::NSTG, PREF = SM::PREF, PW = TL::PW, PLN = TL::PLN, NSLOT = TL::NSLOT, NPX = TL::NPX, NPY = TL::NPY;
  const LevelView<float>& L = a.lv;
  cx<float>* sX = reinterpret_cast<cx<float>*>(smem);
  cx<float>* sD = reinterpret_cast<cx<float>*>(smem + SM::o_d);
  double* sRed = reinterpret_cast<double*>(smem + SM::o_red);
  const unsigned tab = (unsigned)__cvta_generic_to_shared(smem + SM::o_tab);

  const int tid = threadIdx.x;
  const int tx = tid % TL::TXT, ty = tid / TL::TXT;
  const int nx = L.nx, ny = L.ny, nz = L.nz;
  const int nplanes = zb1 - zb0 + 2;
  const long long plane = (long long)nx * ny;
  const long long xs = a.xstride > 0 ? a.xstride : L.N, ys = a.ystride > 0 ? a.ystride : L.N;
  const SegK K = tab_seg<OPK>(a);
  load_table<OPK>(a, smem + SM::o_tab);

  // this thread's columns: (gx0 + i, gy0 + j); addresses are clamped into the
  // grid (a value one past a row's end is read from kappa and 1/diag, which are
  // allocated with a spare element, and never used)
  const int gx0 = x0 + NPX * tx, gy0 = y0 + NPY * ty;
  bool act[NPY][NPX];
  unsigned col[NPY];
#pragma unroll
  for (int j = 0; j < NPY; ++j) {
#pragma unroll
    for (int i = 0; i < NPX; ++i) act[j][i] = gx0 + i <= rx1 && gy0 + j <= ry1;
    col[j] = (unsigned)(min(gy0 + j, ny - 1) * nx + min(gx0, nx - 1));
  }
  // this thread's load slots of every halo plane: byte offsets in the plane; slots
  // outside the grid are zeroed once in every stage and never written again
  unsigned go[NSLOT];
  unsigned in = 0;
#pragma unroll
  for (int j = 0; j < NSLOT; ++j) {
    const int li = tid + j * NT;
    const int ly = li / PW, lx = li - ly * PW;
    const int qx = x0 - 1 + lx, qy = y0 - 1 + ly;
    const bool ok = li < PLN && qx >= 0 && qx < nx && qy >= 0 && qy < ny;
    go[j] = ok ? 8u * (unsigned)(qy * nx + qx) : 0u;
    if (ok) in |= 1u << j;
    if (li < PLN && !ok) {
      for (int s = 0; s < NSTG; ++s) {
#pragma unroll
        for (int r = 0; r < RB; ++r) sX[(s * RB + r) * PLN + li] = mkc<float>(0, 0);
        if constexpr (MODE == M_J2) sD[s * PLN + li] = mkc<float>(0, 0);
      }
    }
  }

  // every slot inside the grid (uniform): only the last one can lie past the tile's plane
  const bool last_ok = tid + (NSLOT - 1) * NT < PLN;
  const bool allin = x0 > 0 && y0 > 0 && x0 + TL::W < nx && y0 + TL::H < ny;
  // group kk (ring stage st): halo plane zb0 - 1 + kk of every right-hand side
  // (and of 1/diag for the Jacobi map); a plane outside the grid is zero
  auto issue = [&](int kk, int st) {
    const int q = zb0 - 1 + kk;
    if ((unsigned)q < (unsigned)nz) {
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const char* src = reinterpret_cast<const char*>(a.x + (long long)(rhs0 + r) * xs + (q - a.xz0) * plane);
        cx<float>* dst = sX + (st * RB + r) * PLN + tid;
        if (allin) {
#pragma unroll
          for (int j = 0; j < NSLOT; ++j)
            if (j < NSLOT - 1 || last_ok) cp8(dst + j * NT, src + go[j]);
        } else {
#pragma unroll
          for (int j = 0; j < NSLOT; ++j)
            if (in >> j & 1) cp8(dst + j * NT, src + go[j]);
        }
      }
      if constexpr (MODE == M_J2) {
        const char* src = reinterpret_cast<const char*>(a.dinv + q * plane);
        cx<float>* dst = sD + st * PLN + tid;
        if (allin) {
#pragma unroll
          for (int j = 0; j < NSLOT; ++j)
            if (j < NSLOT - 1 || last_ok) cp8(dst + j * NT, src + go[j]);
        } else {
#pragma unroll
          for (int j = 0; j < NSLOT; ++j)
            if (in >> j & 1) cp8(dst + j * NT, src + go[j]);
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < NSLOT; ++j)
        if (in >> j & 1) {
#pragma unroll
          for (int r = 0; r < RB; ++r) sX[(st * RB + r) * PLN + tid + j * NT] = mkc<float>(0, 0);
          if constexpr (MODE == M_J2) sD[st * PLN + tid + j * NT] = mkc<float>(0, 0);
        }
    }
    fcp_commit();
  };
  // Jacobi map: y1 / omega = D^-1 g of a landed plane, in place, each thread on
  // the slots it loaded itself
  auto transform = [&](int st) {
#pragma unroll
    for (int j = 0; j < NSLOT; ++j)
      if (allin ? (j < NSLOT - 1 || last_ok) : (in >> j & 1)) {
        const int li = tid + j * NT;
        const cx<float> d = sD[st * PLN + li];
#pragma unroll
        for (int r = 0; r < RB; ++r) sX[(st * RB + r) * PLN + li] = d * sX[(st * RB + r) * PLN + li];
      }
  };

#pragma unroll
  for (int k = 0; k < PREF; ++k) {
    if (k < nplanes) issue(k, k);
    else fcp_commit();
  }
  if constexpr (MODE == M_J2) {
    fcp_wait<PREF - 1>();
    transform(0);
  }

  Column<false> w[RB][NPY][NPX];
  // kappa and own-column values (right-hand side, or what the Jacobi map is added
  // to) of the row completing at the next step: slot = parity of the step that
  // loads them, so that no register move waits for the load
  constexpr bool WANT_G = MODE == M_RESID || MODE == M_JSWEEP || MODE == M_J2;
  float kq[2][NPY][NPX];
  [[maybe_unused]] float2 gq[2][RB][NPY][NPX];
  const cx<float>* gsrc = MODE == M_J2 ? a.base : a.g;
  float nrm2[RB];
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    nrm2[r] = 0.f;
#pragma unroll
    for (int j = 0; j < NPY; ++j)
#pragma unroll
      for (int i = 0; i < NPX; ++i) {
        Column<false>& t = w[r][j][i];
        t.c = t.e = t.k = t.p1 = t.p2 = t.p3 = make_float2(0.f, 0.f);
      }
  }
#pragma unroll
  for (int j = 0; j < NPY; ++j)
#pragma unroll
    for (int i = 0; i < NPX; ++i) {
      kq[0][j][i] = kq[1][j][i] = 0.f;
#pragma unroll
      for (int r = 0; r < RB; ++r) gq[0][r][j][i] = gq[1][r][j][i] = make_float2(0.f, 0.f);
    }
  const float om = a.omega_j, sigma = a.mass_shift.y, inv_l2 = L.inv_ell2;
  int st = 0, stp = NSTG - 1, sti = PREF;  // ring stages of planes k, k - 1 and k + PREF

  auto step = [&](auto Uc, int k) {
    constexpr int U = decltype(Uc)::value, V = 1 - U;  // U = k mod 2
    if constexpr (MODE != M_J2) fcp_wait<PREF - 1>();
    __syncthreads();
    if (k + PREF < nplanes) issue(k + PREF, sti);
    else fcp_commit();
    const int p = zb0 - 2 + k;  // the row that completes with this plane
    const bool fin = k >= 2;
    // (plain loads: a load through the read-only path may be moved past the barrier, down to its use)
    if (k >= 1 && k + 1 < nplanes) {
      const float* kp = L.kappa + (p + 1) * plane;
#pragma unroll
      for (int j = 0; j < NPY; ++j)
#pragma unroll
        for (int i = 0; i < NPX; ++i) kq[U][j][i] = kp[col[j] + i];
      if constexpr (WANT_G) {
        if (gsrc) {
#pragma unroll
          for (int r = 0; r < RB; ++r) {
            const cx<float>* gp = gsrc + (long long)(rhs0 + r) * L.N + (p + 1) * plane;
#pragma unroll
            for (int j = 0; j < NPY; ++j)
#pragma unroll
              for (int i = 0; i < NPX; ++i)
                if (act[j][i]) gq[U][r][j][i] = ldf2(gp + col[j] + i);
          }
        }
      }
    }
    if constexpr (MODE == M_J2) {
      fcp_wait<PREF - 1>();
      if (k + 1 < nplanes) transform(st + 1 == NSTG ? 0 : st + 1);
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      // the plane's rows this thread needs, and their x sums
      const cx<float>* P = sX + (st * RB + r) * PLN + NPY * ty * PW + NPX * tx;
      float2 v[NPY + 2][NPX + 2], hx[NPY + 2][NPX];
#pragma unroll
      for (int q = 0; q < NPY + 2; ++q) {
        static_assert(NPX == 2, "a row's values come as two 128-bit loads");
        const float4 u0 = *reinterpret_cast<const float4*>(P + q * PW);
        const float4 u1 = *reinterpret_cast<const float4*>(P + q * PW + 2);
        v[q][0] = make_float2(u0.x, u0.y);
        v[q][1] = make_float2(u0.z, u0.w);
        v[q][2] = make_float2(u1.x, u1.y);
        v[q][3] = make_float2(u1.z, u1.w);
#pragma unroll
        for (int i = 0; i < NPX; ++i) hx[q][i] = add2(v[q][i], v[q][i + 2]);
      }
#pragma unroll
      for (int j = 0; j < NPY; ++j) {
#pragma unroll
        for (int i = 0; i < NPX; ++i) {
          Sums n;
          n.c = v[j + 1][i + 1];
          n.e = add2(hx[j + 1][i], add2(v[j][i + 1], v[j + 2][i + 1]));
          n.k = add2(hx[j][i], hx[j + 2][i]);
          // the row's weights (before the first row completes: of a row nobody stores)
          const float kap = kq[V][j][i];
          float wt[8];
          row_weights<OPK>(K, tab, kap, wt);
          [[maybe_unused]] const float2 oc = w[r][j][i].c;  // the row's own value
          const float2 h = row_value<OPK, false, false>(wt, kap * kap, inv_l2, sigma, w[r][j][i], n, n.c, n.c, false, n.c, n.c,
                                                        0.f, 0.f);
          if (fin) {
            float2 out;
            if constexpr (MODE == M_APPLY) {
              out = h;
            } else if constexpr (MODE == M_RESID) {
              out = make_float2(gq[V][r][j][i].x - h.x, gq[V][r][j][i].y - h.y);
              if (act[j][i]) nrm2[r] = fmaf(out.x, out.x, fmaf(out.y, out.y, nrm2[r]));
            } else {
              const cx<float> d = MODE == M_J2 ? sD[stp * PLN + (NPY * ty + j + 1) * PW + NPX * tx + i + 1]
                                               : a.dinv[p * plane + col[j] + i];
              if constexpr (MODE == M_J2) {
                out = jacobi2(om, make_float2(d.x, d.y), oc, h);
                out.x += gq[V][r][j][i].x;
                out.y += gq[V][r][j][i].y;
              } else {
                const float rx = gq[V][r][j][i].x - h.x, ry = gq[V][r][j][i].y - h.y;
                out.x = fmaf(om, d.x * rx - d.y * ry, oc.x);
                out.y = fmaf(om, d.x * ry + d.y * rx, oc.y);
              }
            }
            if (act[j][i])
              *reinterpret_cast<float2*>(a.y + (long long)(rhs0 + r) * ys + (p - a.zr0) * plane + col[j] + i) = out;
          }
        }
      }
    }
    stp = st;
    st = (st + 1 == NSTG) ? 0 : st + 1;
    sti = (sti + 1 == NSTG) ? 0 : sti + 1;
  };
  for (int k = 0; k < nplanes; k += 2) {
    step(std::integral_constant<int, 0>{}, k);
    if (k + 1 < nplanes) step(std::integral_constant<int, 1>{}, k + 1);  // uniform across the block
  }
  fcp_wait<0>();

  if constexpr (MODE == M_RESID) reduce_norm<RB>(a, sRed, nrm2, rhs0, bid, nblk);
}

// ----------------------------------------------------------------------------
// the PML-free core, its planes copied by TMA
// ----------------------------------------------------------------------------
// One thread fetches a tile's plane with two tensor copies, signalled on one
// mbarrier per ring stage; a second mbarrier per stage counts the warps that have
// read it, so no block barrier stands in the march (the Jacobi map, which
// transforms each plane in place, keeps one per plane).  Against element-wise
// cp.async this takes a fifth of the instructions out of the compute warps;
// row-wise bulk copies, ten of them per plane, cost their issuing warp more than
// they saved (a copy is a uniform-datapath instruction: a warp issues its lanes'
// copies one after the other).
//
// Rows of nx (odd) 8-byte values have no 16-byte pitch, two rows together have:
// the tensor is the field as lines of two rows, all right-hand sides one after
// the other.  A tile's rows of one parity are then a box of consecutive lines at
// one offset, those of the other parity a second box.  Copies start on a 16-byte
// boundary, so a row sits a = 0 or 1 elements into its shared-memory row; a
// alternates with y and z, and the march alternates two instances of its step.
constexpr int kCoreW = 64;                    // columns of a tile
constexpr unsigned kRowB = 544;               // bytes of a row in shared memory: 68 values

template <int MODE, int NPY, int RB>
struct CoreSmem {
  static constexpr bool J2 = MODE == M_J2, OWN = MODE == M_RESID || MODE == M_JSWEEP;
  static constexpr int H = 4 * NPY, XR = H + 2;
  static constexpr unsigned half = ((XR / 2) * kRowB + 127) & ~127u;  // one box: the rows of one parity
  static constexpr unsigned plane = 2 * half;
  // a stage is refilled one step after every warp has left it
  static constexpr int NSTG = 4, PREF = 2;
  static constexpr unsigned o_d = RB * plane, o_k = o_d + (J2 ? plane : 0), o_g = o_k + NT * NPY * 8;
  static constexpr unsigned stage = (o_g + (OWN ? RB * NPY * NT * 16 : 0) + 127) & ~127u;
  static constexpr unsigned o_bar = NSTG * stage, o_red = o_bar + 2 * NSTG * 8, o_tab = o_red + 32 * 8;
  static constexpr size_t bytes = o_tab + 128;  // and the table, sized at the launch
  static_assert(o_tab % 16 == 0, "");
};
// The tensor maps of one launch (field, 1/diag), their base's offset from the
// 16-byte boundary in elements, and the field's rows per right-hand side.
struct Maps {
  CUtensorMap x, d;
  int sx;
  long long rows;
};

__device__ __forceinline__ bool mbar_try(unsigned b, unsigned ph) {
  unsigned ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(b), "r"(ph)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Once one has given up the thread waits no more (dead, the planes
// asked for by then): the kernel ends with invalid results and the host reports it.
// The limit is a constant: as an argument of the launch it costs the march's J_2 8 %
// (145^3 B 45.0 -> 48.4 us).  A test's waits (a.extra) end sooner.
constexpr unsigned kWaitLimit = 1u << 22, kTestLimit = 4096;  // polls, 64 ns apart
__device__ __forceinline__ void mbar_wait(unsigned b, unsigned ph, int& dead, int armed, const StencilCall<float>& a) {
  if (dead) return;
  for (int i = 0; i < 4; ++i)
    if (mbar_try(b, ph)) return;  // (suspends for a while by itself)
  for (unsigned i = 0; i < kWaitLimit; ++i) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(b), "r"(ph)
        : "memory");
    if (ok) return;
    if (i >= kTestLimit && a.extra) break;
    __nanosleep(64);
  }
  dead = armed;
  if (a.err) atomicExch(a.err, 1);
}
template <int BYTES>
__device__ __forceinline__ void cp_s(unsigned dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(dst), "l"(src), "n"(BYTES));
}
__device__ __forceinline__ void sts64(unsigned a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y));
}

__device__ __forceinline__ void tma_box(unsigned dst, const CUtensorMap* m, int c0, int c1, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(m), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

template <int MODE, int OPK, int NPY, int RB>
__device__ __forceinline__ void core_body(const StencilCall<float>& a, const Maps& mp, unsigned char* smem, int zb0,
                                          int zb1, int x0, int y0, int rx1, int ry1, int rhs0, unsigned bid,
                                          unsigned nblk) {
  using SM = CoreSmem<MODE, NPY, RB>;
  constexpr int NSTG = SM::NSTG, PREF = SM::PREF, XR = SM::XR;
  constexpr bool J2 = SM::J2, OWN = SM::OWN;
  constexpr int NW = OPK == OPK_A ? 4 : 8;
  const LevelView<float>& L = a.lv;
  const unsigned sb = (unsigned)__cvta_generic_to_shared(smem);
  const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
  const int nx = L.nx, nplanes = zb1 - zb0 + 2;
  const long long plane = (long long)nx * L.ny;
  const long long ys = a.ystride > 0 ? a.ystride : L.N;
  const SegK K = tab_seg<OPK>(a);
  load_table<OPK>(a, smem + SM::o_tab);
  const unsigned full = sb + SM::o_bar, empty = full + 8 * NSTG, tab = sb + SM::o_tab;
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < NSTG; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8 * i), "r"(1 + a.extra) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty + 8 * i), "r"(NT / 32) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // Copies of plane k (thread 0).  Global row of the tile's first halo row in
  // plane 0 of right-hand side rhs0; rows of the same parity start at line
  // (row / 2), element (row & 1) nx + x0 - 1 of it.
  // Once a wait of this thread has given up it copies no more: a copy that is only
  // late must not have its stage armed and written a second time.
  int dead = 0;
  const int row0 = (int)(rhs0 * mp.rows) + (zb0 - 1 - a.xz0) * L.ny + y0 - 1;
  const int rowd = (zb0 - 1) * L.ny + y0 - 1;
  auto fetch = [&](int k, int st) {
    const unsigned bar = full + 8 * st, dst = sb + st * SM::stage;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                 "r"((RB + (J2 ? 1 : 0)) * XR * kRowB)
                 : "memory");
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int R = row0 + (int)(r * mp.rows) + k * L.ny + b;
        tma_box(dst + r * SM::plane + b * SM::half, &mp.x, 4 * ((mp.sx + (R & 1) * nx + x0 - 1) >> 1), R >> 1, bar);
      }
    if constexpr (J2) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int R = rowd + k * L.ny + b;
        tma_box(dst + SM::o_d + b * SM::half, &mp.d, 4 * (((R & 1) * nx + x0 - 1) >> 1), R >> 1, bar);
      }
    }
  };
  if (tid == 0)
    for (int k = 0; k < min(PREF, nplanes); ++k) fetch(k, k);

  // this thread's columns (x0 + 2 lane + i, y0 + NPY ty + j); kappa and own values
  // of the row that a plane completes come with it, each thread its own, by
  // cp.async (a ragged tile's threads past its bounds read rows further on, inside
  // the arrays: the core ends before their last plane)
  const int gx0 = x0 + 2 * lane, gy0 = y0 + NPY * ty;
  bool act[NPY][2];
#pragma unroll
  for (int j = 0; j < NPY; ++j) {
    act[j][0] = gx0 <= rx1 && gy0 + j <= ry1;
    act[j][1] = gx0 + 1 <= rx1 && gy0 + j <= ry1;
  }
  const long long own0 = (zb0 - 2) * plane + gy0 * nx + gx0;
  const float* kp = L.kappa + own0;
  const cx<float>* gp = OWN ? a.g + rhs0 * L.N + own0 : nullptr;
  auto own = [&](int st) {
    const unsigned dst = sb + st * SM::stage + SM::o_k + tid * (NPY * 8);
#pragma unroll
    for (int j = 0; j < NPY; ++j) {
      cp_s<4>(dst + 8 * j, kp + j * nx);
      cp_s<4>(dst + 8 * j + 4, kp + j * nx + 1);
    }
    if constexpr (OWN) {
#pragma unroll
      for (int r = 0; r < RB; ++r)
#pragma unroll
        for (int j = 0; j < NPY; ++j) {
          const unsigned d = sb + st * SM::stage + SM::o_g + ((r * NPY + j) * NT + tid) * 16;
          cp_s<8>(d, gp + r * L.N + j * nx);
          cp_s<8>(d + 8, gp + r * L.N + j * nx + 1);
        }
      gp += plane;
    }
    kp += plane;
    fcp_commit();
  };
#pragma unroll
  for (int k = 0; k < PREF; ++k) {
    if (k < nplanes) own(k);
    else fcp_commit();
  }

  // element a of the warp's first halo row in plane 0 (right-hand side rhs0); the
  // rows' places in a stage
  const int a0 = (int)((unsigned)mp.sx + (unsigned)(row0 + NPY * ty) * (unsigned)nx + (unsigned)(x0 - 1)) & 1;
  unsigned xo[NPY + 2];
#pragma unroll
  for (int q = 0; q < NPY + 2; ++q) xo[q] = ((NPY * ty + q) & 1) * SM::half + ((NPY * ty + q) >> 1) * kRowB + 16 * lane;
  cx<float>* yp = a.y + rhs0 * ys + (zb0 - 2 - a.zr0) * plane + gy0 * nx + gx0;
  const float om = a.omega_j, sigma = a.mass_shift.y, inv_l2 = L.inv_ell2;

  // Jacobi map: y1 / omega = D^-1 g of a landed plane, in place
  auto transform = [&](int k, int st) {
    const unsigned xb = sb + st * SM::stage;
    const unsigned px = (unsigned)mp.sx + (unsigned)(row0 + k * L.ny) * (unsigned)nx + (unsigned)(x0 - 1),
                   pd = (unsigned)(rowd + k * L.ny) * (unsigned)nx + (unsigned)(x0 - 1);
    for (int row = ty; row < XR; row += NT / 32) {
      const unsigned ro = xb + (row & 1) * SM::half + (row >> 1) * kRowB + 8 * lane;
      const unsigned ax = 8 * ((px + row * nx) & 1), ad = 8 * ((pd + row * nx) & 1);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (c < 2 || lane < 2) {
          const float2 d = lds64(ro + SM::o_d + ad + 256 * c);
#pragma unroll
          for (int r = 0; r < RB; ++r) {
            const unsigned q = ro + r * SM::plane + (r ? 8 - ax : ax) + 256 * c;
            const float2 g = lds64(q);
            sts64(q, make_float2(d.x * g.x - d.y * g.y, d.x * g.y + d.y * g.x));
          }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before a copy refills the stage
  };

  Column<false> w[RB][NPY][2];
  float nrm2[RB];
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    nrm2[r] = 0.f;
#pragma unroll
    for (int j = 0; j < NPY; ++j)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        Column<false>& t = w[r][j][i];
        t.c = t.e = t.k = t.p1 = t.p2 = t.p3 = make_float2(0.f, 0.f);
      }
  }
  int st = 0;
  unsigned ph = 0;
  if constexpr (J2) {
    mbar_wait(full, 0, dead, min(PREF, nplanes), a);
    transform(0, 0);
  }

  auto step = [&](auto Ac, int k) {
    constexpr int A = decltype(Ac)::value;  // a of this warp's first halo row
    const bool fin = k >= 2;
    const unsigned xb = sb + st * SM::stage;
    const int s2 = st + PREF >= NSTG ? st + PREF - NSTG : st + PREF;
    fcp_wait<PREF - 1>();
    if (k + PREF < nplanes) own(s2);
    else fcp_commit();
    if constexpr (J2) {
      __syncthreads();  // plane k is transformed, every warp has left plane k - 1
      if (tid == 0 && k + PREF < nplanes && !dead) fetch(k + PREF, s2);
      const int sn = st + 1 == NSTG ? 0 : st + 1;
      if (k + 1 < nplanes) {
        mbar_wait(full + 8 * sn, ph ^ (sn == 0), dead, min(k + PREF + 1, nplanes), a);
        transform(k + 1, sn);
      }
    } else {
      if (tid == 0 && k + PREF < nplanes) {
        if (k + PREF >= NSTG)
          mbar_wait(empty + 8 * s2, (unsigned)((k + PREF) / NSTG - 1) & 1, dead, k + PREF, a);
        if (!dead) fetch(k + PREF, s2);
      }
      __syncwarp();
      mbar_wait(full + 8 * st, ph, dead, min(k + PREF + 1, nplanes), a);
    }
    // what the Jacobi map is added to (a ring for it would cost a block per SM)
    [[maybe_unused]] float2 bq[RB][NPY][2];
    if constexpr (J2) {
      if (fin && a.base) {
        const cx<float>* bp = a.base + rhs0 * L.N + own0 + k * plane;
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
          for (int j = 0; j < NPY; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i)
              if (act[j][i]) bq[r][j][i] = ldf2(bp + r * L.N + j * nx + i);
      }
    }
    // weights of the rows that complete; with two right-hand sides once for both
    float kap[NPY][2];
    if constexpr (NPY == 2) {
      const float4 t = lds128(xb + SM::o_k + 16 * tid);
      kap[0][0] = t.x;
      kap[0][1] = t.y;
      kap[NPY - 1][0] = t.z;
      kap[NPY - 1][1] = t.w;
    } else {
      const float2 t = lds64(xb + SM::o_k + 8 * tid);
      kap[0][0] = t.x;
      kap[0][1] = t.y;
    }
    float wt2[RB > 1 ? 2 : 1][NW];
    if constexpr (RB > 1) {
      row_weights<OPK>(K, tab, kap[0][0], wt2[0]);
      row_weights<OPK>(K, tab, kap[0][1], wt2[1]);
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      float2 v[NPY + 2][4], hx[NPY + 2][2];
#pragma unroll
      for (int q = 0; q < NPY + 2; ++q) {
        const unsigned ra = xb + xo[q] + r * SM::plane;
        if ((A ^ q ^ r) & 1) {
          const float4 u = lds128(ra + 16);
          v[q][0] = lds64(ra + 8);
          v[q][1] = make_float2(u.x, u.y);
          v[q][2] = make_float2(u.z, u.w);
          v[q][3] = lds64(ra + 32);
        } else {
          const float4 u0 = lds128(ra), u1 = lds128(ra + 16);
          v[q][0] = make_float2(u0.x, u0.y);
          v[q][1] = make_float2(u0.z, u0.w);
          v[q][2] = make_float2(u1.x, u1.y);
          v[q][3] = make_float2(u1.z, u1.w);
        }
        hx[q][0] = add2(v[q][0], v[q][2]);
        hx[q][1] = add2(v[q][1], v[q][3]);
      }
#pragma unroll
      for (int j = 0; j < NPY; ++j) {
        [[maybe_unused]] float2 gq[2];
        if constexpr (OWN) {
          const float4 t = lds128(xb + SM::o_g + ((r * NPY + j) * NT + tid) * 16);
          gq[0] = make_float2(t.x, t.y);
          gq[1] = make_float2(t.z, t.w);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          Sums n;
          n.c = v[j + 1][i + 1];
          n.e = add2(hx[j + 1][i], add2(v[j][i + 1], v[j + 2][i + 1]));
          n.k = add2(hx[j][i], hx[j + 2][i]);
          float wt1[NW];
          if constexpr (RB == 1) row_weights<OPK>(K, tab, kap[j][i], wt1);
          const float* wt = RB == 1 ? wt1 : wt2[RB == 1 ? 0 : i];
          [[maybe_unused]] const float2 oc = w[r][j][i].c;
          const float2 h = row_value<OPK, false, false>(wt, kap[j][i] * kap[j][i], inv_l2, sigma, w[r][j][i], n, n.c, n.c,
                                                        false, n.c, n.c, 0.f, 0.f);
          if (fin) {
            float2 out = h;
            if constexpr (MODE == M_RESID || MODE == M_JSWEEP) {
              out = make_float2(gq[i].x - h.x, gq[i].y - h.y);
              if constexpr (MODE == M_RESID) {
                if (act[j][i]) nrm2[r] = fmaf(out.x, out.x, fmaf(out.y, out.y, nrm2[r]));
              } else if (act[j][i]) {
                const float2 d = ldf2(a.dinv + own0 + k * plane + j * nx + i);
                out = make_float2(fmaf(om, d.x * out.x - d.y * out.y, oc.x), fmaf(om, d.x * out.y + d.y * out.x, oc.y));
              }
            } else if constexpr (J2) {
              const int sp = st == 0 ? NSTG - 1 : st - 1;
              const unsigned di = ((unsigned)(rowd + (k - 1) * L.ny + NPY * ty + j + 1) * (unsigned)nx + (unsigned)(x0 - 1)) & 1;
              const float2 d = lds64(sb + sp * SM::stage + SM::o_d + xo[j + 1] + 8 * (di + 1 + i));
              out = jacobi2(om, d, oc, h);
              if (a.base) {
                out.x += bq[r][j][i].x;
                out.y += bq[r][j][i].y;
              }
            }
            if (act[j][i]) *reinterpret_cast<float2*>(yp + r * ys + j * nx + i) = out;
          }
        }
      }
    }
    if constexpr (!J2) {
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty + 8 * st) : "memory");
    }
    yp += plane;
    st = st + 1 == NSTG ? 0 : st + 1;
    ph ^= st == 0;
  };
  int k = 0;
  if (a0) step(std::integral_constant<int, 1>{}, k++);
  for (; k < nplanes; k += 2) {
    step(std::integral_constant<int, 0>{}, k);
    if (k + 1 < nplanes) step(std::integral_constant<int, 1>{}, k + 1);
  }
  fcp_wait<0>();
  // A wait of the copying thread gave up: its copies in flight land (bounded, each
  // stage on its own) before the block ends.  A stage's last copy completes the
  // phase of its last plane; a thread that waited for every plane has none left.
  if (tid == 0 && dead) {
    for (int i = 0; i < min(NSTG, dead); ++i) {
      int gone = 0;
      mbar_wait(full + 8 * i, (unsigned)((dead - 1 - i) / NSTG) & 1, gone, 1, a);
    }
  }
  if constexpr (MODE == M_RESID) reduce_norm<RB>(a, reinterpret_cast<double*>(smem + SM::o_red), nrm2, rhs0, bid, nblk);
}

// ----------------------------------------------------------------------------
// PML rows: two columns per thread, tile of w x h columns chosen at the launch
// ----------------------------------------------------------------------------
// FORM 3: y stretched; 1: x stretched, y where a warp meets its PML; 2: any axis
// where a warp meets its PML.  The strips are a few nodes thick, so their tiles
// take the strip's own thickness (a fixed 4-wide tile reads 48-byte row pieces
// and re-reads its halo 1.6 times): w h <= 256, w even, (w + 2)(h + 2) <= kPmlPln.
constexpr int kPmlPln = 384;
constexpr int kSlabW = 32, kSlabH = 8;  // z-PML slabs: the whole x-y range
static_assert((kSlabW + 2) * (kSlabH + 2) <= kPmlPln && kPmlPln <= 3 * NT, "three load slots per thread");
template <int MODE>
struct PmlSmem {
  static constexpr bool J2 = MODE == M_J2, OWN = MODE != M_APPLY;
  // the Jacobi map reads 1/diag of the previous plane and transforms the next
  // one in place, so its ring keeps one more plane than it prefetches
  static constexpr int NSTG = J2 ? 5 : 4, PREF = 3;
  static constexpr unsigned o_d = kPmlPln * 8, o_k = o_d + (J2 ? kPmlPln * 8 : 0), o_g = o_k + NT * 8;
  static constexpr unsigned stage = o_g + (OWN ? NT * 16 : 0);
  static constexpr unsigned o_ez = NSTG * stage, o_red = o_ez + kMaxZb * 16;
  static constexpr unsigned o_tab = o_red + 32 * 8;  // sized at the launch
  static_assert(stage % 16 == 0, "");
};

template <int MODE, int OPK, int FORM>
__device__ __forceinline__ void pml_body(const StencilCall<float>& a, unsigned char* smem, int zb0, int zb1, int x0,
                                         int y0, int tw, int th, int rx1, int ry1, int rhs, unsigned bid,
                                         unsigned nblk) {
  using SM = PmlSmem<MODE>;
  constexpr int NSTG = SM::NSTG, PREF = SM::PREF;
  constexpr bool J2 = SM::J2, OWN = SM::OWN, XC = FORM != 3, ZP = FORM == 2;
  const LevelView<float>& L = a.lv;
  const unsigned sb = (unsigned)__cvta_generic_to_shared(smem);
  float2* sEz = reinterpret_cast<float2*>(smem + SM::o_ez);
  const int tid = threadIdx.x;
  const int nx = L.nx, ny = L.ny, nz = L.nz, nplanes = zb1 - zb0 + 2;
  const int pw = tw + 2, pln = pw * (th + 2);
  const int ty = tid / (tw / 2), tx = 2 * (tid - ty * (tw / 2));
  const long long plane = (long long)nx * ny;
  const long long xs = a.xstride > 0 ? a.xstride : L.N, ys = a.ystride > 0 ? a.ystride : L.N;
  const SegK K = tab_seg<OPK>(a);
  load_table<OPK>(a, smem + SM::o_tab);
  if constexpr (ZP)
    for (int i = tid; i < zb1 - zb0; i += NT) {
      sEz[2 * i] = ldf2(L.eps[2][0] + zb0 + i);
      sEz[2 * i + 1] = ldf2(L.eps[2][1] + zb0 + i);
    }
  // this thread's columns; threads past the tile or its bounds compute columns of
  // the grid that nobody stores
  const bool act0 = ty < th && x0 + tx <= rx1 && y0 + ty <= ry1, act1 = act0 && x0 + tx + 1 <= rx1;
  const int cty = min(ty, th - 1);
  const int gx = min(x0 + tx, nx - 1), gx1 = min(gx + 1, nx - 1), gy = min(y0 + cty, ny - 1);
  const int col = gy * nx + gx;
  // PML factors of the columns: held where every warp needs them, else read where
  // one does (they would cost the others' registers)
  float2 exp_[2], exm_[2], eyp, eym;
  auto load_ex = [&] {
    exp_[0] = ldf2(L.eps[0][0] + gx);
    exm_[0] = ldf2(L.eps[0][1] + gx);
    exp_[1] = ldf2(L.eps[0][0] + gx1);
    exm_[1] = ldf2(L.eps[0][1] + gx1);
  };
  auto load_ey = [&] {
    eyp = ldf2(L.eps[1][0] + gy);
    eym = ldf2(L.eps[1][1] + gy);
  };
  if constexpr (FORM == 1) load_ex();
  if constexpr (FORM == 3) load_ey();
  // (uniform per warp) does it meet the PML of an axis?
  const bool yw = FORM == 3 || __any_sync(0xffffffffu, gy < L.plain_lo[1] || gy > L.plain_hi[1]);
  const bool xw = FORM == 1 || (XC && __any_sync(0xffffffffu, gx < L.plain_lo[0] || gx1 > L.plain_hi[0]));

  // load slots of every halo plane (byte offsets); slots outside the grid are
  // zeroed once in every stage and never written again
  constexpr int NSLOT = (kPmlPln + NT - 1) / NT;
  unsigned go[NSLOT];
  bool in[NSLOT];
#pragma unroll
  for (int j = 0; j < NSLOT; ++j) {
    const int li = tid + j * NT;
    const int ly = li / pw, lx = li - ly * pw;
    const int qx = x0 - 1 + lx, qy = y0 - 1 + ly;
    in[j] = li < pln && qx >= 0 && qx < nx && qy >= 0 && qy < ny;
    go[j] = in[j] ? 8u * (unsigned)(qy * nx + qx) : 0u;
    if (li < pln && !in[j])
      for (int s = 0; s < NSTG; ++s) {
        sts64(sb + s * SM::stage + 8 * li, make_float2(0.f, 0.f));
        if constexpr (J2) sts64(sb + s * SM::stage + SM::o_d + 8 * li, make_float2(0.f, 0.f));
      }
  }
  const cx<float>* gsrc = J2 ? a.base : a.g;
  const char* xp = reinterpret_cast<const char*>(a.x + rhs * xs + (zb0 - 1 - a.xz0) * plane);
  const char* dp = J2 ? reinterpret_cast<const char*>(a.dinv + (zb0 - 1) * plane) : nullptr;
  const float* kp = L.kappa + (zb0 - 2) * plane + col;
  const cx<float>* gp = (OWN && gsrc) ? gsrc + rhs * L.N + (zb0 - 2) * plane + col : nullptr;
  // group k: halo plane zb0 - 1 + k (zero outside the grid), own-column kappa and
  // right-hand side of the row it completes
  auto issue = [&](int k, unsigned so) {
    const unsigned d0 = sb + so + 8 * tid;
    if ((unsigned)(zb0 - 1 + k) < (unsigned)nz) {
#pragma unroll
      for (int j = 0; j < NSLOT; ++j)
        if (in[j]) {
          cp_s<8>(d0 + 8 * NT * j, xp + go[j]);
          if constexpr (J2) cp_s<8>(d0 + SM::o_d + 8 * NT * j, dp + go[j]);
        }
    } else {
#pragma unroll
      for (int j = 0; j < NSLOT; ++j)
        if (in[j]) {
          sts64(d0 + 8 * NT * j, make_float2(0.f, 0.f));
          if constexpr (J2) sts64(d0 + SM::o_d + 8 * NT * j, make_float2(0.f, 0.f));
        }
    }
    if (k >= 2) {
      const unsigned dk = sb + so + SM::o_k + 8 * tid, dg = sb + so + SM::o_g + 16 * tid;
      cp_s<4>(dk, kp);
      cp_s<4>(dk + 4, kp + 1);  // (kappa has a spare element past its end)
      if constexpr (OWN)
        if (gp) {
          if (act0) cp_s<8>(dg, gp);
          if (act1) cp_s<8>(dg + 8, gp + 1);
        }
    }
    xp += 8 * plane;
    if constexpr (J2) dp += 8 * plane;
    kp += plane;
    if constexpr (OWN)
      if (gp) gp += plane;
    fcp_commit();
  };
  // Jacobi map: y1 / omega = D^-1 g of a landed plane, in place, each thread on
  // the slots it loaded itself
  auto transform = [&](unsigned so) {
#pragma unroll
    for (int j = 0; j < NSLOT; ++j)
      if (in[j]) {
        const unsigned q = sb + so + 8 * (tid + NT * j);
        const float2 g = lds64(q), d = lds64(q + SM::o_d);
        sts64(q, make_float2(d.x * g.x - d.y * g.y, d.x * g.y + d.y * g.x));
      }
  };
#pragma unroll
  for (int k = 0; k < PREF; ++k) {
    if (k < nplanes) issue(k, k * SM::stage);
    else fcp_commit();
  }
  if constexpr (J2) {
    fcp_wait<PREF - 1>();
    transform(0);
  }

  Column<true> w[2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
    w[i].c = w[i].e = w[i].k = w[i].p1 = w[i].p2 = w[i].p3 = w[i].A = w[i].B = w[i].BA = w[i].Bm = make_float2(0.f, 0.f);
  float nrm2 = 0.f;
  const float om = a.omega_j, sigma = a.mass_shift.y, inv_l2 = L.inv_ell2;
  const unsigned r0 = sb + 8 * (cty * pw + tx), tab = sb + SM::o_tab;
  cx<float>* yp = a.y + rhs * ys + (zb0 - 2 - a.zr0) * plane + col;
  unsigned so = 0, sop = (NSTG - 1) * SM::stage, soi = PREF * SM::stage;
  auto wrap = [](unsigned s) { return s + SM::stage == NSTG * SM::stage ? 0u : s + SM::stage; };

  auto step = [&](int k) {
    if constexpr (!J2) fcp_wait<PREF - 1>();
    __syncthreads();
    if (k + PREF < nplanes) issue(k + PREF, soi);
    else fcp_commit();
    if constexpr (J2) {
      fcp_wait<PREF - 1>();
      if (k + 1 < nplanes) transform(wrap(so));
    }
    float2 v[3][4], h[3][2], sv[4];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const unsigned qa = r0 + so + 8 * q * pw;
      const float4 u0 = lds128(qa), u1 = lds128(qa + 16);
      v[q][0] = make_float2(u0.x, u0.y);
      v[q][1] = make_float2(u0.z, u0.w);
      v[q][2] = make_float2(u1.x, u1.y);
      v[q][3] = make_float2(u1.z, u1.w);
      h[q][0] = add2(v[q][0], v[q][2]);
      h[q][1] = add2(v[q][1], v[q][3]);
    }
#pragma unroll
    for (int i = XC ? 0 : 1; i < (XC ? 4 : 3); ++i) sv[i] = add2(v[0][i], v[2][i]);
    const bool fin = k >= 2;
    const int p = zb0 - 2 + k;  // the row that completes with this plane
    bool zp = false;
    float2 ezp = make_float2(0.f, 0.f), ezm = ezp;
    if constexpr (ZP) {
      zp = fin && (p < L.plain_lo[2] || p > L.plain_hi[2]);
      if (zp) {
        ezp = sEz[2 * (p - zb0)];
        ezm = sEz[2 * (p - zb0) + 1];
      }
    }
    // in-plane PML corrections
    float2 nA[2], nB[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) nA[i] = nB[i] = make_float2(0.f, 0.f);
    if (yw) {
      if constexpr (FORM != 3) load_ey();
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        cfma2(nA[i], eyp, sub2(v[2][i + 1], v[1][i + 1]));
        cfma2(nA[i], eym, sub2(v[0][i + 1], v[1][i + 1]));
        cfma2(nB[i], eyp, sub2(h[2][i], h[1][i]));
        cfma2(nB[i], eym, sub2(h[0][i], h[1][i]));
      }
    }
    if (XC && xw) {
      if constexpr (FORM != 1) load_ex();
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        cfma2(nA[i], exp_[i], sub2(v[1][i + 2], v[1][i + 1]));
        cfma2(nA[i], exm_[i], sub2(v[1][i], v[1][i + 1]));
        cfma2(nB[i], exp_[i], sub2(sv[i + 2], sv[i + 1]));
        cfma2(nB[i], exm_[i], sub2(sv[i], sv[i + 1]));
      }
    }
    const float2 kap = lds64(sb + so + SM::o_k + 8 * tid);
    float4 gq = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (OWN)
      if (!J2 || gp) gq = lds128(sb + so + SM::o_g + 16 * tid);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      Sums n;
      n.c = v[1][i + 1];
      n.e = add2(h[1][i], sv[i + 1]);
      n.k = add2(h[0][i], h[2][i]);
      const float kp1 = i ? kap.y : kap.x;
      float wt[8], a45[2];
      row_weights<OPK, true>(K, tab, kp1, wt, a45);
      [[maybe_unused]] const float2 oc = w[i].c;  // the row's own value
      const float2 hv = row_value<OPK, true, ZP>(wt, kp1 * kp1, inv_l2, sigma, w[i], n, nA[i], nB[i], zp, ezp, ezm, a45[0], a45[1]);
      if (fin && (i ? act1 : act0)) {
        float2 out = hv;
        if constexpr (OWN) {
          const float2 g = i ? make_float2(gq.z, gq.w) : make_float2(gq.x, gq.y);
          if constexpr (J2) {
            const float2 d = lds64(r0 + sop + SM::o_d + 8 * (pw + 1 + i));
            out = jacobi2(om, d, oc, hv);
            out.x += g.x;
            out.y += g.y;
          } else {
            out = make_float2(g.x - hv.x, g.y - hv.y);
            if constexpr (MODE == M_RESID) {
              nrm2 = fmaf(out.x, out.x, fmaf(out.y, out.y, nrm2));
            } else {
              const float2 d = ldf2(a.dinv + p * plane + col + i);
              out = make_float2(fmaf(om, d.x * out.x - d.y * out.y, oc.x), fmaf(om, d.x * out.y + d.y * out.x, oc.y));
            }
          }
        }
        *reinterpret_cast<float2*>(yp + i) = out;
      }
    }
    yp += plane;
    sop = so;
    so = wrap(so);
    soi = wrap(soi);
  };
  for (int k = 0; k < nplanes; k += 2) {  // (two copies: the state changes registers instead of moving)
    step(k);
    if (k + 1 < nplanes) step(k + 1);
  }
  fcp_wait<0>();
  if constexpr (MODE == M_RESID) reduce_norm<1>(a, reinterpret_cast<double*>(smem + SM::o_red), &nrm2, rhs, bid, nblk);
}

// MB: blocks per SM.  Three, or four where a block carries one row of columns for two
// right-hand sides; the residual of two spills 100 bytes at four, which grids that fill
// the GPU three times over pay for (launch_mode).
template <int MODE, int OPK, int NPY, int RB, int MB>
__global__ void __launch_bounds__(NT, MB) k_march(const __grid_constant__ StencilCall<float> a, const __grid_constant__ Plan pl,
               const __grid_constant__ Maps mp) {
  extern __shared__ __align__(128) unsigned char fsm[];
  const unsigned nb = (unsigned)pl.items;
  const int nf = pl.nfr * a.nrhs;
  if (OPK == OPK_Q || (int)blockIdx.x >= nf) {
    const int ng = a.nrhs / RB, b = (int)blockIdx.x - nf, it = b / ng, rhs0 = (b - it * ng) * RB;
    const int nt = pl.RW * pl.RH;
    const int bz = it / nt, t = it - bz * nt, ty = t / pl.RW, tx = t - ty * pl.RW;
    using TL = CoreT<NPY>;
    const int zb0 = pl.zc0 + bz * pl.zb;
    const int zb1 = min(zb0 + pl.zb, pl.zc1), x0 = pl.fm.px0 + tx * TL::W, y0 = pl.fm.py0 + ty * TL::H;
    const unsigned bid = (unsigned)(pl.nfr + it);
    if constexpr (OPK != OPK_Q) {
      if (pl.rows) {
        core_body<MODE, OPK, NPY, RB>(a, mp, fsm, zb0, zb1, x0, y0, pl.fm.px1, pl.fm.py1, rhs0, bid, nb);
        return;
      }
    }
    tile_body<MODE, OPK, TL, RB>(a, fsm, zb0, zb1, x0, y0, pl.fm.px1, pl.fm.py1, rhs0, bid, nb);
    return;
  }
  if constexpr (OPK != OPK_Q) {
    // PML rows hold more sums per plane: one right-hand side per block
    const int it = (int)blockIdx.x / a.nrhs, rhs = (int)blockIdx.x - it * a.nrhs;
    if (it < pl.nsl) {
      const int nt = pl.SW * pl.SH;
      const int bz = it / nt, t = it - bz * nt, ty = t / pl.SW, tx = t - ty * pl.SW;
      const int zb0 = bz < pl.nlo ? pl.zs0 + bz * pl.zbf : pl.zc1 + (bz - pl.nlo) * pl.zbf;
      pml_body<MODE, OPK, 2>(a, fsm, zb0, min(zb0 + pl.zbf, bz < pl.nlo ? pl.zc0 : pl.zs1), tx * kSlabW, ty * kSlabH,
                             kSlabW, kSlabH, a.lv.nx - 1, a.lv.ny - 1, rhs, it, nb);
      return;
    }
    const int bz = (it - pl.nsl) / pl.fm.count;
    const FrameTile f = decode_frame(pl.fm, it - pl.nsl - bz * pl.fm.count);
    const int zb0 = pl.zc0 + bz * pl.zbf, zb1 = min(zb0 + pl.zbf, pl.zc1);
    if (f.wide) pml_body<MODE, OPK, 3>(a, fsm, zb0, zb1, f.x0, f.y0, pl.fm.ww, pl.fm.wh, f.rx1, f.ry1, rhs, it, nb);
    else pml_body<MODE, OPK, 1>(a, fsm, zb0, zb1, f.x0, f.y0, pl.fm.tw, pl.fm.th, f.rx1, f.ry1, rhs, it, nb);
  }
}

// Dynamic shared memory of a launch: rows of its table without the clamp; the core
// by TMA (tma) or element by element.
template <int MODE, int OPK, int NPY, int RB>
constexpr size_t march_smem(int rows, bool tma) {
  const size_t tab = (size_t)4 * kTabRow<OPK> * (rows + 1);
  const size_t core = (tma ? (size_t)CoreSmem<MODE, NPY, RB>::o_tab : Smem<MODE, CoreT<NPY>, RB>::o_tab) + tab;
  return OPK == OPK_Q ? core : std::max(core, PmlSmem<MODE>::o_tab + tab);
}

}  // namespace march
}  // namespace hz
