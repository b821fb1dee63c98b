// Adjoint 27-point IOFD stencil, the one-sweep Jacobi map, and the dispatch
// of every stencil application (the forward kernels live in hz_fwd.cuh).
//
// Operator (paper Sec. 2.2, Eq. iofd-shell-form / Eq. pml-second-difference):
//   (H x)_i = -ell^-2 sum_j [ abar_j S_j + achk_j D_j ] - s kappa_i^2 ell^-2 (M x)_i
// where, with the transverse weights a4, a5/4, (1-a4-a5)/4 of the row i,
//   T_j(s)  = transverse-weighted sum of x over the plane at offset s along j,
//   S_j     = T_j(+1) + T_j(-1) - 2 T_j(0),   D_j = T_j(+1) - T_j(-1),
//   M x     = a1 N0 + a2/6 N1 + a3/12 N2 + (1-a1-a2-a3)/8 N3 (shell sums N_m),
//   abar_j, achk_j = half sum / half difference of the two PML second-
//   difference weights of row i along j (1 and 0 outside the PML),
//   s = 1 (A_ell) or 1 + i sigma (B_ell, Eq. shifted-iofd-levels).
// Coefficients are evaluated per row from kappa = k ell through the cubic
// Hermite tables at eta* = min(kappa / 2 pi, 0.4) (Eq. iofd-clamped-coordinate).
//
#include <algorithm>
#include <cstdio>
#include <vector>

#include "hz_fwd_launch.cuh"

namespace hz {

// the forward kernels are instantiated in hz_fwd.cu
extern template void launch_fwd<double, M_APPLY>(const StencilCall<double>&, int, cudaStream_t);
extern template void launch_fwd<double, M_RESID>(const StencilCall<double>&, int, cudaStream_t);
extern template void launch_fwd<double, M_J2>(const StencilCall<double>&, int, cudaStream_t);
extern template void launch_fwd<double, M_JSWEEP>(const StencilCall<double>&, int, cudaStream_t);
extern template void launch_fwd<double, M_AWIN>(const StencilCall<double>&, int, cudaStream_t);
extern template void fwd_init_attrs<double, M_APPLY>();
extern template void fwd_init_attrs<double, M_RESID>();
extern template void fwd_init_attrs<double, M_J2>();
extern template void fwd_init_attrs<double, M_JSWEEP>();
extern template void fwd_init_attrs<double, M_AWIN>();

// tiles of the adjoint kernel: 32 x 8 columns, 8 x 8 on very small grids
template <int TX_, int TY_>
struct ATile {
  static constexpr int TX = TX_, TY = TY_, NT = TX_ * TY_, PW = TX_ + 2, PLANE = PW * (TY_ + 2);
};
using ATileL = ATile<32, 8>;
using ATileS = ATile<8, 8>;

// ----------------------------------------------------------------------------
// adjoint kernel
// ----------------------------------------------------------------------------
// (H^H x)_i = sum_j conj(H_j(i - j)) x_j: every source node j spreads its own
// row's weights.  With C_m the shell weights of row j, t_0..t_2 its transverse
// weights and eps the PML factors, node j is turned once into u_m = conj(C_m) x
// (m = 0..3) and, near a PML, v_c = t_c x (c = 0..2); plane q then contributes
//   to its own rows   c(u_0) + e(u_1) + k(u_2),
//   to rows q +- 1    c(u_1) + e(u_2) + k(u_3)
// (c, e, k: centre, face and corner sums over the in-plane neighbours), and each
// stretched axis adds the same sums of the v's along it,
//   conj(eps+(j)) from the node at offset -1, conj(eps-(j)) from that at +1,
//   -conj(eps+ + eps-) from the row's own position.
// A block of 32 x 8 columns marches in z: each plane's nodes with their halo are
// loaded one plane ahead, turned into the u's and v's in shared memory (two
// buffers, one barrier per plane) and summed; a column keeps the partial sums of
// two rows.  Evaluating the weights once per node instead of once per neighbour
// (27 complex coefficients per output node) is what it gains: bound by issue in
// single precision and by the FP64 rate in double.
constexpr int kAdjF = 7;  // fields in shared memory: u_0..u_3, v_0..v_2
template <class R, class AT>
struct AdjSmem {
  static constexpr size_t o_tab = (size_t)2 * kAdjF * AT::PLANE * sizeof(cx<R>);
  static size_t bytes(int opk, int ns) {
    return o_tab + sizeof(R) * (opk == OPK_Q ? (size_t)kCtQ : (size_t)(kCtCA + kCtK + kCtT)) * ns;
  }
};

template <class R, int MODE, int OPK, bool GEN, class AT>
__device__ __forceinline__ void adj_tile(const StencilCall<R>& a, unsigned char* smem, double* sRed, int zblock,
                                         int tiles_x) {
  constexpr bool Q = OPK == OPK_Q, B = OPK == OPK_B;
  constexpr int TX = AT::TX, TY = AT::TY, NT = AT::NT, PW = AT::PW, PLANE = AT::PLANE;
  const LevelView<R>& L = a.lv;
  cx<R>* sF = reinterpret_cast<cx<R>*>(smem);
  R* sT = reinterpret_cast<R*>(smem + AdjSmem<R, AT>::o_tab);
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int ns = a.tab.nseg + 1;
  const R ds = a.tab.ds, inv_ds = a.tab.inv_ds;
  if constexpr (Q) {
    for (int i = tid; i < kCtQ * ns; i += NT) sT[i] = L.ctab[ct_off_Q(ns) + i];
  } else {
    for (int i = tid; i < (kCtCA + kCtK + kCtT) * ns; i += NT) sT[i] = L.ctab[i];
  }
  const int rhs = blockIdx.x % a.nrhs, tile_x = blockIdx.x / a.nrhs;
  const int x0 = tile_x * TX, y0 = blockIdx.y * TY;
  const int nx = L.nx, ny = L.ny, nz = L.nz;
  const int zb0 = blockIdx.z * zblock, zb1 = min(zb0 + zblock, nz);
  const int plane = nx * ny;
  const cx<R>* X = a.x + rhs * L.N;
  const int gx = x0 + tx, gy = y0 + ty;
  const bool active = gx < nx && gy < ny;
  const R sigma = a.mass_shift.y, om = a.omega_j;

  // PML factors along x and y as this column meets them
  const cx<R> zero = mkc<R>(0, 0);
  cx<R> xm = zero, xp = zero, xc = zero, ym = zero, yp = zero, yc = zero;
  bool xw = false, yw = false;
  if constexpr (GEN) {
    xw = x0 - 1 < L.plain_lo[0] || x0 + TX > L.plain_hi[0];
    yw = y0 - 1 < L.plain_lo[1] || y0 + TY > L.plain_hi[1];
    const int xi = min(gx, nx - 1), yi = min(gy, ny - 1);
    xm = conjc(L.eps[0][0][max(xi - 1, 0)]);
    xp = conjc(L.eps[0][1][min(xi + 1, nx - 1)]);
    xc = conjc(L.eps[0][0][xi] + L.eps[0][1][xi]);
    ym = conjc(L.eps[1][0][max(yi - 1, 0)]);
    yp = conjc(L.eps[1][1][min(yi + 1, ny - 1)]);
    yc = conjc(L.eps[1][0][yi] + L.eps[1][1][yi]);
  }

  // this thread's (at most two) nodes of every halo plane, one plane ahead in registers
  int go[2];
  bool in[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int li = tid + j * NT, ly = li / PW, lx = li - ly * PW;
    const int qx = x0 - 1 + lx, qy = y0 - 1 + ly;
    in[j] = li < PLANE && qx >= 0 && qx < nx && qy >= 0 && qy < ny;
    go[j] = in[j] ? qy * nx + qx : 0;
  }
  cx<R> xv[2], dv[2];
  R kv[2];
  auto load = [&](int z) {
    const bool zin = (unsigned)z < (unsigned)nz;
    const long long o = zin ? (long long)z * plane : 0;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const bool ok = zin && in[j];
      xv[j] = ok ? X[o + go[j]] : zero;
      kv[j] = ok ? L.kappa[o + go[j]] : (R)0;
      if constexpr (MODE == M_J2) dv[j] = ok ? a.dinv[o + go[j]] : zero;
    }
  };
  auto stage = [&](int buf) {
    cx<R>* F = sF + (size_t)buf * kAdjF * PLANE;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int li = tid + j * NT;
      if (j && li >= PLANE) break;
      cx<R> v = xv[j];
      if constexpr (MODE == M_J2) v = cjmul(dv[j], v);  // y1 / omega = D^-H g
      R u, C[4];
      const int seg = seg_exact(kv[j], ns, ds, inv_ds, u);
      if constexpr (Q) {
        horner_pm<R, 4, 3>(sT + seg * kCtQ, u, C);
#pragma unroll
        for (int m = 0; m < 4; ++m) F[m * PLANE + li] = C[m] * v;
      } else {
        horner_pm<R, 4, 5>(sT + seg * kCtCA, u, C);
        if constexpr (B) {
          // conj(C - i sigma K) x
          R Km[4];
          horner_pm<R, 4, 5>(sT + ct_off_K(ns) + seg * kCtK, u, Km);
#pragma unroll
          for (int m = 0; m < 4; ++m) F[m * PLANE + li] = mkc<R>(C[m], sigma * Km[m]) * v;
        } else {
#pragma unroll
          for (int m = 0; m < 4; ++m) F[m * PLANE + li] = C[m] * v;
        }
        if constexpr (GEN) {
          const RowT<R> t = eval_t(sT + ct_off_T(ns), seg, u);
          F[4 * PLANE + li] = t.a4 * v;
          F[5 * PLANE + li] = t.q5 * v;
          F[6 * PLANE + li] = t.qb * v;
        }
      }
    }
  };

  R nrm2 = 0;
  const bool want_norm = MODE == M_RESID && a.red.out != nullptr;
  cx<R> pa = zero, pb = zero;  // rows q - 1 and q so far
  load(zb0 - 1);
  __syncthreads();  // table
  const int lc = (ty + 1) * PW + tx + 1;
  for (int q = zb0 - 1; q <= zb1; ++q) {
    const int buf = (q - zb0 + 1) & 1;
    stage(buf);
    if (q < zb1) load(q + 1);
    __syncthreads();
    const cx<R>* F = sF + (size_t)buf * kAdjF * PLANE + lc;
    auto face = [&](const cx<R>* f) { return (f[-1] + f[1]) + (f[-PW] + f[PW]); };
    auto corner = [&](const cx<R>* f) { return (f[-PW - 1] + f[-PW + 1]) + (f[PW - 1] + f[PW + 1]); };
    // (the small terms first: one rounding at the size of the large one)
    cx<R> p0 = (corner(F + 2 * PLANE) + face(F + PLANE)) + F[0];
    cx<R> p1 = (corner(F + 3 * PLANE) + face(F + 2 * PLANE)) + F[PLANE];
    cx<R> pm = p1, pp = p1;
    if constexpr (GEN) {
      const cx<R>*v0 = F + 4 * PLANE, *v1 = F + 5 * PLANE, *v2 = F + 6 * PLANE;
      cx<R> s0 = zero, s1 = zero;
      if (xw) {
        auto X0 = [&](int d) { return v0[d] + (v1[d - PW] + v1[d + PW]); };
        auto X1 = [&](int d) { return v1[d] + (v2[d - PW] + v2[d + PW]); };
        s0 += xm * X0(-1) + xp * X0(1) - xc * X0(0);
        s1 += xm * X1(-1) + xp * X1(1) - xc * X1(0);
      }
      if (yw) {
        auto Y0 = [&](int d) { return v0[d] + (v1[d - 1] + v1[d + 1]); };
        auto Y1 = [&](int d) { return v1[d] + (v2[d - 1] + v2[d + 1]); };
        s0 += ym * Y0(-PW) + yp * Y0(PW) - yc * Y0(0);
        s1 += ym * Y1(-PW) + yp * Y1(PW) - yc * Y1(0);
      }
      p0 += s0;
      pm += s1;
      pp += s1;
      if ((unsigned)q < (unsigned)nz && (q < L.plain_lo[2] || q > L.plain_hi[2])) {
        const cx<R> ep = L.eps[2][0][q], em = L.eps[2][1][q];
        const cx<R> Z = v0[0] + face(v1) + corner(v2);
        pp += conjc(ep) * Z;  // to row q + 1
        pm += conjc(em) * Z;  // to row q - 1
        p0 -= conjc(ep + em) * Z;
      }
    }
    if (q > zb0 && active) {  // row q - 1 is complete
      const cx<R> h = pa + pm;
      const long long idx = (long long)(q - 1) * plane + gy * nx + gx;
      cx<R> out = h;
      if constexpr (MODE == M_RESID) {
        out = a.g[rhs * L.N + idx] - h;
        if (want_norm) nrm2 += abs2(out);
      } else if constexpr (MODE == M_J2) {
        // with y1 = omega D^-H g and h = H^H y1 / omega:
        // y1 + omega D^-H (g - H^H y1) = omega D^-H (2 g - omega h)
        out = om * cjmul(a.dinv[idx], (R)2 * X[idx] - om * h);
        if (a.base) out += a.base[rhs * L.N + idx];
      } else if constexpr (MODE == M_JSWEEP) {
        out = X[idx] + om * cjmul(a.dinv[idx], a.g[rhs * L.N + idx] - h);
      }
      a.y[rhs * L.N + idx] = out;
    }
    pa = pb + p0;
    pb = pp;
  }
  if constexpr (MODE == M_RESID) {
    if (a.red.out) {
      double s = block_sum((double)nrm2, sRed, tid, NT);
      const unsigned nblk = (unsigned)(tiles_x * gridDim.y * gridDim.z);
      const unsigned bid = (unsigned)(tile_x + tiles_x * (blockIdx.y + gridDim.y * blockIdx.z));
      if (tid == 0) a.red.partial[(size_t)rhs * nblk + bid] = s;
      if (last_block_arrive(a.red.count + rhs, nblk, tid)) {
        double t = 0.0;
        for (unsigned b = tid; b < nblk; b += NT) t += __ldcg(a.red.partial + (size_t)rhs * nblk + b);
        t = block_sum(t, sRed, tid, NT);
        if (tid == 0) {
          a.red.out[rhs] = t;
          if (a.red.root) a.red.root[rhs] = sqrt(t);
          if (a.red.inv_root) a.red.inv_root[rhs] = t > 1e-300 ? 1.0 / sqrt(t) : 0.0;
          a.red.count[rhs] = 0;
        }
      }
    }
  }
}

template <class R, int MODE, int OPK, class AT>
__global__ void __launch_bounds__(AT::NT, (sizeof(R) == 4 ? 3 : 1) * (256 / AT::NT)) k_adj(StencilCall<R> a, int zblock, int tiles_x) {
  constexpr int TX = AT::TX, TY = AT::TY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sRed[32];
  if constexpr (OPK == OPK_Q) {
    adj_tile<R, MODE, OPK, false, AT>(a, smem_raw, sRed, zblock, tiles_x);
  } else {
    // a source node in the PML of any axis, the halo's included?
    const LevelView<R>& L = a.lv;
    const int x0 = (blockIdx.x / a.nrhs) * TX, y0 = blockIdx.y * TY;
    const int zb0 = blockIdx.z * zblock, zb1 = min(zb0 + zblock, L.nz);
    const bool plain = x0 - 1 >= L.plain_lo[0] && x0 + TX <= L.plain_hi[0] && y0 - 1 >= L.plain_lo[1] &&
                       y0 + TY <= L.plain_hi[1] && zb0 - 1 >= L.plain_lo[2] && zb1 <= L.plain_hi[2];
    if (plain) adj_tile<R, MODE, OPK, false, AT>(a, smem_raw, sRed, zblock, tiles_x);
    else adj_tile<R, MODE, OPK, true, AT>(a, smem_raw, sRed, zblock, tiles_x);
  }
}

// One Jacobi sweep from zero: y = omega D^-1 g (pointwise; forward or adjoint).
template <class R>
__global__ void k_j1(StencilCall<R> a, int adjoint) {
  const LevelView<R>& L = a.lv;
  const long long n = L.N * a.nrhs;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    long long i = t % L.N;
    int x = (int)(i % L.nx);
    int y = (int)((i / L.nx) % L.ny);
    int z = (int)(i / ((long long)L.nx * L.ny));
    R kap = L.kappa[i];
    R av[5];
    table_eval<R, 0, 5>(a.tab.coef, a.tab.nseg, a.tab.ds, a.tab.inv_ds, eta_star(kap), av);
    cx<R> sab = L.abar[0][x] + L.abar[1][y] + L.abar[2][z];
    cx<R> D = L.inv_ell2 * ((R)2 * av[3] * sab) - (L.inv_ell2 * kap * kap * av[0]) * a.mass_shift;
    if (adjoint) D = conjc(D);
    cx<R> out = a.omega_j * cdiv(a.x[t], D);
    if (a.base) out += a.base[t];
    a.y[t] = out;
  }
}


// ----------------------------------------------------------------------------
// launchers
// ----------------------------------------------------------------------------
// tiling of the adjoint kernel over the whole grid (zblock > 0 forces it)
struct AdjPlan {
  int tw, th, zb, nx, ny, nz;  // tile, planes per block, blocks per axis
};
static AdjPlan adj_plan(int nx, int ny, int nz, int nrhs, int zblock = 0) {
  AdjPlan p;
  const bool small = (long long)nx * ny * nz <= kSmallNodes;
  p.tw = small ? ATileS::TX : ATileL::TX;
  p.th = small ? ATileS::TY : ATileL::TY;
  p.nx = (nx + p.tw - 1) / p.tw;
  p.ny = (ny + p.th - 1) / p.th;
  const long long tiles = (long long)p.nx * p.ny * nrhs, want = 152LL * 2 * 4, nzb = (want + tiles - 1) / tiles;
  p.zb = small ? kMinZblock : std::min(std::max((int)((nz + nzb - 1) / nzb), 4), kMaxZb);
  if (zblock > 0) p.zb = zblock;
  p.nz = (nz + p.zb - 1) / p.zb;
  return p;
}

template <class R, int MODE, int OPK, class AT>
static void launch_adj_at(const StencilCall<R>& c, const AdjPlan& p, cudaStream_t s) {
  count_launch();
  k_adj<R, MODE, OPK, AT><<<dim3(p.nx * c.nrhs, p.ny, p.nz), dim3(AT::TX, AT::TY),
                            AdjSmem<R, AT>::bytes(OPK, c.tab.nseg + 1), s>>>(c, p.zb, p.nx);
}
template <class R, int MODE, int OPK>
static void launch_adj_t(const StencilCall<R>& c, cudaStream_t s) {
  const AdjPlan p = adj_plan(c.lv.nx, c.lv.ny, c.lv.nz, c.nrhs);
  if (p.tw == ATileS::TX) launch_adj_at<R, MODE, OPK, ATileS>(c, p, s);
  else launch_adj_at<R, MODE, OPK, ATileL>(c, p, s);
}

// forward operator kind of a call: A (real shell coefficients) unless the mass
// is shifted, B otherwise
template <class R>
static int fwd_opk(const StencilCall<R>& c, int op) {
  if (op == OP_Q) return OPK_Q;
  return (c.mass_shift.x == (R)1 && c.mass_shift.y == (R)0) ? OPK_A : OPK_B;
}

template <class R>
void launch_stencil(const StencilCall<R>& c, int mode, int op, bool adjoint, cudaStream_t s) {
  if (mode == M_J1) {
    long long n = c.lv.N * c.nrhs;
    int blocks = (int)std::min<long long>((n + 255) / 256, 152LL * 16);
    count_launch();
    k_j1<R><<<blocks, 256, 0, s>>>(c, adjoint ? 1 : 0);
    return;
  }
  if (!adjoint) {
    const int opk = fwd_opk(c, op);
    if constexpr (sizeof(R) == sizeof(float)) {
      if (mode == M_AWIN || march::takes(c.lv, mode, opk == OPK_B, c.nrhs)) march::launch(c, mode, opk, s);
      else gather::launch_fwd_gather(c, mode, op, s);
    } else if (mode != M_AWIN && (c.lv.level > 0 || c.lv.N <= kSmallNodes)) {
      gather::launch_fwd_gather(c, mode, op, s);
    } else if (op == OP_Q) {
      launch_fwd<R, M_APPLY>(c, opk, s);
    } else {
      switch (mode) {
        case M_APPLY: launch_fwd<R, M_APPLY>(c, opk, s); break;
        case M_RESID: launch_fwd<R, M_RESID>(c, opk, s); break;
        case M_J2: launch_fwd<R, M_J2>(c, opk, s); break;
        case M_JSWEEP: launch_fwd<R, M_JSWEEP>(c, opk, s); break;
        case M_AWIN: launch_fwd<R, M_AWIN>(c, opk, s); break;
      }
    }
  } else {
    const int opk = fwd_opk(c, op);
    if (opk == OPK_Q) {
      launch_adj_t<R, M_APPLY, OPK_Q>(c, s);
      return;
    }
    const bool b = opk == OPK_B;
    switch (mode) {
      case M_APPLY: b ? launch_adj_t<R, M_APPLY, OPK_B>(c, s) : launch_adj_t<R, M_APPLY, OPK_A>(c, s); break;
      case M_RESID: b ? launch_adj_t<R, M_RESID, OPK_B>(c, s) : launch_adj_t<R, M_RESID, OPK_A>(c, s); break;
      case M_J2: b ? launch_adj_t<R, M_J2, OPK_B>(c, s) : launch_adj_t<R, M_J2, OPK_A>(c, s); break;
      case M_JSWEEP: b ? launch_adj_t<R, M_JSWEEP, OPK_B>(c, s) : launch_adj_t<R, M_JSWEEP, OPK_A>(c, s); break;
    }
  }
}

// Blocks per right-hand side of a forward stencil launch on this grid (the
// size of the per-block partial-sum array its fused reductions need).
long long stencil_blocks_per_rhs(int level, int nx, int ny, int nz, const int* plain_lo, const int* plain_hi,
                                 int nrhs, int zblock, int zblock_f) {
  if (level > 0 || (long long)nx * ny * nz <= kSmallNodes)
    return gather::gather_blocks_per_rhs(false, nx, ny, nz, plain_lo, plain_hi, nrhs, zblock, zblock_f);
  const int zb = zblock > 0 ? zblock : choose_zblock(nx, ny, nz, nrhs);
  const FwdPlan p = plan_layout(nx, ny, nz, plain_lo, plain_hi, true, zb, zblock_f);
  return p.blocks();
}

// Blocks per right-hand side of an adjoint stencil launch with nrhs
// right-hand sides (zblock > 0: that z-block instead of the launch's own).
long long adj_blocks_per_rhs(int nx, int ny, int nz, int nrhs, int zblock) {
  const AdjPlan p = adj_plan(nx, ny, nz, nrhs, zblock);
  return (long long)p.nx * p.ny * p.nz;
}

// Host replay of the forward launch layout and of the kernels' block and
// thread decode (the plan, the frame tile decode, the thread-to-column map of
// each tile shape, the z-block of every block, the row form each tile takes
// and its block id for fused reductions).  Violations counted: a written
// column outside the grid, a column outside the PML-free range on a row form
// that drops that axis's PML corrections (form 0 both axes, form 1 y, form 3
// x), a block id out of range or repeated.  (The kernels use forms 0, 2, 3.)  counts (nx * ny * nz bytes, or
// null) receives how often each node of right-hand side 0 is written,
// saturating at 255.
long long replay_fwd_layout(int level, int nx, int ny, int nz, const int* plo, const int* phi, int op, int nrhs,
                            int zblock, int zblock_f, unsigned char* counts, long long* blocks) {
  // the single-precision launches have layouts of their own (march, or gather where
  // no mode or not every mode marches)
  long long single = march::replay_layout(nx, ny, nz, plo, phi, op, nrhs, zblock, zblock_f);
  if (!march::takes(M_J2, true, nx, ny, nz, nrhs, plo, phi) || !march::takes(M_J2, false, nx, ny, nz, nrhs, plo, phi))
    single += gather::replay_gather_layout(true, nx, ny, nz, plo, phi, op, nrhs, zblock, zblock_f, nullptr, nullptr);
  if (level > 0 || (long long)nx * ny * nz <= kSmallNodes)
    return single + gather::replay_gather_layout(false, nx, ny, nz, plo, phi, op, nrhs, zblock, zblock_f, counts, blocks);
  const bool ab = op == OP_AB;
  const int zb = zblock > 0 ? zblock : choose_zblock(nx, ny, nz, nrhs);
  const FwdPlan p = plan_layout(nx, ny, nz, plo, phi, ab, zb, zblock_f);
  const long long nblk = p.blocks();
  if (blocks) *blocks = nblk;
  std::vector<unsigned char> seen((size_t)nblk, 0);
  long long bad = single;
  auto plain_x = [&](int x) { return x >= plo[0] && x <= phi[0]; };
  auto plain_y = [&](int y) { return y >= plo[1] && y <= phi[1]; };
  // one block of a tile shape (npx columns per thread, txt x tyt threads)
  auto cta = [&](int npx, int txt, int tyt, int x0, int y0, int rx1, int ry1, int form, int zbk, int bz,
                 long long bid) {
    if (bid < 0 || bid >= nblk || seen[(size_t)bid]++) ++bad;
    const int zb0 = bz * zbk, zb1 = std::min(zb0 + zbk, nz);
    for (int tid = 0; tid < txt * tyt; ++tid) {
      const int tx = tid % txt, ty = tid / txt;
      for (int i = 0; i < npx; ++i) {
        const int gx = x0 + npx * tx + i, gy = y0 + ty;
        if (!(gx <= rx1 && gy <= ry1)) continue;  // inactive column
        if (gx < 0 || gy < 0 || gx >= nx || gy >= ny) {
          ++bad;
          continue;
        }
        if (ab && ((form == 0 && !(plain_x(gx) && plain_y(gy))) || (form == 1 && !plain_y(gy)) ||
                   (form == 3 && !plain_x(gx))))
          ++bad;
        if (counts)
          for (int z = zb0; z < zb1; ++z) {
            unsigned char& c = counts[((size_t)z * ny + gy) * nx + gx];
            if (c < 255) ++c;
          }
      }
    }
  };
  const TileMap& m = p.frame;
  const int rnpx = p.ss ? Shapes<1>::Rect::NPX : Shapes<0>::Rect::NPX;
  const int wnpx = p.ss == 2 ? Shapes<2>::Wide::NPX : (p.ss ? Shapes<1>::Wide::NPX : Shapes<0>::Wide::NPX);
  const int tnpx = p.ss == 2 ? Shapes<2>::Tall::NPX : Shapes<0>::Tall::NPX;
  if (!p.split) {
    for (int bz = 0; bz < p.nzb; ++bz)
      for (int by = 0; by < p.GH; ++by)
        for (int t = 0; t < p.GW; ++t) {
          const int x0 = t * m.rw, y0 = by * m.rh;
          const int form = ab ? (grid_tile_form(x0, y0, m.rw, m.rh, nx, ny, plo, phi) == 0 ? 0 : 2) : 0;
          cta(rnpx, m.rw / rnpx, m.rh, x0, y0, nx - 1, ny - 1, form, p.zb, bz, t + (long long)p.GW * (by + p.GH * bz));
        }
  } else {
    // split: rectangle blocks numbered first, then the frame's; fused (one
    // launch): per z-block, the rectangle tiles and then the frame tiles
    const int px0 = p.frame.px0, py0 = p.frame.py0;
    const long long nrect = (long long)p.RW * p.RH, per_z = nrect + p.frame.count;
    for (int bz = 0; bz < p.nzb; ++bz)
      for (int by = 0; by < p.RH; ++by)
        for (int t = 0; t < p.RW; ++t)
          cta(rnpx, m.rw / rnpx, m.rh, px0 + t * m.rw, py0 + by * m.rh, p.frame.px1, p.frame.py1, 0, p.zb, bz,
              p.fused ? t + (long long)p.RW * by + per_z * bz : t + (long long)p.RW * (by + p.RH * bz));
    const long long off = (long long)p.RW * p.RH * p.nzb;
    for (int bz = 0; bz < p.nzbf; ++bz)
      for (int t = 0; t < p.frame.count; ++t) {
        const FrameTile f = decode_frame(p.frame, t);
        const long long bid = p.fused ? nrect + t + per_z * bz : off + t + (long long)p.frame.count * bz;
        if (f.wide)
          cta(wnpx, m.ww / wnpx, m.wh, f.x0, f.y0, f.rx1, f.ry1, 3, p.zbf, bz, bid);
        else
          cta(tnpx, m.tw / tnpx, m.th, f.x0, f.y0, f.rx1, f.ry1, 2, p.zbf, bz, bid);
      }
  }
  for (unsigned char v : seen)
    if (v != 1) ++bad;
  return bad;
}

// Host replay of the adjoint launch layout (tiles of adj_plan over the whole grid,
// adj_zblock planes per block unless zblock > 0): per-node write counts of
// right-hand side 0 (or null) and the blocks per right-hand side.
long long replay_adj_layout(int nx, int ny, int nz, int nrhs, int zblock, unsigned char* counts, long long* blocks) {
  const AdjPlan p = adj_plan(nx, ny, nz, nrhs, zblock);
  if (blocks) *blocks = (long long)p.nx * p.ny * p.nz;
  if (counts)
    for (int bz = 0; bz < p.nz; ++bz)
      for (int by = 0; by < p.ny; ++by)
        for (int bx = 0; bx < p.nx; ++bx)
          for (int t = 0; t < p.tw * p.th; ++t) {
            const int gx = bx * p.tw + t % p.tw, gy = by * p.th + t / p.tw;
            if (gx >= nx || gy >= ny) continue;
            for (int z = bz * p.zb; z < std::min(bz * p.zb + p.zb, nz); ++z) {
              unsigned char& c = counts[((size_t)z * ny + gy) * nx + gx];
              if (c < 255) ++c;
            }
          }
  return 0;
}

template <class R, int MODE, int OPK>
static void set_adj_attr() {
  cudaFuncSetAttribute(k_adj<R, MODE, OPK, ATileL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)AdjSmem<R, ATileL>::bytes(OPK, kMaxSeg + 1));
  cudaFuncSetAttribute(k_adj<R, MODE, OPK, ATileS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)AdjSmem<R, ATileS>::bytes(OPK, kMaxSeg + 1));
}
template <class R>
static void set_adj_attrs() {
  set_adj_attr<R, M_APPLY, OPK_A>();
  set_adj_attr<R, M_RESID, OPK_A>();
  set_adj_attr<R, M_J2, OPK_A>();
  set_adj_attr<R, M_JSWEEP, OPK_A>();
  set_adj_attr<R, M_APPLY, OPK_B>();
  set_adj_attr<R, M_RESID, OPK_B>();
  set_adj_attr<R, M_J2, OPK_B>();
  set_adj_attr<R, M_JSWEEP, OPK_B>();
  set_adj_attr<R, M_APPLY, OPK_Q>();
}

// Opt the stencil kernels into more than 48 KB of dynamic shared memory where
// they need it.  Called before any launch and outside stream capture.
void init_kernel_attributes() {
  set_adj_attrs<float>();
  set_adj_attrs<double>();
  march::init_attrs();
  fwd_init_attrs<double, M_APPLY>();
  fwd_init_attrs<double, M_RESID>();
  fwd_init_attrs<double, M_J2>();
  fwd_init_attrs<double, M_JSWEEP>();
  fwd_init_attrs<double, M_AWIN>();
}

template void launch_stencil<float>(const StencilCall<float>&, int, int, bool, cudaStream_t);
template void launch_stencil<double>(const StencilCall<double>&, int, int, bool, cudaStream_t);

}  // namespace hz
