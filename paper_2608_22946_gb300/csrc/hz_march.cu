// Launch layout, launchers and host replay of the single-precision forward
// stencil (hz_march.cuh).  Compiled once per part with -DHZ_MARCH_PART=0..3 so
// that its kernels build in parallel; part 0 also holds the dispatch.
#include <vector>

#include "hz_march.cuh"
#include "hz_fwd_launch.cuh"

#ifndef HZ_MARCH_PART
#error "compile with -DHZ_MARCH_PART=<0..3>"
#endif

namespace hz {
namespace march {

// Rows [z0, z1) of one application; npy: rows of columns per thread.
static Plan make_plan(int nx, int ny, const int* plo, const int* phi, const int* strip, bool ab, int zb, int zbf,
                      int npy, int z0, int z1) {
  Plan p;
  p.zb = std::min(zb, kMaxZb);
  p.zbf = std::min(zbf > 0 ? zbf : zb, kMaxZb);
  TileMap& f = p.fm;
  f.nx = nx;
  f.ny = ny;
  f.px0 = ab ? std::max(plo[0], 0) : 0;
  f.px1 = ab ? std::min(phi[0], nx - 1) : nx - 1;
  f.py0 = ab ? std::max(plo[1], 0) : 0;
  f.py1 = ab ? std::min(phi[1], ny - 1) : ny - 1;
  p.zs0 = z0;
  p.zs1 = z1;
  p.zc0 = ab ? std::min(std::max(plo[2], z0), z1) : z0;
  p.zc1 = ab ? std::max(std::min(phi[2] + 1, z1), z0) : z1;
  if (f.px1 < f.px0 || f.py1 < f.py0 || p.zc1 <= p.zc0) p.zc0 = p.zc1 = z1;  // no PML-free core: all rows general
  p.SW = cdiv_i(nx, kSlabW);
  p.SH = cdiv_i(ny, kSlabH);
  p.nlo = cdiv_i(p.zc0 - z0, p.zbf);
  p.nsl = p.SW * p.SH * (p.nlo + cdiv_i(z1 - p.zc1, p.zbf));
  const int nc = p.zc1 - p.zc0;
  if (nc > 0) {
    const int pw = f.px1 - f.px0 + 1, ph = f.py1 - f.py0 + 1;
    f.ww = strip[0];
    f.wh = strip[1];
    f.tw = strip[2];
    f.th = strip[3];
    f.nwx = cdiv_i(pw, f.ww);
    f.nw_lo = cdiv_i(f.py0, f.wh);
    f.nw_hi = cdiv_i(ny - 1 - f.py1, f.wh);
    f.nty = cdiv_i(ny, f.th);
    f.nt_lo = cdiv_i(f.px0, f.tw);
    f.nt_hi = cdiv_i(nx - 1 - f.px1, f.tw);
    f.count = f.nwx * (f.nw_lo + f.nw_hi) + f.nty * (f.nt_lo + f.nt_hi);
    p.RW = cdiv_i(pw, 64);
    p.RH = cdiv_i(ph, 4 * npy);
  }
  p.nfr = p.nsl + f.count * cdiv_i(nc, p.zbf);
  p.items = p.nfr + p.RW * p.RH * cdiv_i(nc, p.zb);
  return p;
}

// Right-hand sides per block (they share its coefficients): two, or one with two
// rows of columns per thread; a thread carries four columns' state either way.
static int pick_rb(int nrhs) { return nrhs % 2 == 0 ? 2 : 1; }

// Planes per block where no tuned value applies: about two waves of three core blocks
// per SM, 8 to 34 planes (two are loaded on top of them: 105^3 A_h 19.8 us at 4, 17.0
// at 12; B with two right-hand sides on 81^3 24.1 at 4, 18.8 at 8).
static int choose_zb(int nx, int ny, int nz, int nrhs) {
  const int rb = pick_rb(nrhs);
  const long long tiles = (long long)cdiv_i(nx, 64) * cdiv_i(ny, rb == 2 ? 4 : 8) * (nrhs / rb);
  const long long nzb = std::max(1LL, 152 * 3 * 2 / tiles);
  return (int)std::min<long long>(std::max<long long>((nz + nzb - 1) / nzb, 8), 34);
}

// Tensor map of a field of `rows` rows of nx complex64 values as lines of two
// rows (CoreSmem's comment); `lines` lines of 68 values per copy.
static bool field_map(CUtensorMap* m, const void* base, int nx, long long rows, int lines) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return (Encode) nullptr;
    }
    return (Encode)f;
  }();
  if (!encode || rows < 2) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)4 * nx, (cuuint64_t)(rows / 2)};
  const cuuint64_t stride[1] = {(cuuint64_t)16 * nx};
  const cuuint32_t box[2] = {kRowB / 4, (cuuint32_t)lines}, one[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)(reinterpret_cast<uintptr_t>(base) & ~(uintptr_t)15), dims,
                stride, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MODE, int OPK, int NPY, int RB, int MB>
static void launch_t(const StencilCall<float>& c, cudaStream_t s) {
  const LevelView<float>& L = c.lv;
  const int zb = L.zb_march > 0 ? L.zb_march : choose_zb(L.nx, L.ny, L.nz, c.nrhs);
  Plan p = make_plan(L.nx, L.ny, L.plain_lo, L.plain_hi, L.strip, OPK != OPK_Q, zb, L.zb_march_f, NPY, c.zr0,
                           c.zr1 > 0 ? c.zr1 : L.nz);
  count_launch();
  // (two right-hand sides per block: the second one's rows must start on the other 8-byte half)
  p.rows = OPK != OPK_Q && L.nx % 2 && L.ny % 2 && p.fm.px0 > 1 && p.fm.px1 < L.nx - 3 && p.fm.py0 > 1 &&
           p.fm.py1 < L.ny - 2 && p.zc0 > 1 && p.zc1 < L.nz - 1;
  Maps mp{};
  if (p.rows) {
    const long long xs = c.xstride > 0 ? c.xstride : L.N;
    mp.sx = (int)(reinterpret_cast<uintptr_t>(c.x) >> 3 & 1);
    mp.rows = xs / L.nx;
    p.rows = (RB == 1 || mp.rows % 2) && field_map(&mp.x, c.x, L.nx, mp.rows * c.nrhs, 2 * NPY + 1);
    if (MODE == M_J2) p.rows = p.rows && field_map(&mp.d, c.dinv, L.nx, L.N / L.nx, 2 * NPY + 1);
  }
  const unsigned blocks = (unsigned)p.nfr * c.nrhs + (unsigned)(p.items - p.nfr) * (c.nrhs / RB);
  k_march<MODE, OPK, NPY, RB, MB><<<blocks, NT, march_smem<MODE, OPK, NPY, RB>(c.tab.nseg * (OPK == OPK_A ? L.nsub : 1), p.rows), s>>>(c, p, mp);
}

template <int MODE, int OPK>
void launch_mode(const StencilCall<float>& c, cudaStream_t s) {
  // residual of two, A, us at three / four blocks per SM: 119^3 62 / 56, 137 x 125 x 113
  // 68 / 64, 153^3 88 / 122, 289^3 347 / 418
  if (pick_rb(c.nrhs) == 2) {
    if constexpr (MODE == M_RESID) {
      if (c.lv.N >= 5LL << 19) {
        launch_t<MODE, OPK, 1, 2, 3>(c, s);
        return;
      }
    }
    launch_t<MODE, OPK, 1, 2, 4>(c, s);
  } else {
    launch_t<MODE, OPK, 2, 1, 3>(c, s);
  }
}

template <int MODE, int OPK, int NPY, int RB, int MB>
static void set_attr() {
  cudaFuncSetAttribute(k_march<MODE, OPK, NPY, RB, MB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)std::max(march_smem<MODE, OPK, NPY, RB>(kMaxParts, true),
                                     march_smem<MODE, OPK, NPY, RB>(kMaxParts, false)));
}
template <int MODE, int OPK>
void mode_attrs() {
  set_attr<MODE, OPK, 1, 2, 4>();
  if constexpr (MODE == M_RESID) set_attr<MODE, OPK, 1, 2, 3>();
  set_attr<MODE, OPK, 2, 1, 3>();
}

#define HZ_MARCH_INST(KW, MODE, OPK)                                                  \
  KW template void launch_mode<MODE, OPK>(const StencilCall<float>&, cudaStream_t); \
  KW template void mode_attrs<MODE, OPK>();
#define HZ_MARCH_PART0(KW) HZ_MARCH_INST(KW, M_APPLY, OPK_A) HZ_MARCH_INST(KW, M_APPLY, OPK_B) HZ_MARCH_INST(KW, M_APPLY, OPK_Q)
#define HZ_MARCH_PART1(KW) HZ_MARCH_INST(KW, M_RESID, OPK_A) HZ_MARCH_INST(KW, M_RESID, OPK_B)
#define HZ_MARCH_PART2(KW) HZ_MARCH_INST(KW, M_J2, OPK_A) HZ_MARCH_INST(KW, M_J2, OPK_B)
#define HZ_MARCH_PART3(KW) HZ_MARCH_INST(KW, M_JSWEEP, OPK_A) HZ_MARCH_INST(KW, M_JSWEEP, OPK_B)

#if HZ_MARCH_PART == 1
HZ_MARCH_PART1()
#elif HZ_MARCH_PART == 2
HZ_MARCH_PART2()
#elif HZ_MARCH_PART == 3
HZ_MARCH_PART3()
#else
HZ_MARCH_PART0()
HZ_MARCH_PART1(extern)
HZ_MARCH_PART2(extern)
HZ_MARCH_PART3(extern)

void launch(const StencilCall<float>& c, int mode, int opk, cudaStream_t s) {
  const bool b = opk == OPK_B;
  if (opk == OPK_Q) launch_mode<M_APPLY, OPK_Q>(c, s);
  else if (mode == M_RESID) b ? launch_mode<M_RESID, OPK_B>(c, s) : launch_mode<M_RESID, OPK_A>(c, s);
  else if (mode == M_J2) b ? launch_mode<M_J2, OPK_B>(c, s) : launch_mode<M_J2, OPK_A>(c, s);
  else if (mode == M_JSWEEP)
    b ? launch_mode<M_JSWEEP, OPK_B>(c, s) : launch_mode<M_JSWEEP, OPK_A>(c, s);
  else b ? launch_mode<M_APPLY, OPK_B>(c, s) : launch_mode<M_APPLY, OPK_A>(c, s);
}

void init_attrs() {
  mode_attrs<M_APPLY, OPK_A>();
  mode_attrs<M_APPLY, OPK_B>();
  mode_attrs<M_APPLY, OPK_Q>();
  mode_attrs<M_RESID, OPK_A>();
  mode_attrs<M_RESID, OPK_B>();
  mode_attrs<M_J2, OPK_A>();
  mode_attrs<M_J2, OPK_B>();
  mode_attrs<M_JSWEEP, OPK_A>();
  mode_attrs<M_JSWEEP, OPK_B>();
}

// Tile of a PML strip `thick` nodes thick and `len` long (alongx: its length runs
// along x): w x h columns, two x-adjacent ones per thread.  Cost per useful node:
// threads the tile leaves idle or past the strip, and its planes' halo loads.
static void strip_tile(int thick, int len, bool alongx, int& w, int& h) {
  double best = 1e30;
  const int nx = alongx ? len : std::max(thick, 1), ny = alongx ? std::max(thick, 1) : len;
  w = 2;
  h = 1;
  for (int pw = 1; pw <= 64; ++pw)
    for (int b = 1; b <= NT / pw && b <= ny; ++b) {
      const int a = 2 * pw;
      if ((a + 2) * (b + 2) > kPmlPln) break;
      const double used = 2.0 * NT * cdiv_i(nx, a) * cdiv_i(ny, b) / ((double)nx * ny);
      const double halo = (double)(a + 2) * (b + 2) / ((double)a * b);
      const double cost = used * (1.0 + 0.25 * halo);
      if (cost < best - 1e-9) {
        best = cost;
        w = a;
        h = b;
      }
    }
}

void strips(int nx, int ny, const int* plo, const int* phi, int* strip) {
  const int px0 = std::max(plo[0], 0), px1 = std::min(phi[0], nx - 1), py0 = std::max(plo[1], 0),
            py1 = std::min(phi[1], ny - 1);
  strip_tile(std::max(py0, ny - 1 - py1), std::max(px1 - px0 + 1, 1), true, strip[0], strip[1]);
  strip_tile(std::max(px0, nx - 1 - px1), ny, false, strip[2], strip[3]);
}

static Plan plan_of(int nx, int ny, int nz, const int* plo, const int* phi, bool ab, int nrhs, int zblock,
                    int zblock_f, const int* strip, int& npy) {
  npy = pick_rb(nrhs) == 2 ? 1 : 2;
  const int zb = zblock > 0 ? zblock : choose_zb(nx, ny, nz, nrhs);
  int own[4];
  if (!strip) {
    strips(nx, ny, plo, phi, own);
    strip = own;
  }
  return make_plan(nx, ny, plo, phi, strip, ab, zb, zblock_f, npy, 0, nz);
}

long long blocks_per_rhs(int nx, int ny, int nz, const int* plo, const int* phi, int nrhs, int zblock, int zblock_f,
                         const int* strip) {
  int npy;
  return plan_of(nx, ny, nz, plo, phi, true, nrhs, zblock, zblock_f, strip, npy).items;
}

// Host replay of k_march's block and thread decode: a written column outside
// the grid, a column inside the PML on a row form that drops that axis's terms,
// a node not written exactly once, or a block id repeated is a violation.
long long replay_layout(int nx, int ny, int nz, const int* plo, const int* phi, int op, int nrhs, int zblock,
                        int zblock_f) {
  const bool ab = op == OP_AB;
  int npy;
  const Plan p = plan_of(nx, ny, nz, plo, phi, ab, nrhs, zblock, zblock_f, nullptr, npy);
  std::vector<unsigned char> cnt((size_t)nx * ny * nz, 0);
  long long bad = 0;
  int th = NT;  // rows of threads
  auto cta = [&](int txt, int npx, int np, int x0, int y0, int rx1, int ry1, int form, int zb0, int zb1) {
    for (int tid = 0; tid < NT; ++tid)
      for (int j = 0; j < np; ++j)
        for (int i = 0; i < npx; ++i) {
          const int gx = x0 + npx * (tid % txt) + i, gy = y0 + np * (tid / txt) + j;
          if (!(tid / txt < th && gx <= rx1 && gy <= ry1)) continue;
          if (gx < 0 || gy < 0 || gx >= nx || gy >= ny) {
            ++bad;
            continue;
          }
          const bool px = gx >= plo[0] && gx <= phi[0], py = gy >= plo[1] && gy <= phi[1];
          if (ab && ((form == 0 && !(px && py)) || (form == 3 && !px))) ++bad;
          for (int z = zb0; z < zb1; ++z) {
            if (ab && form != 2 && (z < plo[2] || z > phi[2])) ++bad;
            unsigned char& c = cnt[((size_t)z * ny + gy) * nx + gx];
            if (c < 255) ++c;
          }
        }
  };
  for (int it = 0; it < p.items; ++it) {
    if (it >= p.nfr) {
      const int nt = p.RW * p.RH, bz = (it - p.nfr) / nt, t = it - p.nfr - bz * nt, ty = t / p.RW, tx = t - ty * p.RW;
      const int zb0 = p.zc0 + bz * p.zb;
      th = NT;
      cta(32, 2, npy, p.fm.px0 + 64 * tx, p.fm.py0 + 4 * npy * ty, p.fm.px1, p.fm.py1, 0, zb0,
          std::min(zb0 + p.zb, p.zc1));
    } else if (it < p.nsl) {
      const int nt = p.SW * p.SH, bz = it / nt, t = it - bz * nt, ty = t / p.SW, tx = t - ty * p.SW;
      th = NT;
      const int zb0 = bz < p.nlo ? p.zs0 + bz * p.zbf : p.zc1 + (bz - p.nlo) * p.zbf;
      cta(kSlabW / 2, 2, 1, tx * kSlabW, ty * kSlabH, nx - 1, ny - 1, 2, zb0,
          std::min(zb0 + p.zbf, bz < p.nlo ? p.zc0 : p.zs1));
    } else {
      const int bz = (it - p.nsl) / p.fm.count;
      const FrameTile f = decode_frame(p.fm, it - p.nsl - bz * p.fm.count);
      const int zb0 = p.zc0 + bz * p.zbf;
      th = f.wide ? p.fm.wh : p.fm.th;
      cta((f.wide ? p.fm.ww : p.fm.tw) / 2, 2, 1, f.x0, f.y0, f.rx1, f.ry1, f.wide ? 3 : 1, zb0,
          std::min(zb0 + p.zbf, p.zc1));
    }
  }
  for (unsigned char c : cnt)
    if (c != 1) ++bad;
  return bad;
}
#endif

}  // namespace march
}  // namespace hz
