// The small solve of the bottom Krylov method C_4h (Sec. 3.2): from the Gram
// entries of the basis p_0 .. p_S, the normal equations of
// min || p_0 - sum_k y_k p_{k+1} || solved by elimination in FP64.
// Shared by the Gram kernel of the launch chain and the persistent bottom
// kernel.
#pragma once

namespace hz {

// sres: Gram entries <p_a, p_b> (a <= b, row by row; re, im interleaved);
// yo: y_0 .. y_{S-1} (re, im).  Called by one whole warp.
//
// The chain of dependent FP64 operations is what this costs (it runs once per
// bottom solve, in one block, with the GPU waiting): one thread working through
// a Cholesky factor in shared memory took most of the Gram kernel's 22 us.  Here
// lane c holds column c of [G_rr | g_r0] in registers, each elimination step is
// one reciprocal, a broadcast of its column and one multiply-add deep, and no
// square roots.  The pivots are those of the Cholesky factor, squared.
template <int KN>
__device__ __forceinline__ void gram_lsq_solve(const double* sres, double* yo, int lane) {
  constexpr int S = KN - 1;
  // index of G[a][b] = <p_a, p_b>, a <= b, in sres (rows a = 0 .. KN - 1, b = a .. KN - 1)
  auto gidx = [](int a, int b) { return a * KN - a * (a - 1) / 2 + (b - a); };
  // normal equations: G_rr y = g_r0 with G_rr = [<p_a, p_b>]_{a,b>=1} (Hermitian),
  // g_r0 = [<p_a, p_0>]_{a>=1}
  const int c = lane < S ? lane : S;
  double re[S], im[S], inv[S];
  double dmax = 0.0;
#pragma unroll
  for (int r = 0; r < S; ++r) {
    const int b = c == S ? 0 : c + 1;  // column's basis vector
    const int lo = min(r + 1, b), hi = max(r + 1, b);
    const double* g = sres + 2 * gidx(lo, hi);
    re[r] = g[0];
    im[r] = r + 1 <= b ? g[1] : -g[1];
    dmax = fmax(dmax, sres[2 * gidx(r + 1, r + 1)]);
  }
  int rank = S;  // (uniform) directions before the first numerically dependent one
#pragma unroll
  for (int j = 0; j < S; ++j) {
    const double d = __shfl_sync(0xffffffffu, re[j], j);
    if (rank == S && !(d > 1e-13 * dmax)) rank = j;
    inv[j] = j < rank ? 1.0 / d : 0.0;
    const double wr = re[j] * inv[j], wi = im[j] * inv[j];
#pragma unroll
    for (int r = j + 1; r < S; ++r) {
      const double mr = __shfl_sync(0xffffffffu, re[r], j), mi = __shfl_sync(0xffffffffu, im[r], j);
      re[r] -= mr * wr - mi * wi;
      im[r] -= mr * wi + mi * wr;
    }
  }
  // back substitution in the right-hand side's lane(s): column a arrives from lane a
#pragma unroll
  for (int a = S - 1; a >= 0; --a) {
    const double yr = a < rank ? re[a] * inv[a] : 0.0, yi = a < rank ? im[a] * inv[a] : 0.0;
    if (lane == S) {
      yo[2 * a] = yr;
      yo[2 * a + 1] = yi;
    }
#pragma unroll
    for (int r = 0; r < a; ++r) {
      const double ur = __shfl_sync(0xffffffffu, re[r], a), ui = __shfl_sync(0xffffffffu, im[r], a);
      if (c == S) {
        re[r] -= ur * yr - ui * yi;
        im[r] -= ur * yi + ui * yr;
      }
    }
  }
}

}  // namespace hz
