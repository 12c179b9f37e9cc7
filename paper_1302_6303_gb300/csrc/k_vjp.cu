// Transposed Jacobian of the residual (the adjoint / vector-Jacobian
// product), at the state of the last linearisation.  Gather form over the rows
// of the frozen Jacobian (Jac), no atomics, deterministic:
//   1. ghost adjoints  gamma_g = the ghost side's flux partials times the face
//                      adjoint lambda_g = +-w of the ghost's cell, less 1/8 of
//                      the coarse cell's at a coarse-fine face (flux matching:
//                      a quarter of the fine face over twice the fine h);
//   2. cell gather     (J^T w)_c = a0 w_c - dt (the own entries, the
//                      neighbours' coefficients for c inside the patch, the
//                      ghost adjoints of every ghost that reads c with the
//                      ghost's stencil weight), and the same for d/dz.
#include <algorithm>

#include "nrd_internal.h"
#include "softfp.h"

namespace {

struct VjpArgs {
  const TileDev* tiles;
  const PatchDev* patches;
  const uint8_t* mask;
  const uint8_t* gtype;
  const uint8_t* gface;
  const int* gcell;
  const int* gzsrc;
  const int* ts_off;   // transposed ghost stencil: cell -> (ghost, weight)
  const int* ts_g;
  const double* ts_w;
  const int* tz_off;   // ghosts taking their z from a cell
  const int* tz_g;
  Jac jac;
  const float* z;
  const double* w;     // [2][N]
  double* gam;         // [3][G]
  double* out;         // [2][N]
  double* dz;          // [N] or null
  double a0, dt;
  int N, G, tx, ty;
};

// adjoint of the face between cell c and its ghost g on side hi: this cell is
// the low side of its high face; zero where flux matching or covering takes
// the face from the cell.  The coarse cell across a coarse-fine face takes
// a quarter of the fine flux (over its own h).
__device__ __forceinline__ double face_adj(const VjpArgs& a, const double* w, int c, int g,
                                           bool hi, uint8_t ty) {
  double l = w[c];
  if (ty == GT_CF) l -= 0.125 * w[a.gzsrc[g]];
  return hi ? l : -l;
}

// 1. ghost adjoints
__global__ void k_vjp_ghosts(VjpArgs a) {
  const int N = a.N;
  const long G = a.G;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    const uint8_t ty = a.gtype[g];
    double gE = 0.0, gT = 0.0, gZ = 0.0;
    const int c = a.gcell[g], f = a.gface[g] & 7;
    const uint8_t m = a.mask[c];
    if ((ty == GT_SIBLING || ty == GT_CF) && !(m & MASK_COVERED) && !(m & (2 << f))) {
      const bool hi = f & 1;   // ghost on the high side of the face
      const double lE = face_adj(a, a.w, c, g, hi, ty), lT = face_adj(a, a.w + N, c, g, hi, ty);
      const long NS = 3L * N + G;
      const double* jf = a.jac.jc + 3L * N + g;
      gE = (hi ? jf[NS] : jf[0]) * lE;
      gT = jf[2 * NS] * lE + (hi ? jf[4 * NS] : jf[3 * NS]) * lT;
      if (a.dz) gZ = jf[5 * NS] * lE;
    }
    a.gam[g] = gE;
    a.gam[G + g] = gT;
    a.gam[2 * G + g] = gZ;
  }
}

// 2. per-cell gather: 26 FP64 instructions and the 19 coefficients of the rows
// per cell (as the forward product), against three kernels with the face
// adjoints through memory before; at 96^3 with 8 fine boxes (1.0M cells) the
// product 134 -> 67 us.
template <bool DZ>
__global__ void __launch_bounds__(256, 6) k_vjp_cells(VjpArgs a) {
  const int N = a.N;
  const long G = a.G;
  const TileDev tile = a.tiles[blockIdx.x];
  const PatchDev P = a.patches[tile.patch];
  const int nx = P.n[0], ny = P.n[1], nz = P.n[2];
  // the tile's extent inside its patch: no lane idles on a cell outside it
  const int ex = min(a.tx, nx - tile.i0), ey = min(a.ty, ny - tile.j0);
  const int nc = ex * ey * (tile.k1 - tile.k0);
  const Jac& J = a.jac;
  const long NS = 3L * N + G;
  const double* wE = a.w;
  const double* wT = a.w + N;
  for (int q = threadIdx.x; q < nc; q += blockDim.x) {
    const int r = q / ex, i = tile.i0 + q - r * ex;
    const int rk = r / ey, j = tile.j0 + r - rk * ey, k = tile.k0 + rk;
    const int idx = P.off + i + nx * (j + ny * k);
    const uint8_t m = a.mask[idx];
    if (m & MASK_COVERED) {
      a.out[idx] = 0.0;
      a.out[N + idx] = 0.0;
      if (DZ) a.dz[idx] = 0.0;
      continue;
    }
    const double wEc = wE[idx], wTc = wT[idx];
    // the four plain products on the integer pipe (bit-identical); the diagonal
    // last, as in the product
    double aE = soft_mul_any(J.cen[3L * N + idx], wTc);
    double aT = soft_mul_any(J.cen[N + idx], wEc);
    double aZ = 0.0;
    const int pos[3] = {i, j, k};
#pragma unroll
    for (int f = 0; f < 6; f++) {
      if (m & (2 << f)) continue;   // flux matching: the neighbour is covered
      const int d = f >> 1, hi = f & 1;
      const int st = (d == 0) ? 1 : (d == 1 ? nx : nx * ny);
      if (pos[d] != (hi ? P.n[d] - 1 : 0)) {
        // the neighbour's row: its coefficient for this cell
        const long n = hi ? idx + st : idx - st;
        const double* jf = J.jc + (long)d * N + (hi ? n : idx);
        const double wn = wE[n];
        aE = fma(hi ? -jf[0] : jf[NS], wn, aE);
        aT = fma(hi ? -jf[2 * NS] : jf[2 * NS], wn, aT);
        aT = fma(hi ? -jf[3 * NS] : jf[4 * NS], wT[n], aT);
        if (DZ) aZ = fma(jf[5 * NS], hi ? wEc - wn : wn - wEc, aZ);
        continue;
      }
      const int g = P.goff + P.fo[f] + pos[(d + 1) % 3] + P.n[(d + 1) % 3] * pos[(d + 2) % 3];
      const uint8_t ty = a.gtype[g];
      if (ty == GT_NEUMANN) continue;
      const double* jf = J.jc + 3L * N + g;
      if (DZ) aZ = fma(jf[5 * NS], face_adj(a, wE, idx, g, hi, ty), aZ);
      if (ty == GT_CF) {
        // the coarse cell's share of this face (the cell's own is in cen)
        const int C = a.gzsrc[g];
        const double lE = (hi ? -0.125 : 0.125) * wE[C], lT = (hi ? -0.125 : 0.125) * wT[C];
        aE = fma(hi ? jf[0] : jf[NS], lE, aE);
        aT = fma(jf[2 * NS], lE, aT);
        aT = fma(hi ? jf[3 * NS] : jf[4 * NS], lT, aT);
      }
    }
    // ghosts that read this cell (sibling copies, coarse-fine stencils)
    for (int t = a.ts_off[idx]; t < a.ts_off[idx + 1]; t++) {
      const int g = a.ts_g[t];
      const double wq = a.ts_w[t];
      aE += wq * a.gam[g];
      aT += wq * a.gam[G + g];
    }
    aE = fma(J.cen[idx], wEc, aE);
    aT = fma(J.cen[2L * N + idx], wTc, aT);
    a.out[idx] = fma(-a.dt, aE, soft_mul_any(a.a0, wEc));
    a.out[N + idx] = fma(-a.dt, aT, soft_mul_any(a.a0, wTc));
    if (DZ) {
      for (int t = a.tz_off[idx]; t < a.tz_off[idx + 1]; t++) aZ += a.gam[2 * G + a.tz_g[t]];
      const double zc = (double)a.z[idx];
      a.dz[idx] = -a.dt * 3.0 * zc * zc * (aZ + J.cZ[idx] * (wEc - wTc));
    }
  }
}

}  // namespace

void launch_vjp(const Hier& H, const Jac& jac, const float* z, const double* w, double* gam,
                double a0, double dt, double* out, double* dz, cudaStream_t s) {
  VjpArgs a;
  a.tiles = H.d_tiles;
  a.patches = H.d_patches;
  a.mask = H.d_mask;
  a.gtype = H.d_gtype;
  a.gface = H.d_gface;
  a.gcell = H.d_gcell;
  a.gzsrc = H.d_gzsrc;
  a.ts_off = H.d_ts_off;
  a.ts_g = H.d_ts_g;
  a.ts_w = H.d_ts_w;
  a.tz_off = H.d_tz_off;
  a.tz_g = H.d_tz_g;
  a.jac = jac;
  a.z = z;
  a.w = w;
  a.gam = gam;
  a.out = out;
  a.dz = dz;
  a.a0 = a0;
  a.dt = dt;
  a.N = H.N;
  a.G = H.G;
  a.tx = H.tile_x;
  a.ty = H.tile_y;
  const int nt = std::max(1, (int)H.tiles.size());
  const int bs = std::min(256, H.tile_x * H.tile_y * H.tile_z);
  int gb = (int)std::min(152L * 8, (H.G + 255L) / 256);
  k_vjp_ghosts<<<std::max(gb, 1), 256, 0, s>>>(a);
  if (dz) k_vjp_cells<true><<<nt, bs, 0, s>>>(a);
  else k_vjp_cells<false><<<nt, bs, 0, s>>>(a);
}
