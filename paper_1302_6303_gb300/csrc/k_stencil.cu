// Stencil kernels of the radiation-diffusion residual (Sec. 3.2, 3.2.1, 3.3)
// and its Jacobian-vector products (Sec. 4.1), all FP64:
//   ghost fill     physical / sibling / coarse-fine ghosts from a work-list
//   k_stencil      one persistent launch over the tiles of every level:
//                  halo staged in shared memory; the residual and the
//                  linearisation as a face launch (each face once) and a
//                  cell launch, the exact and FD Jv in one
//   k_jv_frozen    the frozen Jacobian's product, one row sum per cell and field
//   k_reflux       flux matching at coarse-fine faces
//   k_tag          Sec. 5 refinement indicators
//   k_avgdown      covered cells := mean of their children
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <type_traits>

#include "nrd_internal.h"
#include "softfp.h"

namespace {

struct LevelH {
  double h[NRD_MAX_LEVELS][3];
  double rh[NRD_MAX_LEVELS][3];   // 1/h
  double h3[NRD_MAX_LEVELS][3];   // 3h
  double kh[NRD_MAX_LEVELS][3];   // k/h
  // constants of face_core
  double c1[NRD_MAX_LEVELS][3];   // 1 / (12 h^2)
  double cLh[NRD_MAX_LEVELS][3];  // (cL / 2) h
  double cT[NRD_MAX_LEVELS][3];   // 2^(-5/2) k / h^2 (Tf^(5/2) = 2^(-5/2) Ts^(5/2), Ts = T_a + T_b)
};

struct GhostArgs {
  const uint8_t* gtype;
  const uint8_t* gface;   // face | level << 3
  const int* gcell;
  const int* gt0;
  const int* gidx;
  const double* gw;
  const float* z;
  int N, G;
  double R[6];
  LevelH lh;
};

// Fill ghosts of a two-field vector u (E = u[0..N), T = u[N..2N)) into
// g[0..G) (E) and g[G..2G) (T).  nonlinear = 1 evaluates the Robin ghost of
// Sec. 3.1 Eq. robinbc; nonlinear = 0 copies the interior value there (linear
// uses never read physical ghosts).
__global__ void k_ghost_fill(GhostArgs a, const double* __restrict__ u, double* __restrict__ g,
                             int nonlinear) {
  const int N = a.N, G = a.G;
  for (int gi = blockIdx.x * blockDim.x + threadIdx.x; gi < G; gi += gridDim.x * blockDim.x) {
    uint8_t t = a.gtype[gi];
    int c = a.gcell[gi];
    double e, tt;
    if (t == GT_NEUMANN) {
      e = u[c];
      tt = u[N + c];
    } else if (t == GT_ROBIN) {
      e = u[c];
      tt = u[N + c];
      if (nonlinear) {
        int f = a.gface[gi] & 7, lvl = a.gface[gi] >> 3;
        double h = a.lh.h[lvl][f / 2];
        double T = tt;
        double zc = (double)a.z[c];
        double Db = T * T * T / (3.0 * (zc * zc * zc));
        double aa = Db / (2.0 * h);
        e = (a.R[f] + e * (aa - 0.125)) / (aa + 0.125);
      }
    } else {
      int t0 = a.gt0[gi], t1 = a.gt0[gi + 1];
      double se = 0.0, st = 0.0;
      for (int q = t0; q < t1; q++) {
        int s = a.gidx[q];
        double w = a.gw[q];
        se += w * u[s];
        st += w * u[N + s];
      }
      e = se;
      tt = st;
    }
    g[gi] = e;
    g[G + gi] = tt;
  }
}

__global__ void k_ghost_z(const int* __restrict__ zsrc, const float* __restrict__ z,
                          float* __restrict__ gz, int G) {
  for (int gi = blockIdx.x * blockDim.x + threadIdx.x; gi < G; gi += gridDim.x * blockDim.x)
    gz[gi] = z[zsrc[gi]];
}

struct StArgs {
  const TileDev* tiles;
  const PatchDev* patches;
  const uint8_t* mask;
  const uint8_t* gtype;
  const double* z3;   // z^3 of cells then ghosts (FP64)
  bool soft;          // the faces' constants lie in the soft window
  int ntiles, N, G;
  double cL;      // limiter constant: 4 (Wilson form) or 2 (printed form)
  double R[6];
  LevelH lh;
  StencilIO io;
};

// Linearisation of one face at the iterate, everything divided by h: the
// fluxes, the P1 coefficients X = D_E / h^2 and T25 = D_T / h^2 of Sec. 4.2,
// and the partial derivatives of Phi_E w.r.t. E_a, E_b and T_a (= w.r.t.
// T_b), of Phi_T w.r.t. T_a, T_b, and of Phi_E w.r.t. z_a^3 (= z_b^3)
// (sign(0) = 0).
struct FaceLin {
  double PE, PT, aEa, aEb, aT, bTa, bTb, aZ;
  double X, T25;
};

// 1/x from the PTX approximate FP64 reciprocal (rcp.approx.ftz.f64, a
// seed of about 20 good bits) refined with the second-order series of the
// correction: with e = 1 - x r0, 1/x = r0 / (1 - e) = r0 (1 + e + e^2 + ...),
// so r1 = r0 + r0 (e + e^2) leaves a relative error of e^3 (iterative
// refinement of reciprocals, see e.g. Muller et al., Handbook of
// Floating-Point Arithmetic): about 1e-18 before rounding.  For positive
// x in [2^-997, 2^997) (about 7.5e-301 to 1.3e300); elsewhere (zero,
// subnormal, negative, huge, inf, NaN) the correctly rounded 1/x.  The range
// test looks at the high word of x with integer instructions: FP64 compares
// would take FP64-pipe issue slots, the scarce resource of these kernels.
__device__ __forceinline__ bool in_refine_range(double x) {
  // biased exponent in [26, 2020) and sign bit clear
  const unsigned hi = (unsigned)__double2hiint(x);
  return hi - (26u << 20) < ((2020u - 26u) << 20);
}
__device__ __forceinline__ double rcp_approx(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rsqrt_approx(double x) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rcp_nr(double x) {
  if (!in_refine_range(x)) return 1.0 / x;
  const double r = rcp_approx(x);
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// 1/sqrt(x) from the PTX approximate FP64 reciprocal square root
// (rsqrt.approx.ftz.f64) refined with the second-order series: with
// e = 1 - x y0^2, 1/sqrt(x) = y0 (1 - e)^(-1/2) = y0 (1 + e/2 + 3 e^2/8 + ...),
// a relative error of about (5/16) e^3 before rounding.  For x in the range
// of rcp_nr; elsewhere the correctly rounded 1/sqrt(x).
// SOFT (x in the soft window): the first product on the integer pipe.
template <bool SOFT = false>
__device__ __forceinline__ double rsqrt_nr(double x) {
  if (!in_refine_range(x)) return 1.0 / sqrt(x);
  const double y = rsqrt_approx(x);
  const double e = fma(-Mul<SOFT>::pos(x, y), y, 1.0);
  return fma(__dmul_rn(y, e), fma(0.375, e, 0.5), y);
}

// FP64 -> FP32 with round-to-nearest-even (the IEEE narrowing conversion,
// bit-identical to the (float) cast) from integer instructions: on GB300 the
// conversion instruction issues on the FP64 pipe, which bounds the
// linearisation.  With the FP64 exponent field e in [897, 1150] the result is a
// normal float: its exponent is e - 896 and its 23 mantissa bits are the top
// 23 of the 52; the 29 dropped bits d round up when d > 2^28, or d = 2^28 and
// the kept lsb is odd, i.e. exactly when d + (2^28 - 1) + lsb >= 2^29.  A
// mantissa carry runs into the exponent (up to infinity when the rounded value
// overflows, as IEEE narrowing gives).  Other exponents (zero, subnormal or
// overflowing results, inf, NaN) take the conversion instruction, in a
// function of its own: inlined, the compiler predicates the conversion instead
// of branching around it, and a predicated-off instruction still takes its
// FP64-pipe issue slot.
__device__ __noinline__ float narrow_slow(double x) { return __double2float_rn(x); }
__device__ __forceinline__ float narrow_rn(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - 897u > 253u) return narrow_slow(x);
  const unsigned top = __funnelshift_l(lo, hi & 0x7fffffffu, 3);   // exponent+mantissa bits
  const unsigned rnd = ((lo & 0x1fffffffu) + 0x0fffffffu + (top & 1u)) >> 29;
  return __uint_as_float((hi & 0x80000000u) | (top - (896u << 23) + rnd));
}

// Face flux in the +e_d direction between cells a (low) and b (high), over h
// (its contribution to the divergence of a cell):
//   Phi_E = D_E (E_b - E_a)/h with D_E = D_h/(1 + D_h g) (or the printed form)
//         = 2 Tf^3 S dE / (3 h Zs S + cL Tf^3 |dE|),  S = E_a + E_b,
//           Zs = z_a^3 + z_b^3, dE = E_b - E_a, Tf = (T_a + T_b)/2
//   Phi_T = k Tf^(5/2) (T_b - T_a)/h,
// with the intermediate quantities the partial derivatives reuse.  The
// residual and the linearisation both take their fluxes from here, so the
// two produce bit-identical residuals.
// Evaluated in Ts = T_a + T_b = 2 Tf with the powers of 2 and h folded into
// the constants c1 = 1/(12 h^2), cLh = (cL/2) h, cT = 2^(-5/2) k / h^2:
//   Tc = c1 Ts^3, lt = Tc cLh |dE|, den = Zs S + lt, Q = Tc / den,
//   Phi_E / h = X dE with X = Q S (= D_E / h^2),
//   Phi_T / h = T25 dT with T25 = cT Ts^(5/2) (= D_T / h^2).
// 13 FP64 instructions and 12 products; the products go to the integer pipe
// where SOFT (the same bits, see softfp.h).  Both pipes then take about the
// same time.  Measured at 256^3 (8x8x8 tiles), against the plain formulas on the
// FP64 pipe alone (45 and 26 instructions a face): the linearisation's face
// launch 4.25 -> 2.04 ms, the residual's 2.66 -> 1.37 ms.
struct FaceCore {
  double Ts, dE, S, r, Q, X, lt, PE, y, dT, T25, PT;
};
template <bool SOFT>
__device__ __forceinline__ FaceCore face_core(double Ea, double Eb, double Ta, double Tb,
                                              double za, double zb, double c1, double cLh,
                                              double cT) {
  using M = Mul<SOFT>;
  FaceCore q;
  q.Ts = __dadd_rn(Ta, Tb);
  const double Ts3 = M::pos(M::pos(q.Ts, q.Ts), q.Ts);
  q.dE = __dsub_rn(Eb, Ea);
  q.S = __dadd_rn(Ea, Eb);
  const double Tc = M::pos(c1, Ts3);
  q.lt = M::any(Tc, M::any(cLh, fabs(q.dE)));
  q.r = rcp_nr(fma(__dadd_rn(za, zb), q.S, q.lt));
  q.Q = M::pos(Tc, q.r);
  q.X = M::pos(q.Q, q.S);
  q.PE = M::any(q.X, q.dE);
  q.y = rsqrt_nr<SOFT>(q.Ts);
  q.T25 = M::pos(cT, M::pos(Ts3, q.y));
  q.dT = __dsub_rn(Tb, Ta);
  q.PT = M::any(q.T25, q.dT);
  return q;
}

// Face flux of face_core and its partial derivatives at one iterate (the
// frozen Jacobian).  With w = lt / den (so that Zs S / den = 1 - w):
//   d PE / d E_a = Q (2 w E_b - S),  d PE / d E_b = Q (S - 2 w E_a)
//   d PE / d T_a = d PE / d T_b = 3 (1 - w) PE / Ts
//   d PE / d Zs  = -PE S / den
//   d PT / d T_{a,b} = 2.5 PT / Ts -/+ T25
// (from 4 Tf^3 S dE / den^2 and the like by dividing through by den; the terms
// with sign(dE) combine with |dE|, so dE = 0 gives w = 0).  Ts^(-1) = y^2.
template <bool SOFT>
__device__ __forceinline__ FaceLin flux_lin(double Ea, double Eb, double Ta, double Tb, double za,
                                            double zb, double c1, double cLh, double cT,
                                            bool with_dz) {
  using M = Mul<SOFT>;
  const FaceCore q = face_core<SOFT>(Ea, Eb, Ta, Tb, za, zb, c1, cLh, cT);
  FaceLin r;
  r.PE = q.PE;
  r.PT = q.PT;
  r.X = q.X;
  r.T25 = q.T25;
  const double w = M::any(q.lt, q.r);
  const double wQ2 = M::twice(M::any(w, q.Q));
  r.aEa = fma(wQ2, Eb, -q.X);
  r.aEb = fma(-wQ2, Ea, q.X);
  const double rTs = M::pos(q.y, q.y);
  r.aT = M::any(M::any(q.PE, rTs), fma(-3.0, w, 3.0));
  const double PTr = M::any(q.PT, rTs);
  r.bTa = fma(2.5, PTr, -q.T25);
  r.bTb = fma(2.5, PTr, q.T25);
  r.aZ = with_dz ? -(q.PE * q.r) * q.S : 0.0;
  return r;
}

// Balance of one cell (Eq. nonlinearsystem, per unit volume):
//   F_E = a0 E - b_E - dt (div_E + c),  F_T = a0 T - b_T - dt (div_T - c),
//   c = sigma (T^4 - E), sigma = z^3 / T^3,
// shared by the residual and the linearisation (bit-identical F); returns
// 1/T and sigma for the partial derivatives.
// (SOFT: E, T and z^3 in the soft window; the same bits either way.  At 256^3
// it took the residual's cell launch from 0.89 to 0.63 ms and the linearisation's
// from 1.08 to 0.72; the latter takes 1.25 ms since it also sums the cell's own
// Jacobian entries.)
template <bool SOFT>
__device__ __forceinline__ void cell_balance(double a0, double dt, double E, double T, double z3,
                                             double bE, double bT, double divE, double divT,
                                             double& FE, double& FT, double& rT, double& sig) {
  using M = Mul<SOFT>;
  rT = rcp_nr(T);
  sig = M::pos(M::pos(M::pos(z3, rT), rT), rT);
  const double T2 = M::pos(T, T);
  const double cp = M::any(sig, fma(T2, T2, -E));
  FE = fma(-dt, __dadd_rn(divE, cp), fma(a0, E, -bE));
  FT = fma(-dt, __dsub_rn(divT, cp), fma(a0, T, -bT));
}

// Tangent of the face fluxes in the direction (dEa, dEb, dTa, dTb); sign(0) = 0.
__device__ __forceinline__ void flux_tan(double Ea, double Eb, double Ta, double Tb, double za,
                                         double zb, double h3, double kh, double cL, double vEa,
                                         double vEb, double vTa, double vTb, double& dPE,
                                         double& dPT) {
  double Tf = 0.5 * (Ta + Tb);
  double dTf = 0.5 * (vTa + vTb);
  double Tf2 = Tf * Tf;
  double Tf3 = Tf2 * Tf;
  double dTf3 = 3.0 * Tf2 * dTf;
  double dE = Eb - Ea, ddE = vEb - vEa;
  double S = Ea + Eb, dS = vEa + vEb;
  double Zs = za + zb;
  double sg = (dE > 0.0) ? 1.0 : ((dE < 0.0) ? -1.0 : 0.0);
  double num = 2.0 * Tf3 * dE * S;
  double dnum = 2.0 * (dTf3 * dE * S + Tf3 * (ddE * S + dE * dS));
  double den = h3 * Zs * S + cL * Tf3 * fabs(dE);
  double dden = h3 * Zs * dS + cL * (dTf3 * fabs(dE) + Tf3 * sg * ddE);
  double rden = 1.0 / den;
  double PE = num * rden;
  dPE = (dnum - PE * dden) * rden;
  double sq = sqrt(Tf);
  dPT = kh * ((2.5 * Tf * sq * dTf) * (Tb - Ta) + Tf2 * sq * (vTb - vTa));
}

// Robin face (Sec. 3.1 Eq. robinbc, unlimited D_b = T^3/(3 z^3)): the +e_d
// flux through the boundary face on side s of the cell is
//   Phi = -s D_b (2 E - 8 R) / (4 D_b + h).
__device__ __forceinline__ double robin_flux(double E, double T, double z, double h, double R,
                                             int s) {
  double Db = T * T * T / (3.0 * z);
  return -(double)s * Db * (2.0 * E - 8.0 * R) / (4.0 * Db + h);
}

__device__ __forceinline__ double robin_tan(double E, double T, double z, double h, double R,
                                            int s, double vE, double vT) {
  double Db = T * T * T / (3.0 * z);
  double dDb = T * T * vT / z;
  double m = 2.0 * E - 8.0 * R, dm = 2.0 * vE;
  double q = 4.0 * Db + h;
  return -(double)s * (dDb * m * h + Db * dm * q) / (q * q);
}

// scaled P1 coefficient a = beta C / h^2 (or the Robin diagonal term) in the
// V-cycle precision
__device__ __forceinline__ void put_scaled(const StencilIO& io, long NS, long slot, double aE,
                                           double aT) {
  if (io.a32) {
    io.a32[slot] = (float)aE;
    io.a32[NS + slot] = (float)aT;
  } else {
    io.a64[slot] = aE;
    io.a64[NS + slot] = aT;
  }
}

// the faces' part of a cell's own Jacobian entries
struct OwnSum {
  double EE, ET, TT;
};

// The linearisation's cell outputs: F from cell_balance, the own entries of
// the frozen Jacobian and the P2 data.
template <bool DZ, bool SOFT>
__device__ __forceinline__ void lin_cell(const StencilIO& io, int N, int idx, double a0v,
                                         double dtv, double betav, float betaf, double E,
                                         double T, double z3, double divE, double divT,
                                         const OwnSum& own) {
  using M = Mul<SOFT>;
  double FE, FT, rT, sig;
  cell_balance<SOFT>(a0v, dtv, E, T, z3, io.b[idx], io.b[N + idx], divE, divT, FE, FT, rT, sig);
  io.out[idx] = FE;
  io.out[N + idx] = FT;
  const double T2 = M::pos(T, T), T3 = M::pos(T2, T);
  // coupling tangent dc = -sig vE + cT vT, with the own entries of the faces
  const double cT = M::pos(sig, fma(M::pos(3.0, E), rT, T3));
  double* cen = io.jac.cen;
  cen[idx] = own.EE - sig;
  cen[N + idx] = own.ET + cT;
  cen[2L * N + idx] = own.TT - cT;
  cen[3L * N + idx] = sig;
  if (DZ) io.jac.cZ[idx] = (T2 * T2 - E) * rT * rT * rT;   // d coupling / d z^3
  // P2 of Sec. 4.2 at this iterate: [[1 + sb, -sbt], [-sb, 1 + sbt]]
  // (det = (1 + sb)(1 + sbt) - sbt sb = 1 + sb + sbt), in the
  // preconditioner's precision
  if (io.p2f) {
    const float sb = narrow_rn(sig) * betaf, sbt = sb * narrow_rn(T3);
    io.p2f[idx] = sb;
    io.p2f[N + idx] = sbt;
    io.p2f[2L * N + idx] = 1.0f / (1.0f + sb + sbt);
  } else {
    const double sb = sig * betav, sbt = sb * T3;
    io.p2[idx] = sb;
    io.p2[N + idx] = sbt;
    io.p2[2L * N + idx] = rcp_nr(1.0 + sb + sbt);
  }
}

// covered cell: not an unknown
template <bool DZ>
__device__ __forceinline__ void lin_cell_covered(const StencilIO& io, int N, int idx) {
  io.out[idx] = 0.0;
  io.out[N + idx] = 0.0;
  for (int q = 0; q < 4; q++) io.jac.cen[(long)q * N + idx] = 0.0;
  if (DZ) io.jac.cZ[idx] = 0.0;
  if (io.p2f) {
    io.p2f[idx] = 0.0f;
    io.p2f[N + idx] = 0.0f;
    io.p2f[2L * N + idx] = 0.0f;
  } else {
    io.p2[idx] = 0.0;
    io.p2[N + idx] = 0.0;
    io.p2[2L * N + idx] = 0.0;
  }
}

// Resident blocks per SM the split forms' launches are compiled for.  They
// need warps to cover the latency of their loads and integer products more
// than registers.  Measured at 256^3 (us; the compiler's own choice -> this):
// linearisation faces 2277 -> 2159 (4), cells 1326 -> 1247 (4), residual
// faces 1408 -> 1372 (8), cells on an odd box 40.6 -> 39.7 (5); the cells of
// three levels of ragged patches 603 -> 437 (4).
constexpr int min_blocks(int mode) {
  switch (mode) {
    case ST_LINF: case ST_LINZF: case ST_LINC: case ST_LINZC: return 4;
    case ST_RESF: return 8;
    case ST_RESC: return 5;
    default: return 0;   // no bound
  }
}

// CMP: the cell launches' loop runs over the cells of a tile inside its patch
// only, with index arithmetic in the tile's runtime extent; used where the
// hierarchy has tiles narrower than the tile shape (patches whose sides are not
// multiples of it), so that no lane of a warp idles on a cell outside its patch.
// Without CMP the extents are the compile-time shape (fewer registers: the form
// for hierarchies without such tiles).
template <int MODE, int TX, int TY, int TZ, bool CMP, int MINB>
__global__ void __launch_bounds__(256, MINB) k_stencil(StArgs A) {
  constexpr int HX = TX + 2, HY = TY + 2, HZ = TZ + 2;
  constexpr int NH = HX * HY * HZ;
  constexpr int NFX = (TX + 1) * TY * TZ, NFY = TX * (TY + 1) * TZ, NFZ = TX * TY * (TZ + 1);
  constexpr int NC = TX * TY * TZ;
  constexpr bool TAN = (MODE == ST_JV);
  constexpr bool LIN = (MODE == ST_LINF || MODE == ST_LINZF);   // the linearisation's face launch
  constexpr bool LINC = (MODE == ST_LINC || MODE == ST_LINZC);  // and its cell launch
  constexpr bool FACES = LIN || MODE == ST_RESF;    // split forms: faces only
  constexpr bool CELLS = LINC || MODE == ST_RESC;   // split forms: cells only
  constexpr bool DZ = (MODE == ST_LINZF || MODE == ST_LINZC);   // also the d/dz^3 partials
  extern __shared__ double smem[];
  double* sE = smem;
  double* sT = sE + NH;
  double* svE = sT + NH;                       // tangent direction (JV only)
  double* svT = svE + (TAN ? NH : 0);
  double* fxE = svT + (TAN ? NH : 0);
  double* fxT = fxE + NFX;
  double* fyE = fxT + NFX;
  double* fyT = fyE + NFY;
  double* fzE = fyT + NFY;
  double* fzT = fzE + NFZ;
  double* sZ = FACES ? fxE : fzT + NFZ;       // z^3 of the halo cells

  const int N = A.N, G = A.G;
  const long NS = 3L * N + G;                  // face slots per coefficient array
  const StencilIO& io = A.io;
  // a0, dt, beta: kernel arguments, or device values (graph-captured solves)
  double a0v = io.a0, dtv = io.dt, betav = io.beta;
  if (io.par) {
    a0v = io.par[0];
    dtv = io.par[1];
    betav = io.par[2];
  }
  double eps = 0.0, reps = 0.0;
  if (MODE == ST_FD) {
    eps = *io.eps;
    reps = 1.0 / eps;
  }
  const float betaf = (float)betav;

  for (int t = blockIdx.x; t < A.ntiles; t += gridDim.x) {
    const TileDev tile = A.tiles[t];
    const PatchDev P = A.patches[tile.patch];
    const int nx = P.n[0], ny = P.n[1], nz = P.n[2];
    const int lvl = P.level;
    if (tile.flags & 1) {
      // every cell covered: not unknowns
      for (int c = threadIdx.x; c < NC; c += blockDim.x) {
        int ci = c % TX, cj = (c / TX) % TY, ck = c / (TX * TY);
        int i = tile.i0 + ci, j = tile.j0 + cj, k = tile.k0 + ck;
        if (i >= nx || j >= ny || k >= tile.k1) continue;
        int idx = P.off + i + nx * (j + ny * k);
        io.out[idx] = 0.0;
        io.out[N + idx] = 0.0;
      }
      continue;
    }
    if (CELLS) {
      // the split forms' cell launch: the face fluxes come from pef (written
      // by the face launch, each face once), the divergence is formed in the
      // fused kernel's order, so F is bit-identical to it
      const double* pE = io.pef;
      const double* pT = io.pef + NS;
      const int cex = CMP ? min(TX, nx - tile.i0) : TX, cey = CMP ? min(TY, ny - tile.j0) : TY;
      const int nce = CMP ? cex * cey * (tile.k1 - tile.k0) : NC;
      for (int c = threadIdx.x; c < nce; c += blockDim.x) {
        const int ci = c % cex, cj = (c / cex) % cey, ck = c / (cex * cey);
        const int i = tile.i0 + ci, j = tile.j0 + cj, k = tile.k0 + ck;
        if (i >= nx || j >= ny || k >= tile.k1) continue;
        const int idx = P.off + i + nx * (j + ny * k);
        const uint8_t m = A.mask[idx];
        if (m & MASK_COVERED) {
          if (LINC) {
            lin_cell_covered<DZ>(io, N, idx);
          } else {
            io.out[idx] = 0.0;
            io.out[N + idx] = 0.0;
          }
          continue;
        }
        // face slots: an interior face at dir N + the index of the cell on its
        // high side (the face is that cell's low face: cell idx has its low x
        // face at idx and its high x face at idx + 1); patch faces at 3N +
        // their ghost index
        auto gslot = [&](int ff, int a, int b) {
          return 3L * N + P.goff + P.fo[ff] + a + P.n[((ff >> 1) + 1) % 3] * b;
        };
        const long xl = (i == 0) ? gslot(0, j, k) : (long)idx;
        const long xh = (i == nx - 1) ? gslot(1, j, k) : (long)idx + 1;
        const long yl = (j == 0) ? gslot(2, k, i) : (long)N + idx;
        const long yh = (j == ny - 1) ? gslot(3, k, i) : (long)N + idx + nx;
        const long zl = (k == 0) ? gslot(4, i, j) : 2L * N + idx;
        const long zh = (k == nz - 1) ? gslot(5, i, j) : 2L * N + idx + (long)nx * ny;
        auto pick = [](bool skip, double v) { return skip ? 0.0 : v; };
        const double divE = (pick(m & 4, pE[xh]) - pick(m & 2, pE[xl])) +
                            (pick(m & 16, pE[yh]) - pick(m & 8, pE[yl])) +
                            (pick(m & 64, pE[zh]) - pick(m & 32, pE[zl]));
        const double divT = (pick(m & 4, pT[xh]) - pick(m & 2, pT[xl])) +
                            (pick(m & 16, pT[yh]) - pick(m & 8, pT[yl])) +
                            (pick(m & 64, pT[zh]) - pick(m & 32, pT[zl]));
        // own entries: its side's partials of its six faces
        OwnSum own = {0.0, 0.0, 0.0};
        if (LINC) {
          const double* jc = io.jac.jc;
          auto sum = [&](const double* a, const double* b) {
            return (pick(m & 4, a[xh]) - pick(m & 2, b[xl])) +
                   (pick(m & 16, a[yh]) - pick(m & 8, b[yl])) +
                   (pick(m & 64, a[zh]) - pick(m & 32, b[zl]));
          };
          own.EE = sum(jc, jc + NS);
          own.ET = sum(jc + 2 * NS, jc + 2 * NS);
          own.TT = sum(jc + 3 * NS, jc + 4 * NS);
        }
        const double E = io.u[idx], T = io.u[N + idx];
        const double z3c = A.z3[idx];
        auto cell = [&](auto soft) {
          constexpr bool SOFT = decltype(soft)::value;
          if (LINC) {
            lin_cell<DZ, SOFT>(io, N, idx, a0v, dtv, betav, betaf, E, T, z3c, divE, divT, own);
          } else {
            double FE, FT, rT, sig;
            cell_balance<SOFT>(a0v, dtv, E, T, z3c, io.b[idx], io.b[N + idx], divE, divT, FE, FT,
                               rT, sig);
            io.out[idx] = FE;
            io.out[N + idx] = FT;
          }
        };
        if (soft_window(E) && soft_window(T) && soft_window(z3c)) cell(std::true_type{});
        else cell(std::false_type{});
      }
      continue;
    }
    // ---- halo load (face halos only; edges and corners are never read)
    bool soft_ok = A.soft;   // every staged value in the soft window
    for (int hh = threadIdx.x; hh < NH; hh += blockDim.x) {
      int hx_ = hh % HX, hy_ = (hh / HX) % HY, hz_ = hh / (HX * HY);
      int i = tile.i0 + hx_ - 1, j = tile.j0 + hy_ - 1, k = tile.k0 + hz_ - 1;
      int ox = (i < 0) ? -1 : ((i >= nx) ? 1 : 0);
      int oy = (j < 0) ? -1 : ((j >= ny) ? 1 : 0);
      int oz = (k < 0) ? -1 : ((k >= nz) ? 1 : 0);
      if ((ox != 0) + (oy != 0) + (oz != 0) > 1) continue;
      if (i > nx || j > ny || k > tile.k1) continue;
      double e, tt, ve = 0.0, vt = 0.0;
      double z = 0.0;
      if (!ox && !oy && !oz) {
        int idx = P.off + i + nx * (j + ny * k);
        e = io.u[idx];
        tt = io.u[N + idx];
        z = A.z3[idx];
        if (MODE == ST_JV || MODE == ST_FD) {
          ve = io.v[idx];
          vt = io.v[N + idx];
        }
      } else {
        int f, a, b;
        if (ox) { f = ox < 0 ? 0 : 1; a = j; b = k; }
        else if (oy) { f = oy < 0 ? 2 : 3; a = k; b = i; }
        else { f = oz < 0 ? 4 : 5; a = i; b = j; }
        int d = f / 2;
        int nt1 = P.n[(d + 1) % 3];
        int gi = P.goff + P.fo[f] + a + nt1 * b;
        e = io.gu[gi];
        tt = io.gu[G + gi];
        z = A.z3[(long)N + gi];
        if (MODE == ST_JV || MODE == ST_FD) {
          ve = io.gv[gi];
          vt = io.gv[G + gi];
        }
      }
      if (MODE == ST_FD) {
        e += eps * ve;
        tt += eps * vt;
      }
      sE[hh] = e;
      sT[hh] = tt;
      sZ[hh] = z;
      if (FACES) soft_ok = soft_ok && soft_window(e) && soft_window(tt) && soft_window(z);
      if (TAN) {
        svE[hh] = ve;
        svT[hh] = vt;
      }
    }
    bool soft = false;   // block-uniform: the tile's products on the integer pipe
    if (FACES) soft = __syncthreads_and(soft_ok);
    else __syncthreads();
    // ---- face fluxes, each computed once per tile (split forms: once in the launch:
    // the low faces of the tile's cells, and the patch's high boundary faces
    // where the tile ends the patch, enumerated without gaps so that whole
    // warps skip what is not there)
    const int tzl = tile.k1 - tile.k0;
    // the tile's extent inside its patch (a tile at a patch's high end may be
    // narrower than TX x TY): only its cells' faces are enumerated, so that
    // no lane of a warp idles on a face outside the patch (an idle lane
    // still costs its warp's FP64 issue slots)
    const int ex = min(TX, nx - tile.i0), ey = min(TY, ny - tile.j0);
    const bool full = (ex == TX && ey == TY);
    const int nlow = FACES ? ex * ey * tzl : 0;
    const int nbx = (FACES && tile.i0 + ex == nx) ? ey * tzl : 0;
    const int nby = (FACES && tile.j0 + ey == ny) ? ex * tzl : 0;
    const int nbz = (FACES && tile.k1 == nz) ? ex * ey : 0;
    const int nfaces = FACES ? 3 * nlow + nbx + nby + nbz : NFX + NFY + NFZ;
    auto faces = [&](auto softc) {
    constexpr bool SOFT = decltype(softc)::value;
    for (int f = threadIdx.x; f < nfaces; f += blockDim.x) {
      int dir, fi, fj, fk, slot = 0;
      double* outE = nullptr;
      double* outT = nullptr;
      if (FACES) {
        int q = f;
        if (q < 3 * nlow) {
          dir = q / nlow;
          q -= dir * nlow;
          if (full) {
            fi = q % TX; fj = (q / TX) % TY; fk = q / (TX * TY);
          } else {
            fi = q % ex; fj = (q / ex) % ey; fk = q / (ex * ey);
          }
        } else if ((q -= 3 * nlow) < nbx) {
          dir = 0; fi = ex; fj = q % ey; fk = q / ey;
        } else if ((q -= nbx) < nby) {
          dir = 1; fj = ey; fi = q % ex; fk = q / ex;
        } else {
          q -= nby;
          dir = 2; fk = tzl; fi = q % ex; fj = q / ex;
        }
      } else if (f < NFX) {
        dir = 0; slot = f;
        fi = f % (TX + 1); fj = (f / (TX + 1)) % TY; fk = f / ((TX + 1) * TY);
        outE = fxE; outT = fxT;
      } else if (f < NFX + NFY) {
        dir = 1; slot = f - NFX;
        fi = slot % TX; fj = (slot / TX) % (TY + 1); fk = slot / (TX * (TY + 1));
        outE = fyE; outT = fyT;
      } else {
        dir = 2; slot = f - NFX - NFY;
        fi = slot % TX; fj = (slot / TX) % TY; fk = slot / (TX * TY);
        outE = fzE; outT = fzT;
      }
      // face on the low side of tile cell (fi, fj, fk) along dir
      int i = tile.i0 + fi, j = tile.j0 + fj, k = tile.k0 + fk;
      if (i > nx || j > ny || k > tile.k1) continue;
      if ((dir != 0 && i >= nx) || (dir != 1 && j >= ny) || (dir != 2 && k >= tile.k1)) continue;
      int pos = (dir == 0) ? i : ((dir == 1) ? j : k);
      int nd = P.n[dir];
      int hb = (fi + 1) + HX * ((fj + 1) + HY * (fk + 1));   // high-side cell
      int st = (dir == 0) ? 1 : ((dir == 1) ? HX : HX * HY);
      int ha = hb - st;                                      // low-side cell
      const double h = A.lh.h[lvl][dir];
      double PE = 0.0, PT = 0.0;
      uint8_t gt = GT_SIBLING;
      int gi = -1;
      long fslot;                                            // coefficient slot
      if (pos == 0 || pos == nd) {
        int ff = 2 * dir + (pos == nd ? 1 : 0);
        int a, b;
        if (dir == 0) { a = j; b = k; }
        else if (dir == 1) { a = k; b = i; }
        else { a = i; b = j; }
        gi = P.goff + P.fo[ff] + a + P.n[(dir + 1) % 3] * b;
        gt = A.gtype[gi];
        fslot = 3L * N + gi;
      } else {
        fslot = (long)dir * N + P.off + i + (long)nx * (j + (long)ny * k);
      }
      if (gt == GT_NEUMANN) {
        PE = 0.0;
        PT = 0.0;
        if (LIN) {
          for (int q = 0; q < 6; q++) io.jac.jc[q * NS + fslot] = 0.0;
          put_scaled(io, NS, fslot, 0.0, 0.0);
        }
      } else if (gt == GT_ROBIN) {
        int s = (pos == 0) ? -1 : 1;
        int hc = (pos == 0) ? hb : ha;      // the interior cell
        int ff = 2 * dir + (pos == nd ? 1 : 0);
        const double rh = A.lh.rh[lvl][dir];
        if (TAN) {
          PE = rh * robin_tan(sE[hc], sT[hc], sZ[hc], h, A.R[ff], s, svE[hc], svT[hc]);
        } else {
          PE = rh * robin_flux(sE[hc], sT[hc], sZ[hc], h, A.R[ff], s);
        }
        if (LIN) {
          // dPhi/dE_c and dPhi/dT_c over h, the same on both sides (only the
          // cell's own is read); raw P1 slot holds D_b
          double Ec = sE[hc], Tc = sT[hc], zc = sZ[hc];
          double Db = Tc * Tc * Tc / (3.0 * zc);
          double qd = 4.0 * Db + h;
          double rq = 1.0 / qd;
          double m = 2.0 * Ec - 8.0 * A.R[ff];
          double* jc = io.jac.jc + fslot;
          jc[0] = jc[NS] = rh * (-(double)s * 2.0 * Db * rq);
          jc[2 * NS] = -(double)s * (Tc * Tc / zc) * m * rq * rq;
          jc[3 * NS] = jc[4 * NS] = 0.0;
          if (DZ) jc[5 * NS] = (double)s * m * rq * rq * Db / zc;  // d Phi / d z_c^3
          io.craw[fslot] = Db;
          io.craw[NS + fslot] = 0.0;
          put_scaled(io, NS, fslot, betav * 2.0 * Db * rq / h, 0.0);
        }
        PT = 0.0;
      } else {
        if (TAN) {
          flux_tan(sE[ha], sE[hb], sT[ha], sT[hb], sZ[ha], sZ[hb], A.lh.h3[lvl][dir],
                   A.lh.kh[lvl][dir], A.cL, svE[ha], svE[hb], svT[ha], svT[hb], PE, PT);
          PE *= A.lh.rh[lvl][dir];
          PT *= A.lh.rh[lvl][dir];
        } else if (LIN) {
          FaceLin L = flux_lin<SOFT>(sE[ha], sE[hb], sT[ha], sT[hb], sZ[ha], sZ[hb],
                                     A.lh.c1[lvl][dir], A.lh.cLh[lvl][dir], A.lh.cT[lvl][dir],
                                     DZ);
          PE = L.PE;
          PT = L.PT;
          double* jc = io.jac.jc + fslot;
          jc[0] = L.aEa;
          jc[NS] = L.aEb;
          jc[2 * NS] = L.aT;
          jc[3 * NS] = L.bTa;
          jc[4 * NS] = L.bTb;
          if (DZ) jc[5 * NS] = L.aZ;
          // only the scaled P1 coefficients beta D / h^2: the coarsening
          // averages them (raw values are kept for Robin faces alone)
          if (io.a32) {
            io.a32[fslot] = narrow_rn(L.X) * betaf;
            io.a32[NS + fslot] = narrow_rn(L.T25) * betaf;
          } else {
            io.a64[fslot] = L.X * betav;
            io.a64[NS + fslot] = L.T25 * betav;
          }
        } else {
          const FaceCore q = face_core<SOFT>(sE[ha], sE[hb], sT[ha], sT[hb], sZ[ha], sZ[hb],
                                             A.lh.c1[lvl][dir], A.lh.cLh[lvl][dir],
                                             A.lh.cT[lvl][dir]);
          PE = q.PE;
          PT = q.PT;
        }
        if (gt == GT_CF) {
          io.cfflux[gi] = PE;
          io.cfflux[G + gi] = PT;
        }
      }
      if (FACES) {
        io.pef[fslot] = PE;
        io.pef[NS + fslot] = PT;
      } else {
        outE[slot] = PE;
        outT[slot] = PT;
      }
    }
    };
    if (FACES && soft) faces(std::integral_constant<bool, FACES>{});
    else faces(std::false_type{});
    __syncthreads();
    if (FACES) continue;   // the cell launch forms the balance
    // ---- cell balance
    for (int c = threadIdx.x; c < NC; c += blockDim.x) {
      int ci = c % TX, cj = (c / TX) % TY, ck = c / (TX * TY);
      int i = tile.i0 + ci, j = tile.j0 + cj, k = tile.k0 + ck;
      if (i >= nx || j >= ny || k >= tile.k1) continue;
      int idx = P.off + i + nx * (j + ny * k);
      uint8_t m = A.mask[idx];
      if (m & MASK_COVERED) {
        io.out[idx] = 0.0;
        io.out[N + idx] = 0.0;
        continue;
      }
      int xl = ci + (TX + 1) * (cj + TY * ck);
      int yl = ci + TX * (cj + (TY + 1) * ck);
      int zl = ci + TX * (cj + TY * ck);
      // coarse-side coarse-fine faces take their flux from flux matching
      auto pick = [](bool skip, double v) { return skip ? 0.0 : v; };
      double divE = (pick(m & 4, fxE[xl + 1]) - pick(m & 2, fxE[xl])) +
                    (pick(m & 16, fyE[yl + TX]) - pick(m & 8, fyE[yl])) +
                    (pick(m & 64, fzE[zl + TX * TY]) - pick(m & 32, fzE[zl]));
      double divT = (pick(m & 4, fxT[xl + 1]) - pick(m & 2, fxT[xl])) +
                    (pick(m & 16, fyT[yl + TX]) - pick(m & 8, fyT[yl])) +
                    (pick(m & 64, fzT[zl + TX * TY]) - pick(m & 32, fzT[zl]));
      int hc = (ci + 1) + HX * ((cj + 1) + HY * (ck + 1));
      double E = sE[hc], T = sT[hc], z = sZ[hc];
      double T2 = T * T, T3 = T2 * T;
      if (MODE == ST_JV) {
        double rT = 1.0 / T;
        double sig = z * rT * rT * rT;
        double vE = svE[hc], vT = svT[hc];
        double dc = sig * ((T3 + 3.0 * E * rT) * vT - vE);
        io.out[idx] = a0v * vE - dtv * (divE + dc);
        io.out[N + idx] = a0v * vT - dtv * (divT - dc);
      } else {
        double FE, FT, rT, sig;
        cell_balance<false>(a0v, dtv, E, T, z, io.b[idx], io.b[N + idx], divE, divT, FE, FT, rT, sig);
        FE = (FE - io.F0[idx]) * reps;
        FT = (FT - io.F0[N + idx]) * reps;
        io.out[idx] = FE;
        io.out[N + idx] = FT;
      }
    }
    __syncthreads();
  }
}

struct JvArgs {
  const TileDev* tiles;
  const PatchDev* patches;
  const uint8_t* mask;
  const uint8_t* gtype;
  int N, G, tx, ty;
  Jac jac;
  const double* v;
  const double* gv;
  double* out;
  double* cf;
  double a0, dt;
  const double* par;
};

// Frozen Jv: out = a0 v - dt L v, one row sum per cell and field (25.6 FP64
// instructions, counted) over the 19 coefficients of the cell; fine-side coarse-fine
// fluxes to cf for flux matching.  One tile of the stencil list per block.
// In flux form (each face's two tangent fluxes, then the divergence) a cell
// took 40 FP64 instructions and the kernel was bound by the FP64 pipe; the
// rows move 9% more bytes.  Its four plain products run on the integer pipe.
// At 256^3: 1.30 -> 0.73 ms (six blocks per SM; with five 0.78): 0.93 of the
// FP64 issue rate, the bound left, and 0.63 of HBM.  Rounding: a row's order costs
// 0.04 ms against own entries first, whose error with the coefficients given is a
// fifth larger (2.5e-16 against 2.1e-16 in the 2-norm).  The product's distance
// from a 64-bit evaluation of the whole chain is 2.5-2.6e-16 at 256^3, 2.3e-16 in
// flux form: the own entries are sums, rounded before they meet the vector.
// MINB < 6 (few tiles, launch_jv_frozen): the loads of several faces in flight,
// and every cell by the boundary's path, since the cells of small patches mostly
// take it and a warp holding both takes them in turn.
template <int MINB>
__global__ void __launch_bounds__(256, MINB) k_jv_frozen(JvArgs A) {
  constexpr bool FEW = MINB < 6;
  const int N = A.N, G = A.G;
  double a0 = A.a0, dt = A.dt;
  if (A.par) {
    a0 = A.par[0];
    dt = A.par[1];
  }
  const TileDev tile = A.tiles[blockIdx.x];
  const PatchDev P = A.patches[tile.patch];
  const int nx = P.n[0], ny = P.n[1], nz = P.n[2];
  // the tile's extent inside its patch: no lane idles on a cell outside it
  const int ex = min(A.tx, nx - tile.i0), ey = min(A.ty, ny - tile.j0);
  const int nc = ex * ey * (tile.k1 - tile.k0);
  const long s2 = (long)nx * ny;
  const Jac& J = A.jac;
  for (int c = threadIdx.x; c < nc; c += blockDim.x) {
    const int r = c / ex, i = tile.i0 + c - r * ex;
    const int rk = r / ey, j = tile.j0 + r - rk * ey, k = tile.k0 + rk;
    const long idx = P.off + i + nx * (j + (long)ny * k);
    const uint8_t m = A.mask[idx];
    if (m & MASK_COVERED) {
      A.out[idx] = 0.0;
      A.out[N + idx] = 0.0;
      continue;
    }
    const double* vE = A.v;
    const double* vT = A.v + N;
    const double vEc = vE[idx], vTc = vT[idx];
    // A row's largest terms (the diagonal; in the T row the coupling too) come
    // last: fewer of its roundings are then of its full size.  The plain
    // products run on the integer pipe (bit-identical).
    double LE = soft_mul_any(J.cen[N + idx], vTc), LT = 0.0;
    const bool inner = i > 0 && i < nx - 1 && j > 0 && j < ny - 1 && k > 0 && k < nz - 1;
    const long NS = 3L * N + G;
    if (!FEW && inner && m == 0) {
      const long st[3] = {1, nx, s2};
#pragma unroll
      for (int d = 0; d < 3; d++) {
        const long lo = idx - st[d], hi = idx + st[d];
        const double* jl = J.jc + (long)d * N + idx;   // the low face's slots
        const double* jh = jl + st[d];                 // the high face's
        const double tl = vT[lo], th = vT[hi];
        LE = fma(-jl[0], vE[lo], LE);
        LE = fma(-jl[2 * NS], tl, LE);
        LT = d ? fma(-jl[3 * NS], tl, LT) : soft_mul_any(-jl[3 * NS], tl);
        LE = fma(jh[NS], vE[hi], LE);
        LE = fma(jh[2 * NS], th, LE);
        LT = fma(jh[4 * NS], th, LT);
      }
    } else if (FEW) {
      // Every face's kind first, then the loads without branches, so that those of
      // several faces are in flight: one face after the other, each a chain of
      // dependent loads, took most of the time of a few small patches.
      const int pos[3] = {i, j, k};
      auto ghost = [&](int f) {
        const int d = f >> 1;
        return P.goff + P.fo[f] + pos[(d + 1) % 3] + P.n[(d + 1) % 3] * pos[(d + 2) % 3];
      };
      unsigned bnd = 0, use = 0, cf = 0;   // bit f: patch boundary; enters the row; coarse-fine
#pragma unroll
      for (int f = 0; f < 6; f++) {
        if (pos[f >> 1] == (f & 1 ? P.n[f >> 1] - 1 : 0)) bnd |= 1u << f;
        const uint8_t gt = (bnd >> f & 1) ? A.gtype[ghost(f)] : GT_SIBLING;
        // (not: faces taken by flux matching; physical ones, own entries only)
        if (!(m & (2 << f)) && gt != GT_NEUMANN && gt != GT_ROBIN) use |= 1u << f;
        if (gt == GT_CF) cf |= 1u << f;
      }
#pragma unroll
      for (int f = 0; f < 6; f++) {
        const int d = f >> 1, hi = f & 1;
        const long st = (d == 0) ? 1L : (d == 1 ? (long)nx : s2);
        const bool b = bnd >> f & 1, on = use >> f & 1;
        const long n = hi ? idx + st : idx - st;
        const double* jf = J.jc + (b ? 3L * N + ghost(f) : (long)d * N + (hi ? n : idx));
        const double* nv = b ? A.gv + ghost(f) : vE + n;
        const double cE = on ? jf[hi ? NS : 0] : 0.0, cX = on ? jf[2 * NS] : 0.0;
        const double cT = on ? jf[hi ? 4 * NS : 3 * NS] : 0.0;
        const double nE = on ? nv[0] : 0.0, nT = on ? nv[b ? G : N] : 0.0;
        LE = fma(hi ? cE : -cE, nE, LE);
        LE = fma(hi ? cX : -cX, nT, LE);
        LT = fma(hi ? cT : -cT, nT, LT);
      }
      cf &= use;
#pragma unroll
      for (int f = 0; f < 6; f++) {
        if (!(cf >> f & 1)) continue;
        const int hi = f & 1, g = ghost(f);
        const double* jf = J.jc + 3L * N + g;
        const double nE = A.gv[g], nT = A.gv[G + g];
        const double Ea = hi ? vEc : nE, Eb = hi ? nE : vEc;
        const double Ta = hi ? vTc : nT, Tb = hi ? nT : vTc;
        A.cf[g] = fma(jf[0], Ea, fma(jf[NS], Eb, jf[2 * NS] * (Ta + Tb)));
        A.cf[G + g] = fma(jf[3 * NS], Ta, jf[4 * NS] * Tb);
      }
    } else {
      const int pos[3] = {i, j, k};
#pragma unroll
      for (int f = 0; f < 6; f++) {
        if (m & (2 << f)) continue;   // flux matching
        const int d = f >> 1, hi = f & 1;
        const long st = (d == 0) ? 1L : (d == 1 ? (long)nx : s2);
        double nE, nT;
        const double* jf;
        uint8_t gt = GT_SIBLING;
        int g = 0;
        if (pos[d] != (hi ? P.n[d] - 1 : 0)) {
          const long n = hi ? idx + st : idx - st;
          jf = J.jc + (long)d * N + (hi ? n : idx);
          nE = vE[n];
          nT = vT[n];
        } else {
          g = P.goff + P.fo[f] + pos[(d + 1) % 3] + P.n[(d + 1) % 3] * pos[(d + 2) % 3];
          gt = A.gtype[g];
          if (gt == GT_NEUMANN || gt == GT_ROBIN) continue;   // own entries only
          jf = J.jc + 3L * N + g;
          nE = A.gv[g];
          nT = A.gv[G + g];
        }
        LE = fma(hi ? jf[NS] : -jf[0], nE, LE);
        LE = fma(hi ? jf[2 * NS] : -jf[2 * NS], nT, LE);
        LT = fma(hi ? jf[4 * NS] : -jf[3 * NS], nT, LT);
        if (gt == GT_CF) {
          const double Ea = hi ? vEc : nE, Eb = hi ? nE : vEc;
          const double Ta = hi ? vTc : nT, Tb = hi ? nT : vTc;
          A.cf[g] = fma(jf[0], Ea, fma(jf[NS], Eb, jf[2 * NS] * (Ta + Tb)));
          A.cf[G + g] = fma(jf[3 * NS], Ta, jf[4 * NS] * Tb);
        }
      }
    }
    LE = fma(J.cen[idx], vEc, LE);
    LT = fma(J.cen[3L * N + idx], vEc, LT);
    LT = fma(J.cen[2L * N + idx], vTc, LT);
    A.out[idx] = fma(-dt, LE, soft_mul_any(a0, vEc));
    A.out[N + idx] = fma(-dt, LT, soft_mul_any(a0, vTc));
  }
}

struct RfArgs {
  const int* cell;
  const int* off;
  const int* face;
  const int4* g;
  int nrf, N, G;
};

// Flux matching (Sec. 3.2.1): the coarse face flux is the average of the four
// fine fluxes stored by the fine-side stencil (each over the fine h, half the
// coarse one: the coarse flux over its h is 1/8 of their sum); scale = -dt
// (RESIDUAL, JV) or -dt/eps (FD).
__global__ void k_reflux(RfArgs a, const double* cf, double* out, double dt, const double* par,
                         const double* eps, int mode) {
  if (par) dt = par[1];
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < a.nrf; r += gridDim.x * blockDim.x) {
    int c = a.cell[r];
    double sc = -dt;
    if (mode == ST_FD) sc /= *eps;
    double dE = 0.0, dT = 0.0;
    for (int q = a.off[r]; q < a.off[r + 1]; q++) {
      double s = (a.face[q] % 2) ? 0.125 : -0.125;
      int4 g = a.g[q];
      dE += s * (cf[g.x] + cf[g.y] + cf[g.z] + cf[g.w]);
      dT += s * (cf[a.G + g.x] + cf[a.G + g.y] + cf[a.G + g.z] + cf[a.G + g.w]);
    }
    out[c] += sc * dE;
    out[a.N + c] += sc * dT;
  }
}

// Sec. 5 indicators on every cell.  E holds composite values (covered cells
// already averaged from their children); gE its ghosts.
// The indicator decisions sqrt(s) / b > t (and a / b > t) exactly as the
// correctly rounded formula takes them, with the rounded square root and
// division evaluated only near the threshold: the rounded quotient is within
// 3e-16 relative of the exact one, and t b, (t b)^2 within 7e-16, so away
// from a band of 1e-12 around the threshold the squared comparison decides
// the same.  FP64 square roots and divisions are long instruction sequences
// on GB300's FP64 pipe.
// For non-negative doubles (not NaN) the order of the values is the order of
// their bit patterns as signed 64-bit integers, so the comparisons below take
// integer instructions instead of FP64 compares (which issue on GB300's narrow
// FP64 pipe).  A band of 2^14 units in the last place around the threshold is
// at least 1.8e-12 relative (an ulp step is between 2^-53 and 2^-52
// relative), wider than the 1e-12 the exact-decision argument needs.
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
constexpr long long kBits1em290 = 0x03b8f2b061aea072LL;   // 1e-290
constexpr long long kBits1e290 = 0x7c2485ce9e7a065fLL;    // 1e290
constexpr long long kBits1e300 = 0x7e37e43c8800759cLL;    // 1e300
constexpr long long kBand = 1LL << 14;
__device__ __forceinline__ bool fast_range(double x) {
  const long long xb = dbits(x);
  return xb > kBits1em290 && xb < kBits1e290;
}
__device__ __forceinline__ bool sqrt_ratio_gt(double s, double b, double t) {
  const double tb = t * b, tb2 = tb * tb;
  const long long sb = dbits(s), t2b = dbits(tb2);
  if (dbits(b) > 0 && t >= 0.0 && sb >= 0 && fast_range(tb2) && sb < kBits1e300) {
    if (sb > t2b + kBand) return true;
    if (sb < t2b - kBand) return false;
  }
  return sqrt(s) / b > t;
}
__device__ __forceinline__ bool ratio_gt(double a, double b, double t) {
  const double tb = t * b;
  const long long ab = dbits(a), tbb = dbits(tb);
  if (b > 0.0 && t >= 0.0 && ab >= 0 && fast_range(tb) && ab < kBits1e300) {
    if (ab > tbb + kBand) return true;
    if (ab < tbb - kBand) return false;
  }
  return a / b > t;
}

// x 2^k (k = 1, -1, -2) exactly, by adding k to the exponent field when x is
// normal and stays normal (the product of a power of 2 is then exact, so the
// result is bit-identical to the multiplication), x itself for +-0; other
// values (subnormal, near overflow, inf, NaN) take the multiplication.
__device__ __noinline__ double scale2_slow(double x, double f) { return __dmul_rn(f, x); }
template <int K>
__device__ __forceinline__ double scale2(double x) {
  const long long xb = dbits(x);
  const long long e = (xb >> 52) & 0x7ff;
  if (e >= 3 && e <= 2044) return __longlong_as_double(xb + ((long long)K << 52));
  if ((xb & 0x7fffffffffffffffLL) == 0) return x;
  return scale2_slow(x, K == 1 ? 2.0 : (K == -1 ? 0.5 : 0.25));
}

__global__ void k_tag(const TileDev* tiles, const PatchDev* patches, int ntiles, int tx, int ty, int tz,
                      const double* E, const double* gE, double thr_c, double thr_g,
                      double thr_r, const double* emax_p, uint8_t* tags) {
  const double emax = *emax_p;
  const double sc = 0.1 * emax;
  // an infinite threshold never tags: skip that indicator (uniform branch;
  // the enabled ones keep the plain formulas, so decisions are unchanged)
  const bool want_c = thr_c < INFINITY, want_g = thr_g < INFINITY, want_r = thr_r < INFINITY;
  const int nc = tx * ty * tz;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const TileDev tile = tiles[t];
    const PatchDev P = patches[tile.patch];
    const int nx = P.n[0], ny = P.n[1], nz = P.n[2];
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
      int i = tile.i0 + c % tx, j = tile.j0 + (c / tx) % ty, k = tile.k0 + c / (tx * ty);
      if (i >= nx || j >= ny || k >= tile.k1) continue;
      int idx = P.off + i + nx * (j + ny * k);
      double Ec = E[idx];
      double tc = 0.0, tg = 0.0, gr2 = 0.0;
      int pos[3] = {i, j, k};
      for (int d = 0; d < 3; d++) {
        double Ev[2];
        for (int si = 0; si < 2; si++) {
          int q[3] = {i, j, k};
          q[d] += si ? 1 : -1;
          if (q[d] >= 0 && q[d] < P.n[d]) {
            Ev[si] = E[P.off + q[0] + nx * (q[1] + ny * q[2])];
          } else {
            int f = 2 * d + si;
            int a = pos[(d + 1) % 3], b = pos[(d + 2) % 3];
            Ev[si] = gE[P.goff + P.fo[f] + a + P.n[(d + 1) % 3] * b];
          }
        }
        // no contraction: the same roundings as a plain evaluation (the
        // power-of-2 scalings are exact either way)
        if (want_c) tc += fabs(__dadd_rn(__dsub_rn(Ev[1], scale2<1>(Ec)), Ev[0]));
        const double df = __dsub_rn(Ev[1], Ev[0]);
        if (want_g) tg += scale2<-1>(fabs(df));
        if (want_r) gr2 = __dadd_rn(gr2, __dmul_rn(scale2<-2>(df), df));
      }
      uint8_t tag = 0;
      if (want_c && ratio_gt(tc, sc, thr_c)) tag |= 1;
      if (want_g && ratio_gt(tg, sc, thr_g)) tag |= 2;
      if (want_r && sqrt_ratio_gt(gr2, Ec, thr_r)) tag |= 4;
      tags[idx] = tag;
    }
  }
}

// covered cell := mean of its 8 children (children order: x slowest ... as
// listed), for nfield fields stored fstride apart.
__global__ void k_avgdown(const int4* __restrict__ cov, int n, double* x, int nfield,
                          int fstride) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    int4 c = cov[r];
    for (int f = 0; f < nfield; f++) {
      double* xf = x + (long)f * fstride;
      double s = 0.0;
      for (int a = 0; a < 2; a++)
        for (int b = 0; b < 2; b++)
          for (int e = 0; e < 2; e++) s += xf[c.y + a + b * c.z + e * c.w];
      xf[c.x] = s / 8.0;
    }
  }
}

int blocks_for(long n, int bs) {
  long b = (n + bs - 1) / bs;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (int)b;
}

__global__ void k_check_fastmath(const double* x, long n, double* out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    const double v = x[i];
    out[i] = rcp_nr(v);
    out[n + i] = 1.0 / v;
    out[2 * n + i] = rsqrt_nr(v);
    out[3 * n + i] = 1.0 / sqrt(v);
  }
}

__global__ void k_check_narrow(const double* x, long n, float* out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    const double v = x[i];
    out[i] = narrow_rn(v);
    out[n + i] = __double2float_rn(v);
  }
}

__global__ void k_check_softmul(const double* x, const double* y, long n, double* out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    out[i] = soft_mul(x[i], y[i]);
    out[n + i] = __dmul_rn(x[i], y[i]);
    out[2 * n + i] = soft_twice(x[i]);
    out[3 * n + i] = soft_mul_any(x[i], y[i]);
  }
}

LevelH level_h(const Hier& H, double k = 0.01, double cL = 4.0) {
  LevelH lh;
  for (int l = 0; l < NRD_MAX_LEVELS; l++)
    for (int d = 0; d < 3; d++) {
      double h = (l < H.L) ? H.lev[l].h[d] : 1.0;
      lh.h[l][d] = h;
      lh.rh[l][d] = 1.0 / h;
      lh.h3[l][d] = 3.0 * h;
      lh.kh[l][d] = k / h;
      // from the level's extent n = 1/h, one rounding each
      const long double n = (l < H.L) ? H.lev[l].n[d] : 1;
      lh.c1[l][d] = (double)(n * n / 12.0L);
      lh.cLh[l][d] = (double)(0.5L * cL / n);
      lh.cT[l][d] = (double)(std::sqrt(0.03125L) * k * (n * n));
    }
  return lh;
}

// the constants of the faces in the soft window (softfp.h), so that products
// with in-window cell values stay normal
bool soft_constants(const Hier& H, const LevelH& lh) {
  auto in = [](double x) { return x >= 0x1p-64 && x < 0x1p64; };
  for (int l = 0; l < H.L; l++)
    for (int d = 0; d < 3; d++)
      if (!in(lh.c1[l][d]) || !in(lh.cLh[l][d]) || !in(lh.cT[l][d])) return false;
  return true;
}

template <int MODE, int TX, int TY, int TZ>
size_t stencil_smem() {
  if (MODE == ST_LINC || MODE == ST_LINZC || MODE == ST_RESC) return 0;   // cells and faces from global memory
  constexpr int NH = (TX + 2) * (TY + 2) * (TZ + 2);
  constexpr int NF = (TX + 1) * TY * TZ + TX * (TY + 1) * TZ + TX * TY * (TZ + 1);
  // the split forms' face launches keep no fluxes in shared memory
  const bool faces = MODE == ST_LINF || MODE == ST_LINZF || MODE == ST_RESF;
  size_t d = (size_t)NH * (MODE == ST_JV ? 5 : 3) + (faces ? 0 : 2 * (size_t)NF);
  return d * sizeof(double);
}

template <int MODE, int TX, int TY, int TZ, bool CMP, int MINB>
void run_stencil(const StArgs& a, cudaStream_t s) {
  size_t sm = stencil_smem<MODE, TX, TY, TZ>();
  static bool init = false;
  if (!init) {
    cudaFuncSetAttribute(k_stencil<MODE, TX, TY, TZ, CMP, MINB>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    init = true;
  }
  // one tile per CTA: the block scheduler balances tiles of uneven cost
  int grid = a.ntiles;
  if (grid < 1) return;
  k_stencil<MODE, TX, TY, TZ, CMP, MINB><<<grid, 256, sm, s>>>(a);
}

template <int MODE, bool CMP = false, int MINB = min_blocks(MODE)>
void dispatch_tile(const StArgs& a, int tx, int ty, int tz, cudaStream_t s) {
  if (tx == 32 && ty == 8 && tz == 4) run_stencil<MODE, 32, 8, 4, CMP, MINB>(a, s);
  else if (tx == 32 && ty == 4 && tz == 8) run_stencil<MODE, 32, 4, 8, CMP, MINB>(a, s);
  else if (tx == 32 && ty == 2 && tz == 4) run_stencil<MODE, 32, 2, 4, CMP, MINB>(a, s);
  else if (tx == 16 && ty == 8 && tz == 4) run_stencil<MODE, 16, 8, 4, CMP, MINB>(a, s);
  else if (tx == 16 && ty == 4 && tz == 8) run_stencil<MODE, 16, 4, 8, CMP, MINB>(a, s);
  else if (tx == 16 && ty == 8 && tz == 8) run_stencil<MODE, 16, 8, 8, CMP, MINB>(a, s);
  else if (tx == 16 && ty == 4 && tz == 4) run_stencil<MODE, 16, 4, 4, CMP, MINB>(a, s);
  else if (tx == 8 && ty == 8 && tz == 8) run_stencil<MODE, 8, 8, 8, CMP, MINB>(a, s);
  else if (tx == 8 && ty == 8 && tz == 4) run_stencil<MODE, 8, 8, 4, CMP, MINB>(a, s);
  else run_stencil<MODE, 32, 4, 4, CMP, MINB>(a, s);
}

// the cell launches: the compact-cell form where the hierarchy has ragged tiles;
// up to two blocks per SM, registers for a cell's loads in flight instead of more
// blocks (us, cold caches: 8^3 with fine patches the residual's 6.9 -> 5.9, the
// linearisation's 8.9 -> 7.4; 32^3 7.3 -> 6.4 and 9.8 -> 9.0; 48^3, 864 tiles, 18.5
// against 19.6 so)
template <int MODE>
void dispatch_tile_h(const Hier& H, const StArgs& a, cudaStream_t s) {
  if (a.ntiles <= 2 * 152) {
    if (H.ragged) dispatch_tile<MODE, true, 2>(a, H.tile_x, H.tile_y, H.tile_z, s);
    else dispatch_tile<MODE, false, 2>(a, H.tile_x, H.tile_y, H.tile_z, s);
  } else if (H.ragged) dispatch_tile<MODE, true>(a, H.tile_x, H.tile_y, H.tile_z, s);
  else dispatch_tile<MODE, false>(a, H.tile_x, H.tile_y, H.tile_z, s);
}

}  // namespace

void launch_ghost_fill(const Hier& H, const ModelParams& mp, const float* z, const double* u,
                       double* g, int nonlinear, cudaStream_t s) {
  GhostArgs a;
  a.gtype = H.d_gtype;
  a.gface = H.d_gface;
  a.gcell = H.d_gcell;
  a.gt0 = H.d_gt0;
  a.gidx = H.d_gidx;
  a.gw = H.d_gw;
  a.z = z;
  a.N = H.N;
  a.G = H.G;
  for (int f = 0; f < 6; f++) a.R[f] = mp.bc_R[f];
  a.lh = level_h(H);
  if (H.G == 0) return;
  k_ghost_fill<<<blocks_for(H.G, 256), 256, 0, s>>>(a, u, g, nonlinear);
}

__global__ void k_cube(const float* z, long n, double* z3) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    const double v = (double)z[i];
    z3[i] = v * v * v;
  }
}

void launch_cube(const Hier& H, const float* z, const float* gz, double* z3, cudaStream_t s) {
  k_cube<<<blocks_for(H.N, 256), 256, 0, s>>>(z, H.N, z3);
  if (H.G) k_cube<<<blocks_for(H.G, 256), 256, 0, s>>>(gz, H.G, z3 + H.N);
}

void launch_ghost_z(const Hier& H, const float* z, float* gz, cudaStream_t s) {
  if (H.G == 0) return;
  k_ghost_z<<<blocks_for(H.G, 256), 256, 0, s>>>(H.d_gzsrc, z, gz, H.G);
}

void launch_stencil(const Hier& H, const ModelParams& mp, int mode, const StencilIO& io,
                    cudaStream_t s, const double* z3) {
  StArgs a;
  a.z3 = z3;
  a.tiles = H.d_tiles;
  a.patches = H.d_patches;
  a.mask = H.d_mask;
  a.gtype = H.d_gtype;
  a.ntiles = (int)H.tiles.size();
  a.N = H.N;
  a.G = H.G;
  a.cL = (mp.limiter == NRD_LIM_PAPER_LITERAL) ? 2.0 : 4.0;
  for (int f = 0; f < 6; f++) a.R[f] = mp.bc_R[f];
  a.lh = level_h(H, mp.k, a.cL);
  a.soft = soft_constants(H, a.lh);
  a.io = io;
  if (mode == ST_RESIDUAL) {
    // eight blocks per SM cap the registers: at up to that many tiles in all the
    // face launch is faster with four (us: 16^3 in 32x4x4 tiles 12.2 -> 10.1, 64^3 in
    // 8x8x8 43.3 -> 38.6; 96^3, 2,184 tiles, 92.8 against 94.1 with four, 256^3 1368
    // against 1484)
    if (a.ntiles <= 8 * 152)
      dispatch_tile<ST_RESF, false, 4>(a, H.tile_x, H.tile_y, H.tile_z, s);
    else
      dispatch_tile<ST_RESF>(a, H.tile_x, H.tile_y, H.tile_z, s);
    dispatch_tile_h<ST_RESC>(H, a, s);
  } else if (mode == ST_JV) {
    dispatch_tile<ST_JV>(a, H.tile_x, H.tile_y, H.tile_z, s);
  } else if (mode == ST_LIN) {
    dispatch_tile<ST_LINF>(a, H.tile_x, H.tile_y, H.tile_z, s);
    dispatch_tile_h<ST_LINC>(H, a, s);
  } else if (mode == ST_LINZ) {
    dispatch_tile<ST_LINZF>(a, H.tile_x, H.tile_y, H.tile_z, s);
    dispatch_tile_h<ST_LINZC>(H, a, s);
  } else {
    dispatch_tile<ST_FD>(a, H.tile_x, H.tile_y, H.tile_z, s);
  }
}

void launch_reflux(const Hier& H, const StencilIO& io, int mode, cudaStream_t s) {
  if (H.nrf == 0) return;
  RfArgs a;
  a.cell = H.d_rf_cell;
  a.off = H.d_rf_off;
  a.face = H.d_rf_face;
  a.g = H.d_rf_g;
  a.nrf = H.nrf;
  a.N = H.N;
  a.G = H.G;
  k_reflux<<<blocks_for(H.nrf, 128), 128, 0, s>>>(a, io.cfflux, io.out, io.dt, io.par, io.eps,
                                                   mode);
}

void launch_jv_frozen(const Hier& H, const StencilIO& io, cudaStream_t s) {
  JvArgs a;
  a.tiles = H.d_tiles;
  a.patches = H.d_patches;
  a.mask = H.d_mask;
  a.gtype = H.d_gtype;
  a.N = H.N;
  a.G = H.G;
  a.tx = H.tile_x;
  a.ty = H.tile_y;
  a.jac = io.jac;
  a.v = io.v;
  a.gv = io.gv;
  a.out = io.out;
  a.cf = io.cfflux;
  a.a0 = io.a0;
  a.dt = io.dt;
  a.par = io.par;
  const int nt = (int)H.tiles.size();
  const int cells = H.tile_x * H.tile_y * H.tile_z;
  const int bs = std::min(256, cells);
  // Few tiles are bound by the latency of a cell's chain of loads, not by issue:
  // registers for more of them instead of blocks.  Durations with cold caches, us,
  // six blocks per SM -> this: 8^3 with fine patches (18 tiles) 17.1 -> 12.4, base
  // 16^3 + fine band (160 tiles) 13.6 -> 9.5; base 32^3 + band in 8x8x4 tiles 14.6
  // -> 11.3, 64^3 in 8x8x8 tiles (968) 26.2 -> 19.4.  Beyond, 64^3 in 8x8x4 tiles
  // (1480): 23.7 against 24.9 with four.
  if (nt <= 2 * 152) k_jv_frozen<2><<<nt, bs, 0, s>>>(a);
  else if (nt <= 8 * 152) k_jv_frozen<4><<<nt, bs, 0, s>>>(a);
  else k_jv_frozen<6><<<nt, bs, 0, s>>>(a);
}

void launch_tag(const Hier& H, const double* E, const double* gE, double thr_c, double thr_g,
                double thr_r, const double* emax, uint8_t* tags, cudaStream_t s) {
  // tag tiles: reuse the stencil tile list (tiles are at most 32 x 8 x 8)
  k_tag<<<std::min((int)H.tiles.size(), 152 * 8), 256, 0, s>>>(
      H.d_tiles, H.d_patches, (int)H.tiles.size(), H.tile_x, H.tile_y, H.tile_z, E, gE, thr_c, thr_g, thr_r,
      emax, tags);
}

void launch_average_down(const Hier& H, double* x, int nfield, int fstride, cudaStream_t s) {
  for (int l = H.L - 2; l >= 0; l--) {
    if (H.ncov[l] == 0) continue;
    k_avgdown<<<blocks_for(H.ncov[l], 256), 256, 0, s>>>(H.d_cov[l], H.ncov[l], x, nfield,
                                                          fstride);
  }
}

extern "C" int nrd_check_fastmath(const double* x, int64_t n, double* out, cudaStream_t s) {
  if (!x || !out || n < 0) return NRD_EINVAL;
  if (n == 0) return NRD_OK;
  const int grid = (int)std::min<long>(152L * 8, (n + 255) / 256);
  k_check_fastmath<<<grid, 256, 0, s>>>(x, n, out);
  return cudaGetLastError() == cudaSuccess ? NRD_OK : NRD_ECUDA;
}

extern "C" int nrd_check_softmul(const double* x, const double* y, int64_t n, double* out,
                                 cudaStream_t s) {
  if (!x || !y || !out || n < 0) return NRD_EINVAL;
  if (n == 0) return NRD_OK;
  const int grid = (int)std::min<long>(152L * 8, (n + 255) / 256);
  k_check_softmul<<<grid, 256, 0, s>>>(x, y, n, out);
  return cudaGetLastError() == cudaSuccess ? NRD_OK : NRD_ECUDA;
}

extern "C" int nrd_check_narrow(const double* x, int64_t n, float* out, cudaStream_t s) {
  if (!x || !out || n < 0) return NRD_EINVAL;
  if (n == 0) return NRD_OK;
  const int grid = (int)std::min<long>(152L * 8, (n + 255) / 256);
  k_check_narrow<<<grid, 256, 0, s>>>(x, n, out);
  return cudaGetLastError() == cudaSuccess ? NRD_OK : NRD_ECUDA;
}
