// Fine-grid streaming kernels: static transmissibilities (a1), density and
// linear-system population (a2, Eqs. 3-6 and Eq. 19), the basis operators of
// Eqs. 8-11, residual SpMV with a fused 2-norm, and deterministic reductions.
//
// The assembly and the residual march along z (stencil.h); the others are one
// thread per cell over the x-fastest layout.  Either way every array access
// of a warp is a coalesced 256-byte run; the neighbour reads of the 7-point
// stencil hit L1/L2.  FP64 throughout.
#include <cmath>
#include <cstdlib>
#include <limits>

#include "cams_internal.h"
#include "launch.h"
#include "rcp64.h"
#include "stencil.h"

namespace cams {

namespace {

__device__ __forceinline__ void cell_xyz(const Geo& g, long long i, int& x, int& y, int& z) {
  xyz_of(g, i, x, y, z);
}

// 1/d to the last digits; the division itself where the estimate's range
// ends (subnormal, huge, infinite or not a number).
__device__ __forceinline__ double rcp_any(double d) {
  const unsigned ex = ((unsigned)__double2hiint(d) >> 20) & 0x7ffu;
  if (ex - 1u >= 2043u) return 1.0 / d;
  return rcp_halley(d);
}

// A size (2^-300 to 2^300) whose sums, products of three and reciprocals below
// neither overflow nor lose digits.
__device__ __forceinline__ bool moderate(double v) {
  const unsigned ex = ((unsigned)__double2hiint(v) >> 20) & 0x7ffu;
  return ex - 723u <= 600u;
}

// c = 2 A / (h mu) in two parts, hi + lo (hi NaN: not moderate, no use of it).
struct FaceC {
  double hi, lo;
};

// TPFA: T = A / (h/(2 lambda_a) + h/(2 lambda_b)), as n / s with n = c k_a k_b
// and s = k_a + k_b: one reciprocal a face instead of five divisions, which were
// the kernel's time (an FP64 division is a chain of about ten FP64
// instructions).  n and s are formed with their rounding errors, and the quotient
// is corrected by what it leaves of n, so that T is all but correctly rounded:
// without that, five roundings and a reciprocal's made the root mean square error
// 1.1 to 1.3 units where the formula's is 0.71 to 0.80; it is 0.42 now.  (4M
// cells: 979 us as the formula stands, 203 uncorrected, 407 now.)  Where a factor
// is not moderate, zeros among them, the formula as it stands decides.
__device__ __forceinline__ double face_trans(FaceC c, double area, double h, double mu, double ka,
                                             double kb) {
  if (moderate(ka) && moderate(kb) && !isnan(c.hi)) {
    const bool less = __double_as_longlong(ka) < __double_as_longlong(kb);
    const double s = ka + kb, es = (less ? ka : kb) - (s - (less ? kb : ka));
    const double r = rcp_halley(s);
    const double m = c.hi * ka, em = fma(c.lo, ka, fma(c.hi, ka, -m));
    const double n = m * kb, en = fma(em, kb, fma(m, kb, -n));
    const double t = n * r;
    const double left = fma(-t, s, n) + fma(-t, es, en);
    return fma(left, r, t);
  }
  return area / (h / (2.0 * (ka / mu)) + h / (2.0 * (kb / mu)));
}
// the half cell at a Dirichlet face
__device__ __forceinline__ double half_trans(FaceC c, double area, double h, double mu, double k) {
  if (moderate(k) && !isnan(c.hi)) return fma(c.hi, k, c.lo * k);
  return area / (h / (2.0 * (k / mu)));
}

__global__ void k_transmissibility(Geo g, double mu, const double* __restrict__ kx,
                                   const double* __restrict__ ky, const double* __restrict__ kz,
                                   int dirichlet, FaceC cx, FaceC cy, FaceC cz, double* Tx,
                                   double* Ty, double* Tz, double* Tbw, double* Tbe) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  int x, y, z;
  cell_xyz(g, i, x, y, z);
  const double ax = g.dy * g.dz, ay = g.dx * g.dz, az = g.dx * g.dy;
  Tx[i] = x > 0 ? face_trans(cx, ax, g.dx, mu, kx[i - 1], kx[i]) : 0.0;
  Ty[i] = y > 0 ? face_trans(cy, ay, g.dy, mu, ky[i - g.sy], ky[i]) : 0.0;
  Tz[i] = z > 0 ? face_trans(cz, az, g.dz, mu, kz[i - g.sz], kz[i]) : 0.0;
  if (dirichlet) {
    const long long f = y + (long long)g.ny * z;
    if (x == 0) Tbw[f] = half_trans(cx, ax, g.dx, mu, kx[i]);
    if (x == g.nx - 1) Tbe[f] = half_trans(cx, ax, g.dx, mu, kx[i]);
  }
}

__global__ void k_density(long long N, FluidK fl, const double* __restrict__ p, double* rho) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < N) rho[i] = rho_of(fl, p[i]);
}

// Table 1 step 1: A = C + A~, f, eps (Eq. 19) and per-block sums of eps^2.
// fixm (null when no cell is fixed) marks the prescribed-pressure cells of
// Test Case 2 (Sec. 4.2.2), which are eliminated symmetrically: a face with a
// fixed end stores no coupling, a free cell moves w p_j of a fixed
// neighbour j to its right-hand side (p_j holds the prescribed value), and a
// fixed row reads p_i = p_i with a unit diagonal and eps_i = 0.
//
// full (Reading R22): the full-Jacobian step adds what Eq. 3 leaves out of
// the derivative of the equation over rho, rows times V rho: per face (i, j),
// h = T (p_i - p_j) / 2 gives h rho'_i on the diagonal and h rho'_j at (i, j);
// the diagonal also takes - Phi_i rho'_i / rho_i (Phi_i the mass flux
// leaving i).  A p^{nu+1} = f keeps meaning A dp = -F, so f takes X p^nu over
// the free columns.  A is then not symmetric: Ax.. hold the row's lower
// couplings a_{i,i-e}, Axu.. the transposed ones a_{i-e,i}, both at cell i.
//
// Bound by the FP64 unit, so the instructions are counted: a face takes five
// (the halves of the face density are applied once, to the sums; powers of
// two change no digit), the face below along z comes from the cell below, a
// Dirichlet face takes the place of the missing x face, and the density's
// reciprocal is the pivots' one (rcp64.h).  415 us at 4M cells (650 with
// every face formed twice and a division), about 52 instructions a cell.
struct AsmIn {
  const double *p, *rho, *rhon, *Tx, *Ty, *Tz, *Tbw, *Tbe, *src;
  const unsigned char* fixm;
};
struct AsmOut {
  double *Ad, *Ax, *Ay, *Az, *Cacc, *f, *eps, *Axu, *Ayu, *Azu, *red, *scal, *mail;
  unsigned* tick;
};

template <bool kFix, bool kFull>
__global__ void __launch_bounds__(kColThreads, 3) k_assemble(
    Geo g, ColWork w, FluidK fl, double dt, int dirichlet, double pw, double pe, double rhow2,
    double rhoe2, const __grid_constant__ AsmIn in, const __grid_constant__ AsmOut out) {
  const double* __restrict__ p = in.p;
  const double* __restrict__ rho = in.rho;
  const double phidt = fl.phi * (1.0 / dt), inv_V = 1.0 / g.V, half_inv_V = 0.5 * inv_V;
  const double vphidt = g.V * phidt;
  // d rho / dp: c rho for the exponential law, rho0 c for the linear one
  const double dlin = fl.rho0 * fl.c;
  const double ccst = vphidt * (fl.law == 0 ? fl.c : dlin);
  double e2 = 0.0;
  for (unsigned w0 = blockIdx.x; w0 < w.pieces; w0 += gridDim.x) {
    unsigned j;
    int z0, z1;
    if (!col_of(g, w, w0, j, z0, z1)) continue;
    const unsigned y = j / (unsigned)g.nx, x = j - y * (unsigned)g.nx;
    const bool xl = x > 0, xu = x + 1 < (unsigned)g.nx, yl = y > 0, yu = y + 1 < (unsigned)g.ny;
    long long i = j + g.sz * z0;
    double pi = p[i], ri = rho[i];
    bool fi = kFix && in.fixm[i];
    // the face below: twice its coefficient, p_below - p_i, and the cell's data
    double wz = 0.0, dz = 0.0, pz = 0.0, rz = 0.0, Tzl = 0.0;
    bool fz = false;
    if (z0 > 0) {
      rz = rho[i - g.sz];
      Tzl = in.Tz[i];
      wz = Tzl * (ri + rz);
      pz = p[i - g.sz];
      dz = pz - pi;
      fz = kFix && in.fixm[i - g.sz];
    }
    for (int z = z0; z < z1; ++z, i += g.sz) {
      const bool zu = z + 1 < g.nz;
      const long long fb = y + (long long)g.ny * z;
      // every load of the cell, before the first use
      const double rn = in.rhon[i];
      double Txl, Txu, pxl, pxu, rxl, rxu;
      if (xl) { Txl = in.Tx[i]; pxl = p[i - 1]; rxl = rho[i - 1]; }
      else { Txl = dirichlet ? in.Tbw[fb] : 0.0; pxl = dirichlet ? pw : 0.0; rxl = 0.0; }
      if (xu) { Txu = in.Tx[i + 1]; pxu = p[i + 1]; rxu = rho[i + 1]; }
      else { Txu = dirichlet ? in.Tbe[fb] : 0.0; pxu = dirichlet ? pe : 0.0; rxu = 0.0; }
      const double Tyl = yl ? in.Ty[i] : 0.0, pyl = yl ? p[i - g.sy] : 0.0;
      const double ryl = yl ? rho[i - g.sy] : 0.0;
      const double Tyu = yu ? in.Ty[i + g.sy] : 0.0, pyu = yu ? p[i + g.sy] : 0.0;
      const double ryu = yu ? rho[i + g.sy] : 0.0;
      const double Tzu = zu ? in.Tz[i + g.sz] : 0.0, pzu = zu ? p[i + g.sz] : 0.0;
      const double rzu = zu ? rho[i + g.sz] : 0.0;
      const double q = in.src ? in.src[i] * inv_V : 0.0;
      bool fxl = false, fxu = false, fyl = false, fyu = false, fzu = false;
      if constexpr (kFix) {
        fxl = xl && in.fixm[i - 1]; fxu = xu && in.fixm[i + 1];
        fyl = yl && in.fixm[i - g.sy]; fyu = yu && in.fixm[i + g.sy];
        fzu = zu && in.fixm[i + g.sz];
      }
      // Reading R4: face density = arithmetic mean of the two cell densities
      // (w.. hold twice the face's coefficient; the prescribed density of a
      // Dirichlet face is given doubled)
      const double sxl = ri + rxl, sxu = ri + rxu;
      const double wxl = Txl * (xl ? sxl : rhow2), wxu = Txu * (xu ? sxu : rhoe2);
      const double wyl = Tyl * (ri + ryl), wyu = Tyu * (ri + ryu), wzu = Tzu * (ri + rzu);
      // absent faces: their difference counts as zero whatever p_i is
      const bool bx = dirichlet != 0;
      const double dxl = xl || bx ? pi - pxl : 0.0, dxu = xu || bx ? pi - pxu : 0.0;
      const double dyl = yl ? pi - pyl : 0.0, dyu = yu ? pi - pyu : 0.0;
      const double dzu = zu ? pi - pzu : 0.0;
      double d2 = wxl + wxu;
      d2 += wyl; d2 += wyu; d2 += wz; d2 += wzu;
      double fl2 = wxl * dxl;
      fl2 += wxu * dxu; fl2 += wyl * dyl; fl2 += wyu * dyu; fl2 -= wz * dz; fl2 += wzu * dzu;
      double rhs2 = 0.0;
      if (bx && !(kFix && fi)) {
        if (!xl) rhs2 += wxl * pw;
        if (!xu) rhs2 += wxu * pe;
      }
      const bool cut = kFix && fi;
      if constexpr (kFix) {
        if (!fi) {
          if (fxl) rhs2 += wxl * pxl;
          if (fxu) rhs2 += wxu * pxu;
          if (fyl) rhs2 += wyl * pyl;
          if (fyu) rhs2 += wyu * pyu;
          if (fz) rhs2 += wz * pz;
          if (fzu) rhs2 += wzu * pzu;
        }
      }
      // FP64 divisions are long dependent sequences on this GPU
      const double rinv = rcp_any(ri);
      // Eq. 4 with d phi/dp = 0, then the row scaling V rho (Reading R7):
      // C = V rho phi/dt rho^n rho' / rho^2
      // (rn / ri corrected to its last digit: b is phi/dt times what it differs from 1
      // by, and a product with a reciprocal that may be off by one digit showed there;
      // 721 us for 707 uncorrected, 757 with a division, 4M cells and the density)
      const double t0 = rn * rinv, t = fma(fma(-t0, ri, rn), rinv, t0);
      const double C = ccst * (fl.law == 0 ? rn : t);
      const double b = fma(phidt, t, q - phidt);         // Eq. 5
      const double flux = fl2 * half_inv_V;              // over V
      double xdiag = 0.0, xp = 0.0;
      double ax = xl && !cut && !fxl ? -0.5 * wxl : 0.0;
      double ay = yl && !cut && !fyl ? -0.5 * wyl : 0.0;
      double az = !cut && !fz && z > 0 ? -0.5 * wz : 0.0;
      if constexpr (kFull) {
        const double drho = fl.law == 0 ? fl.c * ri : dlin;
        double axu = 0.0, ayu = 0.0, azu = 0.0;
#define CAMS_JFACE(cond, T, dp, fj, pj, rj, lowslot)                           \
        if (cond) {                                                            \
          const double h = 0.5 * (T) * (dp);                                   \
          xdiag += h * drho;                                                   \
          if (!(kFix && (fi || (fj)))) {                                       \
            const double drj = fl.law == 0 ? fl.c * (rj) : dlin;               \
            xp += h * drj * (pj);                                              \
            lowslot;                                                           \
          }                                                                    \
        }
        // a lower face also gives the transposed entry a_{j,i} = -w - h rho'_i
        CAMS_JFACE(xl, Txl, dxl, fxl, pxl, rxl, (axu = ax - h * drho, ax += h * drj))
        CAMS_JFACE(xu, Txu, dxu, fxu, pxu, rxu, (void)0)
        CAMS_JFACE(yl, Tyl, dyl, fyl, pyl, ryl, (ayu = ay - h * drho, ay += h * drj))
        CAMS_JFACE(yu, Tyu, dyu, fyu, pyu, ryu, (void)0)
        CAMS_JFACE(z > 0, Tzl, -dz, fz, pz, rz, (azu = az - h * drho, az += h * drj))
        CAMS_JFACE(zu, Tzu, dzu, fzu, pzu, rzu, (void)0)
#undef CAMS_JFACE
        xdiag -= 0.5 * fl2 * drho * rinv;
        out.Axu[i] = axu; out.Ayu[i] = ayu; out.Azu[i] = azu;
      }
      out.Ax[i] = ax; out.Ay[i] = ay; out.Az[i] = az;
      out.Cacc[i] = C;
      double e = 0.0;
      if (cut) {
        out.Ad[i] = 1.0;
        out.f[i] = pi;
      } else {
        double fv = fma(g.V * ri, b, C * pi);
        if (kFix || bx) fv += 0.5 * rhs2;
        double ad = fma(0.5, d2, C);
        if constexpr (kFull) {
          ad += xdiag;
          fv += xdiag * pi + xp;
        }
        out.Ad[i] = ad;
        out.f[i] = fv;
        e = fma(-flux, rinv, b);                         // Eq. 19
      }
      out.eps[i] = e;
      e2 += e * e;
      wz = wzu; dz = dzu; pz = pi; fz = fi; rz = ri; Tzl = Tzu;
      pi = pzu; ri = rzu; fi = fzu;
    }
  }
  if (finish_sum(block_sum(e2), out.red, out.tick, out.scal)) out.mail[0] = out.scal[0];
}

// Prescribed cells in list order (a repeated cell keeps its last value):
// mark the cell and put its value into the iterate.
__global__ void k_fix_cells(int n, const int* __restrict__ cell, const double* __restrict__ val,
                            unsigned char* fixm, double* p, long long N) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  for (int k = 0; k < n; ++k) {
    const int c = cell[k];
    if (c >= 0 && c < N) {
      fixm[c] = 1;
      p[c] = val[k];
    }
  }
}

__global__ void k_add_sources(int n, const int* __restrict__ cell, const double* __restrict__ rate,
                              double* src, long long N) {
  // single thread: repeated cells add up in list order (deterministic)
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  for (int k = 0; k < n; ++k) {
    const int c = cell[k];
    if (c >= 0 && c < N) src[c] += rate[k];
  }
}

// r = f - A p and ||r||^2, with the inner loop's bookkeeping by the thread
// that completes the sum.  r32 (null unless wanted): r rounded to FP32 once,
// for the mixed preconditioner's restriction and smoothing steps, which would
// otherwise each round it again (an FP64-unit conversion per cell).
//
// The loop's stopping test (Sec. 4.1.1): scal[0] is ||f - A p||^2 of the
// current iterate, scal[1] the same at the start of the linearisation,
// scal[2] the iterations run.  The test is the host loop's, in the same FP64
// operations: continue while ||r|| >= lin_rtol ||r^0|| (and finite) and fewer
// than max_cams iterations have run.
__global__ void __launch_bounds__(kColThreads, 4) k_residual(
    Geo g, ColWork w, const double* __restrict__ Ad, const double* __restrict__ Ax,
    const double* __restrict__ Ay, const double* __restrict__ Az, const double* __restrict__ Axu,
    const double* __restrict__ Ayu, const double* __restrict__ Azu, const double* __restrict__ f,
    const double* __restrict__ p, double* r, float* r32, double* red, unsigned* tick, double* scal,
    double* mail, LoopCtl ctl) {
  pdl_enter();
  const double s2 = block_sum(residual_columns(g, w, Ad, Ax, Ay, Az, Axu, Ayu, Azu, f, p, r, r32));
  if (!finish_sum(s2, red, tick, scal)) return;
  if (ctl.mode == LoopCtl::kBegin) {
    scal[1] = scal[0];
    scal[2] = 0.0;
  } else if (ctl.mode == LoopCtl::kTest) {
    const double its = scal[2] + 1.0;
    scal[2] = its;
    const double rn = sqrt(scal[0]), r0 = sqrt(scal[1]);
    const bool more = its < (double)ctl.max_cams && isfinite(rn) && !(rn < ctl.lin_rtol * r0);
    cudaGraphSetConditional(ctl.cond, more ? 1u : 0u);
    mail[2] = its;
  }
  mail[0] = scal[0];
}

// Basis operators A_b (Eqs. 8-11, Reading R10: internal faces only).
// Prescribed cells (fixm, null when none) are eliminated as in A: no
// coupling across a face with a fixed end, the free row keeps the face on
// its diagonal, a fixed row is a unit row.
__global__ void k_basis_operator(Geo g, FluidK fl, int kind, double dt,
                                 const double* __restrict__ Tx, const double* __restrict__ Ty,
                                 const double* __restrict__ Tz, const double* __restrict__ rho,
                                 const double* __restrict__ Cacc, const double* __restrict__ pn,
                                 const unsigned char* __restrict__ fixm, double* Abd, double* Abx,
                                 double* Aby, double* Abz) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  int x, y, z;
  cell_xyz(g, i, x, y, z);
  const bool fi = fixm && fixm[i];
  if (fi) {
    Abd[i] = 1.0; Abx[i] = 0.0; Aby[i] = 0.0; Abz[i] = 0.0;
    return;
  }
  // (B1), (B2): rho_f-weighted faces, the couplings of A; (B3), (B4): T
  const double ri = kind <= 2 ? rho[i] : 0.0;
  double bx = 0.0, by = 0.0, bz = 0.0, d = 0.0;
#define CAMS_BFACE(cond, T, j, lowslot)                                 \
  if (cond) {                                                           \
    const double w = kind <= 2 ? (T) * (0.5 * (ri + rho[j])) : (T);     \
    d += w;                                                             \
    if (!(fixm && fixm[j])) { lowslot; }                                \
  }
  CAMS_BFACE(x > 0, Tx[i], i - 1, bx = -w)
  CAMS_BFACE(x < g.nx - 1, Tx[i + 1], i + 1, (void)0)
  CAMS_BFACE(y > 0, Ty[i], i - g.sy, by = -w)
  CAMS_BFACE(y < g.ny - 1, Ty[i + g.sy], i + g.sy, (void)0)
  CAMS_BFACE(z > 0, Tz[i], i - g.sz, bz = -w)
  CAMS_BFACE(z < g.nz - 1, Tz[i + g.sz], i + g.sz, (void)0)
#undef CAMS_BFACE
  if (kind == 1) d += Cacc[i];
  if (kind == 3) {
    const double pp = pn[i];
    const double r = rho_of(fl, pp);
    const double dr = fl.law == 0 ? fl.c * fl.rho0 * exp(fl.c * pp) : fl.rho0 * fl.c;
    d += g.V * (fl.phi * r * dr / (dt * r * r));   // V c^n, Eq. 4 at p = p^n
  }
  Abd[i] = d; Abx[i] = bx; Aby[i] = by; Abz[i] = bz;
}

inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_transmissibility(const Geo& g, double mu, const double* kx, const double* ky,
                                    const double* kz, int dirichlet, Buffers& b, cudaStream_t s) {
  auto factor = [&](double a, double d, double h) {
    const double area = a * d, hm = h * mu, c = 2.0 * area / hm;
    for (double v : {area, hm, c})
      if (!std::isnormal(v) || std::abs(std::ilogb(v)) > 300)
        return FaceC{std::numeric_limits<double>::quiet_NaN(), 0.0};
    // what c leaves of 2 a d / (h mu), products exact
    const double left = std::fma(-c, hm, 2.0 * area) + 2.0 * std::fma(a, d, -area) - c * std::fma(h, mu, -hm);
    return FaceC{c, left / hm};
  };
  k_transmissibility<<<blocks_for(g.N, 256), 256, 0, s>>>(
      g, mu, kx, ky, kz, dirichlet, factor(g.dy, g.dz, g.dx), factor(g.dx, g.dz, g.dy),
      factor(g.dx, g.dy, g.dz), b.Tx, b.Ty, b.Tz, b.Tbw, b.Tbe);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_density(const Geo& g, const FluidK& fl, const double* p, double* rho,
                           cudaStream_t s) {
  k_density<<<blocks_for(g.N, 256), 256, 0, s>>>(g.N, fl, p, rho); count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_assemble(const Geo& g, const FluidK& fl, double dt, int dirichlet, double pw,
                            double pe, const unsigned char* fixm, bool full, Buffers& b,
                            cudaStream_t s) {
  const double rhow = fl.law == 0 ? fl.rho0 * std::exp(fl.c * pw) : fl.rho0 * (1.0 + fl.c * pw);
  const double rhoe = fl.law == 0 ? fl.rho0 * std::exp(fl.c * pe) : fl.rho0 * (1.0 + fl.c * pe);
  const AsmIn in{b.p, b.rho, b.rhon, b.Tx, b.Ty, b.Tz, b.Tbw, b.Tbe, b.src, fixm};
  const AsmOut out{b.Ad, b.Ax, b.Ay, b.Az, b.Cacc, b.f, b.eps, b.Axu, b.Ayu, b.Azu, b.red, b.scal,
                   b.mail, b.tick};
  auto* kern = fixm ? (full ? k_assemble<true, true> : k_assemble<true, false>)
                    : (full ? k_assemble<false, true> : k_assemble<false, false>);
  const ColWork w = col_work(g);
  kern<<<col_grid(w), kColThreads, 0, s>>>(g, w, fl, dt, dirichlet, pw, pe,
                                           dirichlet ? 2.0 * rhow : 0.0,
                                           dirichlet ? 2.0 * rhoe : 0.0, in, out);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_add_sources(int n, const int* cell, const double* rate, double* src,
                               long long N, cudaStream_t s) {
  k_add_sources<<<1, 32, 0, s>>>(n, cell, rate, src, N); count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_fix_cells(int n, const int* cell, const double* val, unsigned char* fixm,
                             double* p, long long N, cudaStream_t s) {
  k_fix_cells<<<1, 32, 0, s>>>(n, cell, val, fixm, p, N); count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_residual(const Geo& g, const Buffers& b, cudaStream_t s, const LoopCtl& ctl) {
  const ColWork w = col_work(g);
  count_launches(1);
  return launch_after(pdl_grid(g), k_residual, dim3(col_grid(w)), kColThreads, 0, s, g, w, b.Ad, b.Ax, b.Ay,
                      b.Az, b.Axu, b.Ayu, b.Azu, b.f, b.p, b.r, b.f32.r, b.red, b.tick, b.scal, b.mail, ctl);
}

cudaError_t launch_basis_operator(const Geo& g, const FluidK& fl, int kind, double dt,
                                  const unsigned char* fixm, Buffers& b, cudaStream_t s) {
  k_basis_operator<<<blocks_for(g.N, 256), 256, 0, s>>>(g, fl, kind, dt, b.Tx, b.Ty, b.Tz, b.rho,
                                                        b.Cacc, b.pn, fixm, b.Abd, b.Abx, b.Aby,
                                                        b.Abz); count_launches(1);
  return cudaGetLastError();
}

}  // namespace cams
