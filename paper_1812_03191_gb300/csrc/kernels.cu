// kernels.cu -- sm_103a kernels of one level step of the nested-mesh solver
// (Velasco Romero & Masset 2018, Sec. 3) and of the inter-level operators.
//
// Each stencil kernel but the fused transport sweeps (whose lanes march through a box) is
// one thread per element of a box (flattened, x fastest, so consecutive threads touch
// consecutive addresses).  A kernel applies its operator
// to the elements of the box where its stencil fits inside the padded array; the
// host picks the box (the active cells plus the margin whose values can still reach
// them before the next ghost fill).  T is the state type (double, or float for the
// FP32-state form); time steps, the force and the frontier flux sums are FP64.
//
// The state is stored as deviations from the uniform background of Sec. 3.4:
// drho = rho - rho0, de = e - e0, dv = v - V.  Every flux is written so that its
// background part cancels exactly (the mass flux F' = F - rho0 V_d A dt, etc.);
// the algebra is that of the plain fields, but rounding scales with the
// perturbation instead of the background, which the FP32 state needs (the drag
// is a small difference of large contributions).
#include "internal.h"

#include <math.h>

#include <type_traits>
#include <utility>

namespace dfn {

namespace {

constexpr int kBlock = kBlockThreads;

// box element t -> (i, j, k); boxes hold fewer than 2^31 elements
__device__ __forceinline__ bool decode(const Box& b, unsigned t, int& i, int& j, int& k) {
  unsigned bx = b.hi[0] - b.lo[0], by = b.hi[1] - b.lo[1], bz = b.hi[2] - b.lo[2];
  if (b.tile == 0) {
    unsigned plane = bx * by;
    if (t >= plane * bz) return false;
    unsigned kk = (unsigned)(((unsigned long long)t * b.mp) >> b.sp);  // t / plane
    unsigned r = t - kk * plane;
    unsigned jj = (unsigned)(((unsigned long long)r * b.mx) >> b.sx);  // r / bx
    i = b.lo[0] + (int)(r - jj * bx);
    j = b.lo[1] + (int)jj;
    k = b.lo[2] + (int)kk;
    return true;
  }
  const unsigned tx = tile_extent(b.tile, 0), ty = tile_extent(b.tile, 1);
  const unsigned tz = tile_extent(b.tile, 2);
  unsigned nx = (bx + tx - 1) / tx, ny = (by + ty - 1) / ty;
  unsigned T = t >> 8, l = t & 255u;
  unsigned Tz = T / (nx * ny), r = T - Tz * nx * ny;
  unsigned Ty = r / nx, Tx = r - Ty * nx;
  unsigned lz = l / (tx * ty), r2 = l - lz * tx * ty;
  unsigned ly = r2 / tx, lx = r2 - ly * tx;
  unsigned ii = Tx * tx + lx, jj = Ty * ty + ly, kk = Tz * tz + lz;
  if (ii >= bx || jj >= by || kk >= bz) return false;
  i = b.lo[0] + (int)ii;
  j = b.lo[1] + (int)jj;
  k = b.lo[2] + (int)kk;
  return true;
}

__device__ __forceinline__ int cidx(const LevelView& L, int i, int j, int k) {
  return (k * L.s[1] + j) * L.s[0] + i;
}

// Division on the hot path.  FP64: one Newton-Raphson refinement of the hardware
// reciprocal estimate (r <- r + r(1 - b r)), then one residual correction
// q <- q + r(a - b q) (Markstein, IBM J. Res. Dev. 34 (1990)): the corrected
// quotient's error is the square of the refined reciprocal's plus the final
// rounding, within one ulp for the normal, non-zero divisors used here (densities,
// 1 + a, and the sum of two same-signed slopes).  FP32: the product with the hardware
// reciprocal estimate.  Its bits were those of __fdividef in all of 4 x 2^22 quotients over
// normal divisors up to 2^126 (relative error at most 1.6e-7), which spends more on larger
// ones; a sum of two slopes whose product is positive is above 2^-74, far from the
// subnormals that the estimate flushes.  Per coarse step, __fdividef and this: three levels
// of 64^3 362 and 333 us, three of 96^3 772 and 735 us, five of 128^3 6.26 and 6.13 ms.
__device__ __forceinline__ double hdiv(double a, double b) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  r = fma(r, fma(-b, r, 1.0), r);
  double q = a * r;
  return fma(r, fma(-b, q, a), q);
}
__device__ __forceinline__ float hdiv(float a, float b) { return a * rcp_est(b); }
__device__ __forceinline__ df64 hdiv(df64 a, df64 b) { return a / b; }
// product and quotient whose result only feeds more arithmetic: in double-float left
// without the final renormalisation (mul_u, div_u in df64.h), in FP32 the plain ones
__device__ __forceinline__ float mul_u(float a, float b) { return a * b; }
__device__ __forceinline__ float div_u(float a, float b) { return a * rcp_est(b); }
// likewise the sum, the difference and p - a of a float p (add_u, sub_u, fsub_u there); a
// sum that is divided by and may cancel (div_sum there)
__device__ __forceinline__ float div_sum(float n, float a, float b) { return div_u(n, a + b); }
__device__ __forceinline__ float add_u(float a, float b) { return a + b; }
__device__ __forceinline__ float sub_u(float a, float b) { return a - b; }
__device__ __forceinline__ float fsub_u(float p, float a) { return p - a; }
__device__ __forceinline__ float norm(float a) { return a; }

// The stencils' arithmetic type C = Arith<T> (internal.h): float for the FP32 state,
// double-float for the FP64 state.  Loads convert the stored value to C, stores round
// C back to the state type.
// The FP64 state is stored as pairs whose values are doubles (dstate, df64.h): loads
// take the pair as it is, stores cut lo onto the pair's grid.
__device__ __forceinline__ float ld(const float* __restrict__ p, int i) { return p[i]; }
__device__ __forceinline__ df64 ld(const df64* __restrict__ p, int i) { return p[i]; }
__device__ __forceinline__ df64 ld(const dstate* __restrict__ p, int i) {
  const dstate v = p[i];
  return df64(v.hi, v.lo);
}
__device__ __forceinline__ void st(df64* p, int i, df64 v) { p[i] = v; }
__device__ __forceinline__ void st(float* p, int i, float v) { p[i] = v; }
__device__ __forceinline__ void st(dstate* p, int i, df64 v) {
  const df64 c = canonical(v);
  p[i] = dstate{c.hi, c.lo};
}
__device__ __forceinline__ bool is0(float v) { return v == 0.f; }
__device__ __forceinline__ bool is0(df64 v) { return v.hi == 0.f; }
// Sums and products with a per-item constant k that is often zero (the background
// wind has one nonzero component): in double-float the operation is skipped when k is
// 0, which gives the same value (a normalised pair plus zero is that pair); in FP32
// the plain expression.  x + k, and x - k y:
__device__ __forceinline__ float add_k(float x, float k) { return k + x; }
__device__ __forceinline__ df64 add_k(df64 x, df64 k) { return k.hi == 0.f ? x : k + x; }
__device__ __forceinline__ float sub_ky(float x, float k, float y) { return x - k * y; }
__device__ __forceinline__ df64 sub_ky(df64 x, df64 k, df64 y) {
  return k.hi == 0.f ? x : x - mul_u(k, y);
}
// k y + z
__device__ __forceinline__ float ky_add(float k, float y, float z) { return k * y + z; }
__device__ __forceinline__ df64 ky_add(df64 k, df64 y, df64 z) {
  return k.hi == 0.f ? z : mul_u(k, y) + z;
}
// e/rho - e0/rho0 of a cell from its deviations, (de - eps0 drho)/(rho0 + drho): one
// expression for every kernel that forms it, so that all give the same bits.  Its
// consumers only take differences of it, so the quotient stays unnormalised; dividend and
// divisor are normalised, since both cancel where the gas is rarefied (left unnormalised,
// the quotient was off by 6e-11 at a hundredth of the background density and by 6e-7 at
// 1e-4, against 1.4e-12 and 1.5e-10, and a FP64 coarse step 0.9 % shorter).
template <class C, class B>
__device__ __forceinline__ C eps_dev(C de, C dr, const B& bg) {
  return div_sum(de - mul_u(bg.eps0, dr), bg.rho0, dr);
}
// a value as a store of the state keeps it (the FP64 state's stores cut lo)
__device__ __forceinline__ float as_stored(float v) { return v; }
__device__ __forceinline__ df64 as_stored(df64 v) { return canonical(v); }
// two neighbouring elements e, e + 1 (e even) in one vector store
__device__ __forceinline__ void st2(float* p, int e, float a, float b) {
  *reinterpret_cast<float2*>(p + e) = make_float2(a, b);
}
__device__ __forceinline__ void st2(dstate* p, int e, df64 a, df64 b) {
  const df64 ca = canonical(a), cb = canonical(b);
  *reinterpret_cast<float4*>(p + e) = make_float4(ca.hi, ca.lo, cb.hi, cb.lo);
}
// A kicked velocity before the fused sweeps.  Where the level step's velocity recovery
// stores the velocity again (`again`), the FP64 state's value stays unrounded until then,
// so that the momenta, which the x sweep forms from it, lose nothing to the cut.
__device__ __forceinline__ void st_kicked(float* p, int i, float v, bool) { p[i] = v; }
__device__ __forceinline__ void st_kicked(dstate* p, int i, df64 v, bool again) {
  const df64 c = canonical(v);
  p[i] = again ? dstate{v.hi, v.lo} : dstate{c.hi, c.lo};
}
// A state value in the state's own type, for the kernels that compute in it (the
// boundary fill, CommMean, the time step, I/O): the float itself, or the exact double
// of a stored pair; put() stores such a value back (a double rounded to the pair).
__device__ __forceinline__ float val(const float* __restrict__ p, int i) { return p[i]; }
__device__ __forceinline__ double val(const dstate* __restrict__ p, int i) {
  return to_double(ld(p, i));
}
__device__ __forceinline__ void put(float* p, int i, float x) { p[i] = x; }
__device__ __forceinline__ void put(dstate* p, int i, double x) { st(p, i, to_df64(x)); }
// exact scalings by 1/2, 2 and other powers of two
__device__ __forceinline__ float pow2_times(float v, float p) { return p * v; }
__device__ __forceinline__ df64 pow2_times(df64 v, float p) { return scale(v, p); }
__device__ __forceinline__ float halve(float v) { return 0.5f * v; }
__device__ __forceinline__ df64 halve(df64 v) { return scale(v, 0.5f); }
__device__ __forceinline__ float twice(float v) { return 2.f * v; }
__device__ __forceinline__ df64 twice(df64 v) { return scale(v, 2.f); }
__device__ __forceinline__ double as_double(float v) { return (double)v; }
__device__ __forceinline__ double as_double(df64 v) { return to_double(v); }
template <class C>
__device__ __forceinline__ C from_double(double x) {
  return (C)x;
}
template <>
__device__ __forceinline__ df64 from_double<df64>(double x) {
  return to_df64(x);
}

// sign tests of the arithmetic types (double-float: df64.h)
__device__ __forceinline__ bool gt0(float v) { return v > 0.f; }
__device__ __forceinline__ bool le0(float v) { return v <= 0.f; }
__device__ __forceinline__ bool lt0(float v) { return v < 0.f; }

// Half the van Leer (1977) harmonic limited slope (Sec. 3.2.1 cites it for the
// interpolation): dl dr / (dl + dr) where dl dr > 0, else 0.  Callers fold the
// factor 2 into their coefficients; scaling by 2 is exact, so the results equal
// those of the full slope bit for bit.  When the product underflows to zero the
// slope is zero, so the divisor dl + dr is never zero or subnormal.  The product and
// the quotient stay unnormalised (mul_u, div_u): the slope only feeds more arithmetic.
template <class C>
__device__ __forceinline__ C hslope(C dl, C dr) {
  C pr = mul_u(dl, dr);
  return le0(pr) ? C(0.f) : div_u(pr, add_u(dl, dr));
}

// The upwind side's value, slopes and coefficient are selected first, so one limiter
// (one division) serves both flow directions: u > 0 gives qm + (1 - cour)/2 * slope,
// u <= 0 gives q0 + (-1 - cour)/2 * slope = q0 - (1 + cour)/2 * slope, with
// (+-1 - cour)/2 * slope = (+-1 - cour) * hslope.  In double-float the operands of
// the two one-sided differences are selected before subtracting (two subtractions of
// 11 instructions, not three); in FP32, where a subtraction costs what a selection does,
// the three differences are formed and the results selected (the same values).  The
// separate transport kernels' form; the fused sweeps have the differences (upwind_d).
template <class C>
__device__ __forceinline__ C upwind_v(C qmm, C qm, C q0, C qp, C u, C cour) {
  const bool up = gt0(u);
  const C a = up ? qm : q0;
  C dl, dr;
  if constexpr (sizeof(C) == 4) {
    const C dm = q0 - qm;
    dl = up ? qm - qmm : dm;
    dr = up ? dm : qp - q0;
  } else {
    dl = a - (up ? qmm : qm);
    dr = (up ? q0 : qp) - a;
  }
  return add_u(a, mul_u(fsub_u(up ? 1.f : -1.f, cour), hslope(dl, dr)));
}

template <class P, class C>
__device__ __forceinline__ C upwind(const P* __restrict__ q, int c, int s, C u, C cour) {
  return upwind_v(ld(q, c - 2 * s), ld(q, c - s), ld(q, c), ld(q, c + s), u, cour);
}

inline unsigned grid_for(long long n) { return (unsigned)((n + kBlock - 1) / kBlock); }

// Programmatic dependent launch: the plan's kernels are launched so that the next
// one is set up while this one drains.  Before touching memory a kernel waits until
// its predecessor has completed and its writes are visible (a no-op for an ordinary
// launch); when a block has done its work it signals that the successor may be
// scheduled.  Stream order is unchanged.  Signalling at the end rather than at the
// start keeps the successor's waiting blocks off the SMs while this grid still runs
// (measured on GB300: signalling at the start slowed the FP64 kernels by 15 % on a
// deep hierarchy of small levels; at the end every workload gained 1-7 %).
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_exit() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// coarse frontier face test: returns side (0/1) and the slot, or -1.  A mirror
// plane is no frontier, and a ghost face across one takes its image's slot.
__device__ __forceinline__ int coarse_frontier(const LevelView& L, int d, int f0, int f1, int f2,
                                               int& slot) {
  int f[3] = {f0, f1, f2};
  int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
  int a = f[t1] - L.G - L.coff[t1], b = f[t2] - L.G - L.coff[t2];
  if (a < 0 && (L.mir >> t1 & 1)) a = -1 - a;
  if (b < 0 && (L.mir >> t2 & 1)) b = -1 - b;
  int h1 = L.cn[t1] >> 1, h2 = L.cn[t2] >> 1;
  if (a < 0 || a >= h1 || b < 0 || b >= h2) return -1;
  int lo = L.G + L.coff[d];
  int side = f[d] == lo && !(L.mir >> d & 1) ? 0 : (f[d] == lo + (L.cn[d] >> 1) ? 1 : -1);
  slot = b * h1 + a;
  return side;
}

// does the low or the high d-face of a cell with d-index gd lie on one of the two
// d-planes that carry the child's frontier faces?
__device__ __forceinline__ bool near_frontier(const LevelView& L, int d, int gd) {
  const int lo = L.G + L.coff[d], hi = lo + (L.cn[d] >> 1);
  return gd == lo || gd == hi || gd + 1 == lo || gd + 1 == hi;
}

// ------------------------------------------------------------------ source S
// S(h) of Eq. 15: v_d -= h [ (p_c - p_m)/(dx rho_face) + (Phi_c - Phi_m)/dx ]
// NC cells per thread (the two-cell form of the compression below): every load of
// all cells first, then the arithmetic and the stores.
template <class T, int NC>
__device__ __forceinline__ void el_source(const LevelView& L, const Box& b, const Scratch& S,
                                          const Arith<T>* __restrict__ dtp, int write_pi,
                                          Arith<T> gm1, const Bg<Arith<T>>& bg,
                                          const Geo<Arith<T>>& g, const Again& ag,
                                          const unsigned* el) {
  using C = Arith<T>;
  int c[NC], c3[NC][3];
  bool ok[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    int i, j, k;
    ok[n] = decode(b, el[n], i, j, k);
    if (NC == 1 && !ok[n]) return;
    if (!ok[n]) i = j = k = 1;
    c[n] = cidx(L, i, j, k);
    c3[n][0] = i;
    c3[n][1] = j;
    c3[n][2] = k;
  }
  const St<T>* __restrict__ rho = (const St<T>*)L.q[F_RHO];
  const St<T>* __restrict__ e = (const St<T>*)L.q[F_E];
  const Arith<T>* __restrict__ phi = (const Arith<T>*)L.phi;
  const C h = halve(dtp[0]);
  C rc[NC], ec[NC], fc[NC], rm[NC][3], em[NC][3], fm[NC][3], vv[NC][3];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    rc[n] = ld(rho, c[n]);
    ec[n] = ld(e, c[n]);
    fc[n] = ld(phi, c[n]);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (c3[n][d] >= 1) {
        const int m = c[n] - L.st[d];
        rm[n][d] = ld(rho, m);
        em[n][d] = ld(e, m);
        fm[n][d] = ld(phi, m);
        vv[n][d] = ld((const St<T>*)L.q[F_VX + d], c[n]);
      }
  }
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    if (!ok[n]) continue;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (c3[n][d] >= 1) {
        C drf = halve(rm[n][d] + rc[n]);
        C rf = bg.rho0 + drf;
        C acc = mul_u(div_u(mul_u(gm1, ec[n] - em[n][d]), rf) + (fc[n] - fm[n][d]),
                      g.inv_dx[d]);
        C vn = vv[n][d] - mul_u(h, acc);
        st_kicked((St<T>*)L.q[F_VX + d], c[n], vn, ag.has(c3[n]));
        // momentum deviation: rf (V + dv) - rho0 V
        if (write_pi)
          st((Arith<T>*)S.pi[d], c[n], mul_u(bg.rho0, vn) + mul_u(drf, add_k(vn, bg.V[d])));
      } else if (write_pi) {
        ((Arith<T>*)S.pi[d])[c[n]] = C(0.f);
      }
    }
  }
}

// ------------------------------------------------------- SubStep2 viscosity
// SubStep2 (Sec. 3.3 stage list, ZEUS naming): the von Neumann-Richtmyer artificial
// viscosity of ZEUS (Stone & Norman 1992).  First pass: along each axis a compressed
// cell (dv = v_d(upper face) - v_d(lower face) < 0) gets q_d = C2 rho dv^2, stored in
// the momentum-flux scratch, and the cell's internal energy loses dt sum_d q_d dv/dx_d
// (from the velocities after the first kick; dv is the same in deviations).
template <class T>
__device__ __forceinline__ void el_visc_q(const LevelView& L, const Box& b, const Scratch& S,
                                          const Arith<T>* __restrict__ dtp, Arith<T> av,
                                          const Bg<Arith<T>>& bg, const Geo<Arith<T>>& g,
                                          unsigned tid) {
  using C = Arith<T>;
  int i, j, k;
  if (!decode(b, tid, i, j, k)) return;
  const int c = cidx(L, i, j, k);
  const int c3[3] = {i, j, k};
  const C rc = bg.rho0 + ld((const St<T>*)L.q[F_RHO], c);
  C heat = C(0.f);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    C q = C(0.f);
    if (c3[d] < L.s[d] - 1) {
      const St<T>* v = (const St<T>*)L.q[F_VX + d];
      const C dv = ld(v, c + L.st[d]) - ld(v, c);
      if (lt0(dv)) q = av * rc * dv * dv;
      heat += q * dv * g.inv_dx[d];
    }
    st((Arith<T>*)S.P[d], c, q);
  }
  St<T>* e = (St<T>*)L.q[F_E];
  st(e, c, ld(e, c) - dtp[0] * heat);
}

// Second pass: v_d -= dt (q_c - q_m) / (dx_d rho_face) on faces 1.. of each axis, and
// the staggered momenta the transport starts from follow the new velocity.
template <class T>
__device__ __forceinline__ void el_visc_v(const LevelView& L, const Box& b, const Scratch& S,
                                          const Arith<T>* __restrict__ dtp, int write_pi,
                                          const Bg<Arith<T>>& bg, const Geo<Arith<T>>& g,
                                          unsigned tid) {
  using C = Arith<T>;
  int i, j, k;
  if (!decode(b, tid, i, j, k)) return;
  const St<T>* __restrict__ rho = (const St<T>*)L.q[F_RHO];
  const int c = cidx(L, i, j, k);
  const int c3[3] = {i, j, k};
  const C dt = dtp[0];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (c3[d] < 1) continue;
    const int m = c - L.st[d];
    const Arith<T>* q = (const Arith<T>*)S.P[d];
    St<T>* v = (St<T>*)L.q[F_VX + d];
    const C drf = halve(ld(rho, m) + ld(rho, c));
    const C vn = ld(v, c) - dt * hdiv(ld(q, c) - ld(q, m), bg.rho0 + drf) * g.inv_dx[d];
    st(v, c, vn);
    if (write_pi) st((Arith<T>*)S.pi[d], c, bg.rho0 * vn + drf * (bg.V[d] + vn));
  }
}

// The compression and diffusion element functions take NC cells per thread: 2 for the
// FP32 state (elements e and e + 256 of a 512-element chunk), 1 otherwise.  Every
// load of both cells is issued before the first store, so a thread keeps twice the
// bytes in flight.  A cell past the end of the box takes an in-bounds stand-in index
// for its loads and stores nothing.  The arithmetic of each cell is unchanged.

// ------------------------------------------------- SubStep3 + luminosity + e/rho
template <class T, int NC>
__device__ __forceinline__ void el_compress_lum(const LevelView& L, const Box& b,
                                                const Scratch& S,
                                                const Arith<T>* __restrict__ dtp, Arith<T> gm1,
                                                Arith<T> lum, int do_ss3, int do_lum, int do_eps,
                                                const Bg<Arith<T>>& bg,
                                                const Geo<Arith<T>>& g, const unsigned* el) {
  using C = Arith<T>;
  int c[NC];
  bool ok[NC], ss3[NC], lm[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    int i, j, k;
    ok[n] = decode(b, el[n], i, j, k);
    if (NC == 1 && !ok[n]) return;
    if (!ok[n]) i = j = k = 0;
    c[n] = cidx(L, i, j, k);
    ss3[n] = do_ss3 && i < L.s[0] - 1 && j < L.s[1] - 1 && k < L.s[2] - 1;
    // active cells and their mirror images in the ghost layers
    lm[n] = do_lum && i >= (L.mir & 1 ? 0 : L.G) && i < L.G + L.n[0] &&
            j >= (L.mir & 2 ? 0 : L.G) && j < L.G + L.n[1] && k >= (L.mir & 4 ? 0 : L.G) &&
            k < L.G + L.n[2];
  }
  St<T>* e = (St<T>*)L.q[F_E];
  const St<T>* vx = (const St<T>*)L.q[F_VX];
  const St<T>* vy = (const St<T>*)L.q[F_VX + 1];
  const St<T>* vz = (const St<T>*)L.q[F_VX + 2];
  C ec[NC], x0[NC], x1[NC], y0[NC], y1[NC], z0[NC], z1[NC], lw[NC], dr[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    ec[n] = ld(e, c[n]);
    if (ss3[n]) {
      x0[n] = ld(vx, c[n]);
      x1[n] = ld(vx, c[n] + L.st[0]);
      y0[n] = ld(vy, c[n]);
      y1[n] = ld(vy, c[n] + L.st[1]);
      z0[n] = ld(vz, c[n]);
      z1[n] = ld(vz, c[n] + L.st[2]);
    }
    if (lm[n]) lw[n] = ld((const Arith<T>*)L.lumw, c[n]);
    if (do_eps) dr[n] = ld((const St<T>*)L.q[F_RHO], c[n]);
  }
  const C dt = dtp[0];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    if (!ok[n]) continue;
    C ecn = ec[n];
    if (ss3[n]) {
      C div = mul_u(x1[n] - x0[n], g.inv_dx[0]) + mul_u(y1[n] - y0[n], g.inv_dx[1]) +
              mul_u(z1[n] - z0[n], g.inv_dx[2]);
      C a = halve(mul_u(mul_u(dt, gm1), div));
      // (e0 + de)(1 - a)/(1 + a) - e0
      ecn = hdiv(mul_u(ecn, C(1.f) - a) - twice(mul_u(a, bg.e0)), C(1.f) + a);
    }
    if (lm[n]) ecn = ecn + mul_u(mul_u(lum, dt), lw[n]);
    st(e, c[n], ecn);
    // e/rho - e0/rho0 = (de - eps0 drho)/(rho0 + drho)
    if (do_eps) st((Arith<T>*)S.eps, c[n], eps_dev(ecn, dr[n], bg));
  }
}

// CommFlux record (Sec. 3.2.3).  A child level writes the flux through each of its
// frontier faces into its record (rec_index), once per sub-cycle; the parent sums the
// entries of a coarse face when it substitutes its own frontier flux, in a fixed
// order: sub-cycle, then the fine faces (u, v) = (0,0), (1,0), (0,1), (1,1).  The
// record is written, never accumulated, so it needs no clearing, and the sub-cycles
// run decide what is summed.

// record a child's flux through the frontier face with index f along d (f = G or
// G + n_d) at transverse position (c1, c2) of the padded array
__device__ __forceinline__ void fr_put(const LevelView& L, int d, int f, int c1, int c2, int q,
                                       int sub, double v) {
  L.acc[rec_index(L.s, d, f == L.G ? 0 : 1, q, sub, c1, c2)] = v;
}

// The parent's substitute for its frontier faces: at the start of its level step
// (in the compression kernel, which every level step that has a consumer runs) one
// thread per (side, quantity, coarse slot) sums the child's record over the
// sub-cycles the child ran (one when the Eq. 55-56 search dropped the second) and
// the 4 fine faces, and the consumers read the sum with one load.
__device__ __forceinline__ void fr_sums(const LevelView& L, const DevScalars* ds, int level,
                                        unsigned tid) {
  if (tid >= 18u * (unsigned)L.cacc_slots) return;
  const int blk = (int)tid / L.cacc_slots, slot = (int)tid - blk * L.cacc_slots;
  const int side = blk / 3, q = blk - 3 * side, d = side >> 1;
  const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
  const int h1 = L.cn[t1] >> 1;
  if (slot >= h1 * (L.cn[t2] >> 1)) return;
  const int a = slot % h1, b = slot / h1;
  const int cs[3] = {L.cn[0] + 2 * L.G, L.cn[1] + 2 * L.G, L.cn[2] + 2 * L.G};
  const bool two = ((ds->xi1 >> level) & 1u) == 0u;
  double sum = 0.0;
  for (int sub = 0; sub < (two ? 2 : 1); ++sub)
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        sum += L.crec[rec_index(cs, d, side & 1, q, sub, L.G + 2 * a + u, L.G + 2 * b + v)];
  L.csum[blk * L.cacc_slots + slot] = sum;
}


// --------------------------------------------------------------- diffusion
// energy moved in +d across a face during dt: -chi rho_f d(e/rho)/dx * area * dt,
// as rho_f (e/rho difference) K_d with K_d = -chi dt area_d / dx_d, one coefficient
// per level step and axis (a level-step constant) instead of three products per face
template <class T>
__device__ __forceinline__ Arith<T> diff_flux(const LevelView& L, const St<T>* __restrict__ rho,
                                              const Arith<T>* __restrict__ eps, int f, int d,
                                              Arith<T> K, Arith<T> rho0, int dfr) {
  using C = Arith<T>;
  int m = f - L.st[d];
  C rf = dfr ? rho0 : rho0 + halve(ld(rho, m) + ld(rho, f));
  return mul_u(rf, ld(eps, f) - ld(eps, m)) * K;
}

// EPSX: the separate transport kernels follow, and the x sweep's preparation (e/rho
// of the diffused state) is done here: written to Scratch::w[0] (a plane the x sweep
// does not use otherwise; neighbours still read Scratch::eps in this launch), for
// every box cell, from e as stored, so with the bits el_tprep would give.
template <class T, int NC, int EPSX>
__device__ __forceinline__ void el_diffuse(const LevelView& L, const Box& b, const Scratch& S,
                                           const Arith<T>* __restrict__ kc,
                                           Arith<T> rho0, int dfr, const Geo<Arith<T>>& g,
                                           const Bg<Arith<T>>& bg, const unsigned* el) {
  using C = Arith<T>;
  int c[NC], c3[NC][3], ce[NC];
  bool ok[NC], edge[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    int i, j, k;
    const bool in = decode(b, el[n], i, j, k);
    ok[n] = in && i >= 1 && j >= 1 && k >= 1 && i < L.s[0] - 1 && j < L.s[1] - 1 &&
            k < L.s[2] - 1;
    edge[n] = EPSX && in && !ok[n];
    if (NC == 1 && !ok[n] && !edge[n]) return;
    ce[n] = in ? cidx(L, i, j, k) : 0;
    if (!ok[n]) i = j = k = 1;
    c[n] = cidx(L, i, j, k);
    c3[n][0] = i;
    c3[n][1] = j;
    c3[n][2] = k;
  }
  const St<T>* __restrict__ rho = (const St<T>*)L.q[F_RHO];
  const Arith<T>* __restrict__ eps = (const Arith<T>*)S.eps;
  C q[NC][3][2];  // flux through the lower and the upper d-face
#pragma unroll
  for (int n = 0; n < NC; ++n)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const C K = kc[K_DIFF + d];
      q[n][d][0] = diff_flux<T>(L, rho, eps, c[n], d, K, rho0, dfr);
      q[n][d][1] = diff_flux<T>(L, rho, eps, c[n] + L.st[d], d, K, rho0, dfr);
    }
  if (L.has_child) {
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (!near_frontier(L, d, c3[n][d])) continue;
        int slot, f3[3] = {c3[n][0], c3[n][1], c3[n][2]};
        int side = coarse_frontier(L, d, f3[0], f3[1], f3[2], slot);
        if (side >= 0)
          q[n][d][0] = from_double<C>(L.cacc[((2 * d + side) * 3 + 2) * L.cacc_slots + slot]);
        f3[d] += 1;
        side = coarse_frontier(L, d, f3[0], f3[1], f3[2], slot);
        if (side >= 0)
          q[n][d][1] = from_double<C>(L.cacc[((2 * d + side) * 3 + 2) * L.cacc_slots + slot]);
      }
  }
  St<T>* e = (St<T>*)L.q[F_E];
  C ev[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) ev[n] = ld(e, c[n]);
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    C div = C(0.f);
#pragma unroll
    for (int d = 0; d < 3; ++d) div += q[n][d][1] - q[n][d][0];
    if (ok[n]) {
      const C en = ev[n] - div * g.inv_vol;
      st(e, c[n], en);
      if (EPSX) {
        const C rc = ld(rho, c[n]);
        st((Arith<T>*)S.w[0], c[n], eps_dev(as_stored(en), rc, bg));
      }
    } else if (edge[n]) {
      const C rc = ld(rho, ce[n]);
      st((Arith<T>*)S.w[0], ce[n], eps_dev(ld(e, ce[n]), rc, bg));
    }
  }
}

// CommFlux record of the diffusive energy fluxes through a child's frontier faces: one
// thread per fine frontier face, in chunks of the diffusion's launch of their own (both
// only read rho and e/rho; as a launch it took 1.5-3 us per child level step)
template <class T>
__device__ __forceinline__ void el_frontier_diff(const LevelView& L, const Scratch& S,
                                                 const Arith<T>* __restrict__ kc,
                                                 Arith<T> rho0, int dfr, int sub, unsigned tid) {
  using C = Arith<T>;
  // one thread per fine face: (side, coarse slot, fine face u, v of the slot)
  if (tid >= 24u * (unsigned)L.acc_slots) return;
  const int u = (int)(tid & 1u), v = (int)((tid >> 1) & 1u);
  const int rest = (int)(tid >> 2);
  const int side = rest / L.acc_slots, slot = rest - side * L.acc_slots;
  const int d = side >> 1, t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
  const int h1 = L.n[t1] >> 1;
  if (slot >= h1 * (L.n[t2] >> 1)) return;
  const int a = slot % h1, b = slot / h1;
  const int fd = (side & 1) ? L.G + L.n[d] : L.G;
  int f3[3];
  f3[d] = fd;
  f3[t1] = L.G + 2 * a + u;
  f3[t2] = L.G + 2 * b + v;
  const int f = (f3[2] * L.s[1] + f3[1]) * L.s[0] + f3[0];
  fr_put(L, d, fd, f3[t1], f3[t2], 2, sub,
         as_double(diff_flux<T>(L, (const St<T>*)L.q[F_RHO], (const Arith<T>*)S.eps, f, d,
                                kc[K_DIFF + d], rho0, dfr)));
}

// --------------------------------------------------------------- transport
template <class T>
__device__ __forceinline__ void el_tprep(const LevelView& L, const Box& b, const Scratch& S,
                                         const Bg<Arith<T>>& bg, int eps_only, unsigned tid) {
  using C = Arith<T>;
  int i, j, k;
  if (!decode(b, tid, i, j, k)) return;
  const St<T>* __restrict__ rho = (const St<T>*)L.q[F_RHO];
  const int c = cidx(L, i, j, k);
  const int c3[3] = {i, j, k};
  const C rc = ld(rho, c);
  const C ec = ld((const St<T>*)L.q[F_E], c);
  if (eps_only) {
    st((Arith<T>*)S.eps, c, eps_dev(ec, rc, bg));
    return;
  }
  // every load first, then the arithmetic and the stores
  C rm[3], pm[3];
#pragma unroll
  for (int m = 0; m < 3; ++m)
    if (c3[m] >= 1) {
      rm[m] = ld(rho, c - L.st[m]);
      pm[m] = ld((const Arith<T>*)S.pi[m], c);
    }
  C wv[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    wv[m] = C(0.f);
    if (c3[m] >= 1) {
      // Pi/rho_face - V = (dPi - V drf)/(rho0 + drf)
      C drf = halve(rm[m] + rc);
      wv[m] = div_u(sub_ky(pm[m], bg.V[m], drf), bg.rho0 + drf);
    }
  }
  st((Arith<T>*)S.eps, c, eps_dev(ec, rc, bg));
#pragma unroll
  for (int m = 0; m < 3; ++m) st((Arith<T>*)S.w[m], c, wv[m]);
}

// mass and energy flux at d-faces 2 <= i_d < s_d - 1
// the sweep direction is a template parameter: every per-axis constant is then a
// fixed kernel-parameter operand instead of a dynamically indexed load
template <class T, int d>
__device__ __forceinline__ void el_tflux(const LevelView& L, const Box& b, const Scratch& S,
                                         const Arith<T>* __restrict__ kc,
                                         const Bg<Arith<T>>& bg, int sub, unsigned tid) {
  using C = Arith<T>;
  int i, j, k;
  if (!decode(b, tid, i, j, k)) return;
  const int c = cidx(L, i, j, k);
  const int c3[3] = {i, j, k};
  C Fv = C(0.f), Ev = C(0.f);
  if (c3[d] >= 2 && c3[d] < L.s[d] - 1) {
    const int sd = L.st[d];
    const C Adt = kc[K_ADT + d];
    const C du = ld((const St<T>*)L.q[F_VX + d], c);
    const C u = add_k(du, bg.V[d]);
    const C cour = mul_u(u, kc[K_DTDX + d]);
    const C F0 = is0(bg.V[d]) ? C(0.f) : kc[K_F0 + d];
    C drs = upwind((const St<T>*)L.q[F_RHO], c, sd, u, cour);
    Fv = (mul_u(bg.rho0, du) + mul_u(drs, u)) * Adt;  // F - rho0 V_d A dt
    C des = upwind((const Arith<T>*)S.eps, c, sd, u, cour);
    Ev = mul_u(bg.eps0, Fv) + mul_u(des, add_k(Fv, F0));  // E - eps0 rho0 V_d A dt
  }
  st((Arith<T>*)S.F, c, Fv);
  st((Arith<T>*)S.E, c, Ev);
  if (L.is_child && (c3[d] == L.G || c3[d] == L.G + L.n[d])) {  // CommFlux record
    constexpr int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
    fr_put(L, d, c3[d], c3[t1], c3[t2], 0, sub, as_double(Fv));
    fr_put(L, d, c3[d], c3[t1], c3[t2], 1, sub, as_double(Ev));
  }
}

// staggered momentum fluxes of sweep d
// staggered momentum fluxes of sweep d (deviation: P - V_m rho0 V_d A dt)
template <class T, int d>
__device__ __forceinline__ void el_tmom(const LevelView& L, const Box& b, const Scratch& S,
                                        const Arith<T>* __restrict__ kc, const Bg<Arith<T>>& bg,
                                        unsigned tid) {
  using C = Arith<T>;
  int i, j, k;
  if (!decode(b, tid, i, j, k)) return;
  const int c = cidx(L, i, j, k);
  const int c3[3] = {i, j, k};
  const int sd = L.st[d];
  const St<T>* __restrict__ vd = (const St<T>*)L.q[F_VX + d];
  const Arith<T>* __restrict__ F = (const Arith<T>*)S.F;
  const C dtdx = kc[K_DTDX + d];
  const C F0 = is0(bg.V[d]) ? C(0.f) : kc[K_F0 + d];
  C Pv[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    C P = C(0.f);
    if (m == d) {
      if (c3[d] >= 2 && c3[d] < L.s[d] - 2) {
        C uc = add_k(halve(ld(vd, c) + ld(vd, c + sd)), bg.V[d]);
        C Fc = halve(ld(F, c) + ld(F, c + sd));
        C ws = d == 0 ? upwind((const St<T>*)S.w[m], c + sd, sd, uc, mul_u(uc, dtdx))
                      : upwind((const Arith<T>*)S.w[m], c + sd, sd, uc, mul_u(uc, dtdx));
        P = ky_add(bg.V[m], Fc, mul_u(ws, add_k(Fc, F0)));
      }
    } else if (c3[d] >= 2 && c3[d] < L.s[d] - 1 && c3[m] >= 1) {
      const int sm = L.st[m];
      C ue = add_k(halve(ld(vd, c - sm) + ld(vd, c)), bg.V[d]);
      C Fe = halve(ld(F, c - sm) + ld(F, c));
      C ws = d == 0 ? upwind((const St<T>*)S.w[m], c, sd, ue, mul_u(ue, dtdx))
                    : upwind((const Arith<T>*)S.w[m], c, sd, ue, mul_u(ue, dtdx));
      P = ky_add(bg.V[m], Fe, mul_u(ws, add_k(Fe, F0)));
    }
    Pv[m] = P;
  }
  // the stores after every load of the three components
#pragma unroll
  for (int m = 0; m < 3; ++m) st((Arith<T>*)S.P[m], c, Pv[m]);
}

// Every load first, then the arithmetic and the stores (a load never waits for a store
// it cannot be reordered with); NC cells per thread as in the compression (one here).
template <class T, int d, int NC>
__device__ __forceinline__ void el_tupdate(const LevelView& L, const Box& b, const Scratch& S,
                                           const Geo<Arith<T>>& g, const unsigned* el) {
  using C = Arith<T>;
  int c[NC], c3[NC][3];
  bool ok[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    int i, j, k;
    ok[n] = decode(b, el[n], i, j, k);
    if (NC == 1 && !ok[n]) return;
    if (!ok[n]) i = j = k = 3;  // an in-bounds stand-in (arrays hold 2 G >= 6 ghosts)
    c[n] = cidx(L, i, j, k);
    c3[n][0] = i;
    c3[n][1] = j;
    c3[n][2] = k;
  }
  const int sd = L.st[d];
  const C iv = g.inv_vol;
  St<T>* rho = (St<T>*)L.q[F_RHO];
  St<T>* e = (St<T>*)L.q[F_E];
  C Flo[NC], Fhi[NC], Elo[NC], Ehi[NC], rv[NC], ev[NC], pv[NC][3], Pa[NC][3], Pb[NC][3];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    Flo[n] = ld((const Arith<T>*)S.F, c[n]);
    Fhi[n] = ld((const Arith<T>*)S.F, c[n] + sd);
    Elo[n] = ld((const Arith<T>*)S.E, c[n]);
    Ehi[n] = ld((const Arith<T>*)S.E, c[n] + sd);
    rv[n] = ld(rho, c[n]);
    ev[n] = ld(e, c[n]);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const Arith<T>* P = (const Arith<T>*)S.P[m];
      pv[n][m] = ld((const Arith<T>*)S.pi[m], c[n]);
      Pa[n][m] = ld(P, m == d ? c[n] - sd : c[n]);
      Pb[n][m] = ld(P, m == d ? c[n] : c[n] + sd);
    }
  }
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    if (!ok[n]) continue;
    if (c3[n][d] >= 2 && c3[n][d] < L.s[d] - 2) {
      if (L.has_child && near_frontier(L, d, c3[n][d])) {
        int slot, f3[3] = {c3[n][0], c3[n][1], c3[n][2]};
        int side = coarse_frontier(L, d, f3[0], f3[1], f3[2], slot);
        if (side >= 0) {
          Flo[n] = from_double<C>(L.cacc[((2 * d + side) * 3 + 0) * L.cacc_slots + slot]);
          Elo[n] = from_double<C>(L.cacc[((2 * d + side) * 3 + 1) * L.cacc_slots + slot]);
        }
        f3[d] += 1;
        side = coarse_frontier(L, d, f3[0], f3[1], f3[2], slot);
        if (side >= 0) {
          Fhi[n] = from_double<C>(L.cacc[((2 * d + side) * 3 + 0) * L.cacc_slots + slot]);
          Ehi[n] = from_double<C>(L.cacc[((2 * d + side) * 3 + 1) * L.cacc_slots + slot]);
        }
      }
      st(rho, c[n], rv[n] - (Fhi[n] - Flo[n]) * iv);
      st(e, c[n], ev[n] - (Ehi[n] - Elo[n]) * iv);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const bool chg = m == d ? (c3[n][d] >= 3 && c3[n][d] < L.s[d] - 2)
                              : (c3[n][d] >= 2 && c3[n][d] < L.s[d] - 2 && c3[n][m] >= 1);
      if (chg) st((Arith<T>*)S.pi[m], c[n], pv[n][m] - (Pb[n][m] - Pa[n][m]) * iv);
    }
  }
}

// coarse-level frontier substitution of the low/high d-face fluxes of cell (g); the
// frontier faces lie on two d-planes, tested first
template <class C>
__device__ __forceinline__ void frontier_fluxes(const LevelView& L, int d, const int g[3], C& Flo,
                                                C& Fhi, C& Elo, C& Ehi) {
  if (!near_frontier(L, d, g[d])) return;
  int slot, f3[3] = {g[0], g[1], g[2]};
  int side = coarse_frontier(L, d, f3[0], f3[1], f3[2], slot);
  if (side >= 0) {
    Flo = from_double<C>(L.cacc[((2 * d + side) * 3 + 0) * L.cacc_slots + slot]);
    Elo = from_double<C>(L.cacc[((2 * d + side) * 3 + 1) * L.cacc_slots + slot]);
  }
  f3[d] += 1;
  side = coarse_frontier(L, d, f3[0], f3[1], f3[2], slot);
  if (side >= 0) {
    Fhi = from_double<C>(L.cacc[((2 * d + side) * 3 + 0) * L.cacc_slots + slot]);
    Ehi = from_double<C>(L.cacc[((2 * d + side) * 3 + 1) * L.cacc_slots + slot]);
  }
}

// ------------------------------------------------------- fused transport sweep
// One sweep along d (Sec. 3.1 transport: the mass flux F = rho* v A dt with the
// time-centred van Leer value rho*, e and the momenta carried as (q/rho)* F) with
// the arithmetic of tprep + tflux + tmom + tupdate in one kernel.  Every warp works by
// itself, without a barrier: a lane holds one position of one row and marches through a
// chunk of planes.
//   y, z sweeps (sweep_march): the march is along the sweep; the stencils' values are
// windows in registers, a chunk starts 3 planes early and ends 2 late.
//   x sweep (sweep_x): the march is along z; the stencils' values come by warp shuffle, a
// chunk starts one plane early (mass flux only).
//   The rows are laid end to end, each with its halo (1 position below; x sweep: 3 below,
// 2 above), and cut into warps that share 1 (5) positions, so that 31/32 W/(W+1) of the
// lanes own a cell of a box W wide (x sweep: 27/32 W/(W+5)): 96 % (81 %) at 136, 94 % (73 %)
// at 32; a grid of 32-wide tiles left 80-85 % (71-80 %) at 136 to 144.  The neighbour below
// in x comes by shuffle; of the row below the mass flux
// is formed again from its rho and v_d (a tenth of the arithmetic), which costs less than
// an exchange between warps: a tile in shared memory with three barriers a plane measured
// 50 us against 37 at 136^3 (FP32, y), with the same arithmetic per cell.
//   Each upwind value takes its one-sided differences from a window (x: from the
// neighbouring lanes), one subtraction per cell and quantity instead of two.
//   State: x reads the level's rho, e and velocities (at its start the staggered momenta
// are those of v and rho, so Pi/rho_face - V is the velocity deviation itself and the
// momenta are formed here), writes Scratch::F, E (rho, e) and Scratch::pi; y reads those
// and writes Scratch::P[0], P[1] and Scratch::w; z reads those and writes the level's
// rho and e and Scratch::pi.  Elements outside a box hold what an earlier op left there;
// no element that is needed later depends on them.
//   EDGE: the box reaches the ends of the array, where the stencils do not fit (faces 0,
// 1 and the last along d, face 0 of the other axes).
//   Bound by instruction issue (FP32 58-71 % of the issue slots, double-float 75-77 %).
// Measured at the first sub-cycle of a 128^3 level (boxes of 136 x 140 x 140, 136 x 136 x
// 140, 136^3; ncu, GB300): FP32 x 46.8, y 41.3, z 34.5 us and 288 / 319 / 326 thread
// instructions per cell, where an earlier form with blocks of 9 warps and a barrier a plane
// took 60-65 us at 144^3 and 363-400; double-float x 143, y 111, z 105 us and 1211 / 1146 /
// 1156.  Over a coarse step of 5 x 128^3 a sweep takes 40 us in FP32 and 113 in
// double-float, where that form took 68 us in FP32 and the four separate kernels 171 in
// double-float.
__device__ __forceinline__ float shfl_up(float v, int k) {
  return __shfl_up_sync(0xffffffffu, v, k);
}
__device__ __forceinline__ float shfl_dn(float v, int k) {
  return __shfl_down_sync(0xffffffffu, v, k);
}
__device__ __forceinline__ df64 shfl_up(df64 v, int k) {
  return df64(__shfl_up_sync(0xffffffffu, v.hi, k), __shfl_up_sync(0xffffffffu, v.lo, k));
}
__device__ __forceinline__ df64 shfl_dn(df64 v, int k) {
  return df64(__shfl_down_sync(0xffffffffu, v.hi, k), __shfl_down_sync(0xffffffffu, v.lo, k));
}

// the upwind value (upwind_v) from the two sides' values and the differences
// dm = q(-1) - q(-2), dc = q(0) - q(-1), dp = q(1) - q(0).  The limiter takes dc and one
// of the others, and is symmetric in the two: one selection.
template <class C>
__device__ __forceinline__ C upwind_d(C qm, C q0, C dm, C dc, C dp, C u, C cour) {
  const bool up = gt0(u);
  return add_u(up ? qm : q0,
               mul_u(fsub_u(up ? 1.f : -1.f, cour), hslope(dc, up ? dm : dp)));
}

// element access by byte offset from a base that is the same for the whole warp (offsets
// stay below 2^32: fewer than 2^31 / 5 elements of 8 bytes)
template <class P>
__device__ __forceinline__ auto ldb(const P* base, unsigned o) {
  return ld((const P*)((const char*)base + o), 0);
}
template <class P, class C>
__device__ __forceinline__ void stb(P* base, unsigned o, C v) {
  st((P*)((char*)base + o), 0, v);
}

// The planes of a march as loaded: the newest, the two before it, and those to come.
//   FP32: in registers, one plane ahead (shared memory measured the same to 1 % slower,
// with four or five blocks an SM alike).
template <class C>
struct Planes {
  static constexpr int kAhead = 1;
  C q[3][kSweepArrays], to_come[kSweepArrays];
  __device__ __forceinline__ explicit Planes(C*) {}
  template <class P>
  __device__ __forceinline__ void fetch(int a, const P* base, unsigned o) {
    to_come[a] = ldb(base, o);
  }
  __device__ __forceinline__ void clear(int a) { to_come[a] = C(0.f); }
  __device__ __forceinline__ void commit() {}
  __device__ __forceinline__ void advance() {
#pragma unroll
    for (int a = 0; a < kSweepArrays; ++a) {
      q[2][a] = q[1][a];
      q[1][a] = q[0][a];
      q[0][a] = to_come[a];
    }
  }
  // array a of the plane `back` before the newest
  __device__ __forceinline__ C get(int back, int a) const { return q[back][a]; }
};
//   Double-float: in shared memory, kSweepAhead planes ahead by asynchronous copies, each
// thread's values in its own column of the buffer (so no barrier).  In registers they
// would take 46: with the planes to come alone in shared memory the march needed 168 and
// spilled, 138 us a sweep of 5 x 128^3 (in chunks) against 124 with 152 (four blocks of 128
// registers spill again, 126).
template <>
struct Planes<df64> {
  static constexpr int kAhead = kSweepAhead, NT = kSweepThreads, SLOT = kSweepArrays * NT;
  df64* buf;  // [slot][array][thread], at this thread
  // slots to fetch to, of the newest plane and of the two before (before the first plane
  // they name slots whose values nothing that is kept depends on)
  int in = 0, s0 = (kSweepSlots - 1) * SLOT, s1 = 0, s2 = 0;
  __device__ __forceinline__ explicit Planes(df64* b) : buf(b) {}
  static __device__ __forceinline__ int next(int s) {
    return s == (kSweepSlots - 1) * SLOT ? 0 : s + SLOT;
  }
  template <class P>
  __device__ __forceinline__ void fetch(int a, const P* base, unsigned o) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(buf + in + a * NT);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"((const char*)base + o)
                 : "memory");
  }
  __device__ __forceinline__ void clear(int a) { buf[in + a * NT] = df64(0.f); }
  __device__ __forceinline__ void commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
    in = next(in);
  }
  // the oldest plane in flight has arrived and becomes the newest
  __device__ __forceinline__ void advance() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
    s2 = s1;
    s1 = s0;
    s0 = next(s0);
  }
  __device__ __forceinline__ df64 get(int back, int a) const {
    return buf[(back == 0 ? s0 : back == 1 ? s1 : s2) + a * NT];
  }
};

template <class T, int d, bool EDGE>
__device__ __forceinline__ void sweep_march(const Item<T>& it, int x, int row, bool own, int m0,
                                            int m1, Arith<T>* __restrict__ buf) {
  using C = Arith<T>;
  constexpr int RA = d == 1 ? 2 : 1;  // row axis
  constexpr unsigned ES = sizeof(C);
  const LevelView& L = it.L;
  const Bg<C> bg = it.bg;
  const int sM = L.s[d];
  const unsigned stM = (unsigned)L.st[d] * ES;
  const unsigned c0 = (unsigned)((EDGE ? min(max(x, 0), L.s[0] - 1) : x) + row * L.st[RA]) * ES;
  const unsigned cb = EDGE && row < 1 ? c0 : c0 - (unsigned)L.st[RA] * ES;
  // between the sweeps rho and e are unrounded (the arithmetic type); the z sweep stores
  // the state
  using D = std::conditional_t<d == 1, C, St<T>>;
  const C* const rhoS = (const C*)(d == 1 ? it.S.F : it.S.P[0]);
  const C* const eS = (const C*)(d == 1 ? it.S.E : it.S.P[1]);
  D* const rhoD = (D*)(d == 1 ? it.S.P[0] : L.q[F_RHO]);
  D* const eD = (D*)(d == 1 ? it.S.P[1] : L.q[F_E]);
  const St<T>* const vd = (const St<T>*)L.q[F_VX + d];
  auto piS = [&](int m) { return (const C*)(d == 1 ? it.S.pi[m] : it.S.w[m]); };
  auto piD = [&](int m) { return (C*)(d == 1 ? it.S.w[m] : it.S.pi[m]); };
  const C* kc = (const C*)it.kc;
  const C Adt = kc[K_ADT + d], dtdx = kc[K_DTDX + d];
  const C F0 = is0(bg.V[d]) ? C(0.f) : kc[K_F0 + d];
  const C iv = it.g.inv_vol;
  const int f0 = L.G, f1 = L.G + L.n[d];

  // fetch plane p: this row's values and, of the row below, rho and v_d
  Planes<C> pl(buf);
  const int r_end = m1 + 2;
  auto fetch = [&](int p) {
    if (p < r_end && (!EDGE || (unsigned)p < (unsigned)sM)) {
      const unsigned c = c0 + (unsigned)p * stM, b = cb + (unsigned)p * stM;
      pl.fetch(0, rhoS, c);
      pl.fetch(1, eS, c);
      pl.fetch(2, vd, c);
#pragma unroll
      for (int m = 0; m < 3; ++m) pl.fetch(3 + m, piS(m), c);
      pl.fetch(6, rhoS, b);
      pl.fetch(7, vd, b);
    } else if (EDGE && p < r_end) {
#pragma unroll
      for (int a = 0; a < kSweepArrays; ++a) pl.clear(a);
    }
    pl.commit();
  };

  // windows at step r (plane r is the newest): x1, x2 the values of planes r-1, r-2, dx0
  // the difference of planes r and r-1, dx1, dx2 the two before
  const C z = C(0.f);
  C dr1 = z, dr2 = z, db1 = z, db2 = z;                     // rho; of the row below
  C e1 = z, e2 = z, de1 = z, de2 = z;                       // e/rho
  C w1[3] = {z, z, z}, w2[3] = {z, z, z};                   // Pi/rho_face - V
  C dw1[3] = {z, z, z}, dw2[3] = {z, z, z};
  C F2 = z, E2 = z, Pp[3] = {z, z, z};                      // fluxes of the face before
  for (int k = 0; k < Planes<C>::kAhead; ++k) fetch(m0 - 3 + k);
#pragma unroll 1
  for (int r = m0 - 3; r < r_end; ++r) {
    // a slot is free again once the plane three before is done with
    pl.advance();
    fetch(r + Planes<C>::kAhead);
    const C rc = pl.get(0, 0), ec = pl.get(0, 1), rb = pl.get(0, 6);
    const C r1 = pl.get(1, 0), b1 = pl.get(1, 6);
    const C pc[3] = {pl.get(0, 3), pl.get(0, 4), pl.get(0, 5)};
    // e/rho and Pi/rho_face - V = (dPi - V drf)/(rho0 + drf) of plane r
    const C ep = eps_dev(ec, rc, bg);
    const C rx = shfl_up(rc, 1);
    C w0[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const C drf = halve((m == 0 ? rx : m == d ? r1 : rb) + rc);
      w0[m] = div_sum(sub_ky(pc[m], bg.V[m], drf), bg.rho0, drf);
      if (EDGE && !(m == 0 ? x >= 1 : m == d ? r >= 1 && r < sM : row >= 1)) w0[m] = z;
    }
    const C dr0 = rc - r1, de0 = ep - e1, db0 = rb - b1;
    C dw0[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) dw0[m] = w0[m] - w1[m];
    C F1 = z, E1 = z;
    if (r >= m0) {
      // mass and energy flux of face r - 1, and the mass flux of the row below
      const int f = r - 1;
      const bool ok = !EDGE || (f >= 2 && f < sM - 1);
      const C r2 = pl.get(2, 0), b2 = pl.get(2, 6), v1 = pl.get(1, 2), vb1 = pl.get(1, 7);
      C Fb = z;
      if (ok) {
        const C u = add_k(v1, bg.V[d]), ub = add_k(vb1, bg.V[d]);
        const C cour = mul_u(u, dtdx);
        const C drs = upwind_d(r2, r1, dr2, dr1, dr0, u, cour);
        F1 = mul_u(add_u(mul_u(bg.rho0, v1), mul_u(drs, u)), Adt);  // F - rho0 V_d A dt
        const C des = upwind_d(e2, e1, de2, de1, de0, u, cour);
        E1 = add_u(mul_u(bg.eps0, F1), mul_u(des, add_k(F1, F0)));
        const C drb = upwind_d(b2, b1, db2, db1, db0, ub, mul_u(ub, dtdx));
        Fb = mul_u(add_u(mul_u(bg.rho0, vb1), mul_u(drb, ub)), Adt);
      }
      if (L.is_child && (f == f0 || f == f1) && own && f >= m0 && (f < m1 || f == it.b.hi[d])) {
        // CommFlux record (transverse axes x and the row axis): the chunk's own faces
        // and, above the last chunk, the box's upper face
        fr_put(L, d, f, x, row, 0, it.sub, as_double(norm(F1)));
        fr_put(L, d, f, x, row, 1, it.sub, as_double(norm(E1)));
      }
      const C Fx = shfl_up(F1, 1), vx = shfl_up(v1, 1);
      C P[3] = {z, z, z};
      if (r >= m0 + 1) {
        // momentum fluxes: on the x and row edges of plane r - 1, along d at cell r - 2
        if (!EDGE || (ok && x >= 1)) {
          const C ue = add_k(halve(vx + v1), bg.V[d]);
          const C Fe = halve(add_u(Fx, F1));
          const C ws = upwind_d(w2[0], w1[0], dw2[0], dw1[0], dw0[0], ue, mul_u(ue, dtdx));
          P[0] = ky_add(bg.V[0], Fe, mul_u(ws, add_k(Fe, F0)));
        }
        if (!EDGE || (ok && row >= 1)) {
          const C ue = add_k(halve(vb1 + v1), bg.V[d]);
          const C Fe = halve(add_u(Fb, F1));
          const C ws = upwind_d(w2[RA], w1[RA], dw2[RA], dw1[RA], dw0[RA], ue, mul_u(ue, dtdx));
          P[RA] = ky_add(bg.V[RA], Fe, mul_u(ws, add_k(Fe, F0)));
        }
        if (!EDGE || (r - 2 >= 2 && r - 2 < sM - 2)) {
          const C uc = add_k(halve(pl.get(2, 2) + v1), bg.V[d]);
          const C Fc = halve(add_u(F2, F1));
          const C ws = upwind_d(w2[d], w1[d], dw2[d], dw1[d], dw0[d], uc, mul_u(uc, dtdx));
          P[d] = ky_add(bg.V[d], Fc, mul_u(ws, add_k(Fc, F0)));
        }
      }
      // conservative update of plane r - 2
      const int u2 = r - 2;
      if (u2 >= m0 && own) {
        const unsigned c = c0 + (unsigned)u2 * stM;
        const bool upd = !EDGE || (u2 >= 2 && u2 < sM - 2);
        C rv = r2, ev = pl.get(2, 1);
        if (upd) {
          C Flo = F2, Fhi = F1, Elo = E2, Ehi = E1;
          if (L.has_child && near_frontier(L, d, u2)) {
            int g[3];
            g[0] = x;
            g[RA] = row;
            g[d] = u2;
            frontier_fluxes(L, d, g, Flo, Fhi, Elo, Ehi);
          }
          rv = rv - mul_u(sub_u(Fhi, Flo), iv);
          ev = ev - mul_u(sub_u(Ehi, Elo), iv);
        }
        stb(rhoD, c, rv);
        stb(eD, c, ev);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          C pv = pl.get(2, 3 + m);
          // P_d of cells r-3, r-2; the others' of planes r-2, r-1
          if (!EDGE || (upd && (m == d ? u2 >= 3 : m == 0 ? x >= 1 : row >= 1)))
            pv = pv - mul_u(sub_u(P[m], Pp[m]), iv);
          stb(piD(m), c, pv);
        }
      }
#pragma unroll
      for (int m = 0; m < 3; ++m) Pp[m] = P[m];
    }
    F2 = F1; E2 = E1;
    dr2 = dr1; dr1 = dr0; db2 = db1; db1 = db0;
    e2 = e1; e1 = ep; de2 = de1; de1 = de0;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      w2[m] = w1[m]; w1[m] = w0[m]; dw2[m] = dw1[m]; dw1[m] = dw0[m];
    }
  }
}

// frontier_fluxes (d = 0) of the cells that a lane of the x sweep marches through: their x
// and y are fixed, so the side and the y-slot are found once.  With the record's running
// address, per coarse step before and after: five levels of 128^3 6.06 and 5.98 ms in FP32,
// 16.74 and 16.64 in FP64; three of 96^3 FP32 728 and 720 us.
struct FrontierLane {
  int side[2];  // of the cell's lower and upper x-face: 0, 1, or -1 (no frontier face)
  int a;        // its coarse slot along y
  __device__ __forceinline__ FrontierLane(const LevelView& L, int x, int row) {
    side[0] = side[1] = -1;
    a = row - L.G - L.coff[1];
    if (a < 0 && (L.mir & 2)) a = -1 - a;
    if (!L.has_child || a < 0 || a >= L.cn[1] >> 1) return;
    const int lo = L.G + L.coff[0], hi = lo + (L.cn[0] >> 1);
#pragma unroll
    for (int k = 0; k < 2; ++k)
      side[k] = x + k == lo && !(L.mir & 1) ? 0 : (x + k == hi ? 1 : -1);
  }
  template <class C>
  __device__ __forceinline__ void substitute(const LevelView& L, int z, C& Flo, C& Fhi, C& Elo,
                                             C& Ehi) const {
    int b = z - L.G - L.coff[2];
    if (b < 0 && (L.mir & 4)) b = -1 - b;
    if (b < 0 || b >= L.cn[2] >> 1) return;
    const double* s = L.cacc + b * (L.cn[1] >> 1) + a;
    if (side[0] >= 0) {
      Flo = from_double<C>(s[side[0] * 3 * L.cacc_slots]);
      Elo = from_double<C>(s[(side[0] * 3 + 1) * L.cacc_slots]);
    }
    if (side[1] >= 0) {
      Fhi = from_double<C>(s[side[1] * 3 * L.cacc_slots]);
      Ehi = from_double<C>(s[(side[1] * 3 + 1) * L.cacc_slots]);
    }
  }
};

// the x sweep
template <class T, bool EDGE>
__device__ __forceinline__ void sweep_x(const Item<T>& it, int x, int row, bool mine, int m0,
                                        int m1, Arith<T>* __restrict__ buf) {
  using C = Arith<T>;
  constexpr unsigned ES = sizeof(C);
  const LevelView& L = it.L;
  const Bg<C> bg = it.bg;
  const bool own = mine && x >= it.b.lo[0] && x < it.b.hi[0];
  const int sx = L.s[0];
  const unsigned stM = (unsigned)L.st[2] * ES;
  const unsigned c0 = (unsigned)((EDGE ? min(max(x, 0), sx - 1) : x) + row * L.st[1]) * ES;
  const unsigned cb = EDGE && row < 1 ? c0 : c0 - (unsigned)L.st[1] * ES;
  const St<T>* const rhoS = (const St<T>*)L.q[F_RHO];
  const St<T>* const eS = (const St<T>*)L.q[F_E];
  const C* kc = (const C*)it.kc;
  const C Adt = kc[K_ADT], dtdx = kc[K_DTDX];
  const C F0 = is0(bg.V[0]) ? C(0.f) : kc[K_F0];
  const C iv = it.g.inv_vol;
  // CommFlux record (transverse axes y and z): the box's own faces and its upper one.  A
  // third to a half of the warps hold such a lane, so its address advances with the march
  const bool rec = L.is_child && mine && (x == L.G || x == L.G + L.n[0]) &&
                   x >= it.b.lo[0] && x <= it.b.hi[0];
  double* recp = rec ? L.acc + rec_index(L.s, 0, x == L.G ? 0 : 1, 0, it.sub, row, m0) : nullptr;
  const int rec_e = rec_index(L.s, 0, 0, 1, 0, 0, 0) - rec_index(L.s, 0, 0, 0, 0, 0, 0);
  const FrontierLane fr(L, x, row);
  const bool okF = !EDGE || (x >= 2 && x < sx - 1);
  const C z = C(0.f);

  Planes<C> pl(buf);
  auto fetch = [&](int p) {
    if (p < m1 && (!EDGE || p >= 0)) {
      const unsigned c = c0 + (unsigned)p * stM, b = cb + (unsigned)p * stM;
      pl.fetch(0, rhoS, c);
      pl.fetch(1, eS, c);
#pragma unroll
      for (int m = 0; m < 3; ++m) pl.fetch(2 + m, (const St<T>*)L.q[F_VX + m], c);
      pl.fetch(5, rhoS, b);
      pl.fetch(6, (const St<T>*)L.q[F_VX], b);
    } else if (EDGE && p < m1) {
#pragma unroll
      for (int a = 0; a < kSweepArrays; ++a) pl.clear(a);
    }
    pl.commit();
  };
  for (int k = 0; k < Planes<C>::kAhead; ++k) fetch(m0 - 1 + k);
  C rp = z, vp = z, Fp = z;  // rho, v_x, F of the plane before
#pragma unroll 1
  for (int p = m0 - 1; p < m1; ++p) {
    pl.advance();
    fetch(p + Planes<C>::kAhead);
    const C rc = pl.get(0, 0), ec = pl.get(0, 1), rb = pl.get(0, 5), vb = pl.get(0, 6);
    const C w[3] = {pl.get(0, 2), pl.get(0, 3), pl.get(0, 4)};
    const C vc = w[0];
    const C r_m1 = shfl_up(rc, 1);
    C Fv = z, Ev = z, Fb = z;
    {
      // each lane forms its difference to the lane below, the neighbours read it
      const C ep = eps_dev(ec, rc, bg);
      const C e_m1 = shfl_up(ep, 1), b_m1 = shfl_up(rb, 1);
      const C dr = rc - r_m1, de = ep - e_m1, db = rb - b_m1;
      const C dr_m = shfl_up(dr, 1), dr_p = shfl_dn(dr, 1);
      const C de_m = shfl_up(de, 1), de_p = shfl_dn(de, 1);
      const C db_m = shfl_up(db, 1), db_p = shfl_dn(db, 1);
      if (!EDGE || (okF && p >= 0)) {
        const C u = add_k(vc, bg.V[0]), ub = add_k(vb, bg.V[0]);
        const C cour = mul_u(u, dtdx);
        const C drs = upwind_d(r_m1, rc, dr_m, dr, dr_p, u, cour);
        Fv = mul_u(add_u(mul_u(bg.rho0, vc), mul_u(drs, u)), Adt);  // F - rho0 V_x A dt
        const C des = upwind_d(e_m1, ep, de_m, de, de_p, u, cour);
        Ev = add_u(mul_u(bg.eps0, Fv), mul_u(des, add_k(Fv, F0)));
        const C drb = upwind_d(b_m1, rb, db_m, db, db_p, ub, mul_u(ub, dtdx));
        Fb = mul_u(add_u(mul_u(bg.rho0, vb), mul_u(drb, ub)), Adt);
      }
    }
    if (p >= m0) {
      if (rec) {
        recp[0] = as_double(norm(Fv));
        recp[rec_e] = as_double(norm(Ev));
        recp += L.s[1];
      }
      const C F_p1 = shfl_dn(Fv, 1), E_p1 = shfl_dn(Ev, 1), v_p1 = shfl_dn(vc, 1);
      // momentum fluxes: P_x cell-centred, P_y and P_z on the x-y and x-z edges
      C P[3] = {z, z, z};
      {
        const C dw = w[0] - shfl_up(w[0], 1);
        const C dw_p = shfl_dn(dw, 1), dw_p2 = shfl_dn(dw, 2);
        if (!EDGE || (x >= 2 && x < sx - 2)) {
          const C uc = add_k(halve(vc + v_p1), bg.V[0]);
          const C Fc = halve(add_u(Fv, F_p1));
          const C ws = upwind_d(w[0], v_p1, dw, dw_p, dw_p2, uc, mul_u(uc, dtdx));
          P[0] = ky_add(bg.V[0], Fc, mul_u(ws, add_k(Fc, F0)));
        }
      }
#pragma unroll
      for (int m = 1; m < 3; ++m) {
        const C w_m1 = shfl_up(w[m], 1), dw = w[m] - w_m1;
        const C dw_m = shfl_up(dw, 1), dw_p = shfl_dn(dw, 1);
        if (!EDGE || (okF && (m == 1 ? row >= 1 : p >= 1))) {
          const C ue = add_k(halve((m == 1 ? vb : vp) + vc), bg.V[0]);
          const C Fe = halve(add_u(m == 1 ? Fb : Fp, Fv));
          const C ws = upwind_d(w_m1, w[m], dw_m, dw, dw_p, ue, mul_u(ue, dtdx));
          P[m] = ky_add(bg.V[m], Fe, mul_u(ws, add_k(Fe, F0)));
        }
      }
      const C Px_m1 = shfl_up(P[0], 1), Py_p1 = shfl_dn(P[1], 1), Pz_p1 = shfl_dn(P[2], 1);
      // conservative update of this cell
      if (own) {
        const unsigned c = c0 + (unsigned)p * stM;
        const bool upd = !EDGE || (x >= 2 && x < sx - 2);
        C rv = rc, ev = ec;
        if (upd) {
          C Flo = Fv, Fhi = F_p1, Elo = Ev, Ehi = E_p1;
          if (fr.side[0] >= 0 || fr.side[1] >= 0) fr.substitute(L, p, Flo, Fhi, Elo, Ehi);
          rv = rv - mul_u(sub_u(Fhi, Flo), iv);
          ev = ev - mul_u(sub_u(Ehi, Elo), iv);
        }
        stb((C*)it.S.F, c, rv);
        stb((C*)it.S.E, c, ev);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          C pv = z;  // the momentum Pi - rho0 V of v
          const bool in = !EDGE || (m == 0 ? x >= 1 : m == 1 ? row >= 1 : p >= 1);
          if (in) {
            const C drf = halve(add_u(m == 0 ? r_m1 : m == 1 ? rb : rp, rc));
            pv = add_u(mul_u(bg.rho0, w[m]), mul_u(drf, add_k(w[m], bg.V[m])));
          }
          if (!EDGE || (upd && in && (m != 0 || x >= 3)))
            pv = pv - mul_u(m == 0 ? sub_u(P[0], Px_m1) : sub_u(m == 1 ? Py_p1 : Pz_p1, P[m]), iv);
          stb((C*)it.S.pi[m], c, pv);
        }
      }
    }
    rp = rc;
    vp = vc;
    Fp = Fv;
  }
}

// planes [m0, m1) of a column.  BATCH, in a pool: every chunk of a box that reaches the ends
// of the march takes the EDGE form, whose multiply-adds the compiler may contract otherwise,
// so that a run's bits do not depend on where its pool's chunks end (FP32 runs with G = 2 or
// 6 differed by roundings; 24 uneven FP32 runs a step, chosen by the chunk and by the box: with
// viscosity 11.47 and 11.47 ms, with G = 6 6.91 and 6.91; chunks by the run alone instead 12.21
// and 7.10).
template <class T, int d, bool BATCH>
__device__ __forceinline__ void sweep_column(const Item<T>& it, int col, int m0, int m1,
                                             Arith<T>* __restrict__ buf) {
  constexpr int MU = d == 0 ? 2 : d;
  const int e0 = BATCH ? it.b.lo[MU] : m0, e1 = BATCH ? it.b.hi[MU] : m1;
  constexpr int RA = d == 1 ? 2 : 1;
  const Box& b = it.b;
  SweepLane p;
  if (!sweep_lane(b, d, col * (kSweepThreads / 32) + (int)(threadIdx.x >> 5),
                  (int)(threadIdx.x & 31), p))
    return;
  if (d == 0) {
    if (b.lo[0] >= 3 && b.hi[0] <= it.L.s[0] - 2 && b.lo[1] >= 1 && e0 >= 1)
      sweep_x<T, false>(it, p.x, p.row, p.mine, m0, m1, buf);
    else
      sweep_x<T, true>(it, p.x, p.row, p.mine, m0, m1, buf);
  } else {
    if (b.lo[0] >= 1 && b.lo[RA] >= 1 && e0 >= 3 && e1 <= it.L.s[d] - 2)
      sweep_march<T, d == 0 ? 1 : d, false>(it, p.x, p.row, p.mine && p.x >= b.lo[0], m0, m1, buf);
    else
      sweep_march<T, d == 0 ? 1 : d, true>(it, p.x, p.row, p.mine && p.x >= b.lo[0], m0, m1, buf);
  }
}

// a unit of a sweep; ENDS: the columns are laid end to end (Box::zc < 0), a form of its own
// because one form for both ran 0.6 % slower where chunks are taken (3 x 64^3 FP64 762 and
// 766 us a coarse step)
template <class T, int d, bool ENDS, bool BATCH>
__device__ __forceinline__ void el_sweep(const Item<T>& it, unsigned unit,
                                         Arith<T>* __restrict__ buf) {
  constexpr int MU = d == 0 ? 2 : d;
  const Box& b = it.b;
  if (ENDS) {
    const int nm = b.hi[MU] - b.lo[MU];
    int pos, end;
    sweep_unit(b, d, (int)unit, pos, end);
    while (pos < end) {
      const int col = pos / nm, m0 = b.lo[MU] + pos - col * nm;
      const int m1 = min(m0 + end - pos, b.hi[MU]);
      sweep_column<T, d, BATCH>(it, col, m0, m1, buf);
      pos += m1 - m0;
    }
  } else {
    const int ncol = sweep_columns(b, d), chunk = (int)unit / ncol;
    const int m0 = b.lo[MU] + chunk * b.zc;
    sweep_column<T, d, BATCH>(it, (int)unit - chunk * ncol, m0, min(m0 + b.zc, b.hi[MU]), buf);
  }
}

// velocity from the transported momenta, then the second half kick S(dt/2); NC cells
// per thread as in el_source.  KICK2: the first sub-cycle of a finest level, whose
// second sub-cycle follows with nothing in between that changes the level: the
// second sub-cycle's first kick S(dt/2) is applied here too, as el_source computes it
// from the stored velocity (so with the same bits), and the momenta its transport
// starts from are written; that sub-cycle runs no kick of its own.
template <class T, int NC, int KICK2>
__device__ __forceinline__ void el_vrec_source(const LevelView& L, const Box& b, const Scratch& S,
                                               const Arith<T>* __restrict__ dtp, Arith<T> gm1,
                                               const Bg<Arith<T>>& bg, const Geo<Arith<T>>& g,
                                               const Again& ag, int write_pi,
                                               const unsigned* el) {
  using C = Arith<T>;
  int c[NC], c3[NC][3];
  bool ok[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    int i, j, k;
    ok[n] = decode(b, el[n], i, j, k);
    if (NC == 1 && !ok[n]) return;
    if (!ok[n]) i = j = k = 1;
    c[n] = cidx(L, i, j, k);
    c3[n][0] = i;
    c3[n][1] = j;
    c3[n][2] = k;
  }
  const St<T>* __restrict__ rho = (const St<T>*)L.q[F_RHO];
  const St<T>* __restrict__ e = (const St<T>*)L.q[F_E];
  const Arith<T>* __restrict__ phi = (const Arith<T>*)L.phi;
  const C h = halve(dtp[0]);
  C rc[NC], ec[NC], fc[NC], rm[NC][3], em[NC][3], fm[NC][3], pv[NC][3];
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    rc[n] = ld(rho, c[n]);
    ec[n] = ld(e, c[n]);
    fc[n] = ld(phi, c[n]);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (c3[n][d] >= 1) {
        const int m = c[n] - L.st[d];
        rm[n][d] = ld(rho, m);
        em[n][d] = ld(e, m);
        fm[n][d] = ld(phi, m);
        pv[n][d] = ld((const C*)S.pi[d], c[n]);
      }
  }
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    if (!ok[n]) continue;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (c3[n][d] < 1) {
        if (KICK2 && write_pi) ((Arith<T>*)S.pi[d])[c[n]] = C(0.f);
        continue;
      }
      C drf = halve(rm[n][d] + rc[n]);
      C rinv = div_u(C(1.f), bg.rho0 + drf);
      C v = mul_u(sub_ky(pv[n][d], bg.V[d], drf), rinv);
      C acc = mul_u(mul_u(mul_u(gm1, ec[n] - em[n][d]), rinv) + (fc[n] - fm[n][d]),
                    g.inv_dx[d]);
      C vn = v - mul_u(h, acc);
      if (KICK2) {  // the same expression as the kick's
        const C rf = bg.rho0 + drf;
        const C acc2 = mul_u(div_u(mul_u(gm1, ec[n] - em[n][d]), rf) + (fc[n] - fm[n][d]),
                             g.inv_dx[d]);
        vn = as_stored(vn) - mul_u(h, acc2);
        if (write_pi)
          st((Arith<T>*)S.pi[d], c[n], mul_u(bg.rho0, vn) + mul_u(drf, add_k(vn, bg.V[d])));
      }
      if (KICK2)
        st_kicked((St<T>*)L.q[F_VX + d], c[n], vn, ag.has(c3[n]));
      else
        st((St<T>*)L.q[F_VX + d], c[n], vn);
    }
  }
}

// ------------------------------------------------------ boundaries, mirror planes
// Fill of the ghost layers by type, axis x, then y, then z, in one launch: where layers of
// several axes meet, an element follows the later axis' source to the earlier axis' (the
// value the axis-by-axis fill would copy), so every element reads active ones only.  One
// thread per element of the shell, all five fields (one launch per axis and a thread per
// field: 1533 of the 6151 launches of a coarse step of nine quadrant levels, 25.2 ms of
// FP32 steps against 23.3; 16 serving runs 0.96 against 0.87).  Sides of type -1 are left
// alone.
//   With as few cells as ghost layers (n = G) a lower wall's last ghost face of v_d, 0,
// mirrors the upper boundary face G + n, which the upper side's fill overwrites; the plan
// then fills axis by axis (bc_by_axis), and the thread of face G + n writes face 0 too.

// source index along axis d of an element with index c; returns 0: the element itself
// (not filled along d), 1: a copy, 2: a copy with the opposite normal velocity, 3: the
// fixed deviation in `fixed`
template <class T>
__device__ __forceinline__ int bc_source(int G, int n, int lo, int hi, int normal, T V, int& c,
                                         T& fixed) {
  const int side = c < G ? 0 : 1;
  const int type = c < G ? lo : (c >= G + n ? hi : -1);
  int how = 0;
  if (type == 0) {  // periodic
    c += side ? -n : n;
    how = 1;
  } else if (type == 1) {  // outflow: the nearest active element; for v_d the boundary
                           // face (G or G + n), which the solver owns on both sides
    if (normal && side && c == G + n) return 0;
    c = side ? (normal ? G + n : G + n - 1) : G;
    how = 1;
  } else if (type == 2) {  // inflow: the background itself
    fixed = T(0);
    return 3;
  } else if (type == 3) {  // reflect
    if (!normal) {
      c = side ? 2 * (G + n) - 1 - c : 2 * G - 1 - c;
      how = 1;
    } else if (side && c == G + n) {  // the wall face
      fixed = -V;
      return 3;
    } else {  // v_ghost = -v_mirror, so dv_ghost = -dv_mirror - 2 V_d
      c = side ? 2 * (G + n) - c : 2 * G - c;
      how = 2;
    }
  }
  // the lower boundary face G of v_d: 0 at a wall, V (zero deviation) on an injection
  // face; the upper boundary face G + n is the first ghost element of the upper side
  if (normal && c == G && lo >= 2) {
    fixed = lo == 3 ? -V : T(0);
    return 3;
  }
  return how;
}

template <class T>
__device__ __forceinline__ void el_bc(const LevelView& L, const int* bc, T V0, T V1, T V2,
                                      unsigned tid) {
  int c[3];
  if (!bc_element(L, bc, tid, c)) return;
  const int dst = (c[2] * L.s[1] + c[1]) * L.s[0] + c[0];
  const T V[3] = {V0, V1, V2};
  // every field's source first, so that no load waits for a store
  int how[5], flip[5];  // flip: the normal velocity changed sign
  T fixed[5];
  St<T> q[5];
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    int src[3] = {c[0], c[1], c[2]};
    how[f] = flip[f] = 0;
    fixed[f] = T(0);
#pragma unroll
    for (int d = 2; d >= 0; --d) {
      if (how[f] == 3) continue;
      const int h = bc_source<T>(L.G, L.n[d], bc[2 * d], bc[2 * d + 1], f == F_VX + d, V[d],
                                 src[d], fixed[f]);
      if (h == 2) flip[f] = 1;
      if (h) how[f] = h;
    }
    if (how[f] == 1 || how[f] == 2)
      q[f] = ((const St<T>*)L.q[f])[(src[2] * L.s[1] + src[1]) * L.s[0] + src[0]];
  }
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    if (!how[f]) continue;
    St<T>* out = (St<T>*)L.q[f];
    const T Vf = f >= F_VX ? V[f - F_VX] : T(0);
    if (f >= F_VX && bc_wraps(L, bc, f - F_VX)) {
      if (c[f - F_VX] == 0) continue;
      if (c[f - F_VX] == L.G + L.n[f - F_VX])
        put(out, dst - c[f - F_VX] * L.st[f - F_VX], T(-1) * val(out, dst) + T(-2) * Vf);
    }
    if (how[f] == 3)  // (a flip found on a later axis than the fixed value's)
      put(out, dst, flip[f] ? -fixed[f] - T(2) * Vf : fixed[f]);
    else if (flip[f])
      put(out, dst, T(-1) * val(&q[f], 0) + T(-2) * Vf);
    else
      out[dst] = q[f];  // a copy keeps the stored value as it is
  }
}

// ---------------------------------------------------------------- CommUp
// A coarse host element holds 2 x 2 x 2 fine elements; CommUp fills the fine ghosts.
// Per field, the hosts with a ghost among their fine elements form the shell of
// their host box around the hosts whose fine elements are all kept (active cells;
// for v_d the faces strictly inside along d, so both frontier faces of v_d are
// filled).  The shell is cut into six disjoint boxes (two slabs across z over the
// whole x-y range, two across y, two across x), each into tiles of at most
// kCuHosts hosts in one host z-plane, one 256-thread chunk per tile.  The z pass
// interpolates each coarse column of a tile and its halo once (to both fine z
// offsets) into shared memory, the y pass each x-column once (to both fine y
// offsets), and the x pass gives a host's 8 fine elements: the arithmetic of
// interpolating each fine element alone along z, then y, then x, with every slope
// computed once per tile.  Along a staggered field's own axis the fine faces lie on
// the host face (copied) or midway to the next one (mean of the two, which favours
// neither side), so a mirror-symmetric coarse state gives mirror-symmetric ghosts.
static_assert(kCuHosts == kBlock, "one thread per host of a CommUp tile");

template <class T>
__device__ __forceinline__ void el_commup(const LevelView& C, const LevelView& F, unsigned tid) {
  using A = Arith<T>;  // the interpolation runs in the stencils' arithmetic type
  __shared__ A s_z[2][kCuZ];  // [fine z offset][column (y, x) of the tile and halo]
  __shared__ A s_y[4][kCuY];  // [fine z offset * 2 + fine y offset][(host y, x column)]
  __shared__ CuBox s_box;
  __shared__ int s_fr[2];     // field (-1: past the last tile) and tile within the box
  const int lt = (int)(tid % kBlock);
  // warp 0 finds the chunk's field and box: lane i takes box i % 6 of field i / 6
  if (lt < 32) {
    const int r = (int)(tid / kBlock);
    const int fb = lt < 30 ? lt : 29;
    const CuBox B = cu_box(F.n, F.G, fb / 6 >= F_VX ? fb / 6 - F_VX : -1, fb % 6);
    const int c = lt < 30 ? B.ez * B.ntx * B.nty : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lt >= o) incl += v;
    }
    const bool hit = r >= incl - c && r < incl;
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    if (hit) {
      s_box = B;
      s_fr[0] = fb / 6;
      s_fr[1] = r - (incl - c);
    }
    if (lt == 0 && m == 0u) s_fr[0] = -1;
  }
  __syncthreads();
  const int f = s_fr[0];
  if (f < 0) return;  // uniform over the block
  const CuBox B = s_box;
  const int r = s_fr[1];
  const int sa = f >= F_VX ? f - F_VX : -1;
  const int per = B.ntx * B.nty;
  const int pz = r / per, rt = r - pz * per;
  const int tyi = rt / B.ntx, txi = rt - tyi * B.ntx;
  const int h2 = B.z0 + pz;
  const int X0 = B.x0 + txi * B.tx, Y0 = B.y0 + tyi * B.ty;
  const int wx = min(B.tx, B.x0 + B.ex - X0), wy = min(B.ty, B.y0 + B.ey - Y0);
  const int P = wx + 2;  // pitch of a row of columns
  // the two centred fine positions lie at -1/4 and +1/4 of a coarse cell: q0 -+ half
  // of the half slope hslope returns
  const St<T>* q = (const St<T>*)C.q[f];
  // z pass: the tile's columns and a halo of one (hosts in [-G/2 - 1, n/2 + G/2])
  for (int e = lt; e < P * (wy + 2); e += kBlock) {
    const int cy = e / P, cx = e - cy * P;
    const int hx = X0 - 1 + cx, hy = Y0 - 1 + cy;
    const int k = ((C.G + F.off[2] + h2) * C.s[1] + C.G + F.off[1] + hy) * C.s[0] + C.G +
                  F.off[0] + hx;
    const A qm = ld(q, k - C.st[2]), q0 = ld(q, k), qp = ld(q, k + C.st[2]);
    if (sa == 2) {
      s_z[0][e] = q0;
      s_z[1][e] = halve(q0 + qp);
    } else {
      const A sl = hslope(q0 - qm, qp - q0);
      s_z[0][e] = q0 - halve(sl);
      s_z[1][e] = q0 + halve(sl);
    }
  }
  __syncthreads();
  // y pass: every x column of the tile's host rows
  for (int e = lt; e < 2 * wy * P; e += kBlock) {
    const int iz = e / (wy * P), rem = e - iz * wy * P;
    const A qm = s_z[iz][rem], q0 = s_z[iz][rem + P], qp = s_z[iz][rem + 2 * P];
    if (sa == 1) {
      s_y[2 * iz][rem] = q0;
      s_y[2 * iz + 1][rem] = halve(q0 + qp);
    } else {
      const A sl = hslope(q0 - qm, qp - q0);
      s_y[2 * iz][rem] = q0 - halve(sl);
      s_y[2 * iz + 1][rem] = q0 + halve(sl);
    }
  }
  __syncthreads();
  // x pass and stores: one host per thread
  if (lt >= wx * wy) return;
  const int ty = lt / wx, tx = lt - ty * wx;
  const int h0 = X0 + tx, h1 = Y0 + ty;
  St<T>* out = (St<T>*)F.q[f];
  const int G = F.G;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int iz = j >> 1, iy = j & 1;
    const A* row = s_y[j] + ty * P + tx;
    const A qm = row[0], q0 = row[1], qp = row[2];
    A v[2];
    if (sa == 0) {
      v[0] = q0;
      v[1] = halve(q0 + qp);
    } else {
      const A sl = hslope(q0 - qm, qp - q0);
      v[0] = q0 - halve(sl);
      v[1] = q0 + halve(sl);
    }
    // the two fine elements along x are neighbours in memory: one vector store when
    // both are ghosts and the pair starts on an even element (aligned)
    const int fi0 = G + 2 * h0, fj = G + 2 * h1 + iy, fk = G + 2 * h2 + iz;
    const bool yz = fj >= G + (sa == 1) && fj < G + F.n[1] && fk >= G + (sa == 2) &&
                    fk < G + F.n[2];
    const bool act0 = yz && fi0 >= G + (sa == 0) && fi0 < G + F.n[0];
    const bool act1 = yz && fi0 + 1 >= G + (sa == 0) && fi0 + 1 < G + F.n[0];
    const int e0 = (fk * F.s[1] + fj) * F.s[0] + fi0;
    if (!act0 && !act1 && (e0 & 1) == 0) {
      st2(out, e0, v[0], v[1]);
      continue;
    }
#pragma unroll
    for (int ix = 0; ix < 2; ++ix) {
      const bool act = ix == 0 ? act0 : act1;
      if (!act) st(out, e0 + ix, v[ix]);
    }
  }
}

// -------------------------------------------------------------- CommMean
__device__ __forceinline__ bool in_band(const LevelView& F, int band, int a0, int a1, int a2) {
  int a3[3] = {a0, a1, a2};
  int dist = 1 << 30;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    int lo = a3[d] - F.off[d], hi = F.off[d] + (F.n[d] >> 1) - 1 - a3[d];
    if (lo < 0 || hi < 0) return false;
    if (F.mir >> d & 1) lo = 1 << 30;  // a mirror face bounds no band
    dist = min(dist, min(lo, hi));
  }
  return dist < band;
}

template <class T>
__device__ __forceinline__ void el_commmean(const LevelView& C, const LevelView& F, int band, unsigned tid) {
  const unsigned t = tid;  // coarse cells of the covered box: fewer than 2^31
  const unsigned h0 = F.n[0] >> 1, h1 = F.n[1] >> 1, h2 = F.n[2] >> 1;
  if (t >= h0 * h1 * h2) return;
  const unsigned q = t / h0;
  int a = (int)(t - q * h0), b = (int)(q % h1), cc = (int)(q / h1);
  int r[3] = {a, b, cc};
  int a3[3] = {a + F.off[0], b + F.off[1], cc + F.off[2]};
  const int Gf = F.G, Gc = C.G;
  int dst = ((Gc + a3[2]) * C.s[1] + Gc + a3[1]) * C.s[0] + Gc + a3[0];
  if (in_band(F, band, a3[0], a3[1], a3[2])) {
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const St<T>* q = (const St<T>*)F.q[f];
      Arith<T> sz[2];
#pragma unroll
      for (int dz = 0; dz < 2; ++dz) {
        Arith<T> sy[2];
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
          int c0 = ((Gf + 2 * cc + dz) * F.s[1] + Gf + 2 * b + dy) * F.s[0] + Gf + 2 * a;
          sy[dy] = ld(q, c0) + ld(q, c0 + 1);
        }
        sz[dz] = sy[0] + sy[1];
      }
      st((St<T>*)C.q[f], dst, pow2_times(sz[0] + sz[1], 0.125f));
    }
  }
#pragma unroll
  for (int sa = 0; sa < 3; ++sa) {
    if (r[sa] == 0) continue;
    int m3[3] = {a3[0], a3[1], a3[2]};
    m3[sa] -= 1;
    if (!in_band(F, band, a3[0], a3[1], a3[2]) && !in_band(F, band, m3[0], m3[1], m3[2])) continue;
    int t1 = sa == 0 ? 1 : 0, t2 = sa == 2 ? 1 : 2;
    const St<T>* q = (const St<T>*)F.q[F_VX + sa];
    Arith<T> sv[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      Arith<T> pair[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        int fi[3];
        fi[sa] = Gf + 2 * r[sa];
        fi[t1] = Gf + 2 * r[t1] + u;
        fi[t2] = Gf + 2 * r[t2] + v;
        pair[u] = ld(q, (fi[2] * F.s[1] + fi[1]) * F.s[0] + fi[0]);
      }
      sv[v] = pair[0] + pair[1];
    }
    st((St<T>*)C.q[F_VX + sa], dst, pow2_times(sv[0] + sv[1], 0.25f));
  }
}

// ------------------------------------------------------------ reductions of a run
// True in the last of a run's `total` chunks of one reduction to get here: every chunk's
// results are then visible (read them past L1).  Each chunk counts itself after its
// results are written; the last one clears the count for the next step.  Nothing waits.
// The final step of a reduction then needs no launch of its own, and the levels share one
// (one 32^3 level: 13 launches, 67.7 us a coarse step -> 10, 66.2; 3 x 64^3 FP64 69, 834
// us -> 62, 800; 16 serving runs 99, 874 us -> 71, 770).  Large levels keep their launches
// (joined_levels).
__device__ __forceinline__ bool last_chunk(unsigned* done, unsigned total) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const bool last = atomicAdd(done, 1u) == total - 1u;
    if (last) *done = 0u;
    __threadfence();
    s_last = last;
  }
  __syncthreads();
  return s_last != 0;
}

// ------------------------------------------------------------- time step
__device__ __forceinline__ float warp_max_t(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// the larger of two double-float values (a total order on normalised pairs: hi, then
// lo); a NaN operand loses, as in fmax
__device__ __forceinline__ df64 dmax(df64 a, df64 b) {
  return (a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo) || b.hi != b.hi) ? a : b;
}
__device__ __forceinline__ df64 warp_max_t(df64 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = dmax(v, df64(__shfl_xor_sync(0xffffffffu, v.hi, o),
                     __shfl_xor_sync(0xffffffffu, v.lo, o)));
  return v;
}
__device__ __forceinline__ df64 dabs(df64 v) { return v.hi < 0.f ? -v : v; }
// Square root in double-float: the float root s refined by one Newton step on the
// square (Heron's method; the double-length form of Karp & Markstein, ACM TOMS 23,
// 1997): s + (x - s^2) / (2 s), with s^2 exact as a product plus its error, so the
// residual is exact up to the low parts and the result good to about 2^-46.  For
// x <= 0 (an unhealthy state, flagged by the caller) the float root of hi.
__device__ __forceinline__ df64 dsqrt(df64 x) {
  const float s = sqrtf(x.hi);
  if (!(x.hi > 0.f)) return df64(s);
  const df64 s2 = two_prod(s, s);
  const float r = ((x.hi - s2.hi) - s2.lo + x.lo) * (0.5f * rcp_est(s));
  return fast_two_sum(s, r);
}

// Per-level Courant limit: min over active cells and axes of cfl dx_d / (cs + |v_d|).
// Division is correctly rounded and monotone, so that minimum equals
// cfl dx_d / max(cs + |v_d|): the kernel reduces the per-axis maxima (one division
// per level instead of three per cell); a maximum is exact in any precision, so it
// is taken in the per-cell type and widened once per block.  Per-cell arithmetic:
// FP32 for the FP32 state (FP32 sound speeds); double-float for the FP64 state (its
// sound speed and |v| within about 2^-44, so the limit is within that of the FP64
// one; the FP64 pipe would take ~40 operations per cell).  The maxima, the minimum
// over levels and dt itself are FP64.  Also flags NaN, rho <= 0 or e <= 0.
constexpr int kDtCells = 4;
template <class T>
__device__ __forceinline__ void el_dt_level(const LevelView& L, const Box& b, int level, double gg,
                                            Arith<T> gga, int hydro, DevScalars* ds,
                                            double rho0, double e0, double V0, double V1,
                                            double V2, const Bg<Arith<T>>& bg,
                                            unsigned tid) {
  using A = Arith<T>;
  __shared__ A sm[3][kBlock / 32];
  __shared__ int bad_s;
  if (threadIdx.x == 0) bad_s = 0;
  __syncthreads();
  A mx[3] = {A(0.f), A(0.f), A(0.f)};
  // kDtCells cells per thread (strided by the block size), every load first: a block
  // then issues one atomic per axis for kBlock kDtCells cells
  int cc[kDtCells];
  bool in[kDtCells];
#pragma unroll
  for (int u = 0; u < kDtCells; ++u) {
    const unsigned t = (tid / kBlock) * kBlock * kDtCells + u * kBlock + threadIdx.x;
    int i, j, k;  // b is the active box: multiply-shift division, no 64-bit divide
    in[u] = decode(b, t, i, j, k);
    cc[u] = in[u] ? (k * L.s[1] + j) * L.s[0] + i : (L.G * L.s[1] + L.G) * L.s[0] + L.G;
  }
  const St<T>* v3[3] = {(const St<T>*)L.q[F_VX], (const St<T>*)L.q[F_VX + 1],
                        (const St<T>*)L.q[F_VX + 2]};
  bool bad = false;
  if constexpr (sizeof(T) == 4) {
    float rho[kDtCells], e[kDtCells], va[kDtCells][3], vb[kDtCells][3];
#pragma unroll
    for (int u = 0; u < kDtCells; ++u) {
      const int c = cc[u];
      rho[u] = val((const St<T>*)L.q[F_RHO], c);
      e[u] = val((const St<T>*)L.q[F_E], c);
      if (hydro)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          va[u][d] = val(v3[d], c);
          vb[u][d] = val(v3[d], c + L.st[d]);
        }
    }
    const float Vb[3] = {(float)V0, (float)V1, (float)V2};
#pragma unroll
    for (int u = 0; u < kDtCells; ++u) {
      if (!in[u]) continue;
      const float r = (float)rho0 + rho[u], ee = (float)e0 + e[u];
      if (!(r > 0.f) || !(ee > 0.f)) bad = true;
      if (hydro) {
        const float cs = sqrtf((float)gg * ee / r);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float v0 = fabsf(Vb[d] + va[u][d]), v1 = fabsf(Vb[d] + vb[u][d]);
          const float m = cs + (v0 > v1 ? v0 : v1);
          mx[d] = m > mx[d] ? m : mx[d];
        }
      }
    }
  } else {
    A rho[kDtCells], e[kDtCells], va[kDtCells][3], vb[kDtCells][3];
#pragma unroll
    for (int u = 0; u < kDtCells; ++u) {
      const int c = cc[u];
      rho[u] = ld((const St<T>*)L.q[F_RHO], c);
      e[u] = ld((const St<T>*)L.q[F_E], c);
      if (hydro)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          va[u][d] = ld(v3[d], c);
          vb[u][d] = ld(v3[d], c + L.st[d]);
        }
    }
#pragma unroll
    for (int u = 0; u < kDtCells; ++u) {
      if (!in[u]) continue;
      const A r = bg.rho0 + rho[u], ee = bg.e0 + e[u];
      if (!gt0(r) || !gt0(ee)) bad = true;
      if (hydro) {
        const A cs = dsqrt(hdiv(gga * ee, r));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const A v0 = dabs(add_k(va[u][d], bg.V[d])), v1 = dabs(add_k(vb[u][d], bg.V[d]));
          mx[d] = dmax(mx[d], cs + dmax(v0, v1));
        }
      }
    }
  }
  if (bad) bad_s = 1;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    A v = warp_max_t(mx[d]);
    if ((threadIdx.x & 31) == 0) sm[d][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      A v = threadIdx.x < kBlock / 32 ? sm[d][threadIdx.x] : A(0.f);
      v = warp_max_t(v);
      // non-negative doubles order like their bit patterns (NaN is caught above)
      const double w = as_double(v);
      if (threadIdx.x == 0 && w > 0.0)
        atomicMax(&ds->dtmin[3 * level + d], (unsigned long long)__double_as_longlong(w));
    }
    if (threadIdx.x == 0 && bad_s) atomicOr(&ds->unhealthy, 1);
  }
}

// Eq. 55: dt = min_l dt_l prod_{m<l} xi_m; resets the per-level maxima.  One block; a
// thread per level and axis, then per level, per sub-cycling word and per constant.
__device__ __forceinline__ void el_dt_finalize(DevScalars* ds, int n_levels, const DtFinal& fin,
                                               double dt_fixed) {
  __shared__ double s_adv[48], s_lim[16], s_prod[16], s_dt;
  __shared__ double s_ratio[kBlock];
  __shared__ int s_word[kBlock];
  const int t = threadIdx.x;
  if (t < 3 * n_levels) {
    const double mx = __longlong_as_double((long long)__ldcg(&ds->dtmin[t]));
    s_adv[t] = fin.cfl_dx[t / 3][t % 3] / mx;  // +inf when the maximum is 0
    ds->dtmin[t] = 0ull;
  }
  __syncthreads();
  if (t < n_levels) {
    double lim = fin.diff_lim[t];
    for (int d = 0; d < 3; ++d)
      if (s_adv[3 * t + d] < lim) lim = s_adv[3 * t + d];
    ds->dtlev[t] = lim;
    s_lim[t] = lim;
    s_prod[t] = fin.prod[t];
  }
  __syncthreads();
  unsigned xi1 = 0;
  if (fin.search && n_levels > 1) {
    // Eq. 55-56: the word xi_m in {1, 2} (bit m of w set: xi_m = 2) with the largest
    // step per unit cost; ties go to the smallest w, as a sequential scan keeps the
    // first maximum
    const int nw = n_levels - 1;
    double best = -1.0;
    int bw = 0;
    for (int w = t; w < (1 << nw); w += kBlock) {
      double dt = INFINITY, C = 0.0, pr = 1.0;
      for (int l = 0; l < n_levels; ++l) {
        if (l > 0) pr *= ((w >> (l - 1)) & 1) ? 2.0 : 1.0;
        const double tl = s_lim[l] * pr;
        if (tl < dt) dt = tl;
        C += fin.cost[l] * pr;
      }
      const double ratio = dt / C;
      if (ratio > best) {
        best = ratio;
        bw = w;
      }
    }
    s_ratio[t] = best;
    s_word[t] = bw;
    __syncthreads();
    for (int h = kBlock / 2; h > 0; h >>= 1) {
      if (t < h) {
        const double r2 = s_ratio[t + h];
        const int w2 = s_word[t + h];
        if (r2 > s_ratio[t] || (r2 == s_ratio[t] && w2 < s_word[t])) {
          s_ratio[t] = r2;
          s_word[t] = w2;
        }
      }
      __syncthreads();
    }
    const int w = s_word[0];
    double pr = 1.0;
    for (int l = 0; l < n_levels; ++l) {
      if (l > 0) {
        const bool two = (w >> (l - 1)) & 1;
        pr *= two ? 2.0 : 1.0;
        if (!two) xi1 |= 1u << (l - 1);
      }
      if (t == 0) s_prod[l] = pr;
    }
  }
  if (t == 0) {
    double dt = INFINITY;
    for (int l = 0; l < n_levels; ++l) {
      const double tl = s_lim[l] * s_prod[l];
      if (tl < dt) dt = tl;
    }
    if (dt_fixed > 0.0) dt = dt_fixed;
    s_dt = dt;
    ds->dt = dt;
    ds->xi1 = xi1;
  }
  __syncthreads();
  // level steps take dt / prod_{m<l} xi_m (a power of two: exact), and their constants
  // are formed once here instead of in every thread of the level step
  for (int i = t; i < 13 * n_levels; i += kBlock) {
    const int l = i / 13, q = i - 13 * l;
    const double dl = s_dt / s_prod[l];
    if (q == 12) {
      ds->dtl[l] = dl;
      ds->dtf[l] = (float)dl;
      ds->dtd[l] = to_df64(dl);
    } else {
      const double c = fin.kfac[l][q] * dl;
      ds->kd[l][q] = to_df64(c);
      ds->kf[l][q] = (float)c;
    }
  }
}

// ------------------------------------------------------------------ force
// Eq. 18 on one level: F += (rho - rho0) w_c over uncovered active cells, with the
// static FP64 weight vectors w_c = GM V_c r_c / (r^2 + eps^2)^(3/2) precomputed
// (x, y and z components in three planes of fw).  Each thread accumulates
// kForceCells cells (strided by the block size) in FP64, then a fixed warp-shuffle
// tree and the 8 warp sums give one partial per block.
constexpr int kForceCells = 8;

template <class T>
__device__ __forceinline__ void el_force_level(const LevelView& L, const Box& b,
                                               const double* __restrict__ fw,
                                               double* partials, unsigned tid) {
  __shared__ double sw[3][kBlock / 32];
  const long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  const double* fx = fw;
  const double* fy = fw + na;
  const double* fz = fw + 2 * na;
  double f[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int u = 0; u < kForceCells; ++u) {
    const unsigned t = (tid / kBlock) * kBlock * kForceCells + u * kBlock + threadIdx.x;
    int i, j, k;  // b is the active box: multiply-shift division, no 64-bit divide
    if (!decode(b, t, i, j, k)) break;
    const int ai = i - L.G, aj = j - L.G, ak = k - L.G;
    bool covered = L.has_child && ai >= L.coff[0] && ai < L.coff[0] + (L.cn[0] >> 1) &&
                   aj >= L.coff[1] && aj < L.coff[1] + (L.cn[1] >> 1) && ak >= L.coff[2] &&
                   ak < L.coff[2] + (L.cn[2] >> 1);
    if (covered) continue;
    double dr = (double)val((const St<T>*)L.q[F_RHO], ((L.G + ak) * L.s[1] + L.G + aj) * L.s[0] + L.G + ai);
    f[0] += dr * fx[t];
    f[1] += dr * fy[t];
    f[2] += dr * fz[t];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f[d] += __shfl_down_sync(0xffffffffu, f[d], o);
    if ((threadIdx.x & 31) == 0) sw[d][threadIdx.x >> 5] = f[d];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kBlock / 32; ++w) s += sw[threadIdx.x][w];
    partials[3 * (tid / kBlock) + threadIdx.x] = s;
  }
}

// static force weights of the active cells; with mirror planes the force is that of
// the unfolded domain: no component along a mirror axis, the others mult times the
// sum over the simulated part (mult = 2^planes scales exactly)
__global__ void __launch_bounds__(kBlock) k_force_weights(LevelView L, double GM, double eps,
                                                          double mult, double* fw) {
  long long t = blockIdx.x * (long long)kBlock + threadIdx.x;
  long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  if (t >= na) return;
  int ai = (int)(t % L.n[0]);
  int aj = (int)((t / L.n[0]) % L.n[1]);
  int ak = (int)(t / ((long long)L.n[0] * L.n[1]));
  double x = L.lo[0] + (ai + 0.5) * L.dx[0];
  double y = L.lo[1] + (aj + 0.5) * L.dx[1];
  double z = L.lo[2] + (ak + 0.5) * L.dx[2];
  double r2 = x * x + y * y + z * z + eps * eps;
  double w = GM * L.vol / (r2 * sqrt(r2));
  fw[t] = L.mir & 1 ? 0.0 : mult * (w * x);
  fw[t + na] = L.mir & 2 ? 0.0 : mult * (w * y);
  fw[t + 2 * na] = L.mir & 4 ? 0.0 : mult * (w * z);
}

constexpr int kPartialsAhead = 8;
// fixed-order compensated (Neumaier) sum of the block partials, one warp per
// component (threads 96.. of the block only take part in the barrier)
__device__ __forceinline__ void el_force_finalize(const double* partials, int n,
                                                  DevScalars* ds, double* ring, int ring_cap,
                                                  long long* ring_pos) {
  int comp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (comp < 3) {
    double s = 0.0, cmp = 0.0;
    for (int p = lane; p < n; p += 32 * kPartialsAhead) {
      double v[kPartialsAhead];  // that many in flight, added in order
#pragma unroll
      for (int k = 0; k < kPartialsAhead; ++k)
        v[k] = p + 32 * k < n ? __ldcg(&partials[3 * (p + 32 * k) + comp]) : 0.0;
#pragma unroll
      for (int k = 0; k < kPartialsAhead; ++k) {
        if (p + 32 * k >= n) break;
        const double tt = s + v[k];
        if (fabs(s) >= fabs(v[k]))
          cmp += (s - tt) + v[k];
        else
          cmp += (v[k] - tt) + s;
        s = tt;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      double so = __shfl_down_sync(0xffffffffu, s, o);
      double co = __shfl_down_sync(0xffffffffu, cmp, o);
      if (lane < o) {
        double tt = s + so;
        if (fabs(s) >= fabs(so))
          cmp += (s - tt) + so;
        else
          cmp += (so - tt) + s;
        s = tt;
        cmp += co;
      }
    }
    if (lane == 0) {
      double F = s + cmp;
      ds->F[comp] = F;
      if (ring) ring[kRingStride * (*ring_pos % ring_cap) + comp] = F;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && ring) {
    // the end of this coarse step
    ds->t += ds->dt;
    ring[kRingStride * (*ring_pos % ring_cap) + 3] = ds->t;
    *ring_pos += 1;
  }
}

// ----------------------------------------------------------- initialisation
template <class T>
__global__ void __launch_bounds__(kBlock) k_init_uniform(LevelView L, T rho0, T e0, T V0, T V1,
                                                         T V2) {
  long long c = blockIdx.x * (long long)kBlock + threadIdx.x;
  if (c >= L.nc) return;
  (void)rho0;
  (void)e0;
  (void)V0;
  (void)V1;
  (void)V2;
#pragma unroll
  for (int f = 0; f < 5; ++f) put((St<T>*)L.q[f], c, T(0));
}

// Plummer potential (Eq. 16, attractive sign) at every cell centre; luminosity
// weights on active cells and on their mirror images in the ghost layers (Gaussian
// weights are normalised afterwards)
template <class T>
__global__ void __launch_bounds__(kBlock) k_static(LevelView L, double GM, double eps,
                                                   double sigma, int vertex_ok, int vx0, int vx1,
                                                   int vx2) {
  long long c = blockIdx.x * (long long)kBlock + threadIdx.x;
  if (c >= L.nc) return;
  int i = (int)(c % L.s[0]), j = (int)((c / L.s[0]) % L.s[1]),
      k = (int)(c / ((long long)L.s[0] * L.s[1]));
  double x = L.lo[0] + (i - L.G + 0.5) * L.dx[0];
  double y = L.lo[1] + (j - L.G + 0.5) * L.dx[1];
  double z = L.lo[2] + (k - L.G + 0.5) * L.dx[2];
  // the static fields are held in the stencils' arithmetic type (double-float for the
  // FP64 state): only the stencils read them
  ((Arith<T>*)L.phi)[c] = from_double<Arith<T>>(-GM / sqrt(x * x + y * y + z * z + eps * eps));
  bool act = i >= (L.mir & 1 ? 0 : L.G) && i < L.G + L.n[0] &&
             j >= (L.mir & 2 ? 0 : L.G) && j < L.G + L.n[1] &&
             k >= (L.mir & 4 ? 0 : L.G) && k < L.G + L.n[2];
  double lw = 0.0;
  if (act) {
    if (sigma > 0.0) {
      lw = exp(-(x * x + y * y + z * z) / (2.0 * sigma * sigma));
    } else if (vertex_ok) {
      int ai = i - L.G, aj = j - L.G, ak = k - L.G;
      if ((ai == vx0 - 1 || ai == vx0) && (aj == vx1 - 1 || aj == vx1) &&
          (ak == vx2 - 1 || ak == vx2))
        lw = 1.0 / (8.0 * L.vol);
    }
  }
  ((Arith<T>*)L.lumw)[c] = from_double<Arith<T>>(lw);
}

// Gaussian weights: fixed-order sum over the active cells (block tree, then one
// block in index order), so every context normalises to the same bits
template <class T>
__global__ void __launch_bounds__(kBlock) k_lum_partials(LevelView L, double* partials) {
  __shared__ double sm[kBlock];
  long long t = blockIdx.x * (long long)kBlock + threadIdx.x;
  long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  double w = 0.0;
  if (t < na) {
    int i = (int)(t % L.n[0]), j = (int)((t / L.n[0]) % L.n[1]),
        k = (int)(t / ((long long)L.n[0] * L.n[1]));
    w = as_double(((const Arith<T>*)L.lumw)[((k + L.G) * L.s[1] + j + L.G) * L.s[0] + i + L.G]);
  }
  sm[threadIdx.x] = w;
  __syncthreads();
  for (int s = kBlock / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = sm[0];
}

__global__ void k_sum_partials(const double* __restrict__ partials, int n, double* out) {
  __shared__ double sm[kBlock];
  double s = 0.0;
  for (int p = threadIdx.x; p < n; p += kBlock) s += partials[p];
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int w = kBlock / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sm[threadIdx.x] += sm[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sm[0];
}

template <class T>
__global__ void __launch_bounds__(kBlock) k_normalise_lum(LevelView L, const double* wsum,
                                                          double mult) {
  long long c = blockIdx.x * (long long)kBlock + threadIdx.x;
  if (c >= L.nc) return;
  Arith<T>* lw = (Arith<T>*)L.lumw;
  // the unfolded domain holds mult copies of the active cells
  lw[c] = from_double<Arith<T>>(as_double(lw[c]) / (mult * wsum[0] * L.vol));
}

// host I/O: full values = background + stored deviation (bgv = 0 for raw state)
template <class T>
__global__ void __launch_bounds__(kBlock) k_pack(LevelView L, int field, double* out, int full,
                                                 double bgv) {
  long long t = blockIdx.x * (long long)kBlock + threadIdx.x;
  const St<T>* q = (const St<T>*)L.q[field];
  if (full) {
    if (t < L.nc) out[t] = bgv + (double)val(q, t);
    return;
  }
  long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  if (t >= na) return;
  int i = (int)(t % L.n[0]), j = (int)((t / L.n[0]) % L.n[1]),
      k = (int)(t / ((long long)L.n[0] * L.n[1]));
  out[t] = bgv + (double)val(q, ((k + L.G) * L.s[1] + j + L.G) * L.s[0] + i + L.G);
}

template <class T>
__global__ void __launch_bounds__(kBlock) k_unpack(LevelView L, int field, const double* in,
                                                   int full, double bgv) {
  long long t = blockIdx.x * (long long)kBlock + threadIdx.x;
  St<T>* q = (St<T>*)L.q[field];
  if (full) {
    if (t < L.nc) put(q, t, (T)(in[t] - bgv));
    return;
  }
  long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  if (t >= na) return;
  int i = (int)(t % L.n[0]), j = (int)((t / L.n[0]) % L.n[1]),
      k = (int)(t / ((long long)L.n[0] * L.n[1]));
  put(q, ((k + L.G) * L.s[1] + j + L.G) * L.s[0] + i + L.G, (T)(in[t] - bgv));
}

// hdiv versus IEEE division on the given operands: max |error| in ulps of the IEEE
// quotient (as a double), over n pairs
__global__ void k_hdiv_check(const double* a, const double* b, int n, double* max_ulp) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  double u = 0.0;
  if (t < n) {
    double q = a[t] / b[t];
    double h = hdiv(a[t], b[t]);
    double aq = fabs(q);
    double ulp = __longlong_as_double(__double_as_longlong(aq) + 1) - aq;
    u = q == h ? 0.0 : fabs(h - q) / ulp;
  }
  for (int o = 16; o > 0; o >>= 1) u = fmax(u, __shfl_xor_sync(0xffffffffu, u, o));
  if ((threadIdx.x & 31) == 0 && u > 0.0)
    atomicMax((unsigned long long*)max_ulp, (unsigned long long)__double_as_longlong(u));
}

// FP64 throughput probe: every thread runs kProbeChains independent chains of
// dependent fused multiply-adds (2 flops each); with a full SM of threads the FP64
// pipe, not the chain latency, sets the rate.  The result is written only when it
// takes an impossible value, so the work cannot be dropped and nothing is stored.
constexpr int kProbeChains = 8;
__global__ void __launch_bounds__(kBlock) k_dfma_probe(int iters, double* sink) {
  double a[kProbeChains];
#pragma unroll
  for (int i = 0; i < kProbeChains; ++i) a[i] = 1.0 + 1e-3 * (threadIdx.x + i);
  const double b = 0.999999999, c = 1e-9;
  for (int k = 0; k < iters; ++k)
#pragma unroll
    for (int i = 0; i < kProbeChains; ++i) a[i] = fma(a[i], b, c);
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < kProbeChains; ++i) s += a[i];
  if (s == -1.0) sink[0] = s;
}

// double-float arithmetic on the device versus FP64 on n operand pairs: the largest
// error of conversion, sum, product and quotient, each in units of its bound
// (2^-45 |a|; 2^-46 (|a| + |b|); 2^-46 |a b| + 2^-120; 2^-42 |a / b| + 2^-120)
constexpr int kDf64Checks = 8;  // entries of df_check_df64's worst[]
__global__ void k_df64_check(const double* a, const double* b, int n, double* worst) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  double w[kDf64Checks] = {};
  if (t < n) {
    const df64 x = to_df64(a[t]), y = to_df64(b[t]);
    const double A = to_double(x), B = to_double(y);
    w[0] = fabs(A - a[t]) / (0x1.0p-45 * fabs(a[t]) + 1e-300);
    w[1] = fabs(to_double(x + y) - (A + B)) / (0x1.0p-46 * (fabs(A) + fabs(B)) + 1e-300);
    w[2] = fabs(to_double(x * y) - A * B) / (0x1.0p-46 * fabs(A * B) + 0x1.0p-120);
    w[3] = fabs(to_double(x / y) - A / B) / (0x1.0p-42 * fabs(A / B) + 0x1.0p-120);
    // the unnormalised product and quotient: their values (hi + lo in FP64) within
    // the same bounds, lo within 2^-21 of hi, and as an operand of the next sum
    const df64 mu = mul_u(x, y), qu = div_u(x, y);
    const double AB = A * B, Q = A / B;
    w[4] = fabs((double)mu.hi + (double)mu.lo - AB) / (0x1.0p-46 * fabs(AB) + 0x1.0p-120);
    w[5] = fabs((double)qu.hi + (double)qu.lo - Q) / (0x1.0p-42 * fabs(Q) + 0x1.0p-120);
    if (mu.hi != 0.f) w[6] = fabs((double)mu.lo) / (0x1.0p-21 * fabs((double)mu.hi));
    if (qu.hi != 0.f) w[6] = fmax(w[6], fabs((double)qu.lo) / (0x1.0p-21 * fabs((double)qu.hi)));
    if (fabs(AB) >= 0x1.0p-100)
      w[7] = fabs(to_double(mu + x) - (AB + A)) /
             (0x1.0p-45 * (fabs(AB) + fabs(A)) + 0x1.0p-120);
  }
  for (int q = 0; q < kDf64Checks; ++q) {
    double u = w[q];
    for (int o = 16; o > 0; o >>= 1) u = fmax(u, __shfl_xor_sync(0xffffffffu, u, o));
    if ((threadIdx.x & 31) == 0 && u > 0.0)
      atomicMax((unsigned long long*)&worst[q], (unsigned long long)__double_as_longlong(u));
  }
}

}  // namespace

int launch_df64_check(const double* a, const double* b, int n, double* worst, cudaStream_t st) {
  k_df64_check<<<(n + 255) / 256, 256, 0, st>>>(a, b, n, worst);
  return 1;
}

long long launch_dfma_probe(int blocks, int iters, double* sink, cudaStream_t st) {
  k_dfma_probe<<<blocks, kBlock, 0, st>>>(iters, sink);
  return 2LL * kProbeChains * iters * (long long)kBlock * blocks;
}

int launch_hdiv_check(const double* a, const double* b, int n, double* max_ulp, cudaStream_t st) {
  k_hdiv_check<<<(n + 255) / 256, 256, 0, st>>>(a, b, n, max_ulp);
  return 1;
}

// =================================================================== work lists

// One op on one work item: maps the item's fields onto the element function.
// items inside a second sub-cycle that the Eq. 55-56 search dropped do nothing
template <class T>
__device__ __forceinline__ bool skipped(const Item<T>& it) {
  return it.br != 0u && (it.br & it.ds->xi1) != 0u;
}

// The chunks of the diffusion that write the frontier record: past the box's.  True if
// this was one.
template <class T, int OP>
__device__ __forceinline__ bool run_record(const Item<T>& it, unsigned chunk) {
  if (OP != OP_DIFFUSE || chunk < it.box_chunks) return false;
  if (!skipped(it))
    el_frontier_diff<T>(it.L, it.S, (const Arith<T>*)it.kc, it.bg.rho0, it.flags & FL_DFR, it.sub,
                        (chunk - it.box_chunks) * kBlock + threadIdx.x);
  return true;
}

template <class T, int OP, int D>
__device__ __forceinline__ void run_op(const Item<T>& it, unsigned tid) {
  if (skipped(it)) return;
  // elements of this thread: tid, or for the two-cell ops the same lane of both
  // halves of its 512-element chunk
  constexpr int NC = cells_per_thread(OP, (int)sizeof(T));
  unsigned el[NC];
  el[0] = NC == 1 ? tid : (tid / kBlock) * (NC * kBlock) + tid % kBlock;
#pragma unroll
  for (int n = 1; n < NC; ++n) el[n] = el[0] + n * kBlock;
  if (OP == OP_SOURCE)
    el_source<T, NC>(it.L, it.b, it.S, (const Arith<T>*)it.dt, it.flags & FL_WRITE_PI, it.gm1,
                     it.bg, it.g, it.again, el);
  else if (OP == OP_COMPRESS) {
    if (it.L.has_child)  // before any consumer
#pragma unroll 1
      for (int n = 0; n < NC; ++n) fr_sums(it.L, it.ds, it.level, el[n]);
    el_compress_lum<T, NC>(it.L, it.b, it.S, (const Arith<T>*)it.dt, it.gm1, it.lum,
                           it.flags & FL_SS3, it.flags & FL_LUM, it.flags & FL_EPS, it.bg, it.g,
                           el);
  }
  else if (OP == OP_DIFFUSE)  // D = 1: with the x sweep's preparation
    el_diffuse<T, NC, D>(it.L, it.b, it.S, (const Arith<T>*)it.kc, it.bg.rho0, it.flags & FL_DFR,
                         it.g, it.bg, el);
  else if (OP == OP_TPREP)
    el_tprep<T>(it.L, it.b, it.S, it.bg, it.flags & FL_EPS_ONLY, tid);
  else if (OP == OP_TFLUX)
    el_tflux<T, D>(it.L, it.b, it.S, (const Arith<T>*)it.kc, it.bg, it.sub, tid);
  else if (OP == OP_TMOM)
    el_tmom<T, D>(it.L, it.b, it.S, (const Arith<T>*)it.kc, it.bg, tid);
  else if (OP == OP_TUPDATE)
    el_tupdate<T, D, NC>(it.L, it.b, it.S, it.g, el);
  else if (OP == OP_VISC_Q)
    el_visc_q<T>(it.L, it.b, it.S, (const Arith<T>*)it.dt, it.av, it.bg, it.g, tid);
  else if (OP == OP_VISC_V)
    el_visc_v<T>(it.L, it.b, it.S, (const Arith<T>*)it.dt, it.flags & FL_WRITE_PI, it.bg, it.g, tid);
  else if (OP == OP_VREC)  // D = 1: with the next sub-cycle's first kick
    el_vrec_source<T, NC, D>(it.L, it.b, it.S, (const Arith<T>*)it.dt, it.gm1, it.bg, it.g,
                             it.again, it.flags & FL_WRITE_PI, el);
  else if (OP == OP_BC)
    el_bc<T>(it.L, it.bc, (T)it.V[0], (T)it.V[1], (T)it.V[2], tid);
  else if (OP == OP_COMMUP)
    el_commup<T>(it.L, it.F, tid);
  else if (OP == OP_COMMMEAN)
    el_commmean<T>(it.L, it.F, it.band, tid);
  else if (OP == OP_DT_LEVEL) {
    el_dt_level<T>(it.L, it.b, it.level, it.gg, it.gga, it.flags & FL_HYDRO, it.ds, it.rho0d, it.e0d,
                   it.V[0], it.V[1], it.V[2], it.bg, tid);
    if (D != kPerLevel && last_chunk(&it.ds->dt_done, it.total))
      el_dt_finalize(it.ds, it.n_levels, *it.fin, it.dt_fixed);
  } else if (OP == OP_FORCE_LEVEL) {
    el_force_level<T>(it.L, it.b, it.L.fw, it.partials, tid);
    if (D != kPerLevel && last_chunk(&it.ds->force_done, it.total))
      el_force_finalize(it.run_partials, it.npart, it.ds, it.ring, it.ring_cap, it.ring_pos);
  } else if (OP == OP_DT_FINAL) {
    el_dt_finalize(it.ds, it.n_levels, *it.fin, it.dt_fixed);
  } else if (OP == OP_FORCE_FINAL) {
    el_force_finalize(it.run_partials, it.npart, it.ds, it.ring, it.ring_cap, it.ring_pos);
  }
}

// Persistent work-list kernel: block b takes the contiguous chunks
// [b*nchunks/grid, (b+1)*nchunks/grid) of the concatenated items, stages the item of
// each chunk in shared memory (re-staging only when the item changes) and runs the
// op on the chunk's elements.  starts[i] is the first chunk of item i.
// (two-cell ops: at least 4 blocks per SM, so as many cells stay in flight as with
// one cell per thread at full occupancy)
template <class T, int OP, int D>
__global__ void __launch_bounds__(kBlock, cells_per_thread(OP, (int)sizeof(T)) == 2 ? 4 : 1)
    k_batch(const Item<T>* __restrict__ items,
                                                  const unsigned* __restrict__ starts, int nitems,
                                                  unsigned nchunks) {
  __shared__ __align__(16) unsigned char s_raw[sizeof(Item<T>)];
  const Item<T>& it = *reinterpret_cast<const Item<T>*>(s_raw);
  pdl_enter();
  unsigned c0 = (unsigned)((unsigned long long)nchunks * blockIdx.x / gridDim.x);
  unsigned c1 = (unsigned)((unsigned long long)nchunks * (blockIdx.x + 1) / gridDim.x);
  int cur = -1;
  for (unsigned ch = c0; ch < c1; ++ch) {
    int lo = cur < 0 ? 0 : cur, hi = nitems - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (starts[mid] <= ch)
        lo = mid;
      else
        hi = mid - 1;
    }
    if (lo != cur) {
      __syncthreads();
      const int4* src = reinterpret_cast<const int4*>(items + lo);
      int4* dst = reinterpret_cast<int4*>(s_raw);
      for (int w = threadIdx.x; w < (int)(sizeof(Item<T>) / 16); w += kBlock) dst[w] = src[w];
      __syncthreads();
      cur = lo;
    }
    // private copy where it scalarises (global stores cannot alias it, so the
    // fields the op uses stay in registers); ops that index the item's arrays with
    // run-time indices read it from shared memory instead
    constexpr bool kLocal =
        !(OP == OP_COMPRESS || OP == OP_BC || OP == OP_COMMUP);
    if (run_record<T, OP>(it, ch - starts[cur])) {
    } else if (kLocal) {
      const Item<T> loc = it;
      run_op<T, OP, D>(loc, (ch - starts[cur]) * kBlock + threadIdx.x);
    } else {
      run_op<T, OP, D>(it, (ch - starts[cur]) * kBlock + threadIdx.x);
    }
    __syncthreads();
  }
  pdl_exit();
}

// One work item: passed by value (kernel-parameter space), one block per chunk.
template <class T, int OP, int D>
__global__ void __launch_bounds__(kBlock) k_single(const Item<T> it) {
  pdl_enter();
  if (!run_record<T, OP>(it, blockIdx.x))
    run_op<T, OP, D>(it, blockIdx.x * kBlock + threadIdx.x);
  pdl_exit();
}

// CommMean and the ghost fill of another level in one launch: both are a few blocks, bound
// by the launch itself (nine quadrant levels 4855 launches a coarse step -> 4665, FP32 20.7 ->
// 20.0 ms, FP64 32.6 -> 31.7; 3 x 64^3 FP32 341 -> 336 us).  Where the fill is the child's,
// whose wall faces CommMean reads, it stays a launch of its own.
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_mean_with_fill(const Item<T> mean, const Item<T> fill, unsigned mean_chunks) {
  pdl_enter();
  if (blockIdx.x < mean_chunks)
    run_op<T, OP_COMMMEAN, 0>(mean, blockIdx.x * kBlock + threadIdx.x);
  else
    run_op<T, OP_BC, 0>(fill, (blockIdx.x - mean_chunks) * kBlock + threadIdx.x);
  pdl_exit();
}

// Reduction over several items (a run's levels, or those of many runs): one block per
// chunk, the item read in place.  The persistent form above, with its staged item, a
// private copy and a barrier per chunk, ran the FP64 time step of 5 x 128^3 in 413 us
// against 222.  Three blocks an SM (80 registers): with two, 275 us.
template <class T, int OP>
__global__ void __launch_bounds__(kBlock, 3) k_reduce(const Item<T>* __restrict__ items,
                                                   const unsigned* __restrict__ starts,
                                                   int nitems) {
  pdl_enter();
  int lo = 0, hi = nitems - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (starts[mid] <= blockIdx.x)
      lo = mid;
    else
      hi = mid - 1;
  }
  run_op<T, OP, 0>(items[lo], (blockIdx.x - starts[lo]) * kBlock + threadIdx.x);
  pdl_exit();
}

// Fused sweep: one block per (column, chunk) unit; the work-list form stages the item as
// k_batch does.
template <class T, int D, bool ENDS>
__global__ void __launch_bounds__(kSweepThreads, sweep_blocks((int)sizeof(T), D))
    k_sweep_single(const Item<T> it) {
  __shared__ Arith<T> s_planes[sweep_buffer((int)sizeof(T))];
  pdl_enter();
  if (skipped(it)) return;
  el_sweep<T, D, ENDS, false>(it, blockIdx.x, s_planes + threadIdx.x);
  pdl_exit();
}

template <class T, int D>
__global__ void __launch_bounds__(kSweepThreads, sweep_blocks((int)sizeof(T), D))
    k_sweep_batch(const Item<T>* __restrict__ items, const unsigned* __restrict__ starts,
                  int nitems, unsigned nchunks) {
  __shared__ Arith<T> s_planes[sweep_buffer((int)sizeof(T))];
  __shared__ __align__(16) unsigned char s_raw[sizeof(Item<T>)];
  const Item<T>& it = *reinterpret_cast<const Item<T>*>(s_raw);
  pdl_enter();
  unsigned c0 = (unsigned)((unsigned long long)nchunks * blockIdx.x / gridDim.x);
  unsigned c1 = (unsigned)((unsigned long long)nchunks * (blockIdx.x + 1) / gridDim.x);
  int cur = -1;
  for (unsigned ch = c0; ch < c1; ++ch) {
    int lo = cur < 0 ? 0 : cur, hi = nitems - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (starts[mid] <= ch)
        lo = mid;
      else
        hi = mid - 1;
    }
    if (lo != cur) {
      __syncthreads();
      const int4* src = reinterpret_cast<const int4*>(items + lo);
      int4* dst = reinterpret_cast<int4*>(s_raw);
      for (int w = threadIdx.x; w < (int)(sizeof(Item<T>) / 16); w += kSweepThreads)
        dst[w] = src[w];
      __syncthreads();
      cur = lo;
    }
    if (!skipped(it)) el_sweep<T, D, false, true>(it, ch - starts[cur], s_planes + threadIdx.x);
    __syncthreads();
  }
  pdl_exit();
}

// launch with the programmatic-stream-serialisation attribute (see pdl_enter); an
// error is left in the runtime's last-error state like that of a <<<>>> launch
template <class... P, class... A>
static void launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block,
                       cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <class T, int D>
static void launch_sweep(const Item<T>* items, const unsigned* starts, int nitems,
                         unsigned nchunks, unsigned grid, cudaStream_t st,
                         const Item<T>* host_item) {
  if constexpr (sizeof(T) == 8)
    if (nitems == 1 && host_item && host_item->b.zc < 0) {
      launch_pdl(k_sweep_single<T, D, true>, nchunks, kSweepThreads, st, *host_item);
      return;
    }
  if (nitems == 1 && host_item)
    launch_pdl(k_sweep_single<T, D, false>, nchunks, kSweepThreads, st, *host_item);
  else  // pools, whose items have chunks (Box::zc > 0)
    launch_pdl(k_sweep_batch<T, D>, grid, kSweepThreads, st, items, starts, nitems, nchunks);
}

template <class T, int OP, int D>
static void launch_one(const Item<T>* items, const unsigned* starts, int nitems, unsigned nchunks,
                       unsigned grid, cudaStream_t st, const Item<T>* host_item) {
  if (nitems == 1 && host_item)
    launch_pdl(k_single<T, OP, D>, nchunks, kBlock, st, *host_item);
  else if constexpr (is_joined_op(OP, D))
    launch_pdl(k_reduce<T, OP>, nchunks, kBlock, st, items, starts, nitems);
  else
    launch_pdl(k_batch<T, OP, D>, grid, kBlock, st, items, starts, nitems, nchunks);
}

template <class T>
int launch_batch(int op, int d, const Item<T>* items, const unsigned* starts, int nitems,
                 unsigned nchunks, unsigned grid, cudaStream_t st, const Item<T>* host_item) {
  if (nchunks == 0 || nitems == 0) return 0;
  if (grid > nchunks) grid = nchunks;
#define DFN_OP(O)                                                          \
  case O:                                                                  \
    launch_one<T, O, 0>(items, starts, nitems, nchunks, grid, st, host_item); \
    break;
#define DFN_OPD(O)                                                         \
  case O:                                                                  \
    if (d == 0) launch_one<T, O, 0>(items, starts, nitems, nchunks, grid, st, host_item); \
    if (d == 1) launch_one<T, O, 1>(items, starts, nitems, nchunks, grid, st, host_item); \
    if (d == 2) launch_one<T, O, 2>(items, starts, nitems, nchunks, grid, st, host_item); \
    break;
  switch (op) {
    DFN_OP(OP_SOURCE)
    DFN_OP(OP_COMPRESS)
    case OP_DIFFUSE:  // d = 1: with the x sweep's preparation
      if (d == 0) launch_one<T, OP_DIFFUSE, 0>(items, starts, nitems, nchunks, grid, st, host_item);
      if (d == 1) launch_one<T, OP_DIFFUSE, 1>(items, starts, nitems, nchunks, grid, st, host_item);
      break;
    DFN_OP(OP_TPREP)
    DFN_OPD(OP_TFLUX)
    DFN_OPD(OP_TMOM)
    DFN_OPD(OP_TUPDATE)
    case OP_VREC:  // d = 1: with the next sub-cycle's first kick
      if (d == 0) launch_one<T, OP_VREC, 0>(items, starts, nitems, nchunks, grid, st, host_item);
      if (d == 1) launch_one<T, OP_VREC, 1>(items, starts, nitems, nchunks, grid, st, host_item);
      break;
    DFN_OP(OP_BC)
    DFN_OP(OP_COMMUP)
    case OP_COMMMEAN:
      if (d == kMeanWithFill && host_item) {  // contexts only
        const unsigned n = (host_item[0].count + kBlock - 1) / kBlock;
        launch_pdl(k_mean_with_fill<T>, nchunks, kBlock, st, host_item[0], host_item[1], n);
      } else {
        launch_one<T, OP_COMMMEAN, 0>(items, starts, nitems, nchunks, grid, st, host_item);
      }
      break;
    case OP_DT_LEVEL:  // d = kPerLevel: contexts only
      if (d == 0) launch_one<T, OP_DT_LEVEL, 0>(items, starts, nitems, nchunks, grid, st, host_item);
      else if (host_item)
        launch_pdl(k_single<T, OP_DT_LEVEL, kPerLevel>, nchunks, kBlock, st, *host_item);
      break;
    case OP_FORCE_LEVEL:
      if (d == 0)
        launch_one<T, OP_FORCE_LEVEL, 0>(items, starts, nitems, nchunks, grid, st, host_item);
      else if (host_item)
        launch_pdl(k_single<T, OP_FORCE_LEVEL, kPerLevel>, nchunks, kBlock, st, *host_item);
      break;
    case OP_DT_FINAL:
      if (host_item) launch_pdl(k_single<T, OP_DT_FINAL, 0>, nchunks, kBlock, st, *host_item);
      break;
    case OP_FORCE_FINAL:
      if (host_item) launch_pdl(k_single<T, OP_FORCE_FINAL, 0>, nchunks, kBlock, st, *host_item);
      break;
    DFN_OP(OP_VISC_Q)
    DFN_OP(OP_VISC_V)
    case OP_SWEEP:
      if (d == 0) launch_sweep<T, 0>(items, starts, nitems, nchunks, grid, st, host_item);
      if (d == 1) launch_sweep<T, 1>(items, starts, nitems, nchunks, grid, st, host_item);
      if (d == 2) launch_sweep<T, 2>(items, starts, nitems, nchunks, grid, st, host_item);
      break;
    default:
      return 0;
  }
#undef DFN_OP
#undef DFN_OPD
  return 1;
}

// elements per chunk of each op (one chunk = one block pass)
int op_chunk_elems(int op, int esz) {
  if (op == OP_DT_LEVEL) return kBlock * kDtCells;
  return op == OP_FORCE_LEVEL ? kBlock * kForceCells : kBlock * cells_per_thread(op, esz);
}

// index-space size of one item of an op (host side, from the item's views)
unsigned op_count(int op, int d, const LevelView& L, const LevelView& F, const Box& b,
                  const int* bc) {
  long long n = 0;
  switch (op) {
    case OP_SOURCE: case OP_COMPRESS: case OP_DIFFUSE: case OP_TPREP: case OP_TFLUX:
    case OP_TMOM: case OP_TUPDATE: case OP_VREC: case OP_VISC_Q: case OP_VISC_V:  // is_box_op
      if (b.tile == 0) {
        n = b.count();
      } else {
        long long nt = 1;
        for (int a = 0; a < 3; ++a) {
          int e = tile_extent(b.tile, a);
          nt *= (b.hi[a] - b.lo[a] + e - 1) / e;
        }
        n = nt * 256;
      }
      break;
    case OP_SWEEP:
      n = (long long)sweep_units(b, d) * kBlock;  // one chunk per (column, chunk) unit
      break;
    case OP_BC: n = bc_elements(L, bc); break;
    case OP_COMMUP:  // one chunk per tile of the ghost hosts' shell
      n = cu_chunks(F.n, F.G) * kBlock;
      break;
    case OP_COMMMEAN: n = (long long)(F.n[0] >> 1) * (F.n[1] >> 1) * (F.n[2] >> 1); break;
    case OP_DT_LEVEL: case OP_FORCE_LEVEL: n = (long long)L.n[0] * L.n[1] * L.n[2]; break;
    default: n = 1; break;
  }
  // the compression kernel also sums the child's CommFlux record (fr_sums): enough
  // threads for it whatever the box (elements beyond the box decode to nothing)
  if (op == OP_COMPRESS && L.has_child && n < 18LL * L.cacc_slots) n = 18LL * L.cacc_slots;
  return (unsigned)n;
}

int force_partials_per_level(const LevelView& L) {
  long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  return (int)((na + kBlock * kForceCells - 1) / (kBlock * kForceCells));
}

int launch_force_weights(const LevelView& L, const Phys& P, cudaStream_t st) {
  k_force_weights<<<grid_for((long long)L.n[0] * L.n[1] * L.n[2]), kBlock, 0, st>>>(
      L, P.GM, P.eps, P.mult, L.fw);
  return 1;
}

template <class T>
int launch_init_uniform(const LevelView& L, const Phys& P, cudaStream_t st) {
  k_init_uniform<T><<<grid_for(L.nc), kBlock, 0, st>>>(L, (T)P.rho0, (T)P.e0, (T)P.V[0],
                                                        (T)P.V[1], (T)P.V[2]);
  return 1;
}

template <class T>
int launch_static_fields(const LevelView& L, const Phys& P, double lum_sigma, double* wsum,
                         double* partials, cudaStream_t st) {
  int v[3], ok = 1;
  for (int d = 0; d < 3; ++d) {
    double o = -L.lo[d] / L.dx[d];
    v[d] = (int)floor(o + 0.5);
    // a vertex on a mirror plane has four of its eight cells in the ghost layer
    if (fabs(o - v[d]) > 1e-9 || v[d] < (L.mir >> d & 1 ? 0 : 1) || v[d] > L.n[d] - 1) ok = 0;
  }
  k_static<T><<<grid_for(L.nc), kBlock, 0, st>>>(L, P.GM, P.eps, lum_sigma, ok, v[0], v[1], v[2]);
  if (lum_sigma <= 0.0) return 1;
  long long na = (long long)L.n[0] * L.n[1] * L.n[2];
  k_lum_partials<T><<<grid_for(na), kBlock, 0, st>>>(L, partials);
  k_sum_partials<<<1, kBlock, 0, st>>>(partials, (int)grid_for(na), wsum);
  return 3;
}

template <class T>
int launch_normalise_lum(const LevelView& L, const double* wsum, double mult, cudaStream_t st) {
  k_normalise_lum<T><<<grid_for(L.nc), kBlock, 0, st>>>(L, wsum, mult);
  return 1;
}

template <class T>
int launch_pack_active(const LevelView& L, int field, double* out, int full, double bgv,
                       cudaStream_t st) {
  long long n = full ? L.nc : (long long)L.n[0] * L.n[1] * L.n[2];
  k_pack<T><<<grid_for(n), kBlock, 0, st>>>(L, field, out, full, bgv);
  return 1;
}

template <class T>
int launch_unpack_active(const LevelView& L, int field, const double* in, int full, double bgv,
                         cudaStream_t st) {
  long long n = full ? L.nc : (long long)L.n[0] * L.n[1] * L.n[2];
  k_unpack<T><<<grid_for(n), kBlock, 0, st>>>(L, field, in, full, bgv);
  return 1;
}

#define DFN_INSTANTIATE(T)                                                                     \
  template int launch_batch<T>(int, int, const Item<T>*, const unsigned*, int, unsigned,       \
                               unsigned, cudaStream_t, const Item<T>*);                        \
  template int launch_init_uniform<T>(const LevelView&, const Phys&, cudaStream_t);            \
  template int launch_static_fields<T>(const LevelView&, const Phys&, double, double*,         \
                                       double*, cudaStream_t);                                 \
  template int launch_normalise_lum<T>(const LevelView&, const double*, double, cudaStream_t); \
  template int launch_pack_active<T>(const LevelView&, int, double*, int, double, cudaStream_t); \
  template int launch_unpack_active<T>(const LevelView&, int, const double*, int, double,      \
                                       cudaStream_t);

DFN_INSTANTIATE(double)
DFN_INSTANTIATE(float)

}  // namespace dfn
