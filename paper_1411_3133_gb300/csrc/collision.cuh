// Arithmetic of the lattice Boltzmann update in generalized metrics (Sec. II of
// the paper): moments, equilibrium, non-equilibrium stress, forcing term, BGK.
// Pure functions of one node's values, without memory access.
#pragma once

#include <type_traits>

#include "lattice.cuh"

namespace lbgm {

// KELT: the theta-resolved double-curved channel -- the ellipsoidal metric
// of each theta node (full Delta^ij, body force with r and phi components),
// the frozen channel's Christoffel symbols, one geometry row per node.
enum MetricKind { KFLAT = 0, KCYL = 1, KELL = 2, KELT = 3 };

// ---------------------------------------------------------------------------
// compile-time loops
// ---------------------------------------------------------------------------
template <int I, int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

template <int P>
struct Pair {
  static constexpr int x = PAIRS[P].x, y = PAIRS[P].y, z = PAIRS[P].z;
  static constexpr double w = PAIRS[P].w;
  static constexpr int s = (x != 0 ? (x < 0 ? -x : x) : (y != 0 ? (y < 0 ? -y : y) : (z < 0 ? -z : z)));
};

template <int L>
struct WeightOf {
  static constexpr double w = L == 0 ? W_REST : PAIRS[(L - 1) / 2].w;
};

// ---------------------------------------------------------------------------
// arithmetic types
// ---------------------------------------------------------------------------
// The update is written once for an arithmetic type V, float or double. Every
// multiply-add is an explicit fmav and the library is compiled with -fmad=false, so the compiler
// fuses no other product into an add: every kernel that inlines these
// functions rounds alike.
__device__ __forceinline__ float fmav(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmav(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rcpv(float a) { return 1.0f / a; }
__device__ __forceinline__ double rcpv(double a) { return 1.0 / a; }
__device__ __forceinline__ bool finite_v(float a) { return fabsf(a) < 1e30f; }
__device__ __forceinline__ bool finite_v(double a) { return fabs(a) < 1e300; }

// acc + C x, compile-time integer C
template <int C, class V>
__device__ __forceinline__ V mac(const V& acc, const V& x) {
  if constexpr (C == 0) return acc;
  else if constexpr (C == 1) return acc + x;
  else if constexpr (C == -1) return acc - x;
  else return fmav(V(double(C)), x, acc);
}
// C x, compile-time integer C != 0
template <int C, class V>
__device__ __forceinline__ V mulc(const V& x) {
  static_assert(C != 0, "mulc by zero");
  if constexpr (C == 1) return x;
  else return V(double(C)) * x;
}
// cx ax + cy ay + cz az; the first non-zero component of every pair's
// representative velocity is positive
template <int CX, int CY, int CZ, class V>
__device__ __forceinline__ V dot3(const V& ax, const V& ay, const V& az) {
  if constexpr (CX != 0) return mac<CZ>(mac<CY>(mulc<CX>(ax), ay), az);
  else if constexpr (CY != 0) return mac<CZ>(mulc<CY>(ay), az);
  else return mulc<CZ>(az);
}

// ---------------------------------------------------------------------------
// moments and collision
// ---------------------------------------------------------------------------
template <typename V>
struct Moments {
  V rho, jx, jy, jz;
  V sxx, syy, szz, sxy, sxz, syz;  // sum_l c^i c^j f_l
};

// Moments pair by pair (the observables, whose FP64 outputs keep their bits).
template <typename V>
__device__ __forceinline__ Moments<V> moments(const V (&f)[Q]) {
  Moments<V> m;
  const V z = V(0.0);
  m.rho = f[0];
  m.jx = m.jy = m.jz = z;
  m.sxx = m.syy = m.szz = m.sxy = m.sxz = m.syz = z;
  static_for<0, NPAIR>([&](auto P_) {
    constexpr int P = decltype(P_)::value;
    using C = Pair<P>;
    const V s = f[2 * P + 1] + f[2 * P + 2];
    const V df = f[2 * P + 1] - f[2 * P + 2];
    m.rho = m.rho + s;
    m.jx = mac<C::x>(m.jx, df);
    m.jy = mac<C::y>(m.jy, df);
    m.jz = mac<C::z>(m.jz, df);
    m.sxx = mac<C::x * C::x>(m.sxx, s);
    m.syy = mac<C::y * C::y>(m.syy, s);
    m.szz = mac<C::z * C::z>(m.szz, s);
    m.sxy = mac<C::x * C::y>(m.sxy, s);
    m.sxz = mac<C::x * C::z>(m.sxz, s);
    m.syz = mac<C::y * C::z>(m.syz, s);
  });
  return m;
}

// The 41 populations (or stored deviations) of a node as moments_shells and
// collide_shells see them: get<L> reads one, put<L> takes its post-collision
// value, each L once and after its get. PopArray holds them in an array.
template <typename V>
struct PopArray {
  V (&f)[Q];
  template <int L>
  __device__ __forceinline__ V get() const { return f[L]; }
  template <int L>
  __device__ __forceinline__ void put(const V& v) const { f[L] = v; }
};

// acc + (C w) x of a shell: with W the shell's weight is part of the
// coefficient (2-byte storage, whose populations are deviations over their
// weight), else the coefficient is C alone.
template <bool W, int C, int P, class V>
__device__ __forceinline__ V acc_shell(const V& acc, const V& x) {
  if constexpr (W) return fmav(V(double(C) * Pair<P>::w), x, acc);
  else return mac<C>(acc, x);
}

// Sums over the four pairs P .. P + 3 of a (1, +-1, +-1)-type shell of
// x = (x0, x1, x2, x3): a 4-point Hadamard transform, so that the shell's
// total and its xy, xz and yz signed sums cost 8 additions.
template <class V>
struct Had4 {
  V t, xy, xz, yz;
  __device__ __forceinline__ Had4(const V& a, const V& b, const V& c, const V& d) {
    const V p = a + b, q = c + d, r = a - b, s = c - d;
    t = p + q;
    xy = p - q;
    xz = r + s;
    yz = r - s;
  }
};

// The moments of the step, shell by shell: pair sums and differences of a
// shell are first combined (4-point Hadamard for the (1,1,1)-type shells, sum
// and difference for the faces), then accumulated once per shell -- 127
// additions and multiply-adds where pair by pair takes 174. With W the
// populations are stored deviations g, f_l = w_l g_l + rho_l, and m0 holds the
// streamed references' moments; without it f are the populations and m0 is
// not read.
template <bool W, typename V, class Pop>
__device__ __forceinline__ Moments<V> moments_shells(const Pop& f, const Moments<V>& m0) {
  Moments<V> m;
#define LB_S(P) (f.template get<2 * (P) + 1>() + f.template get<2 * (P) + 2>())
#define LB_D(P) (f.template get<2 * (P) + 1>() - f.template get<2 * (P) + 2>())
  // |c| = 1 along an axis
  const V s0 = LB_S(0), s1 = LB_S(1), s2 = LB_S(2);
  if constexpr (W) {
    m = m0;
    m.rho = fmav(V(W_REST), f.template get<0>(), m.rho);
    m.sxx = acc_shell<W, 1, 0>(m.sxx, s0);
    m.syy = acc_shell<W, 1, 0>(m.syy, s1);
    m.szz = acc_shell<W, 1, 0>(m.szz, s2);
    m.jx = acc_shell<W, 1, 0>(m.jx, LB_D(0));
    m.jy = acc_shell<W, 1, 0>(m.jy, LB_D(1));
    m.jz = acc_shell<W, 1, 0>(m.jz, LB_D(2));
  } else {
    m.rho = f.template get<0>();
    m.sxx = s0;
    m.syy = s1;
    m.szz = s2;
    m.jx = LB_D(0);
    m.jy = LB_D(1);
    m.jz = LB_D(2);
  }
  m.rho = acc_shell<W, 1, 0>(m.rho, s0 + s1 + s2);
  // (+-1, +-1, 0) faces
  {
    const V axy = LB_S(3), bxy = LB_S(4), axz = LB_S(5), bxz = LB_S(6), ayz = LB_S(7), byz = LB_S(8);
    const V pxy = axy + bxy, pxz = axz + bxz, pyz = ayz + byz;
    m.rho = acc_shell<W, 1, 3>(m.rho, pxy + pxz + pyz);
    m.sxx = acc_shell<W, 1, 3>(m.sxx, pxy + pxz);
    m.syy = acc_shell<W, 1, 3>(m.syy, pxy + pyz);
    m.szz = acc_shell<W, 1, 3>(m.szz, pxz + pyz);
    if constexpr (W) {
      m.sxy = acc_shell<W, 1, 3>(m.sxy, axy - bxy);
      m.sxz = acc_shell<W, 1, 3>(m.sxz, axz - bxz);
      m.syz = acc_shell<W, 1, 3>(m.syz, ayz - byz);
    } else {
      m.sxy = axy - bxy;
      m.sxz = axz - bxz;
      m.syz = ayz - byz;
    }
    const V dxy = LB_D(3), exy = LB_D(4), dxz = LB_D(5), exz = LB_D(6), dyz = LB_D(7), eyz = LB_D(8);
    m.jx = acc_shell<W, 1, 3>(m.jx, (dxy + exy) + (dxz + exz));
    m.jy = acc_shell<W, 1, 3>(m.jy, (dxy - exy) + (dyz + eyz));
    m.jz = acc_shell<W, 1, 3>(m.jz, (dxz - exz) + (dyz - eyz));
  }
  // 3 along an axis
  {
    const V t0 = LB_S(13), t1 = LB_S(14), t2 = LB_S(15);
    m.rho = acc_shell<W, 1, 13>(m.rho, t0 + t1 + t2);
    m.sxx = acc_shell<W, 9, 13>(m.sxx, t0);
    m.syy = acc_shell<W, 9, 13>(m.syy, t1);
    m.szz = acc_shell<W, 9, 13>(m.szz, t2);
    m.jx = acc_shell<W, 3, 13>(m.jx, LB_D(13));
    m.jy = acc_shell<W, 3, 13>(m.jy, LB_D(14));
    m.jz = acc_shell<W, 3, 13>(m.jz, LB_D(15));
  }
  // (+-1, +-1, +-1) and (+-3, +-3, +-3)
  const Had4<V> b1(LB_S(9), LB_S(10), LB_S(11), LB_S(12)), b3(LB_S(16), LB_S(17), LB_S(18), LB_S(19));
  m.rho = acc_shell<W, 1, 16>(acc_shell<W, 1, 9>(m.rho, b1.t), b3.t);
  V T;
  if constexpr (W) T = acc_shell<W, 9, 16>(V(Pair<9>::w) * b1.t, b3.t);
  else T = mac<9>(b1.t, b3.t);
  m.sxx = m.sxx + T;
  m.syy = m.syy + T;
  m.szz = m.szz + T;
  m.sxy = acc_shell<W, 9, 16>(acc_shell<W, 1, 9>(m.sxy, b1.xy), b3.xy);
  m.sxz = acc_shell<W, 9, 16>(acc_shell<W, 1, 9>(m.sxz, b1.xz), b3.xz);
  m.syz = acc_shell<W, 9, 16>(acc_shell<W, 1, 9>(m.syz, b1.yz), b3.yz);
  const Had4<V> e1(LB_D(9), LB_D(10), LB_D(11), LB_D(12)), e3(LB_D(16), LB_D(17), LB_D(18), LB_D(19));
  m.jx = acc_shell<W, 3, 16>(acc_shell<W, 1, 9>(m.jx, e1.t), e3.t);
  m.jy = acc_shell<W, 3, 16>(acc_shell<W, 1, 9>(m.jy, e1.xy), e3.xy);
  m.jz = acc_shell<W, 3, 16>(acc_shell<W, 1, 9>(m.jz, e1.xz), e3.xz);
#undef LB_S
#undef LB_D
  return m;
}

template <typename V>
__device__ __forceinline__ Moments<V> step_moments(V (&f)[Q]) {
  return moments_shells<false, V>(PopArray<V>{f}, Moments<V>{});
}

// Geometry of one node, read for the metric kind K. The Christoffel symbols
// are kept with a minus sign (F^i = F_ext^i - Gamma^i_jk c^j c^k).
template <typename V, int K>
struct NodeGeo {
  V dtt = V(0.0), dpp = V(0.0);
  V n_rtt = V(0.0), n_rpp = V(0.0), n_trt = V(0.0), n_prp = V(0.0), n_ttp = V(0.0), n_ptt = V(0.0);
  V fth = V(1.0);
};

// The theta-resolved ellipsoid adds the off-diagonal and r r components of
// Delta and the r and x3 components of the body force direction.
template <typename V>
struct NodeGeo<V, KELT> : NodeGeo<V, KELL> {
  V drr = V(0.0), drt = V(0.0), drp = V(0.0), dtp = V(0.0);
  V fr = V(0.0), fp = V(0.0);
};

// Per-node coefficients of the equilibrium and of the forcing term.
//   f^eq(+-c) = w (E +- O), forcing(+-c) = w (Fe +- Fo), with
//   E  = e0 + eA c.Delta.c + eB (u.c)^2
//   O  = u.c (oA + eB c.Delta.c + oC (u.c)^2) - Vs.c
//   Fe = fA (u.c)(F.c) - fB (u.F)
//   Fo = (F.c)(t0 + (c.A2s.c) / (2 cs^2)) - F.(A2s c)
// where, from Sec. II,
//   a2 = rho (cs^2 Delta + u u),  tr a2 = rho (cs^2 tr Delta + |u|^2),
//   V^k = a3^{iik} = rho (cs^2 (tr Delta u^k + 2 (Delta u)^k) + |u|^2 u^k),
//   A2 = a2 + kappa Pi,  Pi = sum c c f - rho (cs^2 g^-1 + u u)
//   (sum c c f^eq = rho cs^2 g^ij + rho u^i u^j by the lattice's 4th-moment
//   identity), A2s = A2 / cs^4, F^i = F_ext^i - Gamma^i_jk c^j c^k.
// Stored with signs chosen so that every term is one multiply-add:
// nv = -Vs, nfB = -fB, na = -A2s, and eAt = eA Delta^thth etc.
template <typename V>
struct Coef {
  V ux, uy, uz;
  V rho, uu, trD;           // density, |u|^2, trace of Delta
  V e0, eB, oA, oC;
  V eAt, eAp, eBt, eBp;     // eA dtt, eA dpp, eB dtt, eB dpp
  V nvx, nvy, nvz;
  V fA, nfB, t0;
  V naxx, nayy, nazz, naxy, naxz, nayz;
  V fext_t;
  // theta-resolved ellipsoid: eA and eB times Delta^rr, Delta^{r theta},
  // Delta^{r 3}, Delta^{theta 3}; the body force's r and x3 components
  V eArr, eArt, eArp, eAtp, eBrr, eBrt, eBrp, eBtp;
  V fext_r, fext_p;
};

template <typename V, int K>
__device__ __forceinline__ Coef<V> coefficients(const Moments<V>& m, const NodeGeo<V, K>& g, const V& kappa,
                                                const V& G) {
  const V cs2 = V(CS2);
  const V inv_cs2 = V(1.0 / CS2);
  const V inv_cs4 = V(1.0 / (CS2 * CS2));
  Coef<V> c;
  const V rho = m.rho;
  const V irho = rcpv(rho);
  const V ux = m.jx * irho, uy = m.jy * irho, uz = m.jz * irho;
  c.ux = ux;
  c.uy = uy;
  c.uz = uz;
  const V uu = fmav(uz, uz, fmav(uy, uy, ux * ux));
  V trD = K == KFLAT ? V(0.0) : g.dtt;
  if constexpr (K == KELL || K == KELT) trD = trD + g.dpp;
  if constexpr (K == KELT) trD = trD + g.drr;
  c.rho = rho;
  c.uu = uu;
  c.trD = trD;
  const V tra2 = rho * fmav(cs2, trD, uu);
  c.e0 = fmav(V(-0.5 / CS2), tra2, rho);
  const V eA = rho * V(0.5 / CS2);
  c.eB = rho * V(0.5 / (CS2 * CS2));
  c.eAt = eA * g.dtt;
  c.eAp = eA * g.dpp;
  c.eBt = c.eB * g.dtt;
  c.eBp = c.eB * g.dpp;
  c.oA = rho * inv_cs2;
  c.oC = rho * V(1.0 / (6.0 * CS2 * CS2 * CS2));
  // -V / (2 cs^4), Delta diagonal (dtt on theta, dpp on x3)
  const V nvs = V(-0.5 / (CS2 * CS2)) * rho;
  const V trDc = cs2 * trD;
  if constexpr (K == KELT) {
    // full Delta: V^k / rho = cs^2 (tr Delta u^k + 2 (Delta u)^k) + |u|^2 u^k
    const V c2 = V(2.0 * CS2);
    const V dux = fmav(g.drr, ux, fmav(g.drt, uy, g.drp * uz));
    const V duy = fmav(g.drt, ux, fmav(g.dtt, uy, g.dtp * uz));
    const V duz = fmav(g.drp, ux, fmav(g.dtp, uy, g.dpp * uz));
    c.nvx = nvs * fmav(c2, dux, fmav(trDc, ux, uu * ux));
    c.nvy = nvs * fmav(c2, duy, fmav(trDc, uy, uu * uy));
    c.nvz = nvs * fmav(c2, duz, fmav(trDc, uz, uu * uz));
    c.eArr = eA * g.drr;
    c.eArt = eA * g.drt;
    c.eArp = eA * g.drp;
    c.eAtp = eA * g.dtp;
    c.eBrr = c.eB * g.drr;
    c.eBrt = c.eB * g.drt;
    c.eBrp = c.eB * g.drp;
    c.eBtp = c.eB * g.dtp;
  } else {
    c.nvx = nvs * (fmav(trDc, ux, uu * ux));
    c.nvy = nvs * (fmav(fmav(V(2.0 * CS2), g.dtt, trDc), uy, uu * uy));
    c.nvz = nvs * (fmav(fmav(V(2.0 * CS2), g.dpp, trDc), uz, uu * uz));
  }
  c.fA = rho * inv_cs4;
  c.nfB = rho * V(-1.0 / CS2);
  // -A2s = -A2 / cs^4, A2 = (1 - kappa) rho (cs^2 Delta + u u) + kappa (S - rho cs^2 delta)
  const V nic4 = V(-1.0 / (CS2 * CS2));
  const V rc = rho * cs2;
  const V rk = nic4 * rho * (V(1.0) - kappa);
  const V kn = nic4 * kappa;
  if constexpr (K == KELT) {
    c.naxx = fmav(rk, fmav(cs2, g.drr, ux * ux), kn * (m.sxx - rc));
    c.naxy = fmav(rk, fmav(cs2, g.drt, ux * uy), kn * m.sxy);
    c.naxz = fmav(rk, fmav(cs2, g.drp, ux * uz), kn * m.sxz);
    c.nayz = fmav(rk, fmav(cs2, g.dtp, uy * uz), kn * m.syz);
  } else {
    c.naxx = fmav(rk, ux * ux, kn * (m.sxx - rc));
    c.naxy = fmav(rk, ux * uy, kn * m.sxy);
    c.naxz = fmav(rk, ux * uz, kn * m.sxz);
    c.nayz = fmav(rk, uy * uz, kn * m.syz);
  }
  V yy = uy * uy, zz = uz * uz;
  if constexpr (K != KFLAT) yy = fmav(cs2, g.dtt, yy);
  if constexpr (K == KELL || K == KELT) zz = fmav(cs2, g.dpp, zz);
  c.nayy = fmav(rk, yy, kn * (m.syy - rc));
  c.nazz = fmav(rk, zz, kn * (m.szz - rc));
  c.t0 = fmav(V(0.5), c.naxx + c.nayy + c.nazz, rho * inv_cs2);
  c.fext_t = G * g.fth;
  if constexpr (K == KELT) {
    c.fext_r = G * g.fr;
    c.fext_p = G * g.fp;
  }
  return c;
}

// The post-collision values of a pair (c, -c) from the even and odd parts
// a = omega E + Fe and B = omega O + Fo of the pair:
//   f* = (1 - omega) f + w (a +- B)
// or, with DEV, for the stored deviations g = (f - r) / w of 2-byte storage
//   g* = (1 - omega) g + a +- B
// (a and B then include the stream table's t, see collide_shells).
template <int P, bool DEV, typename V, class Pop>
__device__ __forceinline__ void update_pair(const Pop& f, const V& om1, const V& a, const V& B) {
  const V fp = f.template get<2 * P + 1>(), fm = f.template get<2 * P + 2>();
  if constexpr (DEV) {
    f.template put<2 * P + 1>(fmav(om1, fp, a + B));
    f.template put<2 * P + 2>(fmav(om1, fm, a - B));
  } else {
    const V w = V(Pair<P>::w);
    const V Bw = B * w;
    f.template put<2 * P + 1>(fmav(om1, fp, fmav(a, w, Bw)));
    f.template put<2 * P + 2>(fmav(om1, fm, fmav(a, w, -Bw)));
  }
}

// The two pairs P, P + 1 of a face shell, c = s_i e_i +- s_j e_j: even part
// base +- x, odd part bi s_i + bj s_j.
template <int P, bool DEV, typename V, class Pop>
__device__ __forceinline__ void update_face(const Pop& f, const V& om1, const V& base, const V& x, const V& bi,
                                            const V& bj) {
  update_pair<P, DEV>(f, om1, base + x, bi + bj);
  update_pair<P + 1, DEV>(f, om1, base - x, bi - bj);
}

// The four pairs P .. P + 3 of a (1, +-1, +-1)-type shell: even part
// base + xy s_x s_y + xz s_x s_z + yz s_y s_z, odd part bx s_x + by s_y + bz s_z
// + d s_x s_y s_z, each a 4-point Hadamard transform.
template <int P, bool DEV, typename V, class Pop>
__device__ __forceinline__ void update_body(const Pop& f, const V& om1, const V& base, const V& xy, const V& xz,
                                            const V& yz, const V& bx, const V& by, const V& bz, const V& d) {
  const V ep = base + xy, em = base - xy, eq = xz + yz, er = xz - yz;
  const V op = bx + by, om = bx - by, oq = bz + d, orr = bz - d;
  update_pair<P, DEV>(f, om1, ep + eq, op + oq);
  update_pair<P + 1, DEV>(f, om1, ep - eq, op - oq);
  update_pair<P + 2, DEV>(f, om1, em + er, om + orr);
  update_pair<P + 3, DEV>(f, om1, em - er, om - orr);
}

// Weight of the rest population in the step. In FP32 the nearest floats of the
// 41 weights sum to 1 + 2.4e-8, which the collision adds to the mass of every
// node at every step (omega rho 2.4e-8: the largest part of the FP32 error
// after some tens of steps); the float nearest to 1 minus the sum of the
// other weights' floats leaves 6e-9.
template <typename V>
constexpr double rest_weight() {
  if constexpr (std::is_same<V, float>::value) {
    double others = 0.0;
    for (int P = 0; P < NPAIR; ++P) others += 2.0 * double(float(PAIRS[P].w));
    return double(float(1.0 - others));
  }
  return W_REST;
}
template <typename V>
constexpr double REST_WEIGHT = rest_weight<V>();

// No stream table: populations, not deviations.
struct NoTab {};

// Starting values of a shell's coefficients: with 2-byte storage the stream
// table's t, transformed to the shells' coefficient space (k_stream_table),
// else nothing. E and O of slot P live in entry 3 + P / 2.
template <typename V>
struct TabEntry {
  V x, y, z, w;
};
template <bool DEV, typename V>
struct Start {
  TabEntry<V> t;
  template <int P>
  __device__ __forceinline__ V e(const V& x) const {
    if constexpr (DEV) return x + (P % 2 == 0 ? t.x : t.z);
    else return x;
  }
  template <int P>
  __device__ __forceinline__ V o(const V& x) const {
    if constexpr (DEV) return x + (P % 2 == 0 ? t.y : t.w);
    else return x;
  }
};

// BGK collision with the forcing term, in place (Eq. LB):
//   f* = (1 - omega) f + w (omega E + Fe) +- w (omega O + Fo)
// evaluated shell by shell. omega E + Fe is an even polynomial in c of degree
// 4 and omega O + Fo an odd one of degree 5 whose coefficients do not depend
// on c:
//   a(c) = a0 + c.M.c + (s.c) g3(c),
//     a0 = omega e0 - fB u.f,  s = fA u,  f the body force,
//     M_ij = omega (eA Delta_ij + eB u_i u_j) + fA (u_i f_j + u_j f_i) / 2
//            + sum_k (-fB u_k) n^k_ij,        n^k_ij = -h Gamma^k_ij,
//     g3(c) = c_k n^k_ij c_i c_j = gam1 cx cy^2 + gam2 cx cz^2 + gam3 cy^2 cz;
//   B(c) = L.c + (c.Q.c)(u.c) + hf.c (c.N.c) + q(c).(N c) + g3(c) (t0 + h c.N.c),
//     L = omega (oA u - Vs) + N f + t0 f,  Q_ij = omega (eB Delta_ij + oC u_i u_j),
//     N = -A2s,  h = -1 / (2 cs^2),  hf = h f,  q^k(c) = n^k_ij c_i c_j.
// On a shell c = m s, s_i in {-1, 0, 1}, every power of s_i is 1 or s_i: a face
// shell needs 2 even and 2 odd numbers, a body shell 4 and 4, an axis 1 and
// 1 per pair, and the pairs are their sums and differences. Against
// evaluating both polynomials pair by pair, moments, coefficients and
// collision take 521 instead of 842 FP operations per update on the cylinder
// (ellipsoid 579 / 968, theta-resolved 666 / 1136). The FP64 step, bound by
// its FP64 units, went from 107.6 to 75.6 us on a 64 x 4 x 256 cylinder; FP16
// storage, bound by instruction issue, from 83.2 to 74.6 us on 24 of them
// (FP32 90.3 to 87.2), the theta-resolved ellipsoid (2 x 65 x 64 x 128, FP32)
// from 101 to 86.8.
//
// DEV (2-byte storage): f holds the stored deviations g = (f - r) / w and
//   g* = (1 - omega) g + (a + te) +- (B + to)
// with te, to the even and odd parts of t = ((1 - omega) rho - r) / w from the
// stream table `tab`, in coefficient space: they are added to the shells'
// coefficients instead of to every pair.
template <typename V, int K, class Pop, class Tab = NoTab>
__device__ __forceinline__ void collide_shells(const Pop& f, const Coef<V>& k, const NodeGeo<V, K>& g, const V& omega,
                                               const Tab& tab, const V& t_rest) {
  constexpr bool DEV = !std::is_same<Tab, NoTab>::value;
  constexpr bool curv = K != KFLAT;
  constexpr bool ell = K == KELL || K == KELT;
  constexpr bool gen = K == KELT;
  const V om1 = V(1.0) - omega;
  const V ux = k.ux, uy = k.uy, uz = k.uz, ft = k.fext_t;
  // each table entry is requested one group ahead of its use, so a global
  // load overlaps the arithmetic before it
  using St = Start<DEV, V>;
  auto entry = [&](int j) {
    St s;
    if constexpr (DEV) s.t = tab.at(3 + j);
    return s;
  };
  St T0 = entry(0), T1 = entry(1);

  // equilibrium: omega rho and its multiples
  const V rw = omega * k.rho;
  const V rwc = rw * V(1.0 / CS2);                  // omega oA
  const V weB = rw * V(0.5 / (CS2 * CS2));
  const V a_eq = fmav(V(-0.5) * rwc, fmav(V(CS2), k.trD, k.uu), rw);
  V a0 = fmav(k.nfB * uy, ft, a_eq);
  const V wx = weB * ux, wy = weB * uy, wz = weB * uz;
  const V c3 = V(1.0 / (3.0 * CS2));
  V Mxx = wx * ux, Myy = wy * uy, Mzz = wz * uz;
  V Mxy = (wx + wx) * uy, Mxz = (wx + wx) * uz, Myz = (wy + wy) * uz;   // doubled: 2 M_ij
  V Qxx = c3 * Mxx, Qyy = c3 * Myy, Qzz = c3 * Mzz;
  V Qxy = c3 * Mxy, Qxz = c3 * Mxz, Qyz = c3 * Myz;                     // doubled
  if constexpr (curv) {
    const V dt = weB * g.dtt;
    Qyy = Qyy + dt;
    Myy = fmav(V(CS2), dt, Myy);
  }
  if constexpr (ell) {
    const V dp = weB * g.dpp;
    Qzz = Qzz + dp;
    Mzz = fmav(V(CS2), dp, Mzz);
  }
  if constexpr (gen) {
    const V w2 = weB + weB;
    const V dr = weB * g.drr, drt = w2 * g.drt, drp = w2 * g.drp, dtp = w2 * g.dtp;
    Qxx = Qxx + dr;
    Qxy = Qxy + drt;
    Qxz = Qxz + drp;
    Qyz = Qyz + dtp;
    Mxx = fmav(V(CS2), dr, Mxx);
    Mxy = fmav(V(CS2), drt, Mxy);
    Mxz = fmav(V(CS2), drp, Mxz);
    Myz = fmav(V(CS2), dtp, Myz);
  }
  // L: omega (oA u - Vs) = omega rho u (1 / cs^2 - (cs^2 tr Delta + |u|^2) / (2 cs^4)) - omega oA Delta u
  const V lb = fmav(-weB, fmav(V(CS2), k.trD, k.uu), rwc);
  V Lx = lb * ux, Ly = lb * uy, Lz = lb * uz;
  if constexpr (gen) {
    Lx = fmav(-rwc, fmav(g.drr, ux, fmav(g.drt, uy, g.drp * uz)), Lx);
    Ly = fmav(-rwc, fmav(g.drt, ux, fmav(g.dtt, uy, g.dtp * uz)), Ly);
    Lz = fmav(-rwc, fmav(g.drp, ux, fmav(g.dtp, uy, g.dpp * uz)), Lz);
  } else {
    if constexpr (curv) Ly = fmav(-rwc, g.dtt, lb) * uy;
    if constexpr (ell) Lz = fmav(-rwc, g.dpp, lb) * uz;
  }
  // body force
  const V h = V(-0.5 / CS2);
  const V sx = k.fA * ux, sy = k.fA * uy, sz = k.fA * uz;
  V hx = V(0.0), hz = V(0.0);
  const V hy = h * ft;
  Mxy = fmav(sx, ft, Mxy);
  Myy = fmav(sy, ft, Myy);
  Myz = fmav(sz, ft, Myz);
  Lx = fmav(k.naxy, ft, Lx);
  Ly = fmav(k.nayy + k.t0, ft, Ly);
  Lz = fmav(k.nayz, ft, Lz);
  if constexpr (gen) {
    const V fr = k.fext_r, fp = k.fext_p;
    hx = h * fr;
    hz = h * fp;
    a0 = fmav(k.nfB, fmav(ux, fr, uz * fp), a0);
    Mxx = fmav(sx, fr, Mxx);
    Mzz = fmav(sz, fp, Mzz);
    Mxy = fmav(sy, fr, Mxy);
    Mxz = fmav(sx, fp, fmav(sz, fr, Mxz));
    Myz = fmav(sy, fp, Myz);
    Lx = fmav(k.naxx + k.t0, fr, fmav(k.naxz, fp, Lx));
    Ly = fmav(k.naxy, fr, fmav(k.nayz, fp, Ly));
    Lz = fmav(k.nazz + k.t0, fp, fmav(k.naxz, fr, Lz));
  }
  // inertial forces: n^k_ij and g3
  V n2t = V(0.0), n2p = V(0.0), n2y = V(0.0), gam1 = V(0.0), gam2 = V(0.0), gam3 = V(0.0);
  if constexpr (curv) {
    const V bx = k.nfB * ux, by = k.nfB * uy;
    n2t = g.n_trt + g.n_trt;
    gam1 = g.n_rtt + n2t;
    Myy = fmav(bx, g.n_rtt, Myy);
    Mxy = fmav(by, n2t, Mxy);
    if constexpr (ell) {
      const V bz = k.nfB * uz;
      n2p = g.n_prp + g.n_prp;
      n2y = g.n_ttp + g.n_ttp;
      gam2 = g.n_rpp + n2p;
      gam3 = g.n_ptt + n2y;
      Myy = fmav(bz, g.n_ptt, Myy);
      Mzz = fmav(bx, g.n_rpp, Mzz);
      Mxz = fmav(bz, n2p, Mxz);
      Myz = fmav(by, n2y, Myz);
    }
  }
  const V h2 = V(1.0 - 1.0 / CS2);  // 1 + 2 h

  // rest velocity
  if constexpr (DEV) f.template put<0>(fmav(om1, f.template get<0>(), a0 + t_rest));
  else f.template put<0>(fmav(om1, f.template get<0>(), a0 * V(REST_WEIGHT<V>)));

  // axes, |c| = 1 and 3: even a0 + m^2 M_ii, odd m L_i + m^3 C_i
  {
    V Cx = Qxx * ux, Cy = fmav(Qyy, uy, hy * k.nayy), Cz = Qzz * uz;
    if constexpr (gen) {
      Cx = fmav(hx, k.naxx, Cx);
      Cz = fmav(hz, k.nazz, Cz);
    }
    if constexpr (curv) Cy = fmav(g.n_rtt, k.naxy, Cy);
    if constexpr (ell) {
      Cy = fmav(g.n_ptt, k.nayz, Cy);
      Cz = fmav(g.n_rpp, k.naxz, Cz);
    }
    update_pair<0, DEV>(f, om1, T0.template e<0>(a0 + Mxx), T0.template o<0>(Lx + Cx));
    update_pair<1, DEV>(f, om1, T0.template e<1>(a0 + Myy), T0.template o<1>(Ly + Cy));
    const St T6 = entry(6);
    update_pair<2, DEV>(f, om1, T1.template e<2>(a0 + Mzz), T1.template o<2>(Lz + Cz));
    const St T7 = entry(7);
    const V n9 = V(9.0), n3 = V(3.0);
    update_pair<13, DEV>(f, om1, T6.template e<13>(fmav(n9, Mxx, a0)), T6.template o<13>(n3 * fmav(n9, Cx, Lx)));
    update_pair<14, DEV>(f, om1, T7.template e<14>(fmav(n9, Myy, a0)), T7.template o<14>(n3 * fmav(n9, Cy, Ly)));
    update_pair<15, DEV>(f, om1, T7.template e<15>(fmav(n9, Mzz, a0)), T7.template o<15>(n3 * fmav(n9, Cz, Lz)));
  }
  // faces: s_i^3 = s_i, s_i^2 s_j = s_j
  const V Nxy2 = k.naxy + k.naxy, Nyz2 = k.nayz + k.nayz;
  const V hyNxy = hy * Nxy2, hyNyz = hy * Nyz2;   // hf.c (c.N.c): 2 N_xy hf_y, 2 N_yz hf_y
  const St T2 = entry(2);
  {  // x-y
    const V S = Qxx + Qyy, T = k.naxx + k.nayy;
    V e = a0 + Mxx + Myy, x = Mxy;
    V bi = fmav(S, ux, fmav(Qxy, uy, Lx + hyNxy)), bj = fmav(S, uy, fmav(Qxy, ux, fmav(T, hy, Ly)));
    if constexpr (gen) {
      bi = fmav(T, hx, bi);
      bj = fmav(Nxy2, hx, bj);
    }
    if constexpr (curv) {
      e = fmav(gam1, sx, e);
      x = fmav(gam1, sy, x);
      bi = fmav(gam1, fmav(h, T, k.t0), fmav(g.n_rtt, k.naxx, fmav(n2t, k.nayy, bi)));
      bj = fmav(h2 * gam1, k.naxy, bj);
      if constexpr (ell) {
        bi = fmav(g.n_ptt, k.naxz, bi);
        bj = fmav(g.n_ptt, k.nayz, bj);
      }
    }
    update_face<3, DEV>(f, om1, T1.template e<3>(e), T2.template e<4>(x), T1.template o<3>(bi),
                        T2.template o<4>(bj));
  }
  const St T3 = entry(3);
  {  // x-z
    const V S = Qxx + Qzz;
    V e = a0 + Mxx + Mzz, x = Mxz;
    V bi = fmav(S, ux, fmav(Qxz, uz, Lx)), bj = fmav(S, uz, fmav(Qxz, ux, Lz));
    if constexpr (gen) {
      const V T = k.naxx + k.nazz, Nxz2 = k.naxz + k.naxz;
      bi = fmav(T, hx, fmav(Nxz2, hz, bi));
      bj = fmav(T, hz, fmav(Nxz2, hx, bj));
    }
    if constexpr (ell) {
      const V T = k.naxx + k.nazz;
      e = fmav(gam2, sx, e);
      x = fmav(gam2, sz, x);
      bi = fmav(gam2, fmav(h, T, k.t0), fmav(g.n_rpp, k.naxx, fmav(n2p, k.nazz, bi)));
      bj = fmav(h2 * gam2, k.naxz, bj);
    }
    update_face<5, DEV>(f, om1, T2.template e<5>(e), T3.template e<6>(x), T2.template o<5>(bi),
                        T3.template o<6>(bj));
  }
  const St T4 = entry(4);
  V rho2 = V(0.0);  // n^x on nodes with cy^2 = cz^2 = 1
  if constexpr (curv) rho2 = ell ? g.n_rtt + g.n_rpp : g.n_rtt;
  {  // y-z
    const V S = Qyy + Qzz, T = k.nayy + k.nazz;
    V e = a0 + Myy + Mzz, x = Myz;
    V bi = fmav(S, uy, fmav(Qyz, uz, fmav(T, hy, Ly))), bj = fmav(S, uz, fmav(Qyz, uy, Lz + hyNyz));
    if constexpr (gen) {
      bi = fmav(Nyz2, hz, bi);
      bj = fmav(T, hz, bj);
    }
    if constexpr (curv) {
      bi = fmav(rho2, k.naxy, bi);
      bj = fmav(rho2, k.naxz, bj);
    }
    if constexpr (ell) {
      e = fmav(gam3, sz, e);
      x = fmav(gam3, sy, x);
      bi = fmav(h2 * gam3, k.nayz, bi);
      bj = fmav(gam3, fmav(h, T, k.t0), fmav(n2y, k.nayy, fmav(g.n_ptt, k.nazz, bj)));
    }
    update_face<7, DEV>(f, om1, T3.template e<7>(e), T4.template e<8>(x), T3.template o<7>(bi),
                        T4.template o<8>(bj));
  }
  // bodies: even base + X_ij s_i s_j, odd C.s + C_d s_x s_y s_z; the cubic
  // coefficients C and quintic ones P are shared by |c| = 1 and 3
  const V trQ = Qxx + Qyy + Qzz;
  V Cx = fmav(trQ, ux, fmav(Qxy, uy, fmav(Qxz, uz, hyNxy)));
  V Cy = fmav(trQ, uy, fmav(Qxy, ux, Qyz * uz));
  V Cz = fmav(trQ, uz, fmav(Qxz, ux, fmav(Qyz, uy, hyNyz)));
  V Cd = fmav(Qxy, uz, fmav(Qxz, uy, fmav(Qyz, ux, hy * (k.naxz + k.naxz))));
  const V trN = k.naxx + k.nayy + k.nazz;
  Cy = fmav(trN, hy, Cy);
  V m4 = V(0.0), qxy = V(0.0), qxz = V(0.0), qyz = V(0.0);  // (s.c) g3(c)
  V Px = V(0.0), Py = V(0.0), Pz = V(0.0), Pd = V(0.0);     // h g3 c.N.c
  if constexpr (gen) {
    Cx = fmav(trN, hx, fmav(k.naxz + k.naxz, hz, Cx));
    Cy = fmav(Nxy2, hx, fmav(Nyz2, hz, Cy));
    Cz = fmav(trN, hz, fmav(k.naxz + k.naxz, hx, Cz));
    Cd = fmav(Nyz2, hx, fmav(Nxy2, hz, Cd));
  }
  if constexpr (curv && !ell) {
    Cx = fmav(gam1, k.t0, fmav(g.n_rtt, k.naxx, fmav(n2t, k.nayy, Cx)));
    Cy = fmav(gam1, k.naxy, Cy);
    Cz = fmav(g.n_rtt, k.naxz, Cz);
    Cd = fmav(n2t, k.nayz, Cd);
    const V hg = h * gam1, hg2 = hg + hg;
    Px = hg * trN;
    Py = hg2 * k.naxy;
    Pz = hg2 * k.naxz;
    Pd = hg2 * k.nayz;
    m4 = gam1 * sx;
    qxy = gam1 * sy;
    qxz = gam1 * sz;
  }
  if constexpr (ell) {
    const V g12 = gam1 + gam2;
    Cx = fmav(g12, k.t0, fmav(rho2, k.naxx, fmav(n2t, k.nayy, fmav(g.n_ptt, k.naxz, fmav(n2p, k.nazz, Cx)))));
    Cy = fmav(rho2 + n2t, k.naxy, fmav(gam3, k.nayz, Cy));
    Cz = fmav(gam3, k.t0, fmav(rho2 + n2p, k.naxz, fmav(n2y, k.nayy, fmav(g.n_ptt, k.nazz, Cz))));
    Cd = fmav(n2t + n2p, k.nayz, fmav(n2y, k.naxy, Cd));
    const V hg = h * g12, h3 = h * gam3, hg2 = hg + hg, h32 = h3 + h3;
    Px = fmav(hg, trN, h32 * k.naxz);
    Py = fmav(hg2, k.naxy, h32 * k.nayz);
    Pz = fmav(h3, trN, hg2 * k.naxz);
    Pd = fmav(hg2, k.nayz, h32 * k.naxy);
    m4 = fmav(g12, sx, gam3 * sz);
    qxy = g12 * sy;
    qxz = fmav(g12, sz, gam3 * sx);
    qyz = gam3 * sy;
  }
  const V trM = Mxx + Myy + Mzz;
  const St T5 = entry(5);
  {  // |c_i| = 1
    V e = a0 + trM, x = Mxy, y = Mxz, z = Myz, bx = Lx + Cx, by = Ly + Cy, bz = Lz + Cz, d = Cd;
    if constexpr (curv) {
      e = e + m4;
      x = x + qxy;
      y = y + qxz;
      bx = bx + Px;
      by = by + Py;
      bz = bz + Pz;
      d = d + Pd;
    }
    if constexpr (ell) z = z + qyz;
    update_body<9, DEV>(f, om1, T4.template e<9>(e), T5.template e<10>(x), T5.template e<11>(y),
                        entry(6).template e<12>(z), T4.template o<9>(bx), T5.template o<10>(by),
                        T5.template o<11>(bz), entry(6).template o<12>(d));
  }
  const St T8 = entry(8), T9 = entry(9);
  {  // |c_i| = 3
    const V n9 = V(9.0), n81 = V(81.0), n3 = V(3.0), n27 = V(27.0), n243 = V(243.0);
    V e = fmav(n9, trM, a0), x = n9 * Mxy, y = n9 * Mxz, z = n9 * Myz;
    V bx = fmav(n27, Cx, n3 * Lx), by = fmav(n27, Cy, n3 * Ly), bz = fmav(n27, Cz, n3 * Lz), d = n27 * Cd;
    if constexpr (curv) {
      e = fmav(n81, m4, e);
      x = fmav(n81, qxy, x);
      y = fmav(n81, qxz, y);
      bx = fmav(n243, Px, bx);
      by = fmav(n243, Py, by);
      bz = fmav(n243, Pz, bz);
      d = fmav(n243, Pd, d);
    }
    if constexpr (ell) z = fmav(n81, qyz, z);
    update_body<16, DEV>(f, om1, T8.template e<16>(e), T8.template e<17>(x), T9.template e<18>(y),
                         T9.template e<19>(z), T8.template o<16>(bx), T8.template o<17>(by), T9.template o<18>(bz),
                         T9.template o<19>(d));
  }
}

template <typename V, int K>
__device__ __forceinline__ void collide(V (&f)[Q], const Coef<V>& k, const NodeGeo<V, K>& g, const V& omega) {
  collide_shells<V, K>(PopArray<V>{f}, k, g, omega, NoTab{}, V(0.0));
}

// f^eq(rho, u) for all 41 velocities (initial state, Sec. II).
template <typename V, int K>
__device__ __forceinline__ void equilibrium(const V& rho, const V& ux, const V& uy, const V& uz,
                                            const NodeGeo<V, K>& g, V (&f)[Q]) {
  Moments<V> m;
  m.rho = rho;
  m.jx = rho * ux;
  m.jy = rho * uy;
  m.jz = rho * uz;
  m.sxx = m.syy = m.szz = m.sxy = m.sxz = m.syz = V(0.0);  // unused with kappa = 0
  Coef<V> k = coefficients<V, K>(m, g, V(0.0), V(0.0));
  k.ux = ux;
  k.uy = uy;
  k.uz = uz;
  f[0] = k.e0 * V(W_REST);
  static_for<0, NPAIR>([&](auto P_) {
    constexpr int P = decltype(P_)::value;
    using C = Pair<P>;
    constexpr int cx = C::x, cy = C::y, cz = C::z;
    const V uc = dot3<cx, cy, cz>(ux, uy, uz);
    const V uc2 = uc * uc;
    V E = fmav(k.eB, uc2, k.e0);
    V X = fmav(k.oC, uc2, k.oA);
    if constexpr (cy != 0) {
      E = mac<cy * cy>(E, k.eAt);
      X = mac<cy * cy>(X, k.eBt);
    }
    if constexpr (cz != 0) {
      E = mac<cz * cz>(E, k.eAp);
      X = mac<cz * cz>(X, k.eBp);
    }
    if constexpr (K == KELT) {
      if constexpr (cx != 0) {
        E = mac<cx * cx>(E, k.eArr);
        X = mac<cx * cx>(X, k.eBrr);
      }
      if constexpr (cx * cy != 0) {
        E = mac<2 * cx * cy>(E, k.eArt);
        X = mac<2 * cx * cy>(X, k.eBrt);
      }
      if constexpr (cx * cz != 0) {
        E = mac<2 * cx * cz>(E, k.eArp);
        X = mac<2 * cx * cz>(X, k.eBrp);
      }
      if constexpr (cy * cz != 0) {
        E = mac<2 * cy * cz>(E, k.eAtp);
        X = mac<2 * cy * cz>(X, k.eBtp);
      }
    }
    const V O = fmav(uc, X, dot3<cx, cy, cz>(k.nvx, k.nvy, k.nvz));
    f[2 * P + 1] = (E + O) * V(C::w);
    f[2 * P + 2] = (E - O) * V(C::w);
  });
}

}  // namespace lbgm
