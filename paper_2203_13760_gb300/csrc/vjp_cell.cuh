// Reverse passes of the tiled adjoints (vjp.cuh, vjp3.cuh) cell by cell and
// face by face:
//
//   cell_fwd   both WENO5 face values of a cell along one axis
//   conv_face  the HLLC reverse pass of a face from the two stored values,
//              which it replaces by their cotangents
//   cell_rev   the WENO5 reverse pass of a cell from the cotangents of both of
//              its face values
//   visc_face  the dissipative flux of a face
//
// A cell's two face values share their smoothness indicators and factors
// (weno5_cell), and so do their reverse passes: a face-by-face reverse pass
// evaluates every indicator four times (twice forward, twice in reverse) and
// adds 30 cotangents per face, the cell-by-cell one twice and 25 per cell.
//
// Lanes: FP32 works on pairs of components in packed FP32x2 operations, FP64
// one component at a time; the formulas are written once over both.
#pragma once
#include "stage.cuh"
#include "vjp_math.cuh"

namespace jf {

// Lane arithmetic: float and double scalars and FP32 pairs.
#define JF_LANE(T, fma_, add_, sub_, mul_, rcp_, set_)                              \
  __device__ __forceinline__ T vfma(T a, T b, T c) { return fma_; }                 \
  __device__ __forceinline__ T vadd(T a, T b) { return add_; }                      \
  __device__ __forceinline__ T vsub(T a, T b) { return sub_; }                      \
  __device__ __forceinline__ T vmul(T a, T b) { return mul_; }                      \
  __device__ __forceinline__ T vrcp(T a) { return rcp_; }                           \
  template <> struct Splat<T> { __device__ __forceinline__ static T of(double x) { return set_; } };
template <typename V> struct Splat;
JF_LANE(float, fmaf(a, b, c), a + b, a - b, a * b, trcp(a), (float)x)
JF_LANE(double, fma(a, b, c), a + b, a - b, a * b, trcp(a), x)
JF_LANE(float2, __ffma2_rn(a, b, c), __fadd2_rn(a, b), __ffma2_rn(splat2(-1.0f), b, a), __fmul2_rn(a, b), rcp2(a),
        splat2((float)x))
#undef JF_LANE
template <typename V>
__device__ __forceinline__ V vset(double x) { return Splat<V>::of(x); }

// Reverse of weno5_cell (WENO5-JS): from the cotangents rb of `right` and lb
// of `left`, vb[k] = the cotangent of v[j-2+k].  With u_k = 1/t_k, r_k = u_k^2,
// the weights a = (r0, 6 r1, 3 r2) and c = (3 r0, 6 r1, r2), the candidates'
// offsets E, F and the values' offsets er, el:
//   E_k' = rb a_k / S_r, F_k' = -lb c_k / S_l   (cotangents of E_k, F_k),
//   t_k' = -2 u_k [E_k' (E_k - er) + F_k' (F_k - el)],
// then back through t_k = d_k (4/3 d_k + D) + D^2 + eps and the differences.
template <typename V, typename S>
__device__ __forceinline__ void weno5_cell_rev(V vm2, V vm1, V v0, V vp1, V vp2, S eps, V rb, V lb, V vb[5]) {
  const V D2 = vsub(v0, vm1), D3 = vsub(vp1, v0);
  const V d0 = vadd(D2, vsub(vm2, vm1)), d1 = vsub(D3, D2), d2 = vadd(D3, vsub(vp1, vp2));
  const V ke = vset<V>(eps), k43 = vset<V>(4.0 / 3.0);
  const V q2 = vfma(D2, D2, ke), q3 = vfma(D3, D3, ke);
  const V u0 = vrcp(vfma(d0, vfma(k43, d0, D2), q2));
  const V u1 = vrcp(vfma(d1, vfma(k43, d1, D2), q2));
  const V u2 = vrcp(vfma(d2, vfma(k43, d2, D3), q3));
  const V three = vset<V>(3.0), third = vset<V>(1.0 / 3.0), sixth = vset<V>(1.0 / 6.0), half = vset<V>(0.5);
  const V r0 = vmul(u0, u0), r2 = vmul(u2, u2);
  const V a1 = vmul(vmul(vset<V>(6.0), u1), u1), a2 = vmul(three, r2), c0 = vmul(three, r0);
  const V iR = vrcp(vadd(vadd(r0, a1), a2)), iL = vrcp(vadd(vadd(c0, a1), r2));
  const V h2 = vmul(half, D2), h3 = vmul(half, D3);
  const V E0 = vfma(third, d0, h2), E1 = vfma(third, d1, h2), E2 = vfma(sixth, d2, h3);
  const V F0 = vfma(sixth, d0, h2), F1 = vfma(sixth, d1, h2), F2 = vfma(third, d2, h3);
  const V er = vmul(vfma(a2, E2, vfma(a1, E1, vmul(r0, E0))), iR);
  const V el = vmul(vfma(r2, F2, vfma(a1, F1, vmul(c0, F0))), iL);
  const V sR = vmul(rb, iR), sL = vmul(vmul(vset<V>(-1.0), lb), iL);
  const V E0b = vmul(sR, r0), E1b = vmul(sR, a1), E2b = vmul(sR, a2);
  const V F0b = vmul(sL, c0), F1b = vmul(sL, a1), F2b = vmul(sL, r2);
  const V m2 = vset<V>(-2.0), two = vset<V>(2.0), k83 = vset<V>(8.0 / 3.0);
  const V t0b = vmul(vmul(m2, u0), vfma(E0b, vsub(E0, er), vmul(F0b, vsub(F0, el))));
  const V t1b = vmul(vmul(m2, u1), vfma(E1b, vsub(E1, er), vmul(F1b, vsub(F1, el))));
  const V t2b = vmul(vmul(m2, u2), vfma(E2b, vsub(E2, er), vmul(F2b, vsub(F2, el))));
  const V d0b = vfma(t0b, vfma(k83, d0, D2), vfma(third, E0b, vmul(sixth, F0b)));
  const V d1b = vfma(t1b, vfma(k83, d1, D2), vfma(third, E1b, vmul(sixth, F1b)));
  const V d2b = vfma(t2b, vfma(k83, d2, D3), vfma(third, F2b, vmul(sixth, E2b)));
  V D2b = vfma(half, vadd(vadd(E0b, F0b), vadd(E1b, F1b)), vsub(d0b, d1b));
  D2b = vfma(t0b, vfma(two, D2, d0), D2b);
  D2b = vfma(t1b, vfma(two, D2, d1), D2b);
  V D3b = vfma(half, vadd(E2b, F2b), vadd(d1b, d2b));
  D3b = vfma(t2b, vfma(two, D3, d2), D3b);
  const V m1 = vset<V>(-1.0);
  vb[0] = d0b;
  vb[1] = vsub(vmul(m1, d0b), D2b);
  vb[2] = vadd(vadd(rb, lb), vsub(D2b, D3b));
  vb[3] = vadd(D3b, d2b);
  vb[4] = vmul(m1, d2b);
}

// Position p + n e_D (D a compile-time axis).
template <int D>
struct Along {
  int p[3];
  __device__ __forceinline__ int x(int n) const { return p[0] + (D == 0 ? n : 0); }
  __device__ __forceinline__ int y(int n) const { return p[1] + (D == 1 ? n : 0); }
  __device__ __forceinline__ int z(int n) const { return p[2] + (D == 2 ? n : 0); }
};

// Tile: an accessor with w(c, x, y, z) (primitive c of a cell, tile-relative
// coordinates) and add(c, x, y, z, v) (cotangent accumulation).  rv, lv: a
// cell's slot of the right and left values, component stride cs.
template <typename T, int D, typename Tile>
__device__ __forceinline__ void cell_fwd(const Tile& V, const Along<D>& P, T eps, T* rv, T* lv, int cs) {
  auto val = [&](int c, int n) { return V.w(c, P.x(n), P.y(n), P.z(n)); };
  auto one = [&](int c) {
    T r, l;
    weno5_cell_lean<T>(val(c, -2), val(c, -1), val(c, 0), val(c, 1), val(c, 2), eps, r, l);
    rv[c * cs] = r;
    lv[c * cs] = l;
  };
  if constexpr (sizeof(T) == 4) {
    auto two = [&](int a, int b) {
      auto pr = [&](int n) { return make_float2(val(a, n), val(b, n)); };
      float2 r, l;
      weno5_cell_pair_lean(pr(-2), pr(-1), pr(0), pr(1), pr(2), eps, r, l);
      rv[a * cs] = r.x; rv[b * cs] = r.y;
      lv[a * cs] = l.x; lv[b * cs] = l.y;
    };
    two(0, 4);
    two(1, 2);
    one(3);
  } else {
#pragma unroll
    for (int c = 0; c < 5; ++c) one(c);
  }
}

// vb[n][c]: the cotangent of component c of the cell n - 2 along D.
template <typename T, int D, typename Tile>
__device__ __forceinline__ void cell_rev(const Tile& V, const Along<D>& P, T eps, const T* rv, const T* lv, int cs,
                                         T vb[5][5]) {
  auto val = [&](int c, int n) { return V.w(c, P.x(n), P.y(n), P.z(n)); };
  auto one = [&](int c) {
    T b[5];
    weno5_cell_rev<T>(val(c, -2), val(c, -1), val(c, 0), val(c, 1), val(c, 2), eps, rv[c * cs], lv[c * cs], b);
#pragma unroll
    for (int n = 0; n < 5; ++n) vb[n][c] = b[n];
  };
  if constexpr (sizeof(T) == 4) {
    auto two = [&](int a, int b) {
      auto pr = [&](int n) { return make_float2(val(a, n), val(b, n)); };
      float2 q[5];
      weno5_cell_rev<float2>(pr(-2), pr(-1), pr(0), pr(1), pr(2), eps, make_float2(rv[a * cs], rv[b * cs]),
                             make_float2(lv[a * cs], lv[b * cs]), q);
#pragma unroll
      for (int n = 0; n < 5; ++n) {
        vb[n][a] = q[n].x;
        vb[n][b] = q[n].y;
      }
    };
    two(0, 4);
    two(1, 2);
    one(3);
  } else {
#pragma unroll
    for (int c = 0; c < 5; ++c) one(c);
  }
}

// The face between the cell P and its neighbour along D; nu = dLoss/dNF
// (NF = -F + ...).  rv: the left cell's right values, lv: the right cell's
// left values; replaced by their cotangents.  Safe reconstruction: a side that
// falls back to its cell values hands its cotangents to the cell here.
template <typename T, int D, typename Tile>
__device__ __forceinline__ void conv_face(const Tile& V, const Along<D>& P, const T nu[5], const Gas<T>& g, T* rv,
                                          T* lv, int cs) {
  T WL[5], WR[5], Fb[5], WLb[5], WRb[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    WL[c] = rv[c * cs];
    WR[c] = lv[c * cs];
    Fb[c] = -nu[c];
  }
  bool fm = false, fp = false;
  if (g.safe) {
    fm = !(WL[0] > T(0)) || !(WL[4] > T(0));
    fp = !(WR[0] > T(0)) || !(WR[4] > T(0));
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if (fm) WL[c] = V.w(c, P.x(0), P.y(0), P.z(0));
      if (fp) WR[c] = V.w(c, P.x(1), P.y(1), P.z(1));
    }
  }
  hllc_vjp<T, D>(WL, WR, g, Fb, WLb, WRb);
  if (fm || fp) {
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if (fm) { V.add(c, P.x(0), P.y(0), P.z(0), WLb[c]); WLb[c] = T(0); }
      if (fp) { V.add(c, P.x(1), P.y(1), P.z(1), WRb[c]); WRb[c] = T(0); }
    }
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    rv[c * cs] = WLb[c];
    lv[c * cs] = WRb[c];
  }
}

// Reverse pass of the dissipative flux of the same face (NF = ... + F^d).
// Forward (Sections 2, 3.4), n = the normal axis D, e = an active tangent:
//   du_k/dn = DF4(u_k), dT/dn = DF4(T) along the normal;
//   du_n/de and du_e/de by DC4 along e at the cells -1..2 along n,
//   interpolated to the face with RC4; face velocities RC4(u_k);
//   tau_n = mu (2 du_n/dn - 2/3 div), tau_e = mu (du_n/de + du_e/dn);
//   F^d = [0, tau, u_f . tau + lambda dT/dn] (tau_n in component 1 + D).
// The cotangents are left in `o` for the caller to add (visc_add): those of
// the normal stencils, and those of the cell-centre tangential derivatives,
// which are spread along the tangent once per plane.
template <typename T>
struct ViscCot {
  T g[4], f[3];   // DF4 of u, v, w, T and RC4 of u, v, w along the normal
  T s[3][2];      // per tangent axis e: du_n/de, du_e/de
};
template <typename T, int D, int DIM, typename Tile>
__device__ __forceinline__ void visc_face(const Tile& V, const Along<D>& P, const T nu[5], const Gas<T>& g,
                                          const T inv_h[3], ViscCot<T>& o) {
  constexpr int T1 = D == 0 ? 1 : 0, T2 = D == 2 ? 1 : 2;
  const T hn = inv_h[D];
  // ---- forward ----
  T gn[3], uf[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = V.w(1 + k, P.x(q - 1), P.y(q - 1), P.z(q - 1));
    gn[k] = (T(27.0 / 24.0) * hn) * (v[2] - v[1]) + (T(1.0 / 24.0) * hn) * (v[0] - v[3]);
    uf[k] = T(9.0 / 16.0) * (v[1] + v[2]) - T(1.0 / 16.0) * (v[0] + v[3]);
  }
  T dn_e[3] = {T(0), T(0), T(0)}, div = gn[D];  // du_n/de; the divergence
  auto tangent = [&](auto etag) {
    constexpr int e = decltype(etag)::value;
    auto at = [&](int c, int q, int j) {
      return V.w(c, P.x(q) + (e == 0 ? j : 0), P.y(q) + (e == 1 ? j : 0), P.z(q) + (e == 2 ? j : 0));
    };
    const T k0 = T(9.0 / 192.0) * inv_h[e], k1 = T(-1.0 / 192.0) * inv_h[e];
    if constexpr (sizeof(T) == 4) {  // u_n and u_e in the two lanes
      float2 h[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        auto pr = [&](int j) { return make_float2(at(1 + D, q - 1, j), at(1 + e, q - 1, j)); };
        h[q] = vfma(splat2(8.0f), vsub(pr(1), pr(-1)), vsub(pr(-2), pr(2)));
      }
      const float2 G = vfma(splat2(k0), vadd(h[1], h[2]), vmul(splat2(k1), vadd(h[0], h[3])));
      dn_e[e] = G.x;
      div += G.y;
    } else {
      T G[2];
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int c = s == 0 ? 1 + D : 1 + e;
        T h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          h[q] = vfma(T(8), at(c, q - 1, 1) - at(c, q - 1, -1), at(c, q - 1, -2) - at(c, q - 1, 2));
        G[s] = vfma(k0, h[1] + h[2], k1 * (h[0] + h[3]));
      }
      dn_e[e] = G[0];
      div += G[1];
    }
  };
  if constexpr (T1 < DIM) tangent(std::integral_constant<int, T1>{});
  if constexpr (T2 < DIM) tangent(std::integral_constant<int, T2>{});
  // ---- reverse ----
  T taub[3], ufb[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T tau = k == D ? g.mu * (T(2) * gn[k] - T(2.0 / 3.0) * div) : g.mu * (dn_e[k] + gn[k]);
    taub[k] = g.mu * (nu[1 + k] + nu[4] * uf[k]);  // mu times the cotangent of tau_k
    ufb[k] = nu[4] * tau;
  }
  const T divb = -T(2.0 / 3.0) * taub[D];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    o.g[k] = (k == D ? T(2) * taub[k] + divb : taub[k]) * hn;
    o.f[k] = ufb[k];
  }
  o.g[3] = nu[4] * g.lambda * hn;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    if (e == D || e >= DIM) continue;
    o.s[e][0] = taub[e] * inv_h[e];
    o.s[e][1] = divb * inv_h[e];
  }
}

// The cotangents of visc_face that land on the cell q - 1 along the normal
// (q = 0 .. 3): put(component, value) for the primitives, sep(e, component,
// value) for the centre derivatives along e.
template <typename T, int D, int DIM, typename Put, typename Sep>
__device__ __forceinline__ void visc_add(const ViscCot<T>& o, int q, Put put, Sep sep) {
  const T wg = q == 0 ? T(1.0 / 24.0) : q == 1 ? T(-27.0 / 24.0) : q == 2 ? T(27.0 / 24.0) : T(-1.0 / 24.0);
  const T wf = q == 1 || q == 2 ? T(9.0 / 16.0) : T(-1.0 / 16.0);
#pragma unroll
  for (int k = 0; k < 3; ++k) put(1 + k, wg * o.g[k] + wf * o.f[k]);
  put(5, wg * o.g[3]);
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    if (e == D || e >= DIM) continue;
    sep(e, 1 + D, wf * o.s[e][0]);
    sep(e, 1 + e, wf * o.s[e][1]);
  }
}

}  // namespace jf
