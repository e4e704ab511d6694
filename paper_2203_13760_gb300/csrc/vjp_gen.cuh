// Adjoint (vector-Jacobian product) of one Shu-Osher stage for the run-time
// schemes the tiled adjoint of vjp.cuh does not cover: slip walls, WENO3-JS
// and the Rusanov-NN flux of Section 7.4 (with its parameter gradient), for
// inviscid 1D, 2D and 3D grids.
//
// One stage computes, as the tiled adjoint does (with one more addend),
//   out = a1 x1 + a2 x2 + a3 x3 + m + dt J(Us)^T m,   m = s_in lam,
// with J the Jacobian of the right-hand side L of Eq. (FVD) at Us.
//
// Layout of the work.  A point-wise launch writes the addends and m; then one
// thread per face (every face of every active direction) recomputes the
// face's stencil (6 cells along the normal, mapped through the boundary
// condition), its reconstruction and flux, and runs the reverse pass:
// face cotangent Fb = dt (m_right - m_left) / h (a ghost cell has no
// right-hand side, so its m is 0), flux -> reconstructed states -> stencil
// primitives -> stencil conservative states, each added to `out` of the cell
// the stencil cell maps to (global atomics; with a wall the mirrored normal
// momentum carries its sign back).  For the Rusanov-NN flux the thread also
// writes the face's network input x and the cotangent of the dissipation,
// abar = -1/2 Fb . (U_R - U_L), so that a second launch can form the
// parameter gradient sum_f abar_f d alpha(x_f) / d theta.
//
// This path is built for the small grids of the learned-flux experiment: a
// face thread redoes the full stencil work and the atomics serialise on
// shared cells, which the tiled adjoint avoids.  Atomic summation makes the
// last bits vary from run to run.
#pragma once
#include "stage.cuh"
#include "vjp_math.cuh"

namespace jf {

template <typename T>
struct GVjpArgs {
  const T* Us;        // stage state, [5][nz][ny][nx]
  const T* lam;       // cotangent of the stage output
  const T* x1;        // point-wise addends (may be null)
  const T* x2;
  const T* x3;
  T* out;
  const double* dt;
  T s_in, a1, a2, a3;
  int n[3];
  long long N;
  int periodic[3];
  int wall[3];        // bit 0: wall at the low side, bit 1: at the high side
  T inv_h[3];
  long long nface[3]; // faces per direction (0 for inactive directions)
  T* rec;             // Rusanov-NN: 5 values per face (x0..x3, abar), else null
};

// Up to kMax grids per launch (a batch, or one grid), passed by value in the
// kernel parameters: the grids' arguments and the prefix sums of their faces
// and cells, so that one launch covers every face (cell) of every grid.
template <typename T>
struct GVjpBatch {
  static constexpr int kMax = 32;
  int nsim;
  long long face_base[kMax + 1];
  long long cell_base[kMax + 1];
  GVjpArgs<T> sim[kMax];
};

// The grid an index of [0, base[nsim]) belongs to (base ascending).
__device__ __forceinline__ int find_sim(const long long* base, int nsim, long long i) {
  int lo = 0, hi = nsim - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (base[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// out = a1 x1 + a2 x2 + a3 x3 + s_in lam, every cell of every grid
template <typename T>
__global__ void __launch_bounds__(256) gvjp_point_kernel(const GVjpBatch<T> B) {
  follow_predecessor<sizeof(T) == 4>();
  const long long total = B.cell_base[B.nsim];
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int s = find_sim(B.cell_base, B.nsim, i);
    const GVjpArgs<T>& A = B.sim[s];
    const long long c = i - B.cell_base[s];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const long long q = c + k * A.N;
      T o = A.s_in * A.lam[q];
      if (A.x1) o += A.a1 * A.x1[q];
      if (A.x2) o += A.a2 * A.x2[q];
      if (A.x3) o += A.a3 * A.x3[q];
      A.out[q] = o;
    }
  }
}

// Reciprocal of this file's own divisions (the approximation of trcp, an ulp in
// FP32, serves the functions it shares with the stage kernels).  FP32: one
// Newton step, whose residual is exact, rounds as IEEE division does but for
// arguments within 2^-22 ulp of a tie; 1/0 and 1/inf are the approximation's.
// Without IEEE division's test and branch for subnormal numbers: walled WENO3
// adjoint step, 128^2, 52.2 us with __frcp_rn, 46.4 with this, 45.7 with the
// bare approximation.
__device__ __forceinline__ float rcp_rn(float x) {
  const float y = trcp(x), e = fmaf(-x, y, 1.0f);
  return fabsf(e) < 1.0f ? fmaf(y, e, y) : y;
}
__device__ __forceinline__ double rcp_rn(double x) { return trcp(x); }

// Cotangent of W = (rho, u, v, w, p) -> cotangent of U = (rho, rho u, rho v,
// rho w, E) for an ideal gas, p = (gamma - 1) (E - |m|^2 / (2 rho)).
template <typename T>
__device__ __forceinline__ void prim_vjp(const T W[5], const Gas<T>& g, const T Wb[5], T Ub[5]) {
  const T ir = rcp_rn(W[0]);
  const T u = W[1], v = W[2], w = W[3];
  const T k = g.gm1;
  Ub[0] = Wb[0] - (Wb[1] * u + Wb[2] * v + Wb[3] * w) * ir + Wb[4] * k * T(0.5) * (u * u + v * v + w * w);
  Ub[1] = Wb[1] * ir - Wb[4] * k * u;
  Ub[2] = Wb[2] * ir - Wb[4] * k * v;
  Ub[3] = Wb[3] * ir - Wb[4] * k * w;
  Ub[4] = Wb[4] * k;
}

// Reverse of side_flux<T, D> (flux F and conservative state U of one face
// side from its primitive state W): Wb += (dF/dW)^T Fb + (dU/dW)^T Ub.
template <typename T, int D>
JF_HD void side_flux_vjp(const T W[5], const Gas<T>& g, const T Fb[5], const T Ub[5], T Wb[5]) {
  const T r = W[0], un = W[1 + D], p = W[4];
  const T q2 = W[1] * W[1] + W[2] * W[2] + W[3] * W[3];
  const T E = p * g.inv_gm1 + T(0.5) * r * q2;
  const T mass = r * un;
  const T massb = Fb[0] + Fb[1] * W[1] + Fb[2] * W[2] + Fb[3] * W[3];
  T ub[3] = {Fb[1] * mass + Ub[1] * r, Fb[2] * mass + Ub[2] * r, Fb[3] * mass + Ub[3] * r};
  T pb = Fb[1 + D] + Fb[4] * un;
  T unb = Fb[4] * (E + p) + massb * r;
  const T Eb = Fb[4] * un + Ub[4];
  T rb = Ub[0] + Ub[1] * W[1] + Ub[2] * W[2] + Ub[3] * W[3] + massb * un + Eb * T(0.5) * q2;
  ub[D] += unb;
#pragma unroll
  for (int k = 0; k < 3; ++k) ub[k] += Eb * r * W[1 + k];
  pb += Eb * g.inv_gm1;
  Wb[0] += rb;
  Wb[1] += ub[0];
  Wb[2] += ub[1];
  Wb[3] += ub[2];
  Wb[4] += pb;
}

// NN_HIDDEN values in registers (a hidden layer's values or cotangents), FP32
// as pairs for packed operations.
template <typename T>
struct HRow {
  T v[NN_HIDDEN];
  __device__ __forceinline__ void fill(T x) {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; ++j) v[j] = x;
  }
  __device__ __forceinline__ void load(const T* row) {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) ld4(row + j, v + j);
  }
  // += s w over a row w (16-byte aligned)
  __device__ __forceinline__ void axpy(const T* w, T s) {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      T q[4];
      ld4(w + j, q);
#pragma unroll
      for (int m = 0; m < 4; ++m) v[j + m] += s * q[m];
    }
  }
  // as a 4 x 8 block: += the products of g[0 .. 3] and h[0 .. 7] (16-byte aligned)
  __device__ __forceinline__ void outer(const T* g, const T* h) {
    T a[4], b[8];
    ld4(g, a);
    ld4(h, b);
    ld4(h + 4, b + 4);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int c = 0; c < 8; ++c) v[8 * m + c] += a[m] * b[c];
  }
  __device__ __forceinline__ T get(int j) const { return v[j]; }
  __device__ __forceinline__ void set(int j, T x) { v[j] = x; }
  __device__ __forceinline__ void store(T* row) const {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; ++j) row[j] = v[j];
  }
};
template <>
struct HRow<float> {
  float2 v[NN_HIDDEN / 2];
  __device__ __forceinline__ void fill(float x) {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN / 2; ++j) v[j] = make_float2(x, x);
  }
  __device__ __forceinline__ void load(const float* row) {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      const float4 q = *reinterpret_cast<const float4*>(row + j);
      v[j / 2] = make_float2(q.x, q.y);
      v[j / 2 + 1] = make_float2(q.z, q.w);
    }
  }
  __device__ __forceinline__ void axpy(const float* w, float s) {
    const float2 s2 = make_float2(s, s);
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      const float4 q = *reinterpret_cast<const float4*>(w + j);
      v[j / 2] = __ffma2_rn(make_float2(q.x, q.y), s2, v[j / 2]);
      v[j / 2 + 1] = __ffma2_rn(make_float2(q.z, q.w), s2, v[j / 2 + 1]);
    }
  }
  __device__ __forceinline__ void outer(const float* g, const float* h) {
    const float4 a = *reinterpret_cast<const float4*>(g);
    const float4 p = *reinterpret_cast<const float4*>(h), q = *reinterpret_cast<const float4*>(h + 4);
    const float am[4] = {a.x, a.y, a.z, a.w};
    const float2 b[4] = {make_float2(p.x, p.y), make_float2(p.z, p.w), make_float2(q.x, q.y), make_float2(q.z, q.w)};
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[4 * m + c] = __ffma2_rn(make_float2(am[m], am[m]), b[c], v[4 * m + c]);
  }
  __device__ __forceinline__ float get(int j) const { return j & 1 ? v[j / 2].y : v[j / 2].x; }
  __device__ __forceinline__ void set(int j, float x) {
    if (j & 1) v[j / 2].y = x;
    else v[j / 2].x = x;
  }
  __device__ __forceinline__ void store(float* row) const {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4)
      *reinterpret_cast<float4*>(row + j) =
          make_float4(v[j / 2].x, v[j / 2].y, v[j / 2 + 1].x, v[j / 2 + 1].y);
  }
};

// The network's parameters in shared memory for the adjoint kernels: the flat
// layout (padded to a multiple of 4), then W1, W2 and W3 transposed (inputs by
// outputs), so that every pass over a layer, forward or reverse, adds whole
// rows to a row of register accumulators (HRow::axpy: 16-byte loads that all
// lanes share, FP32 in packed operations).
constexpr int kNnParamsPad = (NN_PARAMS + 3) / 4 * 4;
constexpr int kNnW1 = 0, kNnB1 = kNnW1 + 4 * NN_HIDDEN, kNnW2 = kNnB1 + NN_HIDDEN,
              kNnB2 = kNnW2 + NN_HIDDEN * NN_HIDDEN, kNnW3 = kNnB2 + NN_HIDDEN,
              kNnB3 = kNnW3 + NN_HIDDEN * NN_HIDDEN, kNnW4 = kNnB3 + NN_HIDDEN, kNnB4 = kNnW4 + NN_HIDDEN;
constexpr int kNnTRow = NN_HIDDEN + 4;  // row pitch of W2 and W3 transposed (fewer bank conflicts in nn_stage)
constexpr int kNnT1 = kNnParamsPad, kNnT2 = kNnT1 + 4 * NN_HIDDEN, kNnT3 = kNnT2 + NN_HIDDEN * kNnTRow,
              kNnShared = kNnT3 + NN_HIDDEN * kNnTRow;
template <typename T>
__device__ __forceinline__ void nn_stage(const T* theta, T* th) {
  block_copy(theta, NN_PARAMS, [&](int i, T v) { th[i] = v; });
  __syncthreads();
  for (int i = threadIdx.x; i < 4 * NN_HIDDEN; i += blockDim.x) th[kNnT1 + i % 4 * NN_HIDDEN + i / 4] = th[kNnW1 + i];
  for (int i = threadIdx.x; i < NN_HIDDEN * NN_HIDDEN; i += blockDim.x) {
    const int t = i % NN_HIDDEN * kNnTRow + i / NN_HIDDEN;
    th[kNnT2 + t] = th[kNnW2 + i];
    th[kNnT3 + t] = th[kNnW3 + i];
  }
}

// Row pitch of the per-thread hidden rows in shared memory (a multiple of 4
// for the vector accesses; 36 puts the 16-byte accesses of 8 consecutive
// threads on distinct banks).
constexpr int kHRow = NN_HIDDEN + 4;

// acc += sum_j h[j] W[j][:] over the rows of W (pitch PITCH), h (16-byte
// aligned) read four at a time; a loop, so that the code of a network pass
// stays small.  SPARSE: h holds zeros for inactive units, whose rows FP64 skips
// (the FP64 pipe bounds it, and the faces of a warp share most of them: adjoint
// step with the network, 128^2, 2321 us without, 2050 with; its parameter gradient too
// 4383 and 3807).
template <int PITCH, bool SPARSE = false, typename T>
__device__ __forceinline__ void nn_rows(const T* W, const T* h, HRow<T>& acc) {
#pragma unroll 1
  for (int j = 0; j < NN_HIDDEN; j += 4) {
    T q[4];
    ld4(h + j, q);
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (!SPARSE || sizeof(T) == 4 || q[m] != T(0)) acc.axpy(W + (j + m) * PITCH, q[m]);
  }
}

// The hidden layers for input x: h1, h2 (this thread's rows, shared memory)
// and the third layer's values in `h`; returns the network's output o
// (alpha = exp(o)).
template <typename T>
__device__ __forceinline__ T nn_forward(const T* th, const T x[4], T* h1, T* h2, HRow<T>& h) {
  auto relu = [&]() {
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; ++j) h.set(j, tmax(T(0), h.get(j)));
  };
  h.load(th + kNnB1);
#pragma unroll
  for (int m = 0; m < 4; ++m) h.axpy(th + kNnT1 + m * NN_HIDDEN, x[m]);
  relu();
  h.store(h1);
  h.load(th + kNnB2);
  nn_rows<kNnTRow>(th + kNnT2, h1, h);
  relu();
  h.store(h2);
  h.load(th + kNnB3);
  nn_rows<kNnTRow>(th + kNnT3, h2, h);
  relu();
  T o = th[kNnB4];
#pragma unroll
  for (int j = 0; j < NN_HIDDEN; ++j) o += th[kNnW4 + j] * h.get(j);
  return o;
}

// alpha = exp(NN(x)) (as nn_alpha) and dx = d alpha / dx.  h1, h2: this
// thread's two hidden rows (kHRow pitch, shared memory).
template <typename T>
__device__ __forceinline__ T nn_alpha_grad(const T* th, const T x[4], T dx[4], T* h1, T* h2) {
  HRow<T> h;
  const T alpha = texp(nn_forward(th, x, h1, h2, h));
  // reverse, seed d alpha / d o = alpha: each layer's cotangents masked by
  // its activity and stored over the row of the layer above
  unsigned m1 = 0, m2 = 0;
#pragma unroll
  for (int j = 0; j < NN_HIDDEN; j += 4) {
    T a[4], b[4];
    ld4(h1 + j, a);
    ld4(h2 + j, b);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      m1 |= (a[m] > T(0) ? 1u : 0u) << (j + m);
      m2 |= (b[m] > T(0) ? 1u : 0u) << (j + m);
    }
  }
#pragma unroll
  for (int j = 0; j < NN_HIDDEN; ++j) h.set(j, h.get(j) > T(0) ? alpha * th[kNnW4 + j] : T(0));
  h.store(h2);
  h.fill(T(0));
  nn_rows<NN_HIDDEN, true>(th + kNnW3, h2, h);
#pragma unroll
  for (int j = 0; j < NN_HIDDEN; ++j) h.set(j, (m2 >> j) & 1u ? h.get(j) : T(0));
  h.store(h1);
  h.fill(T(0));
  nn_rows<NN_HIDDEN, true>(th + kNnW2, h1, h);
#pragma unroll
  for (int m = 0; m < 4; ++m) dx[m] = T(0);
#pragma unroll
  for (int k = 0; k < NN_HIDDEN; ++k) {
    const T s = (m1 >> k) & 1u ? h.get(k) : T(0);
    T w[4];
    ld4(th + kNnW1 + 4 * k, w);
#pragma unroll
    for (int m = 0; m < 4; ++m) dx[m] += w[m] * s;
  }
  return alpha;
}

// Reverse of rusanov_nn<T, D>: WLb, WRb += cotangents; rec = (x, abar).
template <typename T, int D>
__device__ __forceinline__ void rusanov_nn_vjp(const T WL[5], const T WR[5], const Gas<T>& g, const T* th,
                                               const T Fb[5], T WLb[5], T WRb[5], T rec[5], T* h1, T* h2) {
  T EL, ER, irL, irR, cL, cR;
  side_state(WL, g, EL, irL, cL);
  side_state(WR, g, ER, irR, cR);
  // nn_inputs, with the entropy jump's sign kept
  const T ds = ((tlog(WR[4]) - tlog(WL[4])) - g.gamma * (tlog(WR[0]) - tlog(WL[0]))) * g.inv_gm1;
  const T x[4] = {fabs(WR[1 + D] - WL[1 + D]), T(0.5) * (WL[1 + D] + WR[1 + D]), T(0.5) * (cL + cR), fabs(ds)};
  T dx[4];
  const T alpha = nn_alpha_grad(th, x, dx, h1, h2);
  T FL[5], FR[5], UL[5], UR[5];
  side_flux<T, D>(WL, EL, FL, UL);
  side_flux<T, D>(WR, ER, FR, UR);
  T abar = T(0), hFb[5], ULb[5], URb[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    abar -= T(0.5) * Fb[q] * (UR[q] - UL[q]);
    hFb[q] = T(0.5) * Fb[q];
    ULb[q] = T(0.5) * alpha * Fb[q];
    URb[q] = -ULb[q];
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) rec[m] = x[m];
  rec[4] = abar;
  side_flux_vjp<T, D>(WL, g, hFb, ULb, WLb);
  side_flux_vjp<T, D>(WR, g, hFb, URb, WRb);
  // through alpha(x): xb = abar d alpha / dx
  T xb[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) xb[m] = abar * dx[m];
  const T du = WR[1 + D] - WL[1 + D];
  const T s0 = du < T(0) ? T(-1) : T(1);  // d|y|/dy, taken as +1 at 0
  WLb[1 + D] += -s0 * xb[0] + T(0.5) * xb[1];
  WRb[1 + D] += s0 * xb[0] + T(0.5) * xb[1];
  // mean sound speed, c = sqrt(gamma p / rho): dc/dp = c / (2 p), dc/drho = -c / (2 rho)
  const T cb = T(0.5) * xb[2];
  const T ipL = rcp_rn(WL[4]), ipR = rcp_rn(WR[4]), idL = rcp_rn(WL[0]), idR = rcp_rn(WR[0]);
  WLb[4] += T(0.5) * cb * cL * ipL;
  WLb[0] -= T(0.5) * cb * cL * idL;
  WRb[4] += T(0.5) * cb * cR * ipR;
  WRb[0] -= T(0.5) * cb * cR * idR;
  // entropy jump, s = (ln p - gamma ln rho) / (gamma - 1), with the sign that
  // the inputs took it with
  const T sb = (ds < T(0) ? T(-1) : T(1)) * xb[3] * g.inv_gm1;
  WLb[4] -= sb * ipL;
  WLb[0] += sb * g.gamma * idL;
  WRb[4] += sb * ipR;
  WRb[0] -= sb * g.gamma * idR;
}

// WENO3-JS reverse (left-biased value from vm1, v0, vp1): vb[k] += yb dy/dv_k.
template <typename T>
__device__ __forceinline__ void weno3_vjp(T vm1, T v0, T vp1, T eps, T yb, T vb[3]) {
  const T q0 = T(0.5) * (T(3) * v0 - vm1), q1 = T(0.5) * (v0 + vp1);
  const T e0 = v0 - vm1, e1 = vp1 - v0;
  const T t0 = eps + e0 * e0, t1 = eps + e1 * e1;
  const T r0 = rcp_rn(t0), r1 = rcp_rn(t1);
  const T a0 = T(1.0 / 3.0) * r0 * r0, a1 = T(2.0 / 3.0) * r1 * r1;
  const T inv = rcp_rn(a0 + a1);
  const T y = (a0 * q0 + a1 * q1) * inv;
  const T s = yb * inv;
  const T qb0 = s * a0, qb1 = s * a1;
  // d alpha_k / d t_k = -2 alpha_k / t_k, d t_k / d e_k = 2 e_k
  const T eb0 = -T(4) * s * (q0 - y) * a0 * r0 * e0;
  const T eb1 = -T(4) * s * (q1 - y) * a1 * r1 * e1;
  vb[0] += -T(0.5) * qb0 - eb0;
  vb[1] += T(1.5) * qb0 + T(0.5) * qb1 + eb0 - eb1;
  vb[2] += T(0.5) * qb1 + eb1;
}

// The reverse pass of one face normal to D whose right cell is c (the left
// cell is c - e_D).  RECON: 0 WENO5-JS, 2 WENO3-JS; FLUX: 0 HLLC (Einfeldt
// speeds), 4 Rusanov-NN.  Worked in the face's frame (the components of a
// cell in the order rho, normal, the two others, E), so that one copy of the
// code serves every axis: the pass is executed once per thread, and with a
// copy per axis the instruction fetch was its largest stall.
template <typename T, int RECON, int FLUX>
__device__ __forceinline__ void gvjp_face(const GVjpArgs<T>& A, const Gas<T>& g, int D, const int c[3], long long f,
                                          T* h1, T* h2) {
  const int n = D == 0 ? A.n[0] : (D == 1 ? A.n[1] : A.n[2]), cD = D == 0 ? c[0] : (D == 1 ? c[1] : c[2]);
  const int per = D == 0 ? A.periodic[0] : (D == 1 ? A.periodic[1] : A.periodic[2]);
  const int wall = D == 0 ? A.wall[0] : (D == 1 ? A.wall[1] : A.wall[2]);
  const long long sD = D == 0 ? 1 : (D == 1 ? (long long)A.n[0] : (long long)A.n[0] * A.n[1]);
  // offset of the face's line (coordinate D = 0) and of the frame's components
  const long long base = c[0] + (long long)A.n[0] * (c[1] + (long long)A.n[1] * c[2]) - cD * sD;
  const long long comp[5] = {0, (1 + D) * A.N, (D == 0 ? 2 : 1) * A.N, (D == 2 ? 2 : 3) * A.N, 4 * A.N};
  // m of the two cells beside the face (a ghost has none)
  const T scale = T(*A.dt) * (D == 0 ? A.inv_h[0] : (D == 1 ? A.inv_h[1] : A.inv_h[2])) * A.s_in;
  T Fb[5];
  {
    int iL = cD - 1;
    const bool hasL = per || iL >= 0, hasR = per || cD < n;
    if (iL < 0 && per) iL += n;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const T mL = hasL ? A.lam[base + iL * sD + comp[q]] : T(0);
      const T mR = hasR ? A.lam[base + cD * sD + comp[q]] : T(0);
      Fb[q] = scale * (mR - mL);
    }
  }
  // primitives of the stencil cells c[D] - 3 .. c[D] + 2 along D, through the
  // boundary map (slot 2 is the left cell, slot 3 the right one)
  T W[6][5];
  long long at[6];
  bool flip[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    if (RECON == 2 && (j == 0 || j == 5)) continue;
    at[j] = base + map_index_bc(cD - 3 + j, n, per, wall, flip[j]) * sD;
    T* w = W[j];
    const T r = A.Us[at[j]], ir = rcp_rn(r);
    w[0] = r;
#pragma unroll
    for (int q = 1; q < 4; ++q) w[q] = A.Us[at[j] + comp[q]] * ir;
    if (flip[j]) w[1] = -w[1];
    w[4] = g.gm1 * (A.Us[at[j] + comp[4]] - T(0.5) * r * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]));
  }
  // face states
  T WL[5], WR[5];
  bool fbL = false, fbR = false;  // safe-reconstruction fallback to the cell values
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    if (RECON == 2) {
      WL[q] = weno3(W[1][q], W[2][q], W[3][q], g.eps);
      WR[q] = weno3(W[4][q], W[3][q], W[2][q], g.eps);
    } else {
      WL[q] = weno5(W[0][q], W[1][q], W[2][q], W[3][q], W[4][q], g.eps, 0);
      WR[q] = weno5(W[5][q], W[4][q], W[3][q], W[2][q], W[1][q], g.eps, 0);
    }
  }
  if (g.safe) {
    fbL = !(WL[0] > T(0)) || !(WL[4] > T(0));
    fbR = !(WR[0] > T(0)) || !(WR[4] > T(0));
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      if (fbL) WL[q] = W[2][q];
      if (fbR) WR[q] = W[3][q];
    }
  }
  T WLb[5] = {T(0), T(0), T(0), T(0), T(0)}, WRb[5] = {T(0), T(0), T(0), T(0), T(0)};
  if constexpr (FLUX == 4) {
    T rec[5];
    rusanov_nn_vjp<T, 0>(WL, WR, g, g.nn, Fb, WLb, WRb, rec, h1, h2);
    if (A.rec)
#pragma unroll
      for (int m = 0; m < 5; ++m) A.rec[f * 5 + m] = rec[m];
  } else {
    hllc_vjp<T, 0>(WL, WR, g, Fb, WLb, WRb);
  }
  // reconstruction reverse
  T Wb[6][5];
#pragma unroll
  for (int j = 0; j < 6; ++j)
#pragma unroll
    for (int q = 0; q < 5; ++q) Wb[j][q] = T(0);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    if (fbL) {
      Wb[2][q] += WLb[q];
    } else if (RECON == 2) {
      T vb[3] = {T(0), T(0), T(0)};
      weno3_vjp(W[1][q], W[2][q], W[3][q], g.eps, WLb[q], vb);
      Wb[1][q] += vb[0]; Wb[2][q] += vb[1]; Wb[3][q] += vb[2];
    } else {
      T vb[5] = {T(0), T(0), T(0), T(0), T(0)};
      weno5_vjp(W[0][q], W[1][q], W[2][q], W[3][q], W[4][q], g.eps, WLb[q], vb);
#pragma unroll
      for (int k = 0; k < 5; ++k) Wb[k][q] += vb[k];
    }
    if (fbR) {
      Wb[3][q] += WRb[q];
    } else if (RECON == 2) {
      T vb[3] = {T(0), T(0), T(0)};
      weno3_vjp(W[4][q], W[3][q], W[2][q], g.eps, WRb[q], vb);
      Wb[4][q] += vb[0]; Wb[3][q] += vb[1]; Wb[2][q] += vb[2];
    } else {
      T vb[5] = {T(0), T(0), T(0), T(0), T(0)};
      weno5_vjp(W[5][q], W[4][q], W[3][q], W[2][q], W[1][q], g.eps, WRb[q], vb);
#pragma unroll
      for (int k = 0; k < 5; ++k) Wb[5 - k][q] += vb[k];
    }
  }
  // primitive -> conservative reverse, back through the boundary map
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    if (RECON == 2 && (j == 0 || j == 5)) continue;
    T Ub[5];
    prim_vjp(W[j], g, Wb[j], Ub);
    if (flip[j]) Ub[1] = -Ub[1];
#pragma unroll
    for (int q = 0; q < 5; ++q) atomicAdd(A.out + at[j] + comp[q], Ub[q]);
  }
}

// One thread per face of every grid of the launch: within a grid, faces of
// direction 0 first, then 1, then 2; within a direction x fastest.  A periodic axis has n faces (face 0 is also face n),
// any other n + 1.  Rusanov-NN: dynamic shared memory of
// gvjp_face_smem_bytes holds the network parameters (nn_stage) and each
// thread's two hidden-layer rows.  Small CTAs spread a training batch's faces
// (42,240 for 20 grids of 32^2) evenly over the SMs.
constexpr int kGvjpThreads = 64;
template <typename T, int FLUX>
constexpr size_t gvjp_face_smem_bytes() {
  return FLUX == 4 ? sizeof(T) * ((size_t)kNnShared + (size_t)kGvjpThreads * 2 * kHRow) : 0;
}

template <typename T, int DIM, int RECON, int FLUX>
__global__ void __launch_bounds__(kGvjpThreads, sizeof(T) == 4 ? 5 : 1) gvjp_face_kernel(const GVjpBatch<T> B, const Gas<T> g) {
  extern __shared__ __align__(16) unsigned char gvjp_smem[];
  follow_predecessor<sizeof(T) == 4>();
  T* th = reinterpret_cast<T*>(gvjp_smem);  // the network parameters (Rusanov-NN)
  T* h1 = th + kNnShared + threadIdx.x * kHRow;
  T* h2 = h1 + kGvjpThreads * kHRow;
  Gas<T> gs = g;
  if constexpr (FLUX == 4) {
    nn_stage(g.nn, th);
    __syncthreads();
    gs.nn = th;
  }
  const long long gf = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gf >= B.face_base[B.nsim]) return;
  const int sidx = find_sim(B.face_base, B.nsim, gf);
  const GVjpArgs<T>& A = B.sim[sidx];
  const long long f = gf - B.face_base[sidx];  // face of this grid (its record index)
  long long r = f;
  int d = 0;
  for (; d < DIM; ++d) {
    if (r < A.nface[d]) break;
    r -= A.nface[d];
  }
  if (d >= DIM) return;
  int ext[3] = {A.n[0], A.n[1], A.n[2]};
  ext[d] += A.periodic[d] ? 0 : 1;
  int c[3];
  c[0] = (int)(r % ext[0]);
  r /= ext[0];
  c[1] = (int)(r % ext[1]);
  c[2] = (int)(r / ext[1]);
  gvjp_face<T, RECON, FLUX>(A, gs, d, c, f, h1, h2);
}

// Parameter gradient of the Rusanov-NN dissipation: grad += sum over the
// face records (x_f, abar_f) of abar_f d alpha(x_f) / d theta.
//
// Persistent blocks of kNnWarps warps; the block stages theta in shared
// memory, and each warp takes chunks of 32 records (one per lane).  Per
// chunk, each lane evaluates the network of its record and the cotangents of
// every layer (seed d alpha / d o = alpha, scaled by abar) into shared rows,
// reusing rows once they are consumed; then the lanes add the weight gradients
// summed over the 32 records (dW[i][k] = sum_f G[f][i] H[f][k]) to accumulators
// kept in registers across chunks, each lane 4 x 8 entries of a 32 x 32 layer.  At the end the block sums its
// warps' accumulators in shared memory and adds them to grad with one atomic
// per parameter.
//
// Bound by the FMA pipe and the shared-memory loads (about 6400 FMA per
// record).  Whole rows in 16-byte loads (pitch 36) and packed FMA: 753 ->
// 505 us for the 1.27 million records of a training step (20 boxes of 32^2, 15
// RK2 steps); 4 x 8 blocks in the place of a row per lane, three loads for 16
// packed multiply-adds and not ten: 464 us.
constexpr int kNnWarps = 6;  // two blocks per SM by shared memory (FP32)
constexpr int kNnWarpElems = 3 * 32 * kHRow + 32 * 5;  // three row sets, inputs, output cotangents
template <typename T>
constexpr size_t nn_grad_smem_bytes() {
  return sizeof(T) * (size_t)(kNnShared + kNnWarps * kNnWarpElems);
}
static_assert(kNnWarpElems >= NN_PARAMS, "the warps' row sets hold their sums at the end");

template <typename T>
__global__ void __launch_bounds__(32 * kNnWarps, sizeof(T) == 4 ? 2 : 1) nn_param_grad_kernel(const T* theta,
                                                                      const T* rec, long long nrec,
                                                                      T* grad) {
  extern __shared__ __align__(16) unsigned char nn_smem[];
  follow_predecessor<sizeof(T) == 4>();
  T* TH = reinterpret_cast<T*>(nn_smem);
  nn_stage(theta, TH);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* base = TH + kNnShared + warp * kNnWarpElems;
  T* R1 = base;                 // H1
  T* R2 = R1 + 32 * kHRow;      // H2
  T* R3 = R2 + 32 * kHRow;      // H3, then G2, then G1
  T* X = R3 + 32 * kHRow;       // [32][4]
  T* OB = X + 32 * 4;           // [32]
  __syncthreads();
  // this lane's 4 x 8 block of the gradients of W3 and W2 and entry `lane` of
  // the others, accumulated over this warp's chunks
  const int br = 4 * (lane >> 2), bc = 8 * (lane & 3);
  HRow<T> a3, a2;
  T a1[4] = {T(0), T(0), T(0), T(0)};
  a3.fill(T(0));
  a2.fill(T(0));
  T ab1 = T(0), ab2 = T(0), ab3 = T(0), a4 = T(0), ab4 = T(0);
  const T w4 = TH[kNnW4 + lane];
  const long long nchunk = (nrec + 31) / 32;
  T* h1 = R1 + lane * kHRow;
  T* h2 = R2 + lane * kHRow;
  T* r3 = R3 + lane * kHRow;
  for (long long ch = (long long)blockIdx.x * kNnWarps + warp; ch < nchunk; ch += (long long)gridDim.x * kNnWarps) {
    const long long f = ch * 32 + lane;
    T x[4] = {T(0), T(0), T(0), T(0)}, abar = T(0);
    if (f < nrec) {
#pragma unroll
      for (int m = 0; m < 4; ++m) x[m] = rec[f * 5 + m];
      abar = rec[f * 5 + 4];
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) X[lane * 4 + m] = x[m];
    HRow<T> v;
    const T o = nn_forward(TH, x, h1, h2, v);
    const T ob = f < nrec ? abar * texp(o) : T(0);  // d alpha / d o = alpha
    OB[lane] = ob;
    v.store(r3);
    __syncwarp();
    // layer 4 (H3 in R3) and b3: G3 = OB W4 where H3 > 0
#pragma unroll 2
    for (int r = 0; r < 32; ++r) {
      const T h3 = R3[r * kHRow + lane], b = OB[r];
      const T g3 = h3 > T(0) ? b * w4 : T(0);
      ab3 += g3;
      a4 += b * h3;
      ab4 += b;
    }
    __syncwarp();
    // layer 3: G3 into R3 (H2 in R2)
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; ++j) v.set(j, v.get(j) > T(0) ? ob * TH[kNnW4 + j] : T(0));
    v.store(r3);
    __syncwarp();
#pragma unroll 2
    for (int r = 0; r < 32; ++r) a3.outer(R3 + r * kHRow + br, R2 + r * kHRow + bc);
    // G2 into R3: g2[j] = [h2_j > 0] sum_i W3[i][j] g3[i]
    v.fill(T(0));
    nn_rows<NN_HIDDEN, true>(TH + kNnW3, r3, v);
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      T q[4];
      ld4(h2 + j, q);
#pragma unroll
      for (int m = 0; m < 4; ++m) v.set(j + m, q[m] > T(0) ? v.get(j + m) : T(0));
    }
    __syncwarp();
    v.store(r3);
    __syncwarp();
    // layer 2 (G2 in R3, H1 in R1)
#pragma unroll 2
    for (int r = 0; r < 32; ++r) {
      ab2 += R3[r * kHRow + lane];
      a2.outer(R3 + r * kHRow + br, R1 + r * kHRow + bc);
    }
    __syncwarp();
    // G1 into R3: g1[k] = [h1_k > 0] sum_j W2[j][k] g2[j]
    v.fill(T(0));
    nn_rows<NN_HIDDEN, true>(TH + kNnW2, r3, v);
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      T q[4];
      ld4(h1 + j, q);
#pragma unroll
      for (int m = 0; m < 4; ++m) v.set(j + m, q[m] > T(0) ? v.get(j + m) : T(0));
    }
    __syncwarp();
    v.store(r3);
    __syncwarp();
    // layer 1 (G1 in R3, inputs in X)
#pragma unroll 2
    for (int r = 0; r < 32; ++r) {
      const T g1 = R3[r * kHRow + lane];
      ab1 += g1;
      T q[4];
      ld4(X + r * 4, q);
#pragma unroll
      for (int m = 0; m < 4; ++m) a1[m] += g1 * q[m];
    }
    __syncwarp();
  }
  // block sum of the warps' rows (the row sets are free now), then one
  // atomic per parameter
  __syncthreads();
  T* S = TH + kNnShared;  // [kNnWarps][kNnWarpElems]
  T* Sw = S + warp * kNnWarpElems;
  const int L = lane;
#pragma unroll
  for (int m = 0; m < 4; ++m) Sw[kNnW1 + 4 * L + m] = a1[m];
  Sw[kNnB1 + L] = ab1;
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      Sw[kNnW2 + NN_HIDDEN * (br + m) + bc + c] = a2.get(8 * m + c);
      Sw[kNnW3 + NN_HIDDEN * (br + m) + bc + c] = a3.get(8 * m + c);
    }
  Sw[kNnB2 + L] = ab2;
  Sw[kNnB3 + L] = ab3;
  Sw[kNnW4 + L] = a4;
  if (L == 0) Sw[kNnB4] = ab4;
  __syncthreads();
  for (int i = threadIdx.x; i < NN_PARAMS; i += blockDim.x) {
    T sum = T(0);
#pragma unroll
    for (int w = 0; w < kNnWarps; ++w) sum += S[w * kNnWarpElems + i];
    if (sum != T(0)) atomicAdd(grad + i, sum);
  }
}

}  // namespace jf
