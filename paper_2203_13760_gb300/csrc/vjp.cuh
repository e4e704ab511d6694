// Adjoint (vector-Jacobian product) of one Shu-Osher stage (Sections 3.1-3.4,
// Section 7.2): the box kernel of 1D and 2D grids (3D grids: the z-marching
// kernel of vjp3.cuh).
//
// One launch computes, for every interior cell,
//   out = a1 x1 + a2 x2 + m + dt J(Us)^T m,   m = s_in lam,
// where J is the Jacobian of the right-hand side L of Eq. (FVD) at the stage
// state Us.  The adjoint of one fixed-dt RK3 step is three such launches
// (see jf_rk3_step_vjp in vjp.cu).
//
// Derivation.  L_c = sum_d (NF_d(c+1/2) - NF_d(c-1/2)) / h_d with the net face
// flux NF = F^d - F, so the face cotangent is nu_f = (m_left - m_right) / h_d
// and (J^T m)_j = (dW/dU)_j^T sum_f (dNF_f/dW_j)^T nu_f.  Each face's reverse
// pass (HLLC -> WENO5 for the convective part, the C4 stencils for the
// dissipative part) yields cotangents of the primitive variables (and T) of
// its stencil cells; the cell then applies the transposed Jacobian of
// W(U) (and of T = p / (rho R)).
//
// Tiling.  A CTA owns a BX (x BY) box of cells.  It stages the primitives of
// a 5-cell halo around the box on every active axis (WENO5 of a cell 3 cells
// outside reads 2 more) and m with a 3-cell halo, and makes three passes over
// each axis (vjp_cell.cuh): the face values of the cells -3 .. B + 2, the
// faces between them, and the reverse reconstruction of the cells
// -2 .. B + 1, whose cotangents accumulate in shared memory; viscous grids
// make a fourth over the dissipative faces.
// Ghost cells follow the boundary condition: with zero gradient a ghost has
// no right-hand side (m = 0) and its cotangent goes to the interior cell it
// copies; with periodic wrap every ghost face is a real face that the owning
// box also evaluates, so only cotangents of the box's own cells are kept.
// The accumulator covers the box and a 5-cell halo, so an addition needs no
// ownership test; boxes near a non-periodic boundary fold their ghost cells
// afterwards.  In 2D the viscous tangential stencil is applied in two
// separable steps (cell-centre derivative cotangents, then a gather pass) and
// the tasks are ordered for conflict-free banks.
//
// A box over which m is uniform (the cotangent has not reached it, or is constant)
// leaves the passes out: the rollout of a uniform one over 128^2 cells in FP64 takes
// 1.9 ms, 4.6 with the passes; a dense one takes the same to within the runs.
//
// Bound by the latency of dependent arithmetic and shared memory (45 % of the
// issue slots at 16 warps per SM) and the barriers between the steps.
// Measured, 256^2 FP32 viscous (256 boxes, one wave, 256 threads): 23.1 us per
// launch; with atomics in the place of the stepped additions 26.8; face by face
// (every face reconstructed and reversed on its own, 30 atomics each) 31.5.
// With 384 threads a step's three launches take 67.2 us, with 256 70.2.
#pragma once
#include "stage.cuh"
#include <type_traits>

#include "vjp_cell.cuh"

namespace jf {

template <typename T>
struct VjpArgs {
  const T* Us;        // stage state, [5][nz][ny][nx]
  const T* lam;       // cotangent of the stage output
  const T* x1;        // point-wise addends (may be null)
  const T* x2;
  T* out;
  const double* dt;
  T s_in, a1, a2;
  int n[3];
  long long N;
  int periodic[3];
  T inv_h[3];
  int* flag;
};

template <int BX, int BY, int DIM, bool VISC>
struct VGeo {
  static constexpr int HX = 5, HY = DIM >= 2 ? 5 : 0;  // W halo
  static constexpr int PX = BX + 2 * HX, PY = BY + 2 * HY, CS = PX * PY;
  static constexpr int NCW = VISC ? 6 : 5;
  static constexpr int MX = 3, MY = DIM >= 2 ? 3 : 0;  // m halo
  static constexpr int MPX = BX + 2 * MX, MPY = BY + 2 * MY, MCS = MPX * MPY;
  // cotangents accumulate over the box and a 5-cell halo (every cell a
  // stencil reaches), with no ownership test per addition; boxes near a
  // non-periodic boundary fold ghost cells onto the cells they copy afterwards
  static constexpr int AX = 5, AY = DIM >= 2 ? 5 : 0;
  static constexpr int APX = BX + 2 * AX, APY = BY + 2 * AY, ACS = APX * APY;
  // face values of the cells -3 .. B + 2 along each axis, then the cotangents
  // of these values: along x [2][5][BY][BX + 6], along y
  // [2][5][BY + 6][BX + 2] (2 columns of padding: every row pitch is 2 mod 4)
  static constexpr int XP = BX + 6, XS = BY * XP;
  static constexpr int YP = BX + 2, YS = DIM >= 2 ? (BY + 6) * YP : 0;
  // 2D viscous: the tangential C4 stencil (DC4 along the tangent at the cells
  // -1..2 along the normal, then RC4 to the face) is separable, so a face
  // adds its cotangents of the four cell-centre derivatives (slots
  // d * 2 + k: k = 0 for du_n/de, 1 for du_e/de) and one gather pass applies
  // the transposed DC4 afterwards: 8 instead of 32 additions per face.
  static constexpr int NCB = DIM == 2 && VISC ? 4 : 0;
  static_assert(DIM <= 2, "3D grids take the z-marching kernel (vjp3.cuh)");
  static_assert(DIM >= 2 || BY == 1, "1D boxes are one row");
};

template <typename T, int DIM, bool VISC, int BX, int BY>
constexpr size_t vjp_smem_bytes() {
  using G = VGeo<BX, BY, DIM, VISC>;
  return sizeof(T) * (size_t)(G::NCW * G::CS + 5 * G::MCS + (6 * DIM + G::NCB) * G::ACS + 10 * (G::XS + G::YS));
}

// 2D task order: a face family covers R rows (y) by C columns (x) of faces.
// Task f goes to row r and column c (0-based) so that a warp takes 16
// consecutive rows of two adjacent columns: every shared array of a box has a
// row pitch of 2 (mod 4) words (26 or 22), so the 16 rows of one column fall
// on 16 distinct even banks (plus the column) and the next column on the odd
// ones, and the warp's loads and atomics are free of bank conflicts.  Rows
// beyond the first 16 follow as a second block in row-fastest order.
template <int R, int C>
__device__ __forceinline__ void task_rc(int f, int& r, int& c) {
  constexpr int RA = R >= 16 ? 16 : 0;
  constexpr int RB = R - RA > 0 ? R - RA : 1;  // rows of the second block (none when R == 16)
  if (f < RA * C) {
    r = f % 16;
    c = f / 16;
  } else {
    const int g = f - RA * C;
    r = RA + g % RB;
    c = g / RB;
  }
}

// Shared-memory views and the boundary-aware accumulator of one box.
template <typename T, int DIM, bool VISC, int BX, int BY>
struct VTile {
  using G = VGeo<BX, BY, DIM, VISC>;
  const T* W;   // [NCW][PY][PX], box cell (0, 0) at (HX, HY)
  const T* M;   // [5][MPY][MPX]
  T* acc;       // per axis of the faces, [DIM][6][APY][APX], box cell (0, 0) at (AX, AY)
  T* cb;        // [NCB][APY][APX]: cotangents of cell-centre tangential derivatives (2D viscous)

  // coordinates along inactive axes are always 0: fold them at compile time
  __device__ __forceinline__ T w(int c, int x, int y, int) const {
    const int yy = DIM >= 2 ? y : 0;
    return W[c * G::CS + (yy + G::HY) * G::PX + x + G::HX];
  }
  __device__ __forceinline__ T m(int c, int x, int y) const {
    const int yy = DIM >= 2 ? y : 0;
    return M[c * G::MCS + (yy + G::MY) * G::MPX + x + G::MX];
  }
  // box coordinate that keeps a cotangent landing on box-relative coordinate
  // x along an axis, or -1 if it is not this box's to keep
  __device__ __forceinline__ int owner(int x, int x0, int nn, int periodic, int B) const {
    const int gxx = x0 + x;
    if (periodic) return (x >= 0 && x < B && gxx < nn) ? x : -1;
    const int c = gxx < 0 ? 0 : (gxx >= nn ? nn - 1 : gxx);
    const int t = c - x0;
    return (t >= 0 && t < B) ? t : -1;
  }
  __device__ __forceinline__ T* at(int d, int c, int x, int y) const {
    const int yy = DIM >= 2 ? y : 0;
    return acc + (d * 6 + c) * G::ACS + (yy + G::AY) * G::APX + x + G::AX;
  }
  // safe reconstruction only
  __device__ __forceinline__ void add(int c, int x, int y, int, T v) const { atomicAdd(at(0, c, x, y), v); }
  // cotangent of the centre derivative of component c along the tangent of a
  // face normal to d: slot d * 2 + k, k = 0 for the normal velocity
  __device__ __forceinline__ T* sep(int d, int c, int x, int y) const {
    return cb + (d * 2 + (c == 1 + d ? 0 : 1)) * G::ACS + (y + G::AY) * G::APX + x + G::AX;
  }
};

// The stage VJP kernel.  blockDim.x == NT >= BX * BY, grid = (ceil(nx/BX), ceil(ny/BY)).
template <typename T, int DIM, bool VISC, int BX, int BY, int MINB, int NT>
__global__ void __launch_bounds__(NT, MINB) vjp_stage_kernel(const VjpArgs<T> A, const Gas<T> g) {
  using G = VGeo<BX, BY, DIM, VISC>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  follow_predecessor<sizeof(T) == 4>();
  T* Wb = reinterpret_cast<T*>(smem_raw);
  T* Mb = Wb + G::NCW * G::CS;
  T* acc = Mb + 5 * G::MCS;
  T* cbuf = acc + 6 * DIM * G::ACS;
  T* EX = cbuf + G::NCB * G::ACS;  // right values, then (5 components on) left values
  T* EY = EX + 10 * G::XS;
  const int g0[3] = {(int)blockIdx.x * BX, (int)blockIdx.y * BY, 0};
  const int tid = threadIdx.x;

  // stage W (halo 5) and m = s_in lam (halo 3; zero on zero-gradient ghosts)
  bool bad = false;
  for (int t = tid; t < G::CS; t += NT) {
    const int lx = t % G::PX, ly = t / G::PX;
    const int gx = map_index(g0[0] + lx - G::HX, A.n[0], A.periodic[0]);
    const int gy = DIM >= 2 ? map_index(g0[1] + ly - G::HY, A.n[1], A.periodic[1]) : 0;
    const long long q = (long long)gy * A.n[0] + gx;
    const T r = A.Us[q];
    const T inv = trcp(r);
    const T u = A.Us[q + A.N] * inv, v = A.Us[q + 2 * A.N] * inv, w = A.Us[q + 3 * A.N] * inv;
    const T p = g.gm1 * (A.Us[q + 4 * A.N] - T(0.5) * r * (u * u + v * v + w * w));
    bad |= !(r > T(0)) || !(p > T(0));
    Wb[t] = r;
    Wb[G::CS + t] = u;
    Wb[2 * G::CS + t] = v;
    Wb[3 * G::CS + t] = w;
    Wb[4 * G::CS + t] = p;
    if (VISC) Wb[5 * G::CS + t] = p * inv * g.inv_R;
  }
  if (bad) atomicOr(A.flag, 1);
  T first[5];  // m of the box's first cell
#pragma unroll
  for (int c = 0; c < 5; ++c) first[c] = A.s_in * A.lam[(long long)g0[1] * A.n[0] + g0[0] + c * A.N];
  bool uneven = false;
  for (int t = tid; t < G::MCS; t += NT) {
    const int lx = t % G::MPX, ly = t / G::MPX;
    const int r[2] = {g0[0] + lx - G::MX, DIM >= 2 ? g0[1] + ly - G::MY : 0};
    bool ghost = false;
#pragma unroll
    for (int a = 0; a < DIM; ++a) ghost |= !A.periodic[a] && (r[a] < 0 || r[a] >= A.n[a]);
    const int gx = map_index(r[0], A.n[0], A.periodic[0]);
    const int gy = DIM >= 2 ? map_index(r[1], A.n[1], A.periodic[1]) : 0;
    const long long q = (long long)gy * A.n[0] + gx;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const T m = ghost ? T(0) : A.s_in * A.lam[q + c * A.N];
      Mb[c * G::MCS + t] = m;
      uneven |= !(m - first[c] == T(0));
    }
  }
  for (int t = tid; t < (6 * DIM + G::NCB) * G::ACS; t += NT) acc[t] = T(0);
  // a box over which m is uniform (no cotangent has reached it yet, say) has no
  // face with one
  const bool live = __syncthreads_or(uneven);

  VTile<T, DIM, VISC, BX, BY> V;
  V.W = Wb;
  V.M = Mb;
  V.acc = acc;
  V.cb = cbuf;
  const T inv_h[3] = {A.inv_h[0], A.inv_h[1], A.inv_h[2]};

  // Three passes over flat task lists, so that every thread takes the same
  // number of tasks (up to one) whatever the per-direction counts.  In 2D the
  // tasks are ordered by task_rc (16 rows of two adjacent columns per warp).
  // Slots along an axis hold the cells -3 .. B + 2 from index 0.
  auto slot = [&](auto dtag, int s, int row) {  // the cell s along the axis, row (x) or column (y) across
    constexpr int d = decltype(dtag)::value;
    return d == 0 ? EX + row * G::XP + s + 3 : EY + (s + 3) * G::YP + row;
  };
  // task f of `along` positions from `first` along the axis by the box's (or
  // `across`) rows (x axis) or columns (y axis) from -off
  auto decode = [&](auto dtag, auto atag, auto ctag, int f, int& s, int& o) {
    if constexpr (DIM == 1) {
      s = f;
      o = 0;
    } else if constexpr (decltype(dtag)::value == 0) {
      task_rc<decltype(ctag)::value, decltype(atag)::value>(f, o, s);
    } else {
      task_rc<decltype(atag)::value, decltype(ctag)::value>(f, s, o);
    }
  };
  using X = std::integral_constant<int, 0>;
  using Y = std::integral_constant<int, 1>;
  auto position = [&](auto dtag, int s, int o) {
    constexpr int d = decltype(dtag)::value;
    return Along<d>{{d == 0 ? s : o, d == 0 ? o : s, 0}};
  };
  constexpr int CX = G::XS / G::XP;  // rows across the x axis

  if (live) {
  // pass 1: face values of the cells -3 .. B + 2
  auto fwd = [&](auto dtag, auto atag, auto ctag, int f) {
    constexpr int d = decltype(dtag)::value, cs = d == 0 ? G::XS : G::YS;
    int s, o;
    decode(dtag, atag, ctag, f, s, o);
    T* e = slot(dtag, s - 3, o);
    cell_fwd<T, d>(V, position(dtag, s - 3, o), g.eps, e, e + 5 * cs, cs);
  };
  constexpr int f0 = (BX + 6) * CX, f1 = DIM >= 2 ? (BY + 6) * BX : 0;
  for (int f = tid; f < f0 + f1; f += NT) {
    if (f < f0) fwd(X{}, std::integral_constant<int, BX + 6>{}, std::integral_constant<int, CX>{}, f);
    else if constexpr (DIM >= 2) fwd(Y{}, std::integral_constant<int, BY + 6>{}, std::integral_constant<int, BX>{}, f - f0);
  }
  __syncthreads();

  // pass 2: the convective faces: left cells -3 .. B + 1 (the cells -2 ..
  // B + 1 reach the box, and a face is theirs on either side), the box's own
  // cells across
  auto face_nu = [&](auto dtag, const int* p, T nu[5]) -> bool {
    constexpr int d = decltype(dtag)::value;
    bool any = false;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      nu[c] = (V.m(c, p[0], p[1]) - V.m(c, p[0] + (d == 0), p[1] + (d == 1))) * inv_h[d];
      any |= nu[c] != T(0);
    }
    return any;
  };
  auto conv = [&](auto dtag, auto atag, auto ctag, int f) {
    constexpr int d = decltype(dtag)::value, cs = d == 0 ? G::XS : G::YS, step = d == 0 ? 1 : G::YP;
    int s, o;
    decode(dtag, atag, ctag, f, s, o);
    const auto P = position(dtag, s - 3, o);
    T* rv = slot(dtag, s - 3, o);
    T* lv = rv + 5 * cs + step;
    T nu[5];
    if (face_nu(dtag, P.p, nu)) {
      conv_face<T, d>(V, P, nu, g, rv, lv, cs);
    } else {
#pragma unroll
      for (int c = 0; c < 5; ++c) rv[c * cs] = lv[c * cs] = T(0);
    }
  };
  constexpr int c0 = (BX + 5) * CX, c1 = DIM >= 2 ? (BY + 5) * BX : 0;
  for (int f = tid; f < c0 + c1; f += NT) {
    if (f < c0) conv(X{}, std::integral_constant<int, BX + 5>{}, std::integral_constant<int, CX>{}, f);
    else if constexpr (DIM >= 2) conv(Y{}, std::integral_constant<int, BY + 5>{}, std::integral_constant<int, BX>{}, f - c0);
  }
  __syncthreads();

  // Additions without atomics (a shared-memory floating-point atomic is a
  // compare-and-swap loop of about seven instructions): the tasks of one axis
  // add to an accumulator of their own, all at the same offset along the axis
  // in one step, so that no two threads meet in a cell; a barrier separates
  // the steps.  Every thread takes part in every step of every round.
  // pass 3: the cells -2 .. B + 1 from the cotangents of their two values
  constexpr int r0 = (BX + 4) * CX, r1 = DIM >= 2 ? (BY + 4) * BX : 0;
#pragma unroll 1
  for (int f0 = 0; f0 < r0 + r1; f0 += NT) {
    const int f = f0 + tid;
    T vb[5][5];
    int s = 0, o = 0;
    if (f < r0) {
      decode(X{}, std::integral_constant<int, BX + 4>{}, std::integral_constant<int, CX>{}, f, s, o);
      const T* e = slot(X{}, s - 2, o);
      cell_rev<T, 0>(V, position(X{}, s - 2, o), g.eps, e, e + 5 * G::XS, G::XS, vb);
    } else if constexpr (DIM >= 2) {
      if (f < r0 + r1) {
        decode(Y{}, std::integral_constant<int, BY + 4>{}, std::integral_constant<int, BX>{}, f - r0, s, o);
        const T* e = slot(Y{}, s - 2, o);
        cell_rev<T, 1>(V, position(Y{}, s - 2, o), g.eps, e, e + 5 * G::YS, G::YS, vb);
      }
    }
    const bool x = f < r0;
    T* a = x ? V.at(0, 0, s - 4, o) : V.at(1, 0, o, s - 4);
    const int step = x ? 1 : G::APX;
#pragma unroll
    for (int n = 0; n < 5; ++n) {
      if (f < r0 + r1) {
#pragma unroll
        for (int c = 0; c < 5; ++c) a[n * step + c * G::ACS] += vb[n][c];
      }
      __syncthreads();
    }
  }
  // pass 4, viscous: the dissipative faces: left cells -2 .. B along the
  // normal, -2 .. B + 1 across on the active tangent
  if constexpr (VISC) {
    constexpr int w = DIM >= 2 ? 4 : 0, o2 = DIM >= 2 ? 2 : 0;
    constexpr int v0 = (BX + 3) * (CX + w), v1 = DIM >= 2 ? (BY + 3) * (BX + 4) : 0;
    auto visc = [&](auto dtag, int s, int o, ViscCot<T>& out) -> bool {
      constexpr int d = decltype(dtag)::value;
      const auto P = position(dtag, s - 2, o - o2);
      T nu[5];
      if (!face_nu(dtag, P.p, nu)) return false;
      visc_face<T, d, DIM>(V, P, nu, g, inv_h, out);
      return true;
    };
#pragma unroll 1
    for (int f0 = 0; f0 < v0 + v1; f0 += NT) {
      const int f = f0 + tid;
      ViscCot<T> out;
      int s = 0, o = 0;
      bool on = false;
      if (f < v0) {
        decode(X{}, std::integral_constant<int, BX + 3>{}, std::integral_constant<int, CX + w>{}, f, s, o);
        on = visc(X{}, s, o, out);
      } else if constexpr (DIM >= 2) {
        if (f < v0 + v1) {
          decode(Y{}, std::integral_constant<int, BY + 3>{}, std::integral_constant<int, BX + 4>{}, f - v0, s, o);
          on = visc(Y{}, s, o, out);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int p = s - 3 + q, r = o - o2;  // the cell q - 1 along the normal
        if (on) {
          if (f < v0)
            visc_add<T, 0, DIM>(out, q, [&](int c, T v) { *V.at(0, c, p, r) += v; },
                                [&](int, int c, T v) { *V.sep(0, c, p, r) += v; });
          else if constexpr (DIM >= 2)
            visc_add<T, 1, DIM>(out, q, [&](int c, T v) { *V.at(1, c, r, p) += v; },
                                [&](int, int c, T v) { *V.sep(1, c, r, p) += v; });
        }
        __syncthreads();
      }
    }
  }
  if constexpr (DIM >= 2) {  // one accumulator from here on
    for (int t = tid; t < 6 * G::ACS; t += NT) acc[t] += acc[6 * G::ACS + t];
    __syncthreads();
  }

  if constexpr (G::NCB > 0) {
    // transposed DC4 along the tangent: cell Y receives
    // sum_o dcw[o] cb(Y - dco[o] e) (dco = -2, -1, 1, 2; dcw = (1, -8, 8, -1) / 12).
    // Slots: x faces (tangent y) 0: du/dy -> u, 1: dv/dy -> v;
    // y faces (tangent x) 2: dv/dx -> v, 3: du/dx -> u.
    for (int t = tid; t < G::ACS; t += NT) {
      const int lx = t % G::APX, ly = t / G::APX;
      // (cells beyond the accumulation region hold no cotangent)
      auto spread = [&](int slot, int step, int pos, int len) {
        const T* s = cbuf + slot * G::ACS + t;
        T v = T(0);
        if (pos + 2 < len) v += (T(1) / T(12)) * s[2 * step];
        if (pos + 1 < len) v += (-T(8) / T(12)) * s[step];
        if (pos >= 1) v += (T(8) / T(12)) * s[-step];
        if (pos >= 2) v += (-T(1) / T(12)) * s[-2 * step];
        return v;
      };
      const T du = spread(0, G::APX, ly, G::APY) + spread(3, 1, lx, G::APX);
      const T dv = spread(1, G::APX, ly, G::APY) + spread(2, 1, lx, G::APX);
      acc[G::ACS + t] += du;
      acc[2 * G::ACS + t] += dv;
    }
    __syncthreads();
  }

  {
    // ghost cells of a non-periodic axis pass their cotangents to the cell
    // they copy (if it is in this box); everything else outside the box (and
    // beyond the grid on a periodic axis) belongs to another box, which
    // evaluates the same faces.  Only boxes within reach of such a boundary
    // (or ragged against it) have ghosts to fold; the test is uniform per CTA.
    bool fold = false;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const int B = a == 0 ? BX : BY, h = a == 0 ? G::AX : G::AY;
      fold |= !A.periodic[a] && (g0[a] - h < 0 || g0[a] + B + h > A.n[a]);
    }
    if (fold) {
      for (int t = tid; t < G::ACS; t += NT) {
        const int lx = t % G::APX - G::AX, ly = t / G::APX - G::AY;
        const int ox = V.owner(lx, g0[0], A.n[0], A.periodic[0], BX);
        const int oy = DIM >= 2 ? V.owner(ly, g0[1], A.n[1], A.periodic[1], BY) : 0;
        if (ox >= 0 && oy >= 0 && (ox != lx || oy != ly)) {
          const int to = (oy + G::AY) * G::APX + ox + G::AX;
#pragma unroll
          for (int c = 0; c < 6; ++c) atomicAdd(acc + c * G::ACS + to, acc[c * G::ACS + t]);
        }
      }
      __syncthreads();
    }
  }

  }  // live

  // cells: cotangent of W (+T) -> cotangent of U, then the stage combination
  const int tx = tid % BX, ty = tid / BX;
  const int gx = g0[0] + tx, gy = g0[1] + ty;
  if (tid < BX * BY && gx < A.n[0] && gy < A.n[1]) {
    const T r = V.w(0, tx, ty, 0), u = V.w(1, tx, ty, 0), v = V.w(2, tx, ty, 0), w = V.w(3, tx, ty, 0);
    const T p = V.w(4, tx, ty, 0);
    const int cell = (ty + G::AY) * G::APX + tx + G::AX;
    T br = acc[cell], bu = acc[G::ACS + cell], bv = acc[2 * G::ACS + cell], bw = acc[3 * G::ACS + cell];
    T bp = acc[4 * G::ACS + cell];
    const T inv = trcp(r);
    if (VISC) {
      const T bT = acc[5 * G::ACS + cell];
      const T Tc = V.w(5, tx, ty, 0);
      br -= bT * Tc * inv;  // T = p / (rho R)
      bp += bT * Tc * trcp(p);
    }
    T bU[5];
    bU[0] = br - (bu * u + bv * v + bw * w) * inv + bp * g.gm1 * T(0.5) * (u * u + v * v + w * w);
    bU[1] = bu * inv - bp * g.gm1 * u;
    bU[2] = bv * inv - bp * g.gm1 * v;
    bU[3] = bw * inv - bp * g.gm1 * w;
    bU[4] = bp * g.gm1;
    const T dt = T(*A.dt);
    const long long q = (long long)gy * A.n[0] + gx;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      T o = V.m(c, tx, ty) + dt * bU[c];
      if (A.x1) o += A.a1 * A.x1[q + c * A.N];
      if (A.x2) o += A.a2 * A.x2[q + c * A.N];
      A.out[q + c * A.N] = o;
    }
  }
}

}  // namespace jf
