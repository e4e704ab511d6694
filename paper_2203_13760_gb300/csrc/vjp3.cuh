// Adjoint of one Shu-Osher stage on 3D grids, marching along z (Sections
// 3.1-3.4, Section 7.2).  Same product as vjp_stage_kernel,
//   out = a1 x1 + a2 x2 + m + dt J(Us)^T m,   m = s_in lam,
// organised like the forward stage kernel instead of in boxes:
//
//  * A CTA owns a BX x BY column of cells and a chunk of planes along z.  Per
//    plane k it makes the three passes of vjp_cell.cuh: the WENO5 face values
//    of the cells along x and y (plane k) and along z (plane k+1); the
//    convective reverse pass of the x and y faces of plane k and of the z face
//    k+1/2, and the dissipative one; the reverse reconstruction of the cells.
//    x and y faces are owned by one CTA: the lower face of each of its cells,
//    and on a non-periodic axis the upper boundary face of the grid's last
//    cell; the rim cells' reverse passes run in both CTAs beside them, each
//    with its own face's cotangent (the pass is linear in them).  Along z a
//    column keeps its cell's upper value and lower cotangent from plane to
//    plane, and the face between two chunks is evaluated by both.
//  * The primitive variables (+T) of the planes k-2 .. k+3 live in a six-slot
//    shared-memory ring with a 3-cell x/y halo, and m = s_in lam of the planes
//    k, k+1 in a two-slot ring with a 1-cell halo (zero on zero-gradient
//    ghosts: ghosts have no right-hand side).
//  * The cotangents of W (+T) land on cells of the planes k-2 .. k+2 (tile
//    plus a 3-cell halo) and are accumulated in a five-slot shared-memory
//    ring with shared-memory atomics.
//  * Plane k-2 then receives nothing more from this CTA: its accumulator slot
//    is added to a global accumulator G[NCW][N] with global atomics, each
//    halo or ghost cell mapped to the cell it stands for (periodic wrap,
//    zero-gradient clamp: a ghost copies the boundary cell, so its cotangent
//    belongs to that cell), and the slot takes plane k+3.
//  * A per-cell pass (vjp3_finish_kernel) applies the transposed Jacobian of
//    W(U) and T = p / (rho R) to G and forms the stage combination.
//
// Summation order of the atomics, and so the last bits, may vary between
// runs.
//
// Planes over which m is uniform have no x and y tasks, and cells between equal
// ones no reverse z pass (24^3 rollout of a uniform cotangent, FP64, 13.8 -> 6.0 ms;
// a dense one the same within 1 %).
//
// Bound by latency at 18 warps per SM (one CTA fills the shared memory): a
// scheduler issues in 50 % of its cycles (44 % with 512 threads), the rest are
// waits for barriers, shared memory and dependent arithmetic.  A warp takes a
// row of a full tile (no bank conflicts along x), and the threads of a CTA
// (vjp_f32.cu) fill the rounds of the passes.  Measured, 128^3 FP32 viscous, a
// step and its adjoint: 3901 us with 512 threads and rows of BX + 1 tasks, 3788
// with the warps on rows, 3583 with 576 threads (adjoint alone 3214 -> 3004 us).
// Its error against 64 bits is half of that of a face-by-face pass.
#pragma once
#include "vjp.cuh"

namespace jf {

template <int BX, int BY, bool VISC>
struct V3Geo {
  static constexpr int H = 3;                        // halo of the W and accumulator planes
  static constexpr int PX = BX + 2 * H, PY = BY + 2 * H, CS = PX * PY;
  static constexpr int NCW = VISC ? 6 : 5;           // rho, u, v, w, p (, T)
  static constexpr int PLANE = NCW * CS;
  static constexpr int RING = 6;                     // W planes k-2 .. k+3
  static constexpr int ARING = 5;                    // accumulator planes k-2 .. k+2
  static constexpr int MPX = BX + 2, MPY = BY + 2, MCS = MPX * MPY;  // m planes, 1-cell halo
  // face values of the cells, then their cotangents: along x [2][5][BY][BX+2]
  // (cells -1 .. BX), along y [2][5][BY+2][BX], along z two planes of
  // [2][5][BY][BX]
  static constexpr int XP = BX + 2, XS = BY * XP, YS = (BY + 2) * BX, ZC = BX * BY;
  // viscous: cotangents of the cell-centre tangential derivatives (the DC4
  // stencil is separable from the face's RC4): the x and y faces of the face
  // plane in 7 slots (spread along y: u, v; along x: u, v; along z: u, v, w),
  // the z faces in a ring of 4 planes (k-1 .. k+2) of 4 slots over the tile's
  // own cells (spread along x: w, u; along y: w, v)
  static constexpr int NXY = VISC ? 7 : 0, NZ = VISC ? 4 : 0, ZRING = 4;
};

template <typename T, bool VISC, int BX, int BY>
constexpr size_t vjp3_smem_bytes() {
  using G = V3Geo<BX, BY, VISC>;
  return sizeof(T) * (size_t)((G::RING + G::ARING) * G::PLANE + 2 * 5 * G::MCS + G::NXY * G::CS +
                              (G::ZRING * G::NZ + 20) * G::ZC + 10 * (G::XS + G::YS) + 5);
}

// Accessor of the rings at face plane k: coordinates relative to the tile
// origin along x, y and to plane k along z (z in -2 .. 3 for W, -2 .. 2 for the
// accumulator, 0 .. 1 for m, -1 .. 2 for the z faces' derivative cotangents).
template <typename T, bool VISC, int BX, int BY>
struct V3Tile {
  using G = V3Geo<BX, BY, VISC>;
  const T* W;
  T* acc;
  const T* M;
  T* cbxy;    // [7][PY][PX]
  T* cbz;     // [4 planes][4][BY][BX]
  int wp[6];  // element offset of the W slot of plane k + z, index z + 2
  int ap[5];  // of the accumulator slot of plane k + z, index z + 2
  int mp[2];  // of the m slot of plane k + z
  int zp[4];  // of the z-face cotangent slot of plane k + z, index z + 1
  __device__ __forceinline__ T w(int c, int x, int y, int z) const {
    return W[wp[z + 2] + c * G::CS + (y + G::H) * G::PX + x + G::H];
  }
  __device__ __forceinline__ void add(int c, int x, int y, int z, T v) const {
    atomicAdd(acc + ap[z + 2] + c * G::CS + (y + G::H) * G::PX + x + G::H, v);
  }
  __device__ __forceinline__ T m(int c, int x, int y, int z) const {
    return M[mp[z] + c * G::MCS + (y + 1) * G::MPX + x + 1];
  }
  // addition to a plane of the own column that no other thread adds to meanwhile
  __device__ __forceinline__ void add_own(int c, int x, int y, int z, T v) const {
    acc[ap[z + 2] + c * G::CS + (y + G::H) * G::PX + x + G::H] += v;
  }
  // cotangent of the centre derivative of component c along axis e at a
  // cell of a face normal to d (x, y faces: plane k; z faces: planes k-1 .. k+2)
  __device__ __forceinline__ void add_sep(int d, int e, int c, int x, int y, int z, T v) const {
    if (d == 2) {
      const int slot = e == 0 ? (c == 3 ? 0 : 1) : (c == 3 ? 2 : 3);
      cbz[zp[z + 1] + slot * G::ZC + y * BX + x] += v;  // the column's own thread
    } else {
      const int slot = e == 1 ? (c == 1 ? 0 : 1) : (e == 0 ? (c == 1 ? 2 : 3) : (c == 1 ? 4 : (c == 2 ? 5 : 6)));
      atomicAdd(cbxy + slot * G::CS + (y + G::H) * G::PX + x + G::H, v);
    }
  }
};

// Transposed DC4 along a line of a cotangent slot: the sum over o of
// dcw[o] src(pos - dco[o]) (dco = -2, -1, 1, 2; dcw = (1, -8, 8, -1) / 12); s
// points at pos, positions outside 0 .. len - 1 hold no cotangent.
template <typename T>
__device__ __forceinline__ T vjp3_pull(const T* s, int pos, int len, int step) {
  auto at = [&](int o) { return (unsigned)(pos + o) < (unsigned)len ? s[o * step] : T(0); };
  return (T(1) / T(12)) * (at(2) - at(-2)) + (T(8) / T(12)) * (at(-1) - at(1));
}

// Primitives (+T) of plane gz (unmapped) into W slot dst.
template <typename T, bool VISC, int BX, int BY, int NT>
__device__ __forceinline__ void vjp3_load_w(const VjpArgs<T>& A, const Gas<T>& g, T* dst, int x0, int y0, int gz,
                                            bool& bad) {
  using G = V3Geo<BX, BY, VISC>;
  const int kz = map_index(gz, A.n[2], A.periodic[2]);
  for (int t = threadIdx.x; t < G::CS; t += NT) {
    const int ly = t / G::PX, lx = t - ly * G::PX;
    const int gx = map_index(x0 + lx - G::H, A.n[0], A.periodic[0]);
    const int gy = map_index(y0 + ly - G::H, A.n[1], A.periodic[1]);
    const long long q = ((long long)kz * A.n[1] + gy) * A.n[0] + gx;
    const T r = A.Us[q];
    const T inv = trcp(r);
    const T u = A.Us[q + A.N] * inv, v = A.Us[q + 2 * A.N] * inv, w = A.Us[q + 3 * A.N] * inv;
    const T p = g.gm1 * (A.Us[q + 4 * A.N] - T(0.5) * r * (u * u + v * v + w * w));
    bad |= !(r > T(0)) || !(p > T(0));
    dst[t] = r;
    dst[G::CS + t] = u;
    dst[2 * G::CS + t] = v;
    dst[3 * G::CS + t] = w;
    dst[4 * G::CS + t] = p;
    if (VISC) dst[5 * G::CS + t] = p * inv * g.inv_R;
  }
}

// m = s_in lam of plane gz (unmapped) into m slot dst; zero on zero-gradient ghosts.
// uneven: whether one of them differs from mref.
template <typename T, bool VISC, int BX, int BY, int NT>
__device__ __forceinline__ void vjp3_load_m(const VjpArgs<T>& A, T* dst, int x0, int y0, int gz, const T mref[5],
                                            bool& uneven) {
  using G = V3Geo<BX, BY, VISC>;
  const bool gzout = !A.periodic[2] && (gz < 0 || gz >= A.n[2]);
  const int kz = map_index(gz, A.n[2], A.periodic[2]);
  for (int t = threadIdx.x; t < G::MCS; t += NT) {
    const int ly = t / G::MPX, lx = t - ly * G::MPX;
    const int rx = x0 + lx - 1, ry = y0 + ly - 1;
    const bool ghost = gzout || (!A.periodic[0] && (rx < 0 || rx >= A.n[0])) ||
                       (!A.periodic[1] && (ry < 0 || ry >= A.n[1]));
    const int gx = map_index(rx, A.n[0], A.periodic[0]);
    const int gy = map_index(ry, A.n[1], A.periodic[1]);
    const long long q = ((long long)kz * A.n[1] + gy) * A.n[0] + gx;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const T m = ghost ? T(0) : A.s_in * A.lam[q + c * A.N];
      dst[c * G::MCS + t] = m;
      uneven |= !(m - mref[c] == T(0));
    }
  }
}

// The next W plane and m plane of the march in registers: their global loads
// are issued right after the face pass (vjp3_fetch), so that their latency
// overlaps with the reverse reconstruction, and converted and stored
// afterwards (vjp3_commit) -- the same values as vjp3_load_w and
// vjp3_load_m.
template <typename T, bool VISC, int BX, int BY, int NT>
struct V3Fetch {
  using G = V3Geo<BX, BY, VISC>;
  static constexpr int PW = (G::CS + NT - 1) / NT, PM = (G::MCS + NT - 1) / NT;
  T w[PW][5];
  T m[PM][5];
  bool ghost[PM];
};

template <typename T, bool VISC, int BX, int BY, int NT>
__device__ __forceinline__ void vjp3_fetch(const VjpArgs<T>& A, V3Fetch<T, VISC, BX, BY, NT>& f, int x0, int y0,
                                           int gzw, int gzm) {
  using G = V3Geo<BX, BY, VISC>;
  using F = V3Fetch<T, VISC, BX, BY, NT>;
  const int kw = map_index(gzw, A.n[2], A.periodic[2]);
#pragma unroll
  for (int i = 0; i < F::PW; ++i) {
    const int t = threadIdx.x + i * NT;
    if (t < G::CS) {
      const int ly = t / G::PX, lx = t - ly * G::PX;
      const int gx = map_index(x0 + lx - G::H, A.n[0], A.periodic[0]);
      const int gy = map_index(y0 + ly - G::H, A.n[1], A.periodic[1]);
      const long long q = ((long long)kw * A.n[1] + gy) * A.n[0] + gx;
#pragma unroll
      for (int c = 0; c < 5; ++c) f.w[i][c] = A.Us[q + c * A.N];
    }
  }
  const bool gzout = !A.periodic[2] && (gzm < 0 || gzm >= A.n[2]);
  const int km = map_index(gzm, A.n[2], A.periodic[2]);
#pragma unroll
  for (int i = 0; i < F::PM; ++i) {
    const int t = threadIdx.x + i * NT;
    if (t < G::MCS) {
      const int ly = t / G::MPX, lx = t - ly * G::MPX;
      const int rx = x0 + lx - 1, ry = y0 + ly - 1;
      f.ghost[i] = gzout || (!A.periodic[0] && (rx < 0 || rx >= A.n[0])) ||
                   (!A.periodic[1] && (ry < 0 || ry >= A.n[1]));
      const int gx = map_index(rx, A.n[0], A.periodic[0]);
      const int gy = map_index(ry, A.n[1], A.periodic[1]);
      const long long q = ((long long)km * A.n[1] + gy) * A.n[0] + gx;
#pragma unroll
      for (int c = 0; c < 5; ++c) f.m[i][c] = f.ghost[i] ? T(0) : A.lam[q + c * A.N];
    }
  }
}

// uneven: whether a value of the m plane differs from mref.
template <typename T, bool VISC, int BX, int BY, int NT>
__device__ __forceinline__ void vjp3_commit(const VjpArgs<T>& A, const Gas<T>& g, const V3Fetch<T, VISC, BX, BY, NT>& f,
                                            T* dstw, T* dstm, const T* mref, bool& bad, bool& uneven) {
  using G = V3Geo<BX, BY, VISC>;
  using F = V3Fetch<T, VISC, BX, BY, NT>;
#pragma unroll
  for (int i = 0; i < F::PW; ++i) {
    const int t = threadIdx.x + i * NT;
    if (t < G::CS) {
      const T r = f.w[i][0];
      const T inv = trcp(r);
      const T u = f.w[i][1] * inv, v = f.w[i][2] * inv, w = f.w[i][3] * inv;
      const T p = g.gm1 * (f.w[i][4] - T(0.5) * r * (u * u + v * v + w * w));
      bad |= !(r > T(0)) || !(p > T(0));
      dstw[t] = r;
      dstw[G::CS + t] = u;
      dstw[2 * G::CS + t] = v;
      dstw[3 * G::CS + t] = w;
      dstw[4 * G::CS + t] = p;
      if (VISC) dstw[5 * G::CS + t] = p * inv * g.inv_R;
    }
  }
#pragma unroll
  for (int i = 0; i < F::PM; ++i) {
    const int t = threadIdx.x + i * NT;
    if (t < G::MCS) {
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        const T m = f.ghost[i] ? T(0) : A.s_in * f.m[i][c];
        dstm[c * G::MCS + t] = m;
        uneven |= !(m - mref[c] == T(0));
      }
    }
  }
}

// Accumulator slot src (plane gz, unmapped) added to Gacc and cleared: a
// thread per plane cell maps the cell once and adds its components.
template <typename T, bool VISC, int BX, int BY, int NT>
__device__ __forceinline__ void vjp3_flush(const VjpArgs<T>& A, T* src, T* __restrict__ Gacc, int x0, int y0,
                                           int gz) {
  using G = V3Geo<BX, BY, VISC>;
  const int kz = map_index(gz, A.n[2], A.periodic[2]);
  for (int t = threadIdx.x; t < G::CS; t += NT) {
    const int ly = t / G::PX, lx = t - ly * G::PX;
    const int gx = map_index(x0 + lx - G::H, A.n[0], A.periodic[0]);
    const int gy = map_index(y0 + ly - G::H, A.n[1], A.periodic[1]);
    const long long q = ((long long)kz * A.n[1] + gy) * A.n[0] + gx;
#pragma unroll
    for (int c = 0; c < G::NCW; ++c) {
      const T v = src[c * G::CS + t];
      if (v != T(0)) {
        atomicAdd(Gacc + (long long)c * A.N + q, v);
        src[c * G::CS + t] = T(0);
      }
    }
  }
}

// The face reverse passes.  blockDim.x == NT; grid = (ceil(nx/BX),
// ceil(ny/BY), ceil(nz/zchunk)).  Gacc [NCW][N] must be zero on entry.
template <typename T, bool VISC, int BX, int BY, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    vjp3_kernel(const VjpArgs<T> A, const Gas<T> g, T* __restrict__ Gacc, int zchunk) {
  using G = V3Geo<BX, BY, VISC>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  follow_predecessor<sizeof(T) == 4>();
  T* Wr = reinterpret_cast<T*>(smem_raw);  // [RING][NCW][PY][PX]
  T* Ar = Wr + G::RING * G::PLANE;         // [ARING][NCW][PY][PX]
  T* Mr = Ar + G::ARING * G::PLANE;        // [2][5][MPY][MPX]
  T* Cxy = Mr + 2 * 5 * G::MCS;            // viscous: [7][PY][PX]
  T* Cz = Cxy + G::NXY * G::CS;            // viscous: [4 planes][4][BY][BX]
  T* EX = Cz + G::ZRING * G::NZ * G::ZC;   // [2][5][BY][BX+2]
  T* EY = EX + 10 * G::XS;                 // [2][5][BY+2][BX]
  T* EZ = EY + 10 * G::YS;                 // [2 planes][2][5][BY][BX]
  T* mref = EZ + 20 * G::ZC;               // m of the tile's first cell, plane z0
  const int nx = A.n[0], ny = A.n[1], nz = A.n[2];
  const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
  const int z0 = blockIdx.z * zchunk, z1 = min(z0 + zchunk, nz);
  const int ex = min(BX, nx - x0), ey = min(BY, ny - y0);
  // owned faces per row / column: the lower faces of the tile's cells, plus
  // the upper boundary face of the grid's last cell on a non-periodic axis;
  // the cells -1 .. f - 1 are beside them
  const int fx = ex + ((!A.periodic[0] && x0 + BX >= nx) ? 1 : 0);
  const int fy = ey + ((!A.periodic[1] && y0 + BY >= ny) ? 1 : 0);
  // task decoding divides by fx and ex (1 .. BX + 1): for d >= 2,
  // r / d = (r m_d) >> 32 with m_d = ceil(2^32 / d) < 2^32, exact for
  // r < 2^16 (the error r (m_d - 2^32/d) / 2^32 < 2^-16 stays below 1/d);
  // d = 1 keeps r (m = 0 flags it)
  auto recip = [](int d) { return d > 1 ? 0xffffffffu / (unsigned)d + 1u : 0u; };
  const unsigned mfx = recip(fx), mex = recip(ex);
  auto divu = [](int r, unsigned m) { return m ? (int)__umulhi((unsigned)r, m) : r; };
  const T inv_h[3] = {A.inv_h[0], A.inv_h[1], A.inv_h[2]};

  bool bad = false;
  for (int q = 0; q < G::RING; ++q)
    vjp3_load_w<T, VISC, BX, BY, NT>(A, g, Wr + q * G::PLANE, x0, y0, z0 - 3 + q, bad);
  for (int t = threadIdx.x; t < G::ARING * G::PLANE; t += NT) Ar[t] = T(0);
  for (int t = threadIdx.x; t < G::NXY * G::CS + G::ZRING * G::NZ * G::ZC; t += NT) Cxy[t] = T(0);
  // a plane over which m is uniform (no cotangent has reached it yet, say) has no
  // x or y face with one: live, live1 for the planes k and k + 1
  T first[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) first[c] = A.s_in * A.lam[((long long)z0 * ny + y0) * nx + x0 + c * A.N];
  bool uneven0 = false, uneven1 = false;
  vjp3_load_m<T, VISC, BX, BY, NT>(A, Mr, x0, y0, z0 - 1, first, uneven0);
  vjp3_load_m<T, VISC, BX, BY, NT>(A, Mr + 5 * G::MCS, x0, y0, z0, first, uneven1);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int c = 0; c < 5; ++c) mref[c] = first[c];
  }
  bool live = __syncthreads_or(uneven0), live1 = __syncthreads_or(uneven1);

  V3Tile<T, VISC, BX, BY> V;
  V.W = Wr;
  V.acc = Ar;
  V.M = Mr;
  V.cbxy = Cxy;
  V.cbz = Cz;
  // plane p sits in W slot (p - z0 + 3) mod 6, accumulator slot
  // (p - z0 + 3) mod 5, z-face cotangent slot (p - z0 + 2) mod 4
  auto zslot = [&](int p) { return ((p - z0 + 2) & 3) * G::NZ * G::ZC; };
  auto set_view = [&](int k) {
    const int q = k - z0 + 1;
#pragma unroll
    for (int z = -2; z <= 3; ++z) V.wp[z + 2] = (q + z + 2) % G::RING * G::PLANE;
#pragma unroll
    for (int z = -2; z <= 2; ++z) V.ap[z + 2] = (q + z + 2) % G::ARING * G::PLANE;
    V.mp[0] = (q & 1) * 5 * G::MCS;
    V.mp[1] = ((q + 1) & 1) * 5 * G::MCS;
#pragma unroll
    for (int z = -1; z <= 2; ++z) V.zp[z + 1] = zslot(k + z);
  };
  auto ez = [&](int k) { return EZ + ((k - z0 + 1) & 1) * 10 * G::ZC; };
  // transposed DC4 along x and y of the z-face cotangents of plane k + z into
  // its accumulator slot, plane cell t
  auto gather_z = [&](int t, int z) {
    const int ly = t / G::PX, lx = t - ly * G::PX, x = lx - G::H, y = ly - G::H;
    const T* src = Cz + V.zp[z + 1] + y * BX + x;
    const bool in_x = (unsigned)x < (unsigned)BX, in_y = (unsigned)y < (unsigned)BY;
    T w = T(0), u = T(0), v = T(0);
    if (in_y) { w += vjp3_pull(src, x, BX, 1); u = vjp3_pull(src + G::ZC, x, BX, 1); }
    if (in_x) { w += vjp3_pull(src + 2 * G::ZC, y, BY, BX); v = vjp3_pull(src + 3 * G::ZC, y, BY, BX); }
    T* dst = Ar + V.ap[z + 2] + t;
    if (in_y) dst[G::CS] += u;
    if (in_x) dst[2 * G::CS] += v;
    if (in_x || in_y) dst[3 * G::CS] += w;
  };
  auto face_nu = [&](auto dtag, const int* p, T nu[5]) -> bool {
    constexpr int d = decltype(dtag)::value;
    bool any = false;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      nu[c] = (V.m(c, p[0], p[1], p[2]) - V.m(c, p[0] + (d == 0), p[1] + (d == 1), p[2] + (d == 2))) * inv_h[d];
      any |= nu[c] != T(0);
    }
    return any;
  };
  auto conv = [&](auto dtag, int x, int y, T* rv, T* lv, int cs) {
    constexpr int d = decltype(dtag)::value;
    const Along<d> P{{x, y, 0}};
    T nu[5];
    if (face_nu(dtag, P.p, nu)) {
      conv_face<T, d>(V, P, nu, g, rv, lv, cs);
    } else {
#pragma unroll
      for (int c = 0; c < 5; ++c) rv[c * cs] = lv[c * cs] = T(0);
    }
  };
  auto visc = [&](auto dtag, int x, int y) {
    constexpr int d = decltype(dtag)::value;
    const Along<d> P{{x, y, 0}};
    T nu[5];
    if (!face_nu(dtag, P.p, nu)) return;
    ViscCot<T> o;
    visc_face<T, d, 3>(V, P, nu, g, inv_h, o);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      visc_add<T, d, 3>(
          o, q,
          [&](int c, T v) {
            if (d == 2 && q != 1 && !g.safe) V.add_own(c, x, y, q - 1, v);
            else V.add(c, P.x(q - 1), P.y(q - 1), P.z(q - 1), v);
          },
          [&](int e, int c, T v) { V.add_sep(d, e, c, P.x(q - 1), P.y(q - 1), P.z(q - 1), v); });
  };
  auto rev = [&](auto dtag, int x, int y, const T* e, int cs) {
    constexpr int d = decltype(dtag)::value;
    const Along<d> P{{x, y, 0}};
    T vb[5][5];
    cell_rev<T, d>(V, P, g.eps, e, e + 5 * cs, cs, vb);
#pragma unroll
    for (int n = 0; n < 5; ++n)
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        if (d == 2 && n != 2) V.add_own(c, x, y, n - 2, vb[n][c]);
        else V.add(c, P.x(n - 2), P.y(n - 2), P.z(n - 2), vb[n][c]);
      }
  };
  using X = std::integral_constant<int, 0>;
  using Y = std::integral_constant<int, 1>;
  using Z = std::integral_constant<int, 2>;
  const int ncol = ex * ey;
  // task r of a pass over the cells: first the tile's own cells along x, so
  // that a warp holds one row of a full tile, then `others`, then the rim
  // cells along x (-1, and ex on a boundary)
  auto x_task = [&](int r, int ncx, int others, int& j, int& i) -> bool {
    if (ncx == 0) return false;
    if (r < ncol) {
      j = divu(r, mex);
      i = r - j * ex;
      return true;
    }
    r -= ncol + others;
    if (r < 0) return false;
    i = r < ey ? -1 : ex;
    j = r < ey ? r : r - ey;
    return true;
  };

  // the upper values of the cells of plane z0 - 1
  set_view(z0 - 1);
  for (int t = threadIdx.x; t < ncol; t += NT) {
    const int j = divu(t, mex), i = t - j * ex;
    T* e = ez(z0 - 1) + j * BX + i;
    cell_fwd<T, 2>(V, Along<2>{{i, j, 0}}, g.eps, e, e + 5 * G::ZC, G::ZC);
  }
  // plane z0 - 1: its upper z face only, and at the bottom of a non-periodic
  // axis the ghost cells' reverse pass; at its top, plane nz: that of the
  // ghost cells above
  const bool bottom = !A.periodic[2] && z0 == 0, top = !A.periodic[2] && z1 == nz;
  const int kend = z1 + (top ? 1 : 0);
#pragma unroll 1
  for (int k = z0 - 1; k < kend; ++k) {
    set_view(k);
    const bool xy = k >= z0 && k < z1 && live;
    const int ncx = xy ? ey * (fx + 1) : 0, ncy = xy ? (fy + 1) * ex : 0, nzf = k < z1 ? ncol : 0;
    // pass 1: face values of the cells along x and y (plane k), z (plane k + 1)
    for (int t = threadIdx.x; t < ncx + ncy + nzf; t += NT) {
      int r = t, j, i;
      if (x_task(r, ncx, ncy + nzf, j, i)) {
        T* e = EX + j * G::XP + i + 1;
        cell_fwd<T, 0>(V, Along<0>{{i, j, 0}}, g.eps, e, e + 5 * G::XS, G::XS);
      } else if ((r -= ncx ? ex * ey : 0) < ncy) {
        const int j = divu(r, mex), i = r - j * ex;  // cell row j - 1
        T* e = EY + j * BX + i;
        cell_fwd<T, 1>(V, Along<1>{{i, j - 1, 0}}, g.eps, e, e + 5 * G::YS, G::YS);
      } else {
        r -= ncy;
        const int j = divu(r, mex), i = r - j * ex;
        T* e = ez(k + 1) + j * BX + i;
        cell_fwd<T, 2>(V, Along<2>{{i, j, 1}}, g.eps, e, e + 5 * G::ZC, G::ZC);
      }
    }
    __syncthreads();
    // pass 2: the faces; values become cotangents (a rim cell's other value,
    // whose face another CTA owns, gets none here)
    const int nfx = xy ? ey * fx : 0, nfy = xy ? fy * ex : 0;
    const int nconv = nfx + nfy + nzf;
    const int nvisc = !VISC ? 0 : (k >= z0 || bottom) ? nconv : 0;
    for (int t = threadIdx.x; t < nconv + nvisc; t += NT) {
      int r = t;
      const bool dissipative = VISC && r >= nconv;
      if (dissipative) r -= nconv;
      if (r < nfx) {  // x face: lower face of cell (x0 + f, y0 + j, k)
        const int j = divu(r, mfx), f = r - j * fx;
        if (dissipative) {
          if constexpr (VISC) visc(X{}, f - 1, j);
        } else {
          T* rv = EX + j * G::XP + f;
          T* lv = rv + 5 * G::XS;
          conv(X{}, f - 1, j, rv, lv + 1, G::XS);
          if (f == 0) {
#pragma unroll
            for (int c = 0; c < 5; ++c) lv[c * G::XS] = T(0);
          }
          if (f == fx - 1) {
#pragma unroll
            for (int c = 0; c < 5; ++c) rv[c * G::XS + 1] = T(0);
          }
        }
      } else if ((r -= nfx) < nfy) {  // y face: lower face of cell (x0 + i, y0 + f, k)
        const int f = divu(r, mex), i = r - f * ex;
        if (dissipative) {
          if constexpr (VISC) visc(Y{}, i, f - 1);
        } else {
          T* rv = EY + f * BX + i;
          T* lv = rv + 5 * G::YS;
          conv(Y{}, i, f - 1, rv, lv + BX, G::YS);
          if (f == 0) {
#pragma unroll
            for (int c = 0; c < 5; ++c) lv[c * G::YS] = T(0);
          }
          if (f == fy - 1) {
#pragma unroll
            for (int c = 0; c < 5; ++c) rv[c * G::YS + BX] = T(0);
          }
        }
      } else {  // z face k + 1/2
        r -= nfy;
        const int j = divu(r, mex), i = r - j * ex, o = j * BX + i;
        if (dissipative) {
          if constexpr (VISC) visc(Z{}, i, j);
        } else {
          T* rv = ez(k) + o;
          T* lv = ez(k + 1) + 5 * G::ZC + o;
          conv(Z{}, i, j, rv, lv, G::ZC);
          if (bottom && k == z0 - 1) {
#pragma unroll
            for (int c = 0; c < 5; ++c) rv[(5 + c) * G::ZC] = T(0);
          }
          if (top && k == z1 - 1) {
#pragma unroll
            for (int c = 0; c < 5; ++c) lv[(c - 5) * G::ZC] = T(0);
          }
        }
      }
    }
    __syncthreads();
    // W of plane k + 4 (the slot of plane k - 2, last read by the pass below)
    // and m of plane k + 2 in flight meanwhile
    V3Fetch<T, VISC, BX, BY, NT> nxt;
    const bool more = k + 1 < kend;
    if (more) vjp3_fetch<T, VISC, BX, BY, NT>(A, nxt, x0, y0, k + 4, k + 2);
    // pass 3: reverse reconstruction of the cells
    const int nz3 = (k >= z0 && k < z1) || k == nz || (bottom && k < z0) ? ncol : 0;
    for (int t = threadIdx.x; t < ncx + ncy + nz3; t += NT) {
      int r = t, j, i;
      if (x_task(r, ncx, ncy + nz3, j, i)) {
        rev(X{}, i, j, EX + j * G::XP + i + 1, G::XS);
      } else if ((r -= ncx ? ex * ey : 0) < ncy) {
        const int j = divu(r, mex), i = r - j * ex;
        rev(Y{}, i, j - 1, EY + j * BX + i, G::YS);
      } else {
        r -= ncy;
        const int j = divu(r, mex), i = r - j * ex;
        const T* e = ez(k) + j * BX + i;
        bool any = false;  // a z face with a cotangent beside it
#pragma unroll
        for (int c = 0; c < 10; ++c) any |= e[c * G::ZC] != T(0);
        if (any) rev(Z{}, i, j, e, G::ZC);
      }
    }
    __syncthreads();
    if constexpr (VISC) {
      // the transposed DC4 of the x and y faces' centre-derivative cotangents
      // (along y and x into plane k, along z into the planes k -+ 1, 2) and of
      // the z faces' of plane k - 1, which are complete; a thread per cell
      for (int r = threadIdx.x; r < G::CS; r += NT) {
        if (xy) {
          const int ly = r / G::PX, lx = r - ly * G::PX;
          T* a0 = Ar + V.ap[2] + r;
          const T* c = Cxy + r;
          a0[G::CS] += vjp3_pull(c, ly, G::PY, G::PX) + vjp3_pull(c + 2 * G::CS, lx, G::PX, 1);
          a0[2 * G::CS] += vjp3_pull(c + G::CS, ly, G::PY, G::PX) + vjp3_pull(c + 3 * G::CS, lx, G::PX, 1);
          constexpr int dco[4] = {-2, -1, 1, 2};
          constexpr T dcw[4] = {T(1) / T(12), -T(8) / T(12), T(8) / T(12), -T(1) / T(12)};
          const T zu = c[4 * G::CS], zv = c[5 * G::CS], zw = c[6 * G::CS];
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            T* ao = Ar + V.ap[dco[o] + 2] + r;
            ao[G::CS] += dcw[o] * zu;
            ao[2 * G::CS] += dcw[o] * zv;
            ao[3 * G::CS] += dcw[o] * zw;
          }
        }
        gather_z(r, -1);
      }
      __syncthreads();
      for (int t = threadIdx.x; t < G::NXY * G::CS; t += NT) Cxy[t] = T(0);
      T* cz = Cz + V.zp[0];  // plane k - 1 becomes plane k + 3
      for (int t = threadIdx.x; t < G::NZ * G::ZC; t += NT) cz[t] = T(0);
    }
    // plane k - 2 is complete: add it to the global accumulator; its slots
    // take the planes k + 3 (cleared accumulator) and k + 4 (W), and the m slot
    // of plane k takes plane k + 2
    vjp3_flush<T, VISC, BX, BY, NT>(A, Ar + V.ap[0], Gacc, x0, y0, k - 2);
    bool uneven = false;
    if (more) vjp3_commit<T, VISC, BX, BY, NT>(A, g, nxt, Wr + V.wp[0], Mr + V.mp[0], mref, bad, uneven);
    live = live1;
    live1 = __syncthreads_or(uneven);
  }
  // the z-face cotangents still held, then the planes still held: kend - 2 ..
  // kend + 1 (the view is plane kend - 1's)
  if constexpr (VISC) {
    for (int t = threadIdx.x; t < 3 * G::CS; t += NT) {
      const int z = t / G::CS, r = t - z * G::CS;
      if (z == 0) gather_z(r, 0);
      else if (z == 1) gather_z(r, 1);
      else gather_z(r, 2);
    }
    __syncthreads();
  }
#pragma unroll
  for (int z = -1; z <= 2; ++z)
    vjp3_flush<T, VISC, BX, BY, NT>(A, Ar + V.ap[z + 2], Gacc, x0, y0, kend - 1 + z);
  if (bad) atomicOr(A.flag, 1);
}

// Per cell: cotangent of W (+T) in Gacc -> cotangent of U (transposed
// Jacobian of W(U), and of T = p / (rho R)), then
// out = m + dt J^T m + a1 x1 + a2 x2.
template <typename T, bool VISC>
__global__ void __launch_bounds__(256) vjp3_finish_kernel(const VjpArgs<T> A, const Gas<T> g,
                                                          const T* Gacc) {
  follow_predecessor<sizeof(T) == 4>();
  const long long N = A.N;
  const T dt = T(*A.dt);
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < N; q += (long long)gridDim.x * blockDim.x) {
    const T r = A.Us[q];
    const T inv = trcp(r);
    const T u = A.Us[q + N] * inv, v = A.Us[q + 2 * N] * inv, w = A.Us[q + 3 * N] * inv;
    const T p = g.gm1 * (A.Us[q + 4 * N] - T(0.5) * r * (u * u + v * v + w * w));
    T br = Gacc[q], bu = Gacc[q + N], bv = Gacc[q + 2 * N], bw = Gacc[q + 3 * N], bp = Gacc[q + 4 * N];
    if (VISC) {
      const T bT = Gacc[q + 5 * N];
      const T Tc = p * inv * g.inv_R;
      br -= bT * Tc * inv;  // T = p / (rho R)
      bp += bT * Tc * trcp(p);
    }
    T bU[5];
    bU[0] = br - (bu * u + bv * v + bw * w) * inv + bp * g.gm1 * T(0.5) * (u * u + v * v + w * w);
    bU[1] = bu * inv - bp * g.gm1 * u;
    bU[2] = bv * inv - bp * g.gm1 * v;
    bU[3] = bw * inv - bp * g.gm1 * w;
    bU[4] = bp * g.gm1;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      T o = A.s_in * A.lam[q + c * N] + dt * bU[c];
      if (A.x1) o += A.a1 * A.x1[q + c * N];
      if (A.x2) o += A.a2 * A.x2[q + c * N];
      A.out[q + c * N] = o;
    }
  }
}

}  // namespace jf
