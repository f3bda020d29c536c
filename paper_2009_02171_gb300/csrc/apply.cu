// Tiled matrix-free operator apply y = A x for VTBE and PPBE (paper eqn:divdiscretization with the
// operators of eqn:tsvelocity, eqn:tstemperature, eqn:tsmag, eqn:tsp, eqn:tspb).
//
// Per cell and component the Laplacian is (1/V) sum_faces F.  The horizontal faces give a 9-point stencil
// whose weights depend only on (j, i): the angular metric is the same on every panel and level, and h_r is
// folded in.  A face on a panel edge carries the mean of the two panels' one-sided fluxes (reading R3); with
// the panel-edge ghosts expanded into their interpolation sources that flux is a fixed linear combination
// of cell values of the same level on two or three panels, tabulated once per grid (build_edge_table).
// The radial faces give a 3-point stencil r_f^2 sigma h_s^2 / h_r (x_{k+1} - x_k) with the wall ghost rules.
//
// One launch, one CTA per (coupled component group, panel, tile of (j, i), chunk of levels k).  Groups: VTBE
// {u_x, u_y, u_z, Theta} (Coriolis, buoyancy and r . u couple them at a cell) and {B_x, B_y, B_z} (the
// pseudo-vacuum wall rule couples them); PPBE {P, P_b}.  A thread owns 16 bytes of consecutive i of one row and
// marches k; the CTA keeps a ring of four planes of its components in shared memory, each own 16 bytes copied by
// one cp.async two levels ahead, halo cells across a panel edge the quadratic ghost interpolants.  Every x value is
// read from HBM once (plus the planes at chunk boundaries) and every y value is written once.
// What bounds it: FP64 its multiply-adds (16 cycles of the SM's FP64 pipe each); FP32 the instructions issued.  So
// the nine horizontal weights and the radial weight carry 1 / sigma in their tables (14 multiply-adds a value and
// level), weights, metric and couplings are shared by a group's components in registers, and shared memory is read
// 16 bytes at a time.  The panel-edge fluxes of a tile are copied beside its planes: as loads behind per-cell tests
// they were 2/3 of the instructions (every warp of a 64-cell panel has an edge lane).
// Against one CTA a component with four rows a thread, both launches, us on GB300: FP64 VTBE 6x64^3 640 -> 517 (FP64
// pipe), PPBE 6x45^2x39 120 -> 62; FP32 VTBE 6x128^2x96 627 -> 353, 6x64^3 134 -> 93, PPBE 6x32^3 25 -> 14.  The tables'
// products are taken in FP64 and rounded once (as FP32 products here the error against 64 bits was above that of
// the earlier kernel: PPBE 6x33^2x17 9.1e-8, then 8.6e-8, now 8.4e-8; VTBE 6x128^2x96 5.0e-8, 5.0e-8, 4.8e-8).
#include <algorithm>
#include <cstdint>
#include <mutex>
#include <vector>

#include "stencil.cuh"

namespace fv {

constexpr int EDGE_BATCH = 12;  // terms read at once: a face has 11 at most on every grid so far
constexpr int EDGE_TERMS = 40;  // bound on the terms of one panel-edge face flux (checked when tabulated)
constexpr int RING = 4;         // planes of the tile ring: levels k - 1 .. k + 2

// tile extents of a grid: ti x tj cells (ti a multiple of the cells a thread owns), at most 32 wide and as many rows
// as the CTA's threads cover, both split evenly over the panel so that a ragged panel leaves few threads idle
struct Tiles {
  int ti, tj, nti, ntj, kchunk, vec;
  long long xs, ys;  // strides of a right-hand side in x and y (grid z = right-hand side * 6 + panel)
};
template <class T>
struct TileT;
template <class T>
__host__ __device__ inline int plane_values(const Tiles& td) {
  constexpr int CPT = 16 / sizeof(T);
  const int tja = (td.tj + CPT - 1) / CPT * CPT;
  return (td.tj + 2) * (td.ti + 2 * CPT) + 2 * tja + 2 * td.ti + CPT;
}
template <class T>
struct TileT {
  static constexpr int CPT = 16 / sizeof(T);                  // cells a thread owns
  static constexpr int THREADS = sizeof(T) == 8 ? 256 : 128;  // 32 x 16 cells
  static constexpr int PAD = CPT;                             // columns left of the tile (the last is its halo)
};

template <class R>
struct EdgeTab {
  const int* cnt;
  const int* off;
  const R* w;
};

// ------------------------------------------------------------------ panel-edge face table
// Records the terms of a face flux as (cell offset within a level, weight), ghosts expanded into their
// interpolation sources (cube-corner ghosts: phi(-1,-1) = phi(-1,0) + phi(0,-1) - phi(0,0)).
struct RecordAcc {
  const Geo* G;
  int n;
  int bad;
  int off[EDGE_TERMS];
  double w[EDGE_TERMS];
  __device__ void cell(double c, int p, int, int j, int i, int) {
    const int o = (p * G->Nr * G->Ns + j) * G->Ns + i;
    for (int m = 0; m < n; ++m)
      if (off[m] == o) {
        w[m] += c;
        return;
      }
    if (n == EDGE_TERMS) {
      bad = 1;
      return;
    }
    off[n] = o, w[n] = c, ++n;
  }
  __device__ void interp(double c, int p, int side, int t) {
    const int Ns = G->Ns, id = (p * 4 + side) * Ns + t, q = G->gq[id];
    for (int m = 0; m < 3; ++m) {
      const int src = G->gsrc[3 * id + m];
      cell(c * G->gw[3 * id + m], q, 0, src / Ns, src % Ns, 0);
    }
  }
  __device__ void ghost(double c, int p, int side, int, int t, int) {
    const int Ns = G->Ns;
    if (t >= 0 && t < Ns) {
      interp(c, p, side, t);
    } else {
      const int jin = t < 0 ? 0 : Ns - 1, iin = side == XI_MIN ? 0 : Ns - 1;
      interp(c, p, side, jin);
      interp(c, p, t < 0 ? ETA_MIN : ETA_MAX, iin);
      cell(-c, p, 0, jin, iin, 0);
    }
  }
};

// one thread per panel-edge face f = (p, side, t): cnt[f], then the terms in term-major slots
// (off[m * nf + f], wt[m * nf + f]), so that neighbouring faces read neighbouring slots
__global__ void edge_table_kernel(Geo G, int* __restrict__ cnt, int* __restrict__ off, double* __restrict__ wt,
                                  int* __restrict__ status) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int nf = 24 * G.Ns;
  if (e >= nf) return;
  const int ps = e / G.Ns, t = e % G.Ns;
  RecordAcc acc;
  acc.G = G.self, acc.n = 0, acc.bad = 0;
  edge_flux(*G.self, acc, 1.0, ps / 4, ps % 4, 0, t, 0);
  if (acc.bad) atomicExch(status, 1);
  int n = 0;
  for (int m = 0; m < acc.n; ++m)  // drop terms that cancelled exactly
    if (acc.w[m] != 0.0) off[n * nf + e] = acc.off[m], wt[n * nf + e] = acc.w[m], ++n;
  cnt[e] = n;
  for (; n < EDGE_BATCH; ++n) off[n * nf + e] = off[e], wt[n * nf + e] = 0.0;  // the first batch is read whole
}

__global__ void to_float_kernel(const double* __restrict__ a, float* __restrict__ b, int n) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) b[e] = (float)a[e];
}

fv_status build_edge_table(fv_grid* g) {
  const int nf = 24 * g->h.Ns;
  int *cnt = nullptr, *off = nullptr, *status = nullptr;
  double* wt = nullptr;
  float* wtf = nullptr;
  FV_CUDA(cudaMalloc(&cnt, nf * sizeof(int)));
  g->allocs.push_back(cnt);
  FV_CUDA(cudaMalloc(&off, (size_t)nf * EDGE_TERMS * sizeof(int)));
  g->allocs.push_back(off);
  FV_CUDA(cudaMalloc(&wt, (size_t)nf * EDGE_TERMS * sizeof(double)));
  g->allocs.push_back(wt);
  FV_CUDA(cudaMalloc(&wtf, (size_t)nf * EDGE_TERMS * sizeof(float)));
  g->allocs.push_back(wtf);
  FV_CUDA(cudaMalloc(&status, sizeof(int)));
  FV_CUDA(cudaMemset(status, 0, sizeof(int)));
  edge_table_kernel<<<(nf + 63) / 64, 64>>>(g->geo, cnt, off, wt, status);
  FV_CUDA(cudaGetLastError());
  to_float_kernel<<<(nf * EDGE_TERMS + 255) / 256, 256>>>(wt, wtf, nf * EDGE_TERMS);
  FV_CUDA(cudaGetLastError());
  int bad = 0;
  FV_CUDA(cudaMemcpy(&bad, status, sizeof(int), cudaMemcpyDeviceToHost));
  cudaFree(status);
  if (bad) return set_error("fv_build_grid: a panel-edge face flux has more terms than the table holds"), FV_EINVAL;
  g->edge_cnt = cnt, g->edge_off = off, g->edge_w = wt, g->edge_wf = wtf;
  return FV_OK;
}

// ------------------------------------------------------------------ tiled apply

// E[(c Nr + k) 24 Ns + f] = flux through panel-edge face f = (p, side, t) at level k, component c, measured
// along p's coordinate: one thread per (level, face); each term's slot is read once for all components.  Bound by
// latency: all slots of the first EDGE_BATCH terms are in flight together, then all their cell values (four terms a
// round trip behind the term count took 8.6 us on the coarse level's 6x32^3, of which 3 are the launch's).
template <int D, class T>
__global__ void __launch_bounds__(128) edge_flux_kernel(int Ns, int Nr, EdgeTab<T> et, const T* __restrict__ x,
                                                        long long xs, T* __restrict__ E) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the tiles' set-up runs beside this
  const int nf = 24 * Ns, N = 6 * Nr * Ns * Ns;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nf * Nr) return;
  x += blockIdx.y * xs, E += blockIdx.y * (long long)D * Nr * nf;
  const int f = e % nf, k = e / nf;
  const T* xk = x + k * Ns * Ns;
  int o[EDGE_BATCH];
  T w[EDGE_BATCH];
#pragma unroll
  for (int u = 0; u < EDGE_BATCH; ++u) o[u] = et.off[u * nf + f], w[u] = et.w[u * nf + f];
  const int n = et.cnt[f];
#pragma unroll
  for (int c = 0; c < D; ++c) {
    T v[EDGE_BATCH], acc = T(0);
#pragma unroll
    for (int u = 0; u < EDGE_BATCH; ++u) v[u] = xk[c * N + o[u]];
#pragma unroll
    for (int u = 0; u < EDGE_BATCH; ++u) acc = fma(w[u], w[u] != T(0) ? v[u] : T(0), acc);
    for (int m = EDGE_BATCH; m < n; ++m) acc = fma(et.w[m * nf + f], xk[c * N + et.off[m * nf + f]], acc);
    E[(c * Nr + k) * nf + f] = acc;
  }
}

template <class T>
__device__ __forceinline__ void async_copy(unsigned dst, const T* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(sizeof(T)) : "memory");
}
__device__ __forceinline__ void async_copy16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// CPT values at a 16-byte aligned address
template <class T>
struct Vals;
template <>
struct Vals<float> {
  __device__ __forceinline__ static void load(const float* p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
  }
  __device__ __forceinline__ static void store(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct Vals<double> {
  __device__ __forceinline__ static void load(const double* p, double (&v)[2]) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    v[0] = q.x, v[1] = q.y;
  }
  __device__ __forceinline__ static void store(double* p, const double (&v)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
};

// the rotation of panel p applied to a local vector: entries in {-1, 0, 1}, so selections and signs, no arithmetic
template <class R>
__device__ __forceinline__ void rotate_exact(int p, const R (&l)[3], R (&v)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int m0 = kPM[p][3 * a], m1 = kPM[p][3 * a + 1], m2 = kPM[p][3 * a + 2];
    const R t = m0 ? l[0] : (m1 ? l[1] : l[2]);
    v[a] = m0 + m1 + m2 < 0 ? -t : t;
  }
}

// components C0 .. C0 + NG - 1 of one tile and level chunk: y = A x, or y = b - A x when b is given
template <int KIND, int C0, int NG, class T, class GT>
__device__ __forceinline__ void tile_body(const GT& G, const Coefs<T>& cf, const Tiles& td, int tile, const T* __restrict__ x,
                                          const T* __restrict__ b, T* __restrict__ y, const T* __restrict__ E) {
  constexpr int CPT = TileT<T>::CPT, PAD = TileT<T>::PAD;
  constexpr bool UT = KIND == FV_VTBE && C0 == 0, BG = KIND == FV_VTBE && C0 == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* const sh = reinterpret_cast<T*>(smem_raw);
  const int Ns = G.Ns, Nr = G.Nr, Ns2 = Ns * Ns, NP = Nr * Ns2, N = 6 * NP;
  const int i0 = tile % td.nti * td.ti, j0 = tile / td.nti * td.tj, p = blockIdx.z % 6, rhs = blockIdx.z / 6;
  const int wi = min(td.ti, Ns - i0), wj = min(td.tj, Ns - j0);  // cells of this tile
  const int kb = blockIdx.y * td.kchunk, ke = min(Nr, kb + td.kchunk);
  const int pitch = td.ti + 2 * PAD, PL = (td.tj + 2) * pitch;
  // a component's plane, then the fluxes through the tile's panel-edge faces: xi-min, xi-max rows, eta-min, eta-max
  // columns, and a zero
  const int tja = (td.tj + CPT - 1) / CPT * CPT, CS = plane_values<T>(td), SLOT = NG * CS;
  const int tid = threadIdx.x, gpr = td.ti / CPT, row = tid / gpr, ig = (tid - row * gpr) * CPT;
  const bool act = row < wj && ig < wi;
  const int own = act ? (j0 + row) * Ns + i0 + ig : 0;  // first own cell within a level
  const int pos = (row + 1) * pitch + PAD + ig;
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(sh);
  const bool vec = td.vec;
  x += rhs * td.xs + C0 * N, y += rhs * td.ys + C0 * N;
  E += (long long)rhs * (KIND == FV_VTBE ? 7 : 2) * Nr * 24 * Ns;
  if (b) b += C0 * N;

  // halo cell of this thread: a cell of the panel (one source), a panel-edge ghost (its three interpolation
  // sources), or nothing (cube corners: zero, no weight reads them)
  int hmode = 0, hpos = 0, spos = 0, eoff = -1, ho[3] = {0, 0, 0};
  T hw[3] = {T(0), T(0), T(0)};
  if (tid < 2 * wj + 2 * (wi + 2)) {
    int hj, hi;
    if (tid < wj) hj = tid, hi = -1;
    else if (tid < 2 * wj) hj = tid - wj, hi = wi;
    else if (tid < 2 * wj + wi + 2) hj = -1, hi = tid - 2 * wj - 1;
    else hj = wj, hi = tid - 2 * wj - wi - 3;
    hpos = (hj + 1) * pitch + PAD + hi;
    const int j = j0 + hj, i = i0 + hi;
    const bool in_i = i >= 0 && i < Ns, in_j = j >= 0 && j < Ns;
    int side = -1, t = 0;
    if (in_i && in_j) ho[0] = p * NP + j * Ns + i, hmode = 1;
    else if (in_j) side = i < 0 ? XI_MIN : XI_MAX, t = j;
    else if (in_i) side = j < 0 ? ETA_MIN : ETA_MAX, t = i;
    if (side >= 0) {
      const int id = (p * 4 + side) * Ns + t, q = G.gq[id];
      hmode = 3;
#pragma unroll
      for (int m = 0; m < 3; ++m) ho[m] = q * NP + G.gsrc[3 * id + m], hw[m] = G.gw[3 * id + m];
      // the face between this ghost and the tile's cell (a ghost beyond a corner of the tile has none here)
      if (side < 2 ? hj >= 0 && hj < wj : hi >= 0 && hi < wi) {
        eoff = (p * 4 + side) * Ns + t;
        spos = PL + (side < 2 ? side * tja + hj : 2 * tja + (side - 2) * td.ti + hi);
      }
    }
    if (hmode == 0)
      for (int s = 0; s < RING * NG; ++s) sh[s * CS + hpos] = T(0);
  }
  if (tid < CPT)
    for (int s = 0; s < RING * NG; ++s) sh[s * CS + PL + 2 * tja + 2 * td.ti + tid] = T(0);
  // level k into its slot: own cells and panel halo cells by asynchronous copies
  auto copy_level = [&](int k) {
    const unsigned slot = sbase + (unsigned)((k & (RING - 1)) * SLOT * sizeof(T));
    const T* xk = x + k * Ns2;
    if (act) {
#pragma unroll
      for (int c = 0; c < NG; ++c) {
        const T* src = xk + c * N + p * NP + own;
        const unsigned dst = slot + (unsigned)((c * CS + pos) * sizeof(T));
        if (vec) {
          async_copy16(dst, src);
        } else {
#pragma unroll
          for (int m = 0; m < CPT; ++m)
            if (ig + m < wi) async_copy(dst + m * sizeof(T), src + m);
        }
      }
    }
    if (hmode == 1)
#pragma unroll
      for (int c = 0; c < NG; ++c) async_copy(slot + (unsigned)((c * CS + hpos) * sizeof(T)), xk + c * N + ho[0]);
    if (eoff >= 0)
#pragma unroll
      for (int c = 0; c < NG; ++c)
        async_copy(slot + (unsigned)((c * CS + spos) * sizeof(T)), E + ((C0 + c) * Nr + k) * 24 * Ns + eoff);
  };
  T hv[NG];
  auto ghost_values = [&](int k) {
    const T* xk = x + k * Ns2;
    if (hmode == 3)
#pragma unroll
      for (int c = 0; c < NG; ++c) hv[c] = hw[0] * xk[c * N + ho[0]] + hw[1] * xk[c * N + ho[1]] + hw[2] * xk[c * N + ho[2]];
  };
  auto ghost_store = [&](int k) {
    if (hmode == 3)
#pragma unroll
      for (int c = 0; c < NG; ++c) sh[(k & (RING - 1)) * SLOT + c * CS + hpos] = hv[c];
  };
  // per-cell constants: weights over sigma, unit radius vector
  T w[CPT][9], rh[CPT][3];
#pragma unroll
  for (int m = 0; m < CPT; ++m) {
    const int ji = act && ig + m < wi ? own + m : 0;
#pragma unroll
    for (int q = 0; q < 9; ++q) w[m][q] = G.w9[9 * ji + q];
    if constexpr (KIND == FV_VTBE) {
      const T xl[3] = {G.xhat[3 * ji], G.xhat[3 * ji + 1], G.xhat[3 * ji + 2]};
      rotate_exact(p, xl, rh[m]);
    }
  }
  const int i = i0 + ig, j = j0 + row;
  // panel-edge faces: + flux at the max sides, - at the min sides.  xi: at most the first or the last cell of the
  // thread has one, every thread reads its row's place (the zero where it has none); eta: whole rows
  const bool xmin = act && i == 0, xmax = act && i + CPT >= Ns;
  const int xat = PL - pos + (xmin ? row : xmax ? tja + row : 2 * tja + 2 * td.ti);
  const int last = xmax ? Ns - 1 - i : CPT - 1;
  const bool both = xmin && xmax;  // a row of one thread: the max side is added apart
  const T ex = xmin ? -G.invsig[own] : xmax ? G.invsig[own + last] : T(0);
  const int xcell = xmin ? 0 : last;
  const bool jmin = act && j == 0, jmax = act && j == Ns - 1;
  const int jat = PL - pos + 2 * tja + ig;

  const int kl = min(ke, Nr - 1);  // last level the chunk reads
  // the launch overlaps the edge-flux kernel (which itself began after all earlier work): its results from here on
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int k = max(kb - 1, 0); k <= min(kb + 1, kl); ++k) copy_level(k), ghost_values(k), ghost_store(k);

  const T r2v = cf.r2 * (G.hs * G.hs * G.hr);  // invr2 = 1 / (r^2 h_s^2 h_r)
  for (int k = kb; k < ke; ++k) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // level k + 1 has landed, level k - 2 is no longer read
    const bool more = k + 2 <= kl;
    if (more) copy_level(k + 2), ghost_values(k + 2);
    if (act) {
      const T* s0 = sh + (k & (RING - 1)) * SLOT + pos;
      const T* sm = sh + ((k - 1) & (RING - 1)) * SLOT + pos;
      const T* sp = sh + ((k + 1) & (RING - 1)) * SLOT + pos;
      const T q = G.invr2[k], rb = G.rf2[k], rt = G.rf2[k + 1], rk = G.rc[k];
      const T r1k = UT ? cf.r1 * rk : T(0), b2 = UT ? r2v * q : T(0);  // r_1 r_k, r_2 / r_k^2
      T rdot[CPT], thk[CPT];  // r_hat . u or (at a wall) r_hat . B; r_1 r_k Theta
      if (UT || (BG && (k == 0 || k == Nr - 1))) {
        T a0[CPT], a1[CPT], a2[CPT], a3[CPT];
        Vals<T>::load(s0, a0), Vals<T>::load(s0 + CS, a1), Vals<T>::load(s0 + (NG > 2 ? 2 : 0) * CS, a2);
        if constexpr (UT) Vals<T>::load(s0 + (NG - 1) * CS, a3);
#pragma unroll
        for (int m = 0; m < CPT; ++m) {
          rdot[m] = rh[m][0] * a0[m] + rh[m][1] * a1[m] + rh[m][2] * a2[m];
          if constexpr (UT) thk[m] = r1k * a3[m];
        }
      }
      // FP64 keeps one component's code (4 to 8 % faster: registers), FP32 all of them
#pragma unroll(sizeof(T) == 8 ? 1 : NG)
      for (int c = 0; c < NG; ++c) {
        T x0[CPT], up[CPT], dn[CPT], lo[CPT], hi[CPT], h[CPT];
        Vals<T>::load(s0 + c * CS, x0);
        // wall rule of this component: odd (-x), even (+x), pseudo-vacuum B: -B + fac (B . r_hat) r_hat
        auto wall = [&](T fac, T (&g)[CPT]) {
#pragma unroll
          for (int m = 0; m < CPT; ++m) {
            g[m] = KIND == FV_PPBE && c == 0 ? x0[m] : -x0[m];
            if constexpr (BG) g[m] += fac * rdot[m] * (c == 0 ? rh[m][0] : c == 1 ? rh[m][1] : rh[m][2]);
          }
        };
        if (k + 1 < Nr) Vals<T>::load(sp + c * CS, up);
        else wall(G.wall_out, up);
        if (k > 0) Vals<T>::load(sm + c * CS, dn);
        else wall(G.wall_in, dn);
        const T* v = s0 + c * CS;
        Vals<T>::load(v - pitch, lo);
        Vals<T>::load(v + pitch, hi);
        const T l0 = v[-pitch - 1], l1 = v[-1], l2 = v[pitch - 1], r0 = v[-pitch + CPT], r1 = v[CPT], r2 = v[pitch + CPT];
#pragma unroll
        for (int m = 0; m < CPT; ++m) {
          T a = w[m][0] * (m ? lo[m ? m - 1 : 0] : l0);
          a = fma(w[m][1], lo[m], a);
          a = fma(w[m][2], m + 1 < CPT ? lo[m + 1 < CPT ? m + 1 : 0] : r0, a);
          a = fma(w[m][3], m ? x0[m ? m - 1 : 0] : l1, a);
          a = fma(w[m][4], x0[m], a);
          a = fma(w[m][5], m + 1 < CPT ? x0[m + 1 < CPT ? m + 1 : 0] : r1, a);
          a = fma(w[m][6], m ? hi[m ? m - 1 : 0] : l2, a);
          a = fma(w[m][7], hi[m], a);
          h[m] = fma(w[m][8], m + 1 < CPT ? hi[m + 1 < CPT ? m + 1 : 0] : r2, a);
        }
        const T fx = v[xat];
        T hx = h[0];
#pragma unroll
        for (int m = 1; m < CPT; ++m) hx = m == xcell ? h[m] : hx;
        hx = fma(ex, fx, hx);
#pragma unroll
        for (int m = 0; m < CPT; ++m) h[m] = m == xcell ? hx : h[m];
        if (both) h[CPT - 1] = fma(G.invsig[own + last], v[PL - pos + tja + row], h[CPT - 1]);  // Ns = CPT: last = CPT - 1
        if (jmin | jmax) {
#pragma unroll
          for (int m = 0; m < CPT; ++m)
            if (ig + m < wi) {
              const T is = G.invsig[own + m];
              if (jmin) h[m] = fma(-is, v[jat + m], h[m]);
              if (jmax) h[m] = fma(is, v[jat + td.ti + m], h[m]);
            }
        }
        const T cd = q * (KIND == FV_PPBE ? cf.pp : (BG ? cf.hpm : (c == 3 ? cf.hpr : cf.h)));
        T out[CPT], uo[CPT];  // uo: the other horizontal velocity of the Coriolis term
        if constexpr (UT)
          if (c < 2) Vals<T>::load(s0 + (1 - c) * CS, uo);
#pragma unroll
        for (int m = 0; m < CPT; ++m) {
          const T lap = fma(G.crad, rt * (up[m] - x0[m]) - rb * (x0[m] - dn[m]), h[m]);
          T o = KIND == FV_PPBE ? cd * lap : fma(cd, lap, x0[m]);
          if constexpr (UT) {
            if (c < 3) o = fma(c == 0 ? rh[m][0] : c == 1 ? rh[m][1] : rh[m][2], thk[m], o);
            if (c < 2) o = fma(c == 0 ? cf.cor : -cf.cor, uo[m], o);
            if (c == 3) o = fma(b2, rdot[m], o);
          }
          out[m] = o;
        }
        const int e = c * N + p * NP + k * Ns2 + own;
        if (vec) {
          if (b) {
            T bv[CPT];
            Vals<T>::load(b + e, bv);
#pragma unroll
            for (int m = 0; m < CPT; ++m) out[m] = bv[m] - out[m];
          }
          Vals<T>::store(y + e, out);
        } else {
#pragma unroll
          for (int m = 0; m < CPT; ++m)
            if (ig + m < wi) y[e + m] = b ? b[e + m] - out[m] : out[m];
        }
      }
    }
    if (more) ghost_store(k + 2);
  }
}

// blockIdx: x = tile and component group, y = level chunk, z = panel
template <int KIND, class T, class GT>
__global__ void __launch_bounds__(TileT<T>::THREADS, sizeof(T) == 8 ? 2 : 4)
    tile_apply_kernel(const __grid_constant__ GT G, const __grid_constant__ Coefs<T> cf, const __grid_constant__ Tiles td,
                      const T* __restrict__ x, const T* __restrict__ b, T* __restrict__ y, const T* __restrict__ E) {
  if constexpr (KIND == FV_VTBE) {
    if (blockIdx.x % 2 == 0) tile_body<KIND, 0, 4, T>(G, cf, td, blockIdx.x / 2, x, b, y, E);
    else tile_body<KIND, 4, 3, T>(G, cf, td, blockIdx.x / 2, x, b, y, E);
  } else {
    tile_body<KIND, 0, 2, T>(G, cf, td, blockIdx.x, x, b, y, E);
  }
}

template <int KIND, class T, class GT>
static fv_status launch_tiled(const GT& G, const Coefs<T>& cf, const EdgeTab<T>& et, const T* x, const T* b, T* E, T* y,
                              cudaStream_t st, int cat, int nrhs = 1, long long xs = 0, long long ys = 0) {
  constexpr int D = KIND == FV_VTBE ? 7 : 2, GROUPS = KIND == FV_VTBE ? 2 : 1, NG = KIND == FV_VTBE ? 4 : 2;
  constexpr int CPT = TileT<T>::CPT, THREADS = TileT<T>::THREADS;
  static std::once_flag once[64];
  static cudaError_t attr_err[64];
  int dev = 0;
  FV_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return set_error("apply: device ordinal out of range"), FV_EINVAL;
  std::call_once(once[dev], [&] {
    attr_err[dev] = cudaFuncSetAttribute(tile_apply_kernel<KIND, T, GT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  });
  FV_CUDA(attr_err[dev]);
  Tiles td{};
  const int Ns = G.Ns;
  td.nti = (Ns + 31) / 32;
  td.ti = ((Ns + td.nti - 1) / td.nti + CPT - 1) / CPT * CPT;
  td.nti = (Ns + td.ti - 1) / td.ti;
  const int rows = THREADS / (td.ti / CPT);
  td.ntj = (Ns + rows - 1) / rows;
  td.tj = (Ns + td.ntj - 1) / td.ntj;
  td.vec = Ns % CPT == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(b)) & 15) == 0 &&
           xs % CPT == 0 && ys % CPT == 0;
  td.xs = xs, td.ys = ys;
  // threads of the tile, and one for every halo cell
  const int threads = (std::max(td.ti / CPT * td.tj, 2 * td.tj + 2 * (td.ti + 2)) + 31) / 32 * 32;
  const size_t smem = (size_t)RING * NG * plane_values<T>(td) * sizeof(T);
  if (threads > THREADS || smem > 200 * 1024) return set_error("apply: tile out of range"), FV_EINVAL;
  // about eight CTAs per SM of the 152, chunks of at least 2 levels (a chunk re-reads a plane at either end)
  const int per_chunk = td.nti * td.ntj * GROUPS * 6 * nrhs;
  int nchunk = std::max(1, std::min((152 * 8 + per_chunk - 1) / per_chunk, std::max(1, G.Nr / 2)));
  td.kchunk = (G.Nr + nchunk - 1) / nchunk;
  nchunk = (G.Nr + td.kchunk - 1) / td.kchunk;
  {
    ProfScope ps(FV_K_GHOST + (cat & ~15), st);
    const int ne = 24 * Ns * G.Nr;
    edge_flux_kernel<D, T><<<dim3((ne + 127) / 128, nrhs), 128, 0, st>>>(Ns, G.Nr, et, x, xs, E);
  }
  FV_CUDA(cudaGetLastError());
  {
    ProfScope ps(cat, st);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(td.nti * td.ntj * GROUPS, nchunk, 6 * nrhs), cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem, cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at, cfg.numAttrs = 1;
    FV_CUDA(cudaLaunchKernelEx(&cfg, tile_apply_kernel<KIND, T, GT>, G, cf, td, x, b, y, (const T*)E));
  }
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

// y = A x, or y = b - A x
fv_status apply_op(const fv_system* s, const double* x, double* y, cudaStream_t st, const double* b) {
  const fv_grid* g = s->grid;
  const Coefs<double> cf = make_coefs<double>(Phys{s->phys.E, s->phys.Ra, s->phys.Pr, s->phys.Pm, s->phys.dt},
                                               g->h.ri, g->h.ro);
  const EdgeTab<double> et{g->edge_cnt, g->edge_off, g->edge_w};
  const int cat = (s->kind == FV_VTBE ? FV_K_APPLY_VTBE : FV_K_APPLY_PPBE) + FV_K_COARSE * s->level;
  if (s->kind == FV_VTBE) return launch_tiled<FV_VTBE>(g->geo, cf, et, x, b, s->ghost, y, st, cat);
  return launch_tiled<FV_PPBE>(g->geo, cf, et, x, b, s->ghost, y, st, cat);
}

// y_r = A x_r for nrhs vectors with strides xs and ys; E: nrhs edge-flux buffers
fv_status apply_op_batch(const fv_system* s, int nrhs, const double* x, long long xs, double* y, long long ys, double* E,
                         cudaStream_t st) {
  const fv_grid* g = s->grid;
  const Coefs<double> cf = make_coefs<double>(Phys{s->phys.E, s->phys.Ra, s->phys.Pr, s->phys.Pm, s->phys.dt},
                                               g->h.ri, g->h.ro);
  const EdgeTab<double> et{g->edge_cnt, g->edge_off, g->edge_w};
  const double* none = nullptr;
  if (s->kind == FV_VTBE) return launch_tiled<FV_VTBE>(g->geo, cf, et, x, none, E, y, st, FV_K_APPLY_VTBE, nrhs, xs, ys);
  return launch_tiled<FV_PPBE>(g->geo, cf, et, x, none, E, y, st, FV_K_APPLY_PPBE, nrhs, xs, ys);
}

// FP32 operator (mixed-precision inner solves): FP32 tables, FP32 arithmetic
fv_status apply_op32(const fv_system* s, const float* x, float* y, cudaStream_t st, const float* b) {
  const fv_grid* g = s->grid;
  const Coefs<float> cf = make_coefs<float>(Phys{s->phys.E, s->phys.Ra, s->phys.Pr, s->phys.Pm, s->phys.dt},
                                             g->h.ri, g->h.ro);
  const EdgeTab<float> et{g->edge_cnt, g->edge_off, g->edge_wf};
  const int cat = (s->kind == FV_VTBE ? FV_K_APPLY_VTBE : FV_K_APPLY_PPBE) + FV_K_COARSE * s->level + FV_K_FP32;
  if (s->kind == FV_VTBE) return launch_tiled<FV_VTBE>(g->geof, cf, et, x, b, s->ghost32, y, st, cat);
  return launch_tiled<FV_PPBE>(g->geof, cf, et, x, b, s->ghost32, y, st, cat);
}

}  // namespace fv

extern "C" fv_status fv_apply_op_fp32(const fv_system* s, const float* x, float* y, void* stream) {
  if (!s || !x || !y) return fv::set_error("fv_apply_op_fp32: null argument"), FV_EINVAL;
  if (!s->prec32) return fv::set_error("fv_apply_op_fp32: the system was not assembled with FV_PREC_FP32"), FV_EINVAL;
  return fv::apply_op32(s, x, y, (cudaStream_t)stream);
}
