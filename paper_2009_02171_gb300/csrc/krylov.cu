// Restarted right-preconditioned flexible GMRES on the GPU (paper Sec. 3.3).
//
// Right preconditioning A M^{-1} (M x) = b (eqn:newlinear): the residual of
// the preconditioned system is the true residual b - A x; stop when
// ||b - A x|| <= max(eps_a, eps_r ||b - A x_0||).  The flexible form stores
// Z_j = M^{-1} v_j and updates x = x_0 + Z y, which allows the variable
// two-level preconditioner (inner GMRES on the coarse mesh) and, in mixed
// precision, an FP32 inner solve as preconditioner of the FP64 outer solve.
// Arnoldi uses classical Gram-Schmidt applied twice (CGS2), a whole step in one
// cooperative launch where the vectors' slices fit in shared memory, else one
// fused sweep over the basis a pass (multi-dot, then update-and-dot, then
// update-and-norm), with deterministic two-stage reductions (per-block
// partials in FP64 summed in a fixed order).  Hessenberg, Givens rotations and
// the small least-squares solve of the outer solves run on the host in FP64.
//
// The vector type T is double (FP64 path, outer solve of mixed precision) or
// float (inner solves of mixed precision).  For float vectors each thread sums
// at most 32 products in FP32 before adding them into its FP64 accumulators;
// block and grid reductions are FP64.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/fv_net.h"
#include "fv_internal.h"

namespace fv {

constexpr int KMAX = 32;     // max basis vectors in one fused pass
constexpr int RBLOCKS = 304; // reduction blocks of the weighted sums (2 per SM)
constexpr int CGS_BMAX = 608; // reduction blocks of a basis pass at most (4 per SM)
constexpr int RTHREADS = 256;

// Arnoldi bookkeeping of a device-driven solve (no host synchronisation)
struct ArnoldiDev {
  double H[KMAX * KMAX];  // upper Hessenberg after rotations, column-major H[j * KMAX + i]
  double cs[KMAX], sn[KMAX], g[KMAX + 1], y[KMAX];
  double scale;           // 1 / norm of the newest basis vector (0 after a breakdown)
  int k_eff;              // number of usable columns (first breakdown)
};

template <class T>
struct KrylovT {
  int m = 0;
  long long n = 0;
  T *V = nullptr, *Z = nullptr, *w = nullptr, *r = nullptr;
  double* part = nullptr;   // [KMAX][CGS_BMAX]
  double* h = nullptr;      // [3][KMAX]: h1, h2, nrm2
  double* hhost = nullptr;  // pinned [3][KMAX]
  ArnoldiDev* ad = nullptr; // device-driven solves
  unsigned* ticket = nullptr; // last-block counter of the fused reductions (returns to 0 after each use)
  unsigned* bar = nullptr;    // [3] grid barrier of the one-launch Gram-Schmidt step: arrivals, generation, ran out
  int* err = nullptr;         // the system's word (device address): a grid barrier ran out
  unsigned spins = 0;         // bound of a barrier's wait
  int sms = 0, smem = 0;
};

struct Krylov {
  KrylovT<double> d;
  KrylovT<float> f;
  unsigned long long moves = 0;  // times the FP32 workspace has been allocated
};

// Changes when a buffer of the FP32 inner solve of s (its own or a coarser level's) is allocated anew: a coarse system
// is also a system of its own (fv_coarse_system), whose solves may need more vectors than its place in the hierarchy.
unsigned long long inner_buffers(const fv_system* s) {
  unsigned long long n = 0;
  for (; s; s = s->coarse) n += s->kry ? s->kry->moves : 0;
  return n;
}

template <class T>
static void free_kt(KrylovT<T>& k) {
  cudaFree(k.V), cudaFree(k.Z), cudaFree(k.w), cudaFree(k.r), cudaFree(k.part), cudaFree(k.h), cudaFree(k.ad), cudaFree(k.ticket), cudaFree(k.bar);
  cudaFreeHost(k.hhost);
  k = KrylovT<T>();
}

void free_krylov(Krylov* k) {
  if (!k) return;
  free_kt(k->d);
  free_kt(k->f);
  delete k;
}

template <class T>
static KrylovT<T>& kt(Krylov* k);
template <>
KrylovT<double>& kt<double>(Krylov* k) { return k->d; }
template <>
KrylovT<float>& kt<float>(Krylov* k) { return k->f; }

template <class T>
static fv_status gs_limits(KrylovT<T>& k);

template <class T>
static fv_status ensure_krylov(const fv_system* s, int m) {
  fv_system* sm = const_cast<fv_system*>(s);
  if (!sm->kry) sm->kry = new Krylov();
  KrylovT<T>& k = kt<T>(sm->kry);
  k.spins = s->wait_limit;
  if (k.m >= m && k.n == s->n) return FV_OK;
  free_kt(k);
  k.spins = s->wait_limit;
  if (sizeof(T) == 4) ++sm->kry->moves;
  k.m = m, k.n = s->n;
  const size_t n = (size_t)s->n;
  if (cudaMalloc(&k.V, (m + 1) * n * sizeof(T)) != cudaSuccess || cudaMalloc(&k.Z, m * n * sizeof(T)) != cudaSuccess ||
      cudaMalloc(&k.w, n * sizeof(T)) != cudaSuccess || cudaMalloc(&k.r, n * sizeof(T)) != cudaSuccess ||
      cudaMalloc(&k.part, KMAX * CGS_BMAX * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&k.h, 3 * KMAX * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&k.ad, sizeof(ArnoldiDev)) != cudaSuccess || cudaMalloc(&k.ticket, sizeof(unsigned)) != cudaSuccess ||
      cudaMemset(k.ticket, 0, sizeof(unsigned)) != cudaSuccess ||
      cudaMalloc(&k.bar, 3 * sizeof(unsigned)) != cudaSuccess || cudaMemset(k.bar, 0, 3 * sizeof(unsigned)) != cudaSuccess ||
      cudaMallocHost(&k.hhost, 3 * KMAX * sizeof(double)) != cudaSuccess) {
    free_kt(k);
    return set_error("fv_gmres_solve: device allocation of the Krylov basis failed"), FV_ENOMEM;
  }
  k.err = s->words_dev + (sizeof(T) == 4 ? WORD_GS32 : WORD_GS64);
  return gs_limits<T>(k);
}

// Whether a grid barrier of s's workspaces (either type) or of its coarse levels' ran out, in work on st, since the last
// call.  The words are cleared and the barriers made usable again.
static fv_status gs_failed(const fv_system* s, cudaStream_t st, bool* bad) {
  auto check = [&](auto& k, int word) -> fv_status {
    if (!*(volatile int*)(s->words + word)) return FV_OK;
    *bad = true, s->words[word] = 0;
    if (!k.bar) return FV_OK;
    FV_CUDA(cudaMemsetAsync(k.bar, 0, 3 * sizeof(unsigned), st));
    FV_CUDA(cudaStreamSynchronize(st));
    return FV_OK;
  };
  fv_status rc;
  for (; s; s = s->coarse)
    if (s->kry && ((rc = check(s->kry->d, WORD_GS64)) || (rc = check(s->kry->f, WORD_GS32)))) return rc;
  return FV_OK;
}

fv_status waits_failed(const fv_system* s, const char* where, cudaStream_t st) {
  bool grid = false;
  fv_status rc = gs_failed(s, st, &grid);
  const bool sweep = sweep_failed(s);
  if (rc) return rc;
  if (grid || sweep)
    return set_error(std::string(where) + (grid ? "a wait of the Gram-Schmidt steps ran out" : "a wait of the subdomain sweeps ran out")),
           FV_ECUDA;
  return FV_OK;
}

// ------------------------------------------------------------------ vector kernels
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// block-reduce acc[0..nv) into part[v * gridDim.x + blockIdx.x]
__device__ __forceinline__ void block_store(double (&acc)[KMAX], int nv, double* part) {
  __shared__ double sm[RTHREADS / 32][KMAX];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int v = 0; v < KMAX; ++v) {
    if (v < nv) {
      double t = warp_sum(acc[v]);
      if (lane == 0) sm[wid][v] = t;
    }
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    double t = 0.0;
    for (int q = 0; q < RTHREADS / 32; ++q) t += sm[q][threadIdx.x];
    part[threadIdx.x * gridDim.x + blockIdx.x] = t;
  }
}

// block-reduce acc[0..nv) (nv <= NA) into part[v * gridDim.x + blockIdx.x]
template <int NA>
__device__ __forceinline__ void block_store_n(double (&acc)[NA], int nv, double* part) {
  __shared__ double sm[RTHREADS / 32][NA];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int v = 0; v < NA; ++v) {
    if (v < nv) {
      double t = warp_sum(acc[v]);
      if (lane == 0) sm[wid][v] = t;
    }
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    double t = 0.0;
    for (int q = 0; q < RTHREADS / 32; ++q) t += sm[q][threadIdx.x];
    part[threadIdx.x * gridDim.x + blockIdx.x] = t;
  }
}

// the rotation (c, s) that takes (a, b) to (den, 0); returns den
__device__ __forceinline__ double givens_rotation(double a, double b, double& c, double& s) {
  const double big = fmax(fabs(a), fabs(b));
  const double den = big > 1e-140 && big < 1e140 ? sqrt(a * a + b * b) : hypot(a, b);
  const double rden = den > 0.0 ? 1.0 / den : 0.0;
  c = den > 0.0 ? a * rden : 1.0, s = b * rden;
  return den;
}

// Givens update of column j of the device-driven Arnoldi (thread 0 of one block):
// h = h1 + h2 (CGS2), h_{j+1,j} = hn; previous rotations, new rotation,
// right-hand side update; scale = rhn = 1 / hn (0 for hn = 0)
__device__ void givens_update(int j, const double* h, double hn, double rhn, ArnoldiDev* ad) {
  double col[KMAX + 1];
  for (int i = 0; i <= j; ++i) col[i] = h[i] + h[KMAX + i];
  col[j + 1] = hn;
  for (int i = 0; i < j; ++i) {
    const double a = ad->cs[i] * col[i] + ad->sn[i] * col[i + 1];
    col[i + 1] = -ad->sn[i] * col[i] + ad->cs[i] * col[i + 1];
    col[i] = a;
  }
  double c, s;
  const double den = givens_rotation(col[j], col[j + 1], c, s);
  ad->cs[j] = c, ad->sn[j] = s;
  col[j] = den;
  ad->g[j + 1] = -s * ad->g[j];
  ad->g[j] = c * ad->g[j];
  for (int i = 0; i <= j; ++i) ad->H[j * KMAX + i] = col[i];
  if (!(den > 0.0) && ad->k_eff > j) ad->k_eff = j;              // no usable column j
  else if (!(hn > 0.0) && ad->k_eff > j + 1) ad->k_eff = j + 1;  // lucky breakdown after column j
  ad->scale = rhn;
}

// y = H^{-1} g on the first min(m, k_eff) columns (back substitution), zero beyond
__device__ void least_squares(int m, ArnoldiDev* ad) {
  const int kk = m < ad->k_eff ? m : ad->k_eff;
  for (int i = KMAX - 1; i >= kk; --i) ad->y[i] = 0.0;
  for (int i = kk - 1; i >= 0; --i) {
    double s = ad->g[i];
    for (int q = i + 1; q < kk; ++q) s -= ad->H[q * KMAX + i] * ad->y[q];
    ad->y[i] = s / ad->H[i * KMAX + i];
  }
}

// sum of the nb partials p[0..nb) by one warp in a fixed order; the loads of a lane are issued
// together (L2, written by other blocks of this launch) before they are added
__device__ __forceinline__ double last_block_sum(const double* p, int nb, int lane) {
  double t = 0.0;
  for (int b0 = 0; b0 < nb; b0 += 32 * 8) {
    double q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int b = b0 + u * 32 + lane;
      q[u] = b < nb ? __ldcg(p + b) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) t += q[u];
  }
  return warp_sum(t);
}

// 16-byte vector of T: four floats or two doubles
template <class T>
struct Vec16;
template <>
struct Vec16<float> {
  static constexpr int L = 4;
  __device__ static void load(const float* p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
  }
  __device__ static void ldg(const float* p, float (&v)[4]) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
  }
  __device__ static void store(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct Vec16<double> {
  static constexpr int L = 2;
  __device__ static void load(const double* p, double (&v)[2]) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    v[0] = q.x, v[1] = q.y;
  }
  __device__ static void ldg(const double* p, double (&v)[2]) {
    const double2 q = __ldg(reinterpret_cast<const double2*>(p));
    v[0] = q.x, v[1] = q.y;
  }
  __device__ static void store(double* p, const double (&v)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
};

// mode 0: part = V^T w
// mode 1: w -= V h; part = V^T w
// mode 2: w -= V h; part[0] = w^T w
// NV (the number of basis vectors) is a template parameter so the loops over
// the basis unroll exactly; h is staged in shared memory.  With `vec` (n a
// multiple of the 16-byte width and 16-byte aligned bases) a thread moves 16
// bytes of every vector per iteration, which keeps enough loads in flight to
// stream the basis at HBM rate; otherwise one element at a time.  FP32
// products are summed in FP32 for up to 32 elements of a thread, then in FP64;
// FP64 products go straight into the FP64 accumulators.  With `out`, the last
// block to finish sums the per-block partials in a fixed order into
// out[0..nv) (and, for mode 2 with `ad`, applies the Givens update of column
// gj), so no separate reduction launch is needed.
template <int NV, class T>
__global__ void __launch_bounds__(RTHREADS, (NV > (sizeof(T) == 8 ? 18 : 14) ? 1 : 2)) cgs_kernel(long long n, int vec, const T* __restrict__ V,
                                                          const double* __restrict__ h, T* __restrict__ w,
                                                          double* __restrict__ part, int mode, double* out,
                                                          unsigned* ticket, ArnoldiDev* ad, int gj,
                                                          const double* __restrict__ hg) {
  constexpr int NA = NV > 0 ? NV : 1;
  constexpr int L = Vec16<T>::L;
  constexpr bool F32 = sizeof(T) == 4;
  __shared__ T hs[NA];
  if (mode > 0)
    for (int v = threadIdx.x; v < NV; v += blockDim.x) hs[v] = (T)h[v];
  __syncthreads();
  double acc[NA];
  T cur[NA];
#pragma unroll
  for (int v = 0; v < NA; ++v) acc[v] = 0.0, cur[v] = T(0);
  double accn = 0.0;
  T curn = T(0);
  int cnt = 0;
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  const long long ng = vec ? n / L : 0;
  for (long long g = tid; g < ng; g += stride) {
    const long long e = g * L;
    T we[L];
    Vec16<T>::load(w + e, we);
    if (mode > 0 && NV > 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T vv[L];
        Vec16<T>::ldg(V + v * n + e, vv);
        const T hv = hs[v];
#pragma unroll
        for (int l = 0; l < L; ++l) we[l] -= hv * vv[l];
      }
      Vec16<T>::store(w + e, we);
    }
    if (mode < 2) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T vv[L];
        Vec16<T>::ldg(V + v * n + e, vv);
#pragma unroll
        for (int l = 0; l < L; ++l) {
          if constexpr (F32) cur[v] += vv[l] * we[l];
          else acc[v] += vv[l] * we[l];
        }
      }
    } else {
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if constexpr (F32) curn += we[l] * we[l];
        else accn += we[l] * we[l];
      }
    }
    if constexpr (F32) {  // FP32 partial sums go into the FP64 accumulators every 32 elements
      cnt += L;
      if (cnt >= 32) {
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] += (double)cur[v], cur[v] = T(0);
        accn += (double)curn, curn = T(0);
        cnt = 0;
      }
    }
  }
  for (long long e = ng * L + tid; e < n; e += stride) {
    T we = w[e];
    if (mode > 0 && NV > 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) we -= hs[v] * V[v * n + e];
      w[e] = we;
    }
    if (mode < 2) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        if constexpr (F32) cur[v] += V[v * n + e] * we;
        else acc[v] += V[v * n + e] * we;
      }
    } else {
      if constexpr (F32) curn += we * we;
      else accn += we * we;
    }
    if constexpr (F32) {  // FP32 partial sums go into the FP64 accumulators every 32 elements
      cnt += 1;
      if (cnt >= 32) {
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] += (double)cur[v], cur[v] = T(0);
        accn += (double)curn, curn = T(0);
        cnt = 0;
      }
    }
  }
  if constexpr (F32) {
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] += (double)cur[v];
    accn += (double)curn;
  }
  if (mode == 2) acc[0] = accn;
  const int nvv = mode < 2 ? NV : 1;
  block_store_n<NA>(acc, nvv, part);
  if (!out) return;
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int v = wid; v < nvv; v += nw) out[v] = last_block_sum(part + v * gridDim.x, (int)gridDim.x, lane);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (mode == 2 && ad) {
      const double hn = sqrt(out[0]);
      givens_update(gj, hg, hn, hn > 0.0 ? 1.0 / hn : 0.0, ad);
    }
    *ticket = 0u;
  }
}

// reduction blocks of a basis pass over n elements: about four 16-byte groups (or elements) a
// thread, at most CGS_BMAX blocks (short vectors: fewer partials for the final sum); consumers of
// the partials take the same count
template <class T>
static int cgs_blocks(long long n, bool vec) {
  const long long g = vec ? n / Vec16<T>::L : n;
  return (int)std::min<long long>(std::max<long long>((g + 4 * RTHREADS - 1) / (4 * RTHREADS), 1), CGS_BMAX);
}

template <class T>
static bool cgs_vec(long long n, const T* V, const T* w) {
  return n % Vec16<T>::L == 0 && (reinterpret_cast<uintptr_t>(V) & 15) == 0 && (reinterpret_cast<uintptr_t>(w) & 15) == 0;
}

// ------------------------------------------------------------------ Gram-Schmidt step in one launch
// One Arnoldi step's orthogonalization (one or two classical Gram-Schmidt passes), norm, Givens update and the
// next basis vector, v = w / ||w||, with a grid barrier between its reductions, for vectors whose slice per SM
// fits in shared memory: w is read from memory once and kept there, only the basis is read again.  At the sizes
// of the coarse level (n = 393,216 FP32: 1.5 MB a vector, all in L2) the separate passes were bound by their
// launches, drains and the FP64 arithmetic of the block reductions (five dependent DADDs a warp and value, 16
// cycles of the SM's FP64 pipe each); here a value's 512 partial sums go through shared memory, where one warp
// adds 16 a lane before its butterfly, a quarter of the operations.  Measured: see gs_step().
constexpr int GS_THREADS = 512;          // threads a block at most
// FP64: 512, half of them above 16 basis vectors (registers).  FP32: 256, since every thread's partial sums are
// converted to FP64 on the slow pipe (coarse level, 5 vectors: 24.6 us with 512 threads, see gs_step())
__host__ __device__ constexpr int gs_threads(int nv, int es) { return es == 4 || nv > 16 ? GS_THREADS / 2 : GS_THREADS; }
constexpr int GS_CHUNK = 8;              // values reduced together: [GS_CHUNK][GS_THREADS] doubles of shared memory

struct GsArgs {
  long long n, slice;   // elements; elements a block
  int keep;             // the block's slice of the basis is kept in shared memory for the later passes
  int passes;           // Gram-Schmidt passes (0: norm and scaling alone)
  int start;            // 1: the norm starts a cycle (ad->g = ||w|| e_1)
  int last;             // 1: after this column solve the least-squares problem into ad->y
  int gj;
  double* part;         // [3][KMAX][blocks]
  double* h;            // [3][KMAX]: the two passes' coefficients, ||w||^2
  ArnoldiDev* ad;       // device-driven solves
  unsigned* bar;
  int* err;
  unsigned spins;
};

// All blocks (co-resident: cooperative launch) meet.  The wait is bounded.  A block whose wait runs out goes on with
// incomplete sums (every access stays in range), says so through err, and marks the barrier: later barriers, whose
// count no longer fits, return at once, until the host has read err and reset the words (gs_failed).
__device__ __forceinline__ void grid_barrier(unsigned* bar, int* err, unsigned spins) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned gen, cur, lost;
    asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(gen) : "l"(bar + 1) : "memory");
    asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(lost) : "l"(bar + 2) : "memory");
    __threadfence();
    const unsigned before = atomicAdd(bar, 1u);  // the marks are read beside it, not before it
    if (lost) {
      *err = 1;
    } else if (before == gridDim.x - 1) {
      bar[0] = 0;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      unsigned t = 0;
      do {
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(bar + 1) : "memory");
      } while (cur == gen && ++t < spins);
      if (cur == gen) *err = 1, atomicExch(bar + 2, 1u);
    }
    __threadfence();
  }
  __syncthreads();
}

// sums of acc[0..nv) over the block into part[v * gridDim.x + blockIdx.x], fixed order
template <int NA, int TH>
__device__ __forceinline__ void gs_reduce(double (&acc)[NA], int nv, double* red, double* part) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int v0 = 0; v0 < NA; v0 += GS_CHUNK) {
    if (v0 >= nv) break;
    if (v0) __syncthreads();
#pragma unroll
    for (int u = 0; u < GS_CHUNK; ++u)
      if (v0 + u < NA && v0 + u < nv) red[u * TH + threadIdx.x] = acc[v0 + u < NA ? v0 + u : 0];
    __syncthreads();
    if (wid < GS_CHUNK && v0 + wid < nv) {
      const double* q = red + wid * TH + lane;
      double t0 = 0.0, t1 = 0.0;
#pragma unroll
      for (int u = 0; u < TH / 32; u += 2) t0 += q[32 * u], t1 += q[32 * (u + 1)];
      const double t = warp_sum(t0 + t1);
      if (lane == 0) part[(v0 + wid) * gridDim.x + blockIdx.x] = t;
    }
  }
}

// the grid's sums out[0..nv) from the blocks' partials, the same order in every block
template <int TH>
__device__ __forceinline__ void gs_total(const double* part, int nv, double* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int v = wid; v < nv; v += TH / 32) {
    const double t = last_block_sum(part + v * gridDim.x, (int)gridDim.x, lane);
    if (lane == 0) out[v] = t;
  }
  __syncthreads();
}

template <int NV, class T>
__global__ void __launch_bounds__(gs_threads(NV, sizeof(T)), 1) gs_kernel(GsArgs A, const T* __restrict__ V, const T* w, T* vout) {
  constexpr int NA = NV > 0 ? NV : 1, L = Vec16<T>::L, TH = gs_threads(NV, sizeof(T));
  constexpr bool F32 = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char gs_smem[];
  double* red = reinterpret_cast<double*>(gs_smem);
  T* ws = reinterpret_cast<T*>(gs_smem + GS_CHUNK * GS_THREADS * sizeof(double));
  T* vs = ws + A.slice;  // [NV][slice] when A.keep
  __shared__ double tot[NA], coef[NA];
  __shared__ T hs[NA];
  // what the Givens update of block 0 needs of the earlier columns, fetched now
  __shared__ double rot[2][NA], Hs[NA * NA], gj0;
  const bool givens = blockIdx.x == 0 && A.ad && !A.start;
  if (givens) {
    if (threadIdx.x < A.gj) rot[0][threadIdx.x] = A.ad->cs[threadIdx.x], rot[1][threadIdx.x] = A.ad->sn[threadIdx.x];
    if (threadIdx.x == TH - 1) gj0 = A.ad->g[A.gj];
    if (A.last)
      for (int e = threadIdx.x; e < A.gj * A.gj; e += TH) Hs[e / A.gj * NA + e % A.gj] = A.ad->H[e / A.gj * KMAX + e % A.gj];
  }
  const long long n = A.n, b0 = blockIdx.x * A.slice;
  const int len = (int)(n - b0 < A.slice ? (n > b0 ? n - b0 : 0) : A.slice);
  const bool vec = n % L == 0 && ((reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(w)) & 15) == 0;
  const int ng = vec ? len / L : 0;
  const T* Vb = V + b0;
  const T* wb = w + b0;
  double acc[NA];
  T cur[NA];
  // FP32 products are summed in FP32 for at most 32 elements of a thread, then in FP64
  auto clear = [&]() {
#pragma unroll
    for (int v = 0; v < NA; ++v) acc[v] = 0.0, cur[v] = T(0);
  };
  auto flush = [&]() {
    if constexpr (F32)
#pragma unroll
      for (int v = 0; v < NA; ++v) acc[v] += (double)cur[v], cur[v] = T(0);
  };
  auto add = [&](int v, T a, T b) {
    if constexpr (F32) cur[v] += a * b;
    else acc[v] += a * b;
  };
  // one pass over the slice.  sub: w -= V h;  dots: V^T w, else w^T w;  first: w comes from memory
  auto pass = [&](auto first, bool sub, bool dots) {
    clear();
    int cnt = 0;
#pragma unroll(NV <= 8 ? 2 : 1)
    for (int g = threadIdx.x; g < ng; g += TH) {
      const int e = g * L;
      T we[L];
      if constexpr (decltype(first)::value) Vec16<T>::load(wb + e, we);
      else Vec16<T>::load(ws + e, we);
      T vv[NA][L];
      if (decltype(first)::value || !A.keep) {
#pragma unroll
        for (int v = 0; v < NV; ++v) Vec16<T>::ldg(Vb + v * n + e, vv[v]);
        if (A.keep) {
#pragma unroll
          for (int v = 0; v < NV; ++v) Vec16<T>::store(vs + v * (int)A.slice + e, vv[v]);
        }
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) Vec16<T>::load(vs + v * (int)A.slice + e, vv[v]);
      }
      if (sub) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int l = 0; l < L; ++l) we[l] -= hs[v] * vv[v][l];
      }
      if (decltype(first)::value || sub) Vec16<T>::store(ws + e, we);
      if (dots) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int l = 0; l < L; ++l) add(v, vv[v][l], we[l]);
      } else {
#pragma unroll
        for (int l = 0; l < L; ++l) add(0, we[l], we[l]);
      }
      cnt += L;
      if (F32 && cnt >= 32) flush(), cnt = 0;
    }
    for (int e = ng * L + threadIdx.x; e < len; e += TH) {  // unaligned vectors, or a ragged end
      T we;
      if constexpr (decltype(first)::value) we = wb[e];
      else we = ws[e];
      if (sub) {
#pragma unroll
        for (int v = 0; v < NV; ++v) we -= hs[v] * Vb[v * n + e];
      }
      if (decltype(first)::value || sub) ws[e] = we;
      if (dots) {
#pragma unroll
        for (int v = 0; v < NV; ++v) add(v, Vb[v * n + e], we);
      } else {
        add(0, we, we);
      }
      if (F32 && ++cnt >= 32) flush(), cnt = 0;
    }
    flush();
  };
  double* part = A.part;
  if (A.passes > 0) {
    pass(std::true_type(), false, true);
    gs_reduce<NA, TH>(acc, NV, red, part);
    for (int q = 0; q < A.passes; ++q) {
      grid_barrier(A.bar, A.err, A.spins);
      gs_total<TH>(part, NV, tot);
      if (threadIdx.x < NV) {
        hs[threadIdx.x] = (T)tot[threadIdx.x];
        coef[threadIdx.x] = (q ? coef[threadIdx.x] : 0.0) + tot[threadIdx.x];
        if (blockIdx.x == 0) A.h[q * KMAX + threadIdx.x] = tot[threadIdx.x];
      }
      __syncthreads();
      part += KMAX * gridDim.x;
      const bool more = q + 1 < A.passes;
      pass(std::false_type(), true, more);
      gs_reduce<NA, TH>(acc, more ? NV : 1, red, part);
    }
    if (A.passes == 1 && blockIdx.x == 0 && threadIdx.x < NV) A.h[KMAX + threadIdx.x] = 0.0;
  } else {
    pass(std::true_type(), false, false);
    gs_reduce<NA, TH>(acc, 1, red, part);
  }
  grid_barrier(A.bar, A.err, A.spins);
  gs_total<TH>(part, 1, tot);
  // one thread takes the square root and the reciprocal: on the FP64 pipe (16 cycles a warp instruction) every
  // warp doing so cost more than a pass over the basis
  __shared__ T inv;
  double hn = 0.0, rhn = 0.0;
  if (threadIdx.x == 0) {
    hn = sqrt(tot[0]);
    rhn = hn > 0.0 ? 1.0 / hn : 0.0;
    inv = (T)rhn;
  }
  if (vout) {
    __syncthreads();
    const T a = inv;
    T* vb = vout + b0;
    for (int g = threadIdx.x; g < ng; g += TH) {
      T we[L];
      Vec16<T>::load(ws + g * L, we);
  #pragma unroll
      for (int l = 0; l < L; ++l) we[l] *= a;
      Vec16<T>::store(vb + g * L, we);
    }
    for (int e = ng * L + threadIdx.x; e < len; e += TH) vb[e] = a * ws[e];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    A.h[2 * KMAX] = tot[0];
    if (A.ad && A.start) {
      for (int i = 0; i <= KMAX; ++i) A.ad->g[i] = 0.0;
      A.ad->g[0] = hn;
      A.ad->scale = rhn;
      A.ad->k_eff = hn > 0.0 ? KMAX : 0;
    } else if (A.ad) {
      // as givens_update(), from shared memory
      const int j = A.gj;
      double c0 = coef[0];
      for (int i = 0; i < j; ++i) {
        const double c1 = coef[i + 1 < NA ? i + 1 : 0];
        coef[i] = rot[0][i] * c0 + rot[1][i] * c1;
        c0 = -rot[1][i] * c0 + rot[0][i] * c1;
      }
      double c, s;
      const double den = givens_rotation(c0, hn, c, s);
      coef[j] = den;
      for (int i = 0; i <= j; ++i) A.ad->H[j * KMAX + i] = coef[i];
      A.ad->cs[j] = c, A.ad->sn[j] = s;
      A.ad->g[j + 1] = -s * gj0;
      A.ad->g[j] = c * gj0;
      int k_eff = A.ad->k_eff;
      if (!(den > 0.0) && k_eff > j) k_eff = j;              // no usable column j
      else if (!(hn > 0.0) && k_eff > j + 1) k_eff = j + 1;  // lucky breakdown after column j
      A.ad->k_eff = k_eff;
      A.ad->scale = rhn;
      if (A.last) {
        const int kk = min(j + 1, k_eff);
        double y[NA];
        for (int i = KMAX - 1; i >= kk; --i) A.ad->y[i] = 0.0;
#pragma unroll
        for (int i = NA - 1; i >= 0; --i) {
          if (i >= kk) continue;
          double t = i == j ? c * gj0 : A.ad->g[i];
#pragma unroll
          for (int q = i + 1; q < NA; ++q)
            if (q < kk) t -= (q == j ? coef[i] : Hs[q * NA + i]) * y[q];
          y[i] = t / (i == j ? coef[i] : Hs[i * NA + i]);
          A.ad->y[i] = y[i];
        }
      }
    }
  }
}

template <int NV, class T>
static const void* gs_kernel_ptr() { return reinterpret_cast<const void*>(&gs_kernel<NV, T>); }

template <class T, int... I>
static const void* gs_kernel_of(int nv, std::integer_sequence<int, I...>) {
  using F = const void* (*)();
  static const F table[] = {&gs_kernel_ptr<I, T>...};
  return table[nv]();
}

template <class T>
static fv_status gs_limits(KrylovT<T>& k) {
  int dev = 0, limit = 0;
  FV_CUDA(cudaGetDevice(&dev));
  FV_CUDA(cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  FV_CUDA(cudaDeviceGetAttribute(&k.sms, cudaDevAttrMultiProcessorCount, dev));
  k.smem = limit - 12 * 1024;  // less the kernel's static shared memory
  for (int v = 0; v < KMAX; ++v)
    FV_CUDA(cudaFuncSetAttribute(gs_kernel_of<T>(v, std::make_integer_sequence<int, KMAX>{}),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem));
  return FV_OK;
}

// Blocks and shared memory of the one-launch step for vectors of n; 0 blocks: the slice does not fit (the separate
// passes below stream such vectors at HBM rate: FP64 above 3.5M, FP32 above 7.1M elements).  At least 1024 elements
// a block: fewer only add partials and arrivals at the barrier.
template <class T>
static int gs_blocks(const KrylovT<T>& k, long long n, long long* slice, size_t* smem) {
  const long long blocks = std::max<long long>(1, std::min<long long>(k.sms, n / 1024));
  *slice = ((n + blocks - 1) / blocks + 15) / 16 * 16;
  *smem = GS_CHUNK * GS_THREADS * sizeof(double) + (size_t)*slice * sizeof(T);
  return *smem <= (size_t)k.smem ? (int)((n + *slice - 1) / *slice) : 0;
}

struct CgsFuse {
  double* out = nullptr;       // fused final reduction target (null: partials only)
  unsigned* ticket = nullptr;
  ArnoldiDev* ad = nullptr;    // mode 2: Givens update of column gj in the last block
  int gj = 0;
  const double* hg = nullptr;  // CGS2 coefficients h1 [0, KMAX), h2 [KMAX, 2 KMAX) of that column
};

template <int NV, class T>
static void cgs_launch_t(long long n, const T* V, const double* h, T* w, double* part, int mode, CgsFuse f,
                         cudaStream_t st) {
  const bool vec = cgs_vec<T>(n, V, w);
  cgs_kernel<NV, T><<<cgs_blocks<T>(n, vec), RTHREADS, 0, st>>>(n, vec ? 1 : 0, V, h, w, part, mode, f.out, f.ticket,
                                                                 f.ad, f.gj, f.hg);
}

template <class T, int... I>
static void cgs_dispatch(int nv, long long n, const T* V, const double* h, T* w, double* part, int mode, CgsFuse f,
                         cudaStream_t st, std::integer_sequence<int, I...>) {
  using F = void (*)(long long, const T*, const double*, T*, double*, int, CgsFuse, cudaStream_t);
  static const F table[] = {&cgs_launch_t<I, T>...};
  table[nv](n, V, h, w, part, mode, f, st);
}

template <class T>
static void cgs_launch(int nv, long long n, const T* V, const double* h, T* w, double* part, int mode,
                       cudaStream_t st, CgsFuse f = CgsFuse()) {
  cgs_dispatch<T>(nv, n, V, h, w, part, mode, f, st, std::make_integer_sequence<int, KMAX>{});
}

// out[v] = sum_b part[v * nb + b]: one warp per vector, fixed summation order
__global__ void reduce_kernel(const double* __restrict__ part, int nb, int nv, double* __restrict__ out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int v = wid; v < nv; v += nw) {
    double t = 0.0;
    for (int b = lane; b < nb; b += 32) t += part[v * nb + b];
    t = warp_sum(t);
    if (lane == 0) out[v] = t;
  }
}

// beta = ||r|| from the norm partials; g = (beta, 0, ...); scale = 1/beta
__global__ void start_kernel(const double* __restrict__ part, int nb, ArnoldiDev* ad) {
  const int lane = threadIdx.x;
  double t = 0.0;
  for (int b = lane; b < nb; b += 32) t += part[b];
  t = warp_sum(t);
  if (lane == 0) {
    const double beta = sqrt(t);
    for (int i = 0; i <= KMAX; ++i) ad->g[i] = 0.0;
    ad->g[0] = beta;
    ad->scale = beta > 0.0 ? 1.0 / beta : 0.0;
    ad->k_eff = beta > 0.0 ? KMAX : 0;
  }
}

__global__ void lsq_kernel(int m, ArnoldiDev* ad) {
  if (threadIdx.x == 0) least_squares(m, ad);
}

template <class T>
__global__ void dscale_kernel(long long n, const T* __restrict__ x, const double* __restrict__ scale, T* __restrict__ out) {
  const T a = (T)*scale;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = a * x[e];
}

// out = x / sqrt(*nrm2) (zero for a zero norm)
template <class T>
__global__ void rscale_kernel(long long n, const T* __restrict__ x, const double* __restrict__ nrm2, T* __restrict__ out) {
  const double hn = sqrt(*nrm2);
  const T a = (T)(hn > 0.0 ? 1.0 / hn : 0.0);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = a * x[e];
}

static int vblocks(long long n) { return (int)std::min<long long>(std::max<long long>((n + 255) / 256, 1), 152LL * 16); }

// One Arnoldi step's orthogonalization of k.w against the first nv basis vectors (`passes` passes) and the next basis
// vector into vout (null: none); with ad, the Givens update of column nv - 1 (last: and the least-squares solve).
// nv = 0: the norm of w and w / ||w|| (with ad: the start of a cycle).  One cooperative launch where the slices of w
// fit in shared memory, else the separate passes.
// A step against the separate passes, us on GB300 (mean over a cycle): FP32 coarse level 6x32^3 (one pass) 28.5 -> 21,
// 6x64^2x48 59 -> 38; FP32 6x64^3 72 -> 55; FP64 (two passes) 6x45^2x39 218 -> 137, 6x16^3 64 -> 40.
template <class T>
static fv_status gs_step(const KrylovT<T>& k, int nv, long long n, const T* w, T* vout, int passes, ArnoldiDev* ad,
                         bool last, cudaStream_t st) {
  GsArgs a{};
  size_t smem = 0;
  const int blocks = gs_blocks<T>(k, n, &a.slice, &smem);
  if (blocks) {
    // basis and w in shared memory: short vectors (the coarse level) read nothing twice
    const size_t keep = (size_t)nv * a.slice * sizeof(T);
    a.keep = nv > 0 && n % Vec16<T>::L == 0 && smem + keep <= (size_t)k.smem;
    if (a.keep) smem += keep;
    a.n = n, a.passes = nv > 0 ? passes : 0, a.start = nv == 0, a.last = last, a.gj = nv - 1;
    a.part = k.part, a.h = k.h, a.ad = ad, a.bar = k.bar, a.err = k.err, a.spins = k.spins;
    const T* V = nv > 0 ? k.V : w;
    void* args[] = {&a, &V, &w, &vout};
    FV_CUDA(cudaLaunchCooperativeKernel(gs_kernel_of<T>(nv, std::make_integer_sequence<int, KMAX>{}), dim3(blocks),
                                        dim3(gs_threads(nv, sizeof(T))), args, smem, st));
    return FV_OK;
  }
  T* wm = const_cast<T*>(w);
  if (nv == 0) {
    cgs_launch<T>(0, n, w, nullptr, wm, k.part, 2, st);
    const int nb = cgs_blocks<T>(n, cgs_vec<T>(n, w, w));
    if (ad) start_kernel<<<1, 32, 0, st>>>(k.part, nb, ad);
    else reduce_kernel<<<1, RTHREADS, 0, st>>>(k.part, nb, 1, k.h + 2 * KMAX);
  } else {
    CgsFuse f;
    f.ticket = k.ticket;
    f.out = k.h;
    cgs_launch<T>(nv, n, k.V, nullptr, wm, k.part, 0, st, f);
    if (passes == 2) {
      f.out = k.h + KMAX;
      cgs_launch<T>(nv, n, k.V, k.h, wm, k.part, 1, st, f);
    } else if (nv == 1) {
      FV_CUDA(cudaMemsetAsync(k.h + KMAX, 0, KMAX * sizeof(double), st));
    }
    f.out = k.h + 2 * KMAX, f.ad = ad, f.gj = nv - 1, f.hg = k.h;
    cgs_launch<T>(nv, n, k.V, passes == 2 ? k.h + KMAX : k.h, wm, k.part, 2, st, f);
    if (last && ad) lsq_kernel<<<1, 32, 0, st>>>(nv, ad);
  }
  if (vout) {
    if (ad) dscale_kernel<T><<<vblocks(n), 256, 0, st>>>(n, w, &ad->scale, vout);
    else rscale_kernel<T><<<vblocks(n), 256, 0, st>>>(n, w, k.h + 2 * KMAX, vout);
  }
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

// four consecutive values, moved 16 bytes at a time
template <class T>
struct alignas(16) Pack4 {
  T v[4];
};
static bool pack4(long long n, const void* a, const void* b, const void* c) {
  return n >= 4 && ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & 15) == 0;
}

// out = a x + b y (y unread for b = 0).  Bound by memory: 16-byte accesses, four values a thread and turn (packs:
// all pointers 16-byte aligned), the rest one by one; y may be out.  All vector kernels of a mixed step on 6x64^3:
// 5.1 -> 4.5 ms one value against four a turn
template <class T, class U>
__global__ void axpby_kernel(long long n, long long packs, double a, const U* x, double b, const T* y, T* out) {
  const T at = (T)a, bt = (T)b;
  const bool has_y = b != 0.0;
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long g = tid; g < packs; g += stride) {
    const Pack4<U> p = reinterpret_cast<const Pack4<U>*>(x)[g];
    Pack4<T> o;
    if (has_y) {
      const Pack4<T> q = reinterpret_cast<const Pack4<T>*>(y)[g];
#pragma unroll
      for (int l = 0; l < 4; ++l) o.v[l] = at * (T)p.v[l] + bt * q.v[l];
    } else {
#pragma unroll
      for (int l = 0; l < 4; ++l) o.v[l] = at * (T)p.v[l] + T(0);
    }
    reinterpret_cast<Pack4<T>*>(out)[g] = o;
  }
  for (long long e = 4 * packs + tid; e < n; e += stride) out[e] = at * (T)x[e] + (has_y ? bt * y[e] : T(0));
}

template <class T>
struct Coef {
  T c[KMAX];
};

// x += sum_v y_v Z_v (add = 1) or x = sum_v y_v Z_v, the sum of an element in basis order
template <int NV, class T>
__device__ __forceinline__ void combine(long long n, long long packs, const T* __restrict__ Z, const T (&c)[NV > 0 ? NV : 1],
                                        bool add, T* __restrict__ x) {
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long g = tid; g < packs; g += stride) {
    Pack4<T> s{};
    if (add) s = reinterpret_cast<const Pack4<T>*>(x)[g];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const Pack4<T> z = reinterpret_cast<const Pack4<T>*>(Z + v * n)[g];
#pragma unroll
      for (int l = 0; l < 4; ++l) s.v[l] += c[v] * z.v[l];
    }
    reinterpret_cast<Pack4<T>*>(x)[g] = s;
  }
  for (long long e = 4 * packs + tid; e < n; e += stride) {
    T s = add ? x[e] : T(0);
#pragma unroll
    for (int v = 0; v < NV; ++v) s += c[v] * Z[v * n + e];
    x[e] = s;
  }
}

template <int NV, class T>
__global__ void update_kernel(long long n, long long packs, const T* __restrict__ Z, Coef<T> y, T* __restrict__ x) {
  T c[NV > 0 ? NV : 1];
#pragma unroll
  for (int v = 0; v < NV; ++v) c[v] = y.c[v];
  combine<NV, T>(n, packs, Z, c, true, x);
}

template <int NV, class T>
static void update_launch_t(long long n, const T* Z, const Coef<T>& y, T* x, cudaStream_t st) {
  const long long packs = n % 4 == 0 && pack4(n, Z, x, nullptr) ? n / 4 : 0;
  update_kernel<NV, T><<<vblocks(packs ? packs : n), 256, 0, st>>>(n, packs, Z, y, x);
}

template <class T, int... I>
static void update_dispatch(int nv, long long n, const T* Z, const Coef<T>& y, T* x, cudaStream_t st,
                            std::integer_sequence<int, I...>) {
  using F = void (*)(long long, const T*, const Coef<T>&, T*, cudaStream_t);
  static const F table[] = {&update_launch_t<I, T>...};
  table[nv](n, Z, y, x, st);
}

template <class T, class U>
static void axpby_launch(long long n, double a, const U* x, double b, const T* y, T* out, cudaStream_t st) {
  const long long packs = pack4(n, x, b != 0.0 ? y : nullptr, out) ? n / 4 : 0;
  axpby_kernel<T, U><<<vblocks(packs ? (n + 3) / 4 : n), 256, 0, st>>>(n, packs, a, x, b, y, out);
}

fv_status axpby(long long n, double a, const double* x, double b, const double* y, double* out, cudaStream_t st) {
  ProfScope ps(FV_K_VEC, st);
  axpby_launch<double, double>(n, a, x, b, y, out, st);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

fv_status axpby32(long long n, double a, const float* x, double b, const float* y, float* out, cudaStream_t st) {
  ProfScope ps(FV_K_VEC, st);
  axpby_launch<float, float>(n, a, x, b, y, out, st);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

fv_status to_fp32(long long n, const double* x, float* out, cudaStream_t st) {
  ProfScope ps(FV_K_VEC, st);
  axpby_launch<float, double>(n, 1.0, x, 0.0, nullptr, out, st);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

fv_status to_fp64(long long n, const float* x, double* out, cudaStream_t st) {
  ProfScope ps(FV_K_VEC, st);
  axpby_launch<double, float>(n, 1.0, x, 0.0, nullptr, out, st);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

// ||x||, and x / ||x|| into vout (null: none)
template <class T>
static fv_status norm2(KrylovT<T>& k, long long n, const T* x, T* vout, cudaStream_t st, double* out) {
  if (fv_status rc = gs_step<T>(k, 0, n, x, vout, 0, nullptr, false, st)) return rc;
  FV_CUDA(cudaMemcpyAsync(k.hhost, k.h + 2 * KMAX, sizeof(double), cudaMemcpyDeviceToHost, st));
  FV_CUDA(cudaStreamSynchronize(st));
  *out = std::sqrt(k.hhost[0]);
  return FV_OK;
}

// y = A x, or y = b - A x
template <class T>
static fv_status apply_t(const fv_system* s, const T* x, T* y, cudaStream_t st, const T* b = nullptr);
template <>
fv_status apply_t<double>(const fv_system* s, const double* x, double* y, cudaStream_t st, const double* b) {
  return apply_op(s, x, y, st, b);
}
template <>
fv_status apply_t<float>(const fv_system* s, const float* x, float* y, cudaStream_t st, const float* b) {
  return apply_op32(s, x, y, st, b);
}

template <class T>
static fv_status precond_t(const fv_system* s, const T* r, T* z, cudaStream_t st);
template <>
fv_status precond_t<double>(const fv_system* s, const double* r, double* z, cudaStream_t st) {
  return precond_apply(s, r, z, st);
}
template <>
fv_status precond_t<float>(const fv_system* s, const float* r, float* z, cudaStream_t st) {
  return precond_apply32(s, r, z, st);
}

// ------------------------------------------------------------------ device-driven FGMRES
// x = sum_v y_v Z_v with y in device memory
template <int NV, class T>
__global__ void dupdate_kernel(long long n, long long packs, const T* __restrict__ Z, const double* __restrict__ y, T* __restrict__ x) {
  T c[NV > 0 ? NV : 1];
#pragma unroll
  for (int v = 0; v < NV; ++v) c[v] = (T)y[v];
  combine<NV, T>(n, packs, Z, c, false, x);
}

template <int NV, class T>
static void dupdate_launch_t(long long n, const T* Z, const double* y, T* x, cudaStream_t st) {
  const long long packs = n % 4 == 0 && pack4(n, Z, x, nullptr) ? n / 4 : 0;
  dupdate_kernel<NV, T><<<vblocks(packs ? packs : n), 256, 0, st>>>(n, packs, Z, y, x);
}

template <class T, int... I>
static void dupdate_dispatch(int nv, long long n, const T* Z, const double* y, T* x, cudaStream_t st,
                             std::integer_sequence<int, I...>) {
  using F = void (*)(long long, const T*, const double*, T*, cudaStream_t);
  static const F table[] = {&dupdate_launch_t<I, T>...};
  table[nv](n, Z, y, x, st);
}

// Exactly m FGMRES iterations from x0 = 0, driven entirely on the device (no host
// synchronisation, so the call can be captured in a CUDA graph).  A flexible outer
// solve accepts this as a (variable) preconditioner.
template <class T>
static fv_status gmres_fixed_t(const fv_system* s, const T* b, T* x, int m, cudaStream_t st) {
  if (m < 1 || m > KMAX - 1) return set_error("fixed-iteration FGMRES: iterations must be in [1, 31]"), FV_EINVAL;
  fv_status rc = ensure_krylov<T>(s, m);
  if (rc) return rc;
  KrylovT<T>& k = kt<T>(s->kry);
  const long long n = s->n;
  const int lvl = FV_K_COARSE * s->level + (sizeof(T) == 4 ? FV_K_FP32 : 0);
  const bool once = s->pc.inner_gs_passes == 1;
  {
    ProfScope ps(FV_K_CGS + lvl, st);
    if ((rc = gs_step<T>(k, 0, n, b, k.V, 0, k.ad, false, st))) return rc;
  }
  for (int j = 0; j < m; ++j) {
    T* vj = k.V + (size_t)j * n;
    T* zj = k.Z + (size_t)j * n;
    if ((rc = precond_t<T>(s, vj, zj, st))) return rc;
    if ((rc = apply_t<T>(s, zj, k.w, st))) return rc;
    ProfScope ps(FV_K_CGS + lvl, st);
    if ((rc = gs_step<T>(k, j + 1, n, k.w, j + 1 < m ? k.V + (size_t)(j + 1) * n : nullptr, once ? 1 : 2, k.ad, j + 1 == m, st)))
      return rc;
  }
  ProfScope ps(FV_K_VEC, st);
  dupdate_dispatch<T>(m, n, k.Z, k.ad->y, x, st, std::make_integer_sequence<int, KMAX>{});
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

fv_status gmres_fixed32(const fv_system* s, const float* b, float* x, int m, cudaStream_t st) {
  return gmres_fixed_t<float>(s, b, x, m, st);
}

// ------------------------------------------------------------------ FGMRES
template <class T>
static fv_status gmres_t(const fv_system* s, const T* b, T* x, const fv_gmres_opts* o, fv_solve_stats* stats,
                         cudaStream_t st, bool inner) {
  auto t0 = std::chrono::steady_clock::now();
  const int m = o->restart;
  if (m < 1 || m > KMAX - 1 || o->max_it < 0) return set_error("fv_gmres_solve: restart must be in [1, 31]"), FV_EINVAL;
  fv_status rc = ensure_krylov<T>(s, m);
  if (rc) return rc;
  KrylovT<T>& k = kt<T>(s->kry);
  const long long n = s->n;
  const int lvl = FV_K_COARSE * s->level + (sizeof(T) == 4 ? FV_K_FP32 : 0);
  if (!inner) s->last_inner = 0;
  // r = b - A x
  if ((rc = apply_t<T>(s, x, k.r, st, b))) return rc;
  double beta;
  if ((rc = norm2<T>(k, n, k.r, k.V, st, &beta))) return rc;
  // the stream has been waited for and x is as it was: what fv_precond_apply calls before this one left
  if (!inner && (rc = waits_failed(s, "fv_gmres_solve: not begun, in an earlier call ", st))) return rc;
  const double r0 = beta, target = std::max(o->atol, o->rtol * r0);
  int its = 0;
  bool nan = !std::isfinite(beta);
  std::vector<double> H((m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
  while (!nan && beta > target && its < o->max_it) {
    std::fill(g.begin(), g.end(), 0.0);
    g[0] = beta;
    int j = 0;
    bool breakdown = false;
    for (; j < m; ++j) {
      T* vj = k.V + (size_t)j * n;
      T* zj = k.Z + (size_t)j * n;
      if ((rc = precond_t<T>(s, vj, zj, st))) return rc;
      if ((rc = apply_t<T>(s, zj, k.w, st))) return rc;
      const int nv = j + 1;
      {
        ProfScope ps(FV_K_CGS + lvl, st);
        // with the next basis vector (k.V holds m + 1)
        if ((rc = gs_step<T>(k, nv, n, k.w, k.V + (size_t)(j + 1) * n, 2, nullptr, false, st))) return rc;
      }
      FV_CUDA(cudaGetLastError());
      FV_CUDA(cudaMemcpyAsync(k.hhost, k.h, 3 * KMAX * sizeof(double), cudaMemcpyDeviceToHost, st));
      FV_CUDA(cudaStreamSynchronize(st));
      std::vector<double> col(j + 2);
      for (int i = 0; i <= j; ++i) col[i] = k.hhost[i] + k.hhost[KMAX + i];  // CGS2: h = h1 + h2
      const double hn = std::sqrt(k.hhost[2 * KMAX]);
      col[j + 1] = hn;
      for (int i = 0; i < j; ++i) {
        const double t = cs[i] * col[i] + sn[i] * col[i + 1];
        col[i + 1] = -sn[i] * col[i] + cs[i] * col[i + 1];
        col[i] = t;
      }
      const double den = std::hypot(col[j], col[j + 1]);
      cs[j] = col[j] / den, sn[j] = col[j + 1] / den;
      col[j] = den, col[j + 1] = 0.0;
      g[j + 1] = -sn[j] * g[j];
      g[j] = cs[j] * g[j];
      for (int i = 0; i <= j; ++i) H[i * m + j] = col[i];
      ++its;
      if (!std::isfinite(hn) || !std::isfinite(g[j + 1])) {
        nan = true;
        ++j;
        break;
      }
      if (hn == 0.0) breakdown = true;
      if (std::fabs(g[j + 1]) <= target || its >= o->max_it || breakdown) {
        ++j;
        break;
      }
    }
    const int kk = std::min(j, m);
    if (!nan) {
      for (int i = kk - 1; i >= 0; --i) {
        double sacc = g[i];
        for (int q = i + 1; q < kk; ++q) sacc -= H[i * m + q] * y[q];
        y[i] = sacc / H[i * m + i];
      }
      Coef<T> c{};
      for (int i = 0; i < kk; ++i) c.c[i] = (T)y[i];
      ProfScope ps(FV_K_VEC, st);
      update_dispatch<T>(kk, n, k.Z, c, x, st, std::make_integer_sequence<int, KMAX>{});
      FV_CUDA(cudaGetLastError());
    }
    if ((rc = apply_t<T>(s, x, k.r, st, b))) return rc;
    if ((rc = norm2<T>(k, n, k.r, k.V, st, &beta))) return rc;
    if (!std::isfinite(beta)) nan = true;
    if (breakdown) break;
  }
  if ((rc = waits_failed(s, "fv_gmres_solve: ", st))) return rc;
  const bool conv = !nan && beta <= target;
  if (stats) {
    stats->iters = its;
    stats->fallback = 0;
    stats->inner_iters = s->last_inner;
    stats->converged = conv ? 1 : 0;
    stats->r0 = r0;
    stats->rfinal = beta;
    stats->time_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  }
  if (nan) return set_error("fv_gmres_solve: NaN or Inf residual"), FV_ENAN;
  if (!conv) return set_error("fv_gmres_solve: max_it reached before the tolerance"), FV_ENOCONV;
  return FV_OK;
}

// Top-level solves of a system with a learned coarse correction: optional
// learned initial guess, then FGMRES for at most one restart cycle; if that
// ends without convergence, the plain coarse solve finishes from the last
// finite iterate with the original absolute target max(atol, rtol ||b - A x0||)
// and the iterations left.
static fv_status gmres_learned(const fv_system* s, const double* b, double* x, const fv_gmres_opts* o,
                               fv_solve_stats* stats, cudaStream_t st) {
  fv_system* sm = const_cast<fv_system*>(s);
  const size_t bytes = (size_t)s->n * sizeof(double);
  FV_CUDA(cudaMemcpyAsync(s->xbak, x, bytes, cudaMemcpyDeviceToDevice, st));
  fv_solve_stats s1{};
  fv_status rc = FV_OK;
  double r0 = -1.0;
  if (s->learned_flags & FV_LEARN_GUESS) {
    // the tolerance stays relative to the caller's x0
    const fv_gmres_opts o0{o->restart, 0, o->atol, o->rtol};
    fv_status rr = gmres_t<double>(s, b, x, &o0, &s1, st, false);
    if (rr && rr != FV_ENOCONV && rr != FV_ENAN) return rr;
    r0 = s1.r0;
    if ((rc = learned_guess(s, b, x, st))) return rc;
  }
  fv_gmres_opts o1 = *o;
  if (r0 >= 0.0) o1.atol = std::max(o->atol, o->rtol * r0), o1.rtol = 0.0;
  // the learned preconditioner gets one restart cycle; a solve it has not finished by then
  // (a stall, or a network that does not fit this problem) goes on with the plain one
  o1.max_it = std::min(o->max_it, o->restart);
  rc = gmres_t<double>(s, b, x, &o1, &s1, st, false);
  int inner = s->last_inner;
  if (r0 >= 0.0) s1.r0 = r0;
  if (rc == FV_ENOCONV || rc == FV_ENAN) {
    if (rc == FV_ENAN) FV_CUDA(cudaMemcpyAsync(x, s->xbak, bytes, cudaMemcpyDeviceToDevice, st));
    fv_gmres_opts o2 = *o;
    o2.max_it = std::max(0, o->max_it - s1.iters);
    o2.atol = std::max(o->atol, o->rtol * s1.r0), o2.rtol = 0.0;
    fv_solve_stats s2{};
    set_learned_active(sm, 0);
    rc = gmres_t<double>(s, b, x, &o2, &s2, st, false);
    set_learned_active(sm, 1);
    inner += s->last_inner;
    s1.iters += s2.iters, s1.converged = s2.converged, s1.rfinal = s2.rfinal, s1.time_ms += s2.time_ms;
    s1.fallback = 1;
  }
  s->last_inner = inner;
  s1.inner_iters = inner;
  if (stats) *stats = s1;
  return rc;
}

fv_status gmres(const fv_system* s, const double* b, double* x, const fv_gmres_opts* o, fv_solve_stats* stats,
                cudaStream_t st, bool inner) {
  if (!inner && s->net) return gmres_learned(s, b, x, o, stats, st);
  return gmres_t<double>(s, b, x, o, stats, st, inner);
}

fv_status gmres32(const fv_system* s, const float* b, float* x, const fv_gmres_opts* o, fv_solve_stats* stats,
                  cudaStream_t st) {
  return gmres_t<float>(s, b, x, o, stats, st, true);
}

// volume-weighted mean removal of the first component (Neumann pressure gauge)
// I: the index type, 32-bit whenever N allows (32-bit divisions in the index decomposition)
template <class T, class I>
__global__ void wsum_kernel(long long N, int Ns, int Nr, const double* __restrict__ crf,
                            const double* __restrict__ rc, double hr2, const T* __restrict__ x, double* __restrict__ part) {
  double acc[KMAX];
  acc[0] = 0.0, acc[1] = 0.0;
  const I ns2 = (I)Ns * Ns;
  for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < (I)N; e += (I)gridDim.x * blockDim.x) {
    const int ij = (int)(e % ns2);
    const int k = (int)((e / ns2) % Nr);
    // sigma h_s^2 / h_r times (r h_r)^2: multiplications (a division an element was a third of the kernel's FP64 work)
    const double V = crf[ij] * (rc[k] * rc[k] * hr2);
    acc[0] += V * (double)x[e];
    acc[1] += V;
  }
  block_store(acc, 2, part);
}

template <class T>
__global__ void shift_kernel(long long N, const double* __restrict__ sums, T* __restrict__ x) {
  const T mean = (T)(sums[0] / sums[1]);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < N; e += (long long)gridDim.x * blockDim.x)
    x[e] -= mean;
}

template <class T>
static fv_status wmr(const fv_grid* g, T* x, cudaStream_t st, double* part, double* sums) {
  const Geo& G = g->geo;
  ProfScope ps(FV_K_VEC, st);
  if (G.N < (1LL << 31) - (1LL << 24))
    wsum_kernel<T, int><<<RBLOCKS, RTHREADS, 0, st>>>(G.N, G.Ns, G.Nr, G.crf, G.rc, G.hr * G.hr, x, part);
  else
    wsum_kernel<T, long long><<<RBLOCKS, RTHREADS, 0, st>>>(G.N, G.Ns, G.Nr, G.crf, G.rc, G.hr * G.hr, x, part);
  reduce_kernel<<<1, RTHREADS, 0, st>>>(part, RBLOCKS, 2, sums);
  shift_kernel<T><<<vblocks(G.N), 256, 0, st>>>(G.N, sums, x);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

fv_status weighted_mean_remove(const fv_grid* g, double* x, cudaStream_t st, double* part, double* sums) {
  return wmr<double>(g, x, st, part, sums);
}

fv_status weighted_mean_remove32(const fv_grid* g, float* x, cudaStream_t st, double* part, double* sums) {
  return wmr<float>(g, x, st, part, sums);
}

}  // namespace fv
