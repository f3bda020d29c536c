// Many right-hand sides of one system solved together (fv_gmres_solve_batch).
//
// The same right-preconditioned restarted FGMRES as fv_gmres_solve (paper
// Sec. 3.3), run in lock-step for nrhs right-hand sides: one batched launch per
// step for all of them, each right-hand side with its own Hessenberg matrix,
// Givens rotations, tolerance and convergence flag (columns of a converged
// right-hand side are no longer used).  The preconditioner is the system's
// one-level RAS: FP64 subdomain solves, or FP32 subdomain solves inside the
// FP64 outer FGMRES when the system was assembled with FV_PREC_FP32.
//
// Batched RAS sweeps: the streamed sweeps over (subdomain, right-hand side) tasks.  Subdomains too wide for them: each
// CTA takes a (subdomain, group of G right-hand sides) task and applies every factor it loads to the G right-hand
// sides; the launch is persistent, as many CTAs as fit on the GPU pull tasks from an atomic counter in decreasing
// subdomain size, and G is chosen by timing each candidate on the first call for a given nrhs (kept in the system).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <vector>

#include "stencil.cuh"

namespace fv {

constexpr int BK = 32;        // max basis vectors
constexpr int BBLOCKS = 152;  // reduction blocks per right-hand side at most
// about four blocks an SM over all right-hand sides: every block adds a reduction of its FP64 partial sums (five
// DADDs a warp and value on the slow pipe), which with 152 blocks a right-hand side was over half of a pass
static int rblocks(int nrhs) { return std::max(16, std::min(BBLOCKS, 608 / nrhs)); }
constexpr int BTHREADS = 256;

// device-side Arnoldi bookkeeping of one right-hand side (Hessenberg column-major H[j * BK + i])
struct BatchArn {
  double H[BK * BK];
  double cs[BK], sn[BK], g[BK + 1], y[BK];
  double beta, r0, target;
  int its, kk, done;
  int max_it;  // of this solve: kept here, since a captured cycle is replayed by solves with other limits
};

struct BatchWork {
  int nrhs = 0, m = 0, G = 0;
  long long n = 0;
  double *gh = nullptr, *V = nullptr, *Z = nullptr, *w = nullptr, *r = nullptr;
  double *part = nullptr, *h = nullptr, *hhost = nullptr, *coef = nullptr, *coef_host = nullptr;
  unsigned* ticket = nullptr;
  void* loc = nullptr;     // [nrhs][total_cells * d] sweep vectors (factor type)
  void* ring = nullptr;    // global rings when they do not fit in shared memory
  int* task = nullptr;     // persistent-launch task counters (fwd, bwd)
  int ctas = 0;            // persistent CTAs
  size_t smem = 0;
  int ring_in_smem = 0;
  BatchArn* arn = nullptr;       // [nrhs] device Arnoldi state
  BatchArn* arn_host = nullptr;  // pinned copy for the convergence check after a cycle
  cudaGraphExec_t cycle = nullptr;  // one restart cycle, captured for (B, X, m)
  const double* gB = nullptr;
  double* gX = nullptr;
  int gm = 0, warm = 0;
};

void free_batch(BatchWork* b) {
  if (!b) return;
  cudaFree(b->gh), cudaFree(b->V), cudaFree(b->Z), cudaFree(b->w), cudaFree(b->r), cudaFree(b->part), cudaFree(b->h);
  cudaFree(b->coef), cudaFree(b->ticket), cudaFree(b->loc), cudaFree(b->ring), cudaFree(b->task);
  cudaFreeHost(b->hhost), cudaFreeHost(b->coef_host);
  cudaFree(b->arn), cudaFreeHost(b->arn_host);
  if (b->cycle) cudaGraphExecDestroy(b->cycle);
  delete b;
}

// ------------------------------------------------------------------ batched RAS
__device__ __forceinline__ void tables(int nx, int ny, int nz, int levels, int* lvl, int* rowoff) {
  for (int L = threadIdx.x; L < levels; L += blockDim.x) {
    int cnt = 0;
    for (int j = 0; j < ny; ++j) {
      rowoff[L * ny + j] = cnt;
      const int lo = max(0, L - 2 * j - (nz - 1)), hi = min(nx - 1, L - 2 * j);
      if (hi >= lo) cnt += hi - lo + 1;
    }
    lvl[L + 1] = cnt;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    lvl[0] = 0;
    for (int L = 0; L < levels; ++L) lvl[L + 1] += lvl[L];
  }
  __syncthreads();
}

struct BatchRas {
  const long long* cell_off;
  const int* dims;
  const int* lpt;
  const long long* gmap_p;
  const unsigned char* owned_p;
  int count, ngroups, nrhs, max_cols;
  long long N, rs, zs, total;  // cells per component, input / output stride per rhs, packed box cells
  int ring_in_smem;
};

// task -> (subdomain in decreasing size, group of right-hand sides)
__device__ __forceinline__ bool next_task(int* counter, const BatchRas& R, int* sd, int* grp) {
  __shared__ int t;
  if (threadIdx.x == 0) t = atomicAdd(counter, 1);
  __syncthreads();
  const int task = t;
  __syncthreads();
  if (task >= R.count * R.ngroups) return false;
  *sd = R.lpt[task / R.ngroups];
  *grp = task % R.ngroups;
  return true;
}

// forward sweep with the gather of R_i^delta r fused in; ring = [4][cols][D][Gc]
template <class T, int D, int GC>
__global__ void __launch_bounds__(512) ras_fwd_batch_kernel(BatchRas R, const T* __restrict__ F, T* __restrict__ loc,
                                                            T* ring_g, const double* __restrict__ r, int* counter) {
  extern __shared__ __align__(16) unsigned char smem[];
  const size_t rb = R.ring_in_smem ? ((4 * (size_t)R.max_cols * D * GC * sizeof(T) + 15) / 16 * 16) : 0;
  T* ring = R.ring_in_smem ? (T*)smem : ring_g + (size_t)blockIdx.x * 4 * R.max_cols * D * GC;
  int sd, grp;
  while (next_task(counter, R, &sd, &grp)) {
    const int nx = R.dims[3 * sd], ny = R.dims[3 * sd + 1], nz = R.dims[3 * sd + 2];
    const int levels = (nx - 1) + 2 * (ny - 1) + (nz - 1) + 1, ncols = nx * ny;
    int* lvl = (int*)(smem + rb);
    int* rowoff = lvl + levels + 1;
    tables(nx, ny, nz, levels, lvl, rowoff);
    const long long base = R.cell_off[sd], nc = R.cell_off[sd + 1] - base;
    const T* Fb = F + base * (10 * D + D * D);
    const int r0 = grp * GC, gn = min(GC, R.nrhs - r0);
    for (int L = 0; L < levels; ++L) {
      for (int col = threadIdx.x; col < ncols; col += blockDim.x) {
        const int j = col / nx, i = col - j * nx, k = L - i - 2 * j;
        if (k < 0 || k >= nz) continue;
        const long long pos = lvl[L] + rowoff[L * ny + j] + i - max(0, L - 2 * j - (nz - 1));
        T fl[5 * D], fd[D * D];
#pragma unroll
        for (int q = 0; q < 5 * D; ++q) fl[q] = Fb[q * nc + pos];
#pragma unroll
        for (int a = 1; a < D; ++a)
#pragma unroll
          for (int c = 0; c < a; ++c) fd[a * D + c] = Fb[(5 * D + a * D + c) * nc + pos];
        const long long g = R.gmap_p[base + pos];
        T* rp = ring + (size_t)((k & 3) * ncols) * D * GC;
        const T* rm = ring + (size_t)(((k - 1) & 3) * ncols + col) * D * GC;
        for (int gg = 0; gg < gn; ++gg) {
          const int rhs = r0 + gg;
          T y[D];
#pragma unroll
          for (int a = 0; a < D; ++a) y[a] = g >= 0 ? (T)r[rhs * R.rs + a * R.N + g] : T(0);
#pragma unroll
          for (int a = 0; a < D; ++a) {
            if (k > 0) y[a] -= fl[0 * D + a] * rm[a * GC + gg];
            if (i > 0 && j > 0) y[a] -= fl[1 * D + a] * rp[((col - nx - 1) * D + a) * GC + gg];
            if (j > 0) y[a] -= fl[2 * D + a] * rp[((col - nx) * D + a) * GC + gg];
            if (j > 0 && i + 1 < nx) y[a] -= fl[3 * D + a] * rp[((col - nx + 1) * D + a) * GC + gg];
            if (i > 0) y[a] -= fl[4 * D + a] * rp[((col - 1) * D + a) * GC + gg];
#pragma unroll
            for (int c = 0; c < a; ++c) y[a] -= fd[a * D + c] * y[c];
          }
          T* lb = loc + rhs * R.total * D + base * D;
#pragma unroll
          for (int a = 0; a < D; ++a) rp[(col * D + a) * GC + gg] = y[a], lb[a * nc + pos] = y[a];
        }
      }
      __syncthreads();
    }
  }
}

// backward sweep with the scatter of the owned cells, (R_i^0)^T, fused in
template <class T, int D, int GC>
__global__ void __launch_bounds__(512) ras_bwd_batch_kernel(BatchRas R, const T* __restrict__ F, T* __restrict__ loc,
                                                            T* ring_g, double* __restrict__ z, int* counter) {
  extern __shared__ __align__(16) unsigned char smem[];
  const size_t rb = R.ring_in_smem ? ((4 * (size_t)R.max_cols * D * GC * sizeof(T) + 15) / 16 * 16) : 0;
  T* ring = R.ring_in_smem ? (T*)smem : ring_g + (size_t)blockIdx.x * 4 * R.max_cols * D * GC;
  constexpr int U = 5 * D + D * D;
  int sd, grp;
  while (next_task(counter, R, &sd, &grp)) {
    const int nx = R.dims[3 * sd], ny = R.dims[3 * sd + 1], nz = R.dims[3 * sd + 2];
    const int levels = (nx - 1) + 2 * (ny - 1) + (nz - 1) + 1, ncols = nx * ny;
    int* lvl = (int*)(smem + rb);
    int* rowoff = lvl + levels + 1;
    tables(nx, ny, nz, levels, lvl, rowoff);
    const long long base = R.cell_off[sd], nc = R.cell_off[sd + 1] - base;
    const T* Fb = F + base * (10 * D + D * D);
    const int r0 = grp * GC, gn = min(GC, R.nrhs - r0);
    for (int L = levels - 1; L >= 0; --L) {
      for (int col = threadIdx.x; col < ncols; col += blockDim.x) {
        const int j = col / nx, i = col - j * nx, k = L - i - 2 * j;
        if (k < 0 || k >= nz) continue;
        const long long pos = lvl[L] + rowoff[L * ny + j] + i - max(0, L - 2 * j - (nz - 1));
        T fu[5 * D], fd[D * D];
#pragma unroll
        for (int q = 0; q < 5 * D; ++q) fu[q] = Fb[(U + q) * nc + pos];
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int c = a; c < D; ++c) fd[a * D + c] = Fb[(5 * D + a * D + c) * nc + pos];
        const bool own = R.owned_p[base + pos];
        const long long g = R.gmap_p[base + pos];
        T* rp = ring + (size_t)((k & 3) * ncols) * D * GC;
        const T* rq = ring + (size_t)(((k + 1) & 3) * ncols + col) * D * GC;
        for (int gg = 0; gg < gn; ++gg) {
          const int rhs = r0 + gg;
          T* lb = loc + rhs * R.total * D + base * D;
          T x[D];
#pragma unroll
          for (int a = 0; a < D; ++a) x[a] = lb[a * nc + pos];
#pragma unroll
          for (int a = D - 1; a >= 0; --a) {
#pragma unroll
            for (int c = a + 1; c < D; ++c) x[a] -= fd[a * D + c] * x[c];
            if (i + 1 < nx) x[a] -= fu[0 * D + a] * rp[((col + 1) * D + a) * GC + gg];
            if (i > 0 && j + 1 < ny) x[a] -= fu[1 * D + a] * rp[((col + nx - 1) * D + a) * GC + gg];
            if (j + 1 < ny) x[a] -= fu[2 * D + a] * rp[((col + nx) * D + a) * GC + gg];
            if (i + 1 < nx && j + 1 < ny) x[a] -= fu[3 * D + a] * rp[((col + nx + 1) * D + a) * GC + gg];
            if (k + 1 < nz) x[a] -= fu[4 * D + a] * rq[a * GC + gg];
            x[a] *= fd[a * D + a];  // 1 / U_aa
          }
#pragma unroll
          for (int a = 0; a < D; ++a) rp[(col * D + a) * GC + gg] = x[a];
          if (own)
#pragma unroll
            for (int a = 0; a < D; ++a) z[rhs * R.zs + a * R.N + g] = (double)x[a];
        }
      }
      __syncthreads();
    }
  }
}

static size_t batch_tables_bytes(const fv_system* s) {
  // widest level table over the boxes, as in the single-RHS sweeps
  const Subdomains& S = s->subs;
  std::vector<int> dims(3 * S.count);
  cudaMemcpy(dims.data(), S.dims, dims.size() * sizeof(int), cudaMemcpyDeviceToHost);
  size_t tab = 0;
  for (int sd = 0; sd < S.count; ++sd) {
    const int nx = dims[3 * sd], ny = dims[3 * sd + 1], nz = dims[3 * sd + 2];
    const int levels = (nx - 1) + 2 * (ny - 1) + (nz - 1) + 1;
    tab = std::max(tab, (size_t)(levels + 1 + levels * ny) * sizeof(int));
  }
  return tab;
}

template <class T, int D, int GC>
static fv_status ras_batch_t(const fv_system* s, BatchWork* bw, int nrhs, const double* r, long long rs, double* z,
                             long long zs, cudaStream_t st) {
  const Subdomains& S = s->subs;
  BatchRas R{S.cell_off, S.dims, S.lpt, S.gmap_p, S.owned_p, S.count, (nrhs + GC - 1) / GC, nrhs, S.max_cols,
             s->grid->geo.N, rs, zs, S.total_cells, bw->ring_in_smem};
  const int threads = std::min(512, ((S.max_cols + 31) / 32) * 32);
  FV_CUDA(cudaMemsetAsync(bw->task, 0, 2 * sizeof(int), st));
  {
    ProfScope ps(s->kind == FV_VTBE ? FV_K_RAS_FWD_VTBE : FV_K_RAS_FWD_PPBE, st);
    ras_fwd_batch_kernel<T, D, GC><<<bw->ctas, threads, bw->smem, st>>>(R, (const T*)S.F, (T*)bw->loc, (T*)bw->ring,
                                                                      r, bw->task);
  }
  FV_CUDA(cudaGetLastError());
  {
    ProfScope ps(s->kind == FV_VTBE ? FV_K_RAS_BWD_VTBE : FV_K_RAS_BWD_PPBE, st);
    ras_bwd_batch_kernel<T, D, GC><<<bw->ctas, threads, bw->smem, st>>>(R, (const T*)S.F, (T*)bw->loc, (T*)bw->ring,
                                                                      z, bw->task + 1);
  }
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

template <class T, int D, int GC>
static fv_status setup_batch_ras(const fv_system* s, BatchWork* bw, size_t tab) {
  const Subdomains& S = s->subs;
  const int threads = std::min(512, ((S.max_cols + 31) / 32) * 32);
  const size_t ring = 4 * (size_t)S.max_cols * D * GC * sizeof(T), ring_al = (ring + 15) / 16 * 16;
  int dev = 0, limit = 0, sms = 0;
  FV_CUDA(cudaGetDevice(&dev));
  FV_CUDA(cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  FV_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // the dynamic limit is the opt-in maximum less the kernel's static shared memory
  cudaFuncAttributes fa{}, fb{};
  FV_CUDA(cudaFuncGetAttributes(&fa, ras_fwd_batch_kernel<T, D, GC>));
  FV_CUDA(cudaFuncGetAttributes(&fb, ras_bwd_batch_kernel<T, D, GC>));
  const int dyn = limit - (int)std::max(fa.sharedSizeBytes, fb.sharedSizeBytes);
  bw->ring_in_smem = ring_al + tab <= (size_t)dyn;
  bw->smem = (bw->ring_in_smem ? ring_al : 0) + tab;
  if (bw->smem > (size_t)dyn) return set_error("fv_gmres_solve_batch: sweep tables exceed shared memory"), FV_EINVAL;
  FV_CUDA(cudaFuncSetAttribute(ras_fwd_batch_kernel<T, D, GC>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
  FV_CUDA(cudaFuncSetAttribute(ras_bwd_batch_kernel<T, D, GC>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
  int per_sm = 0;
  FV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ras_fwd_batch_kernel<T, D, GC>, threads, bw->smem));
  const int tasks = S.count * ((bw->nrhs + GC - 1) / GC);
  bw->ctas = std::max(1, std::min(tasks, std::max(1, per_sm) * sms));
  if (!bw->ring_in_smem) {
    cudaFree(bw->ring);
    bw->ring = nullptr;
    if (cudaMalloc(&bw->ring, (size_t)bw->ctas * ring) != cudaSuccess)
      return set_error("fv_gmres_solve_batch: ring allocation failed"), FV_ENOMEM;
  }
  return FV_OK;
}

template <class T, int D>
static fv_status ras_batch_g(const fv_system* s, BatchWork* bw, int nrhs, const double* r, long long rs, double* z,
                             long long zs, cudaStream_t st) {
  switch (bw->G) {
    case 1: return ras_batch_t<T, D, 1>(s, bw, nrhs, r, rs, z, zs, st);
    case 2: return ras_batch_t<T, D, 2>(s, bw, nrhs, r, rs, z, zs, st);
    case 4: return ras_batch_t<T, D, 4>(s, bw, nrhs, r, rs, z, zs, st);
    default: return ras_batch_t<T, D, 8>(s, bw, nrhs, r, rs, z, zs, st);
  }
}

template <class T, int D>
static fv_status setup_g(const fv_system* s, BatchWork* bw, size_t tab) {
  switch (bw->G) {
    case 1: return setup_batch_ras<T, D, 1>(s, bw, tab);
    case 2: return setup_batch_ras<T, D, 2>(s, bw, tab);
    case 4: return setup_batch_ras<T, D, 4>(s, bw, tab);
    default: return setup_batch_ras<T, D, 8>(s, bw, tab);
  }
}

static fv_status ras_batch(const fv_system* s, BatchWork* bw, int nrhs, const double* r, long long rs, double* z,
                           long long zs, cudaStream_t st) {
  if (s->subs.st.on) {
    ProfScope ps(s->kind == FV_VTBE ? FV_K_RAS_FWD_VTBE : FV_K_RAS_FWD_PPBE, st);
    return ras_stream64(s, nrhs, r, rs, z, zs, bw->loc, st);
  }
  if (s->d == 2)
    return s->subs.fp32 ? ras_batch_g<float, 2>(s, bw, nrhs, r, rs, z, zs, st)
                        : ras_batch_g<double, 2>(s, bw, nrhs, r, rs, z, zs, st);
  return s->subs.fp32 ? ras_batch_g<float, 7>(s, bw, nrhs, r, rs, z, zs, st)
                      : ras_batch_g<double, 7>(s, bw, nrhs, r, rs, z, zs, st);
}

static fv_status setup_ras(const fv_system* s, BatchWork* bw, size_t tab) {
  if (s->d == 2) return s->subs.fp32 ? setup_g<float, 2>(s, bw, tab) : setup_g<double, 2>(s, bw, tab);
  return s->subs.fp32 ? setup_g<float, 7>(s, bw, tab) : setup_g<double, 7>(s, bw, tab);
}

// ------------------------------------------------------------------ batched vectors
__device__ __forceinline__ double bwarp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// per right-hand side (grid.y): mode 0 dots V^T w, mode 1 w -= V h then dots, mode 2 w -= V h then
// ||w||^2; the last block of each right-hand side sums the partials in a fixed order into out
template <int NV>
__global__ void __launch_bounds__(BTHREADS) cgs_batch_kernel(long long n, const double* __restrict__ V,
                                                             long long vstride, const double* __restrict__ h,
                                                             double* __restrict__ w, double* __restrict__ part,
                                                             double* __restrict__ out, unsigned* ticket, int mode) {
  const int rhs = blockIdx.y;
  V += rhs * vstride;
  w += rhs * n;
  h += rhs * 3 * BK;
  part += (size_t)rhs * BK * gridDim.x;
  out += rhs * 3 * BK;
  double acc[NV > 0 ? NV : 1], hv[NV > 0 ? NV : 1], nrm = 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0, hv[v] = mode > 0 ? h[v] : 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    double we = w[e];
    if (mode > 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) we -= hv[v] * V[v * n + e];
      w[e] = we;
    }
    if (mode < 2) {
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += V[v * n + e] * we;
    } else {
      nrm += we * we;
    }
  }
  // eight values at a time through shared memory: a warp adds eight partial sums a lane, then its butterfly
  __shared__ double red[8][BTHREADS];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nvv = mode < 2 ? NV : 1;
  if (mode == 2) acc[0] = nrm;
#pragma unroll
  for (int v0 = 0; v0 < (NV > 0 ? NV : 1); v0 += 8) {
    if (v0 >= nvv) break;
    if (v0) __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v0 + u < (NV > 0 ? NV : 1)) red[u][threadIdx.x] = acc[v0 + u < (NV > 0 ? NV : 1) ? v0 + u : 0];
    __syncthreads();
    if (v0 + wid < nvv) {
      double t = 0.0;
#pragma unroll
      for (int u = 0; u < BTHREADS / 32; ++u) t += red[wid][32 * u + lane];
      t = bwarp_sum(t);
      if (lane == 0) part[(v0 + wid) * gridDim.x + blockIdx.x] = t;
    }
  }
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket + rhs, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int v = wid; v < nvv; v += BTHREADS / 32) {
    double t = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + v * gridDim.x + b);
    t = bwarp_sum(t);
    if (lane == 0) out[(mode == 2 ? 2 * BK : mode * BK) + v] = t;
  }
  if (threadIdx.x == 0) ticket[rhs] = 0u;
}

template <int... I>
static void cgs_batch_dispatch(int nv, dim3 grid, long long n, const double* V, long long vs, const double* h, double* w,
                               double* part, double* out, unsigned* ticket, int mode, cudaStream_t st,
                               std::integer_sequence<int, I...>) {
  using Fn = void (*)(long long, const double*, long long, const double*, double*, double*, double*, unsigned*, int);
  static const Fn table[] = {&cgs_batch_kernel<I>...};
  table[nv]<<<grid, BTHREADS, 0, st>>>(n, V, vs, h, w, part, out, ticket, mode);
}

// out_r = a_r x_r + b y_r  (a per right-hand side from coef[rhs]; coef null: a = -1)
__global__ void scale_batch_kernel(long long n, const double* __restrict__ coef, const double* __restrict__ x,
                                   long long xs, double b, const double* __restrict__ y, double* __restrict__ out,
                                   long long os) {
  const int rhs = blockIdx.y;
  const double a = coef ? coef[rhs] : -1.0;
  x += rhs * xs, out += rhs * os;
  if (y) y += rhs * n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = a * x[e] + (y ? b * y[e] : 0.0);
}

// x_r += sum_v y_{r,v} Z_{r,v}
__global__ void update_batch_kernel(long long n, int kk, const double* __restrict__ Z, long long zs,
                                    const double* __restrict__ y, double* __restrict__ x) {
  const int rhs = blockIdx.y;
  Z += rhs * zs, x += rhs * n, y += rhs * BK;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    double s = x[e];
    for (int v = 0; v < kk; ++v) s += y[v] * Z[v * n + e];
    x[e] = s;
  }
}

static int bblocks(long long n) { return (int)std::min<long long>((n + 255) / 256, 1024); }

static fv_status ensure_batch(const fv_system* s, int nrhs, int m) {
  fv_system* sm = const_cast<fv_system*>(s);
  BatchWork* bw = sm->batch;
  if (bw && bw->nrhs == nrhs && bw->m >= m) return FV_OK;
  free_batch(bw);
  bw = sm->batch = new BatchWork();
  bw->nrhs = nrhs, bw->m = m, bw->n = s->n;
  const size_t n = (size_t)s->n, R = (size_t)nrhs;
  const size_t gsz = (size_t)s->d * 6 * 4 * s->grid->h.Nr * (s->grid->h.Ns + 2);
  const size_t es = s->subs.fp32 ? 4 : 8;
  const long long cells = s->subs.st.on ? s->subs.st.sT : s->subs.total_cells;
  if (cudaMalloc(&bw->gh, gsz * R * 8) || cudaMalloc(&bw->V, (m + 1) * n * R * 8) || cudaMalloc(&bw->Z, m * n * R * 8) ||
      cudaMalloc(&bw->w, n * R * 8) || cudaMalloc(&bw->r, n * R * 8) || cudaMalloc(&bw->part, R * BK * BBLOCKS * 8) ||
      cudaMalloc(&bw->h, R * 3 * BK * 8) || cudaMalloc(&bw->coef, R * BK * 8) || cudaMalloc(&bw->ticket, R * 4) ||
      cudaMalloc(&bw->loc, (size_t)cells * s->d * R * es) || cudaMalloc(&bw->task, 2 * sizeof(int)) ||
      cudaMallocHost(&bw->hhost, R * 3 * BK * 8) || cudaMallocHost(&bw->coef_host, R * BK * 8) ||
      cudaMalloc(&bw->arn, R * sizeof(BatchArn)) || cudaMallocHost(&bw->arn_host, R * sizeof(BatchArn)) ||
      cudaMemset(bw->ticket, 0, R * 4)) {
    free_batch(bw);
    sm->batch = nullptr;
    return set_error("fv_gmres_solve_batch: device allocation failed"), FV_ENOMEM;
  }
  if (s->subs.st.on) {
    FV_CUDA(cudaMemset(bw->loc, 0, (size_t)cells * s->d * R * es));  // padding cells are copied, never used
    return FV_OK;
  }
  // autotune the right-hand-side group G of the RAS sweeps on this system and batch size
  const size_t tab = batch_tables_bytes(s);
  FV_CUDA(cudaMemset(bw->r, 0, n * R * 8));
  float best = 1e30f;
  int bestG = 1;
  cudaEvent_t e0, e1;
  FV_CUDA(cudaEventCreate(&e0));
  FV_CUDA(cudaEventCreate(&e1));
  const int cand[4] = {1, 2, 4, 8};
  fv_status rc = FV_OK;
  for (int G : cand) {
    if (G > nrhs && G != 1) break;
    bw->G = G;
    if ((rc = setup_ras(s, bw, tab))) break;
    if ((rc = ras_batch(s, bw, nrhs, bw->r, n, bw->w, n, 0))) break;  // warm-up
    cudaEventRecord(e0);
    for (int t = 0; t < 3; ++t)
      if ((rc = ras_batch(s, bw, nrhs, bw->r, n, bw->w, n, 0))) break;
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) best = ms, bestG = G;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  bw->G = bestG;
  return setup_ras(s, bw, tab);
}

// after r = B - A X and its squared norm (h[2 BK] per right-hand side): beta, the target and the iteration limit on
// the first call (atol, rtol and max_it are read there only: a captured cycle holds those of the solve that captured
// it), the convergence flag, 1 / beta into coef, g = beta e_1 (one thread per right-hand side)
__global__ void batch_start_kernel(int nrhs, BatchArn* __restrict__ arn, const double* __restrict__ h,
                                   double* __restrict__ coef, int first, double atol, double rtol, int max_it) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nrhs) return;
  BatchArn& a = arn[t];
  const double beta = sqrt(h[t * 3 * BK + 2 * BK]);
  if (first) a.r0 = beta, a.target = fmax(atol, rtol * beta), a.its = 0, a.max_it = max_it;
  a.beta = beta;
  a.done = !(isfinite(beta) && beta > a.target && a.its < a.max_it);
  a.kk = 0;
  for (int i = 0; i <= BK; ++i) a.g[i] = 0.0;
  for (int i = 0; i < BK; ++i) a.y[i] = 0.0;
  a.g[0] = a.done ? 0.0 : beta;
  coef[t] = a.done ? 0.0 : 1.0 / beta;
}

// column j of every active right-hand side's Hessenberg from the two Gram-Schmidt passes (h = h1 + h2,
// h_{j+1,j} = sqrt(||w||^2)), previous rotations, a new rotation, the right-hand side update; the next basis
// vector's scale 1 / h_{j+1,j} into coef, 0 once converged (its later columns are zero and unused)
__global__ void batch_givens_kernel(int nrhs, int j, BatchArn* __restrict__ arn, const double* __restrict__ h,
                                    double* __restrict__ coef) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nrhs) return;
  BatchArn& a = arn[t];
  if (a.done) {
    coef[t] = 0.0;
    return;
  }
  const double* hh = h + t * 3 * BK;
  double col[BK + 1];
  for (int i = 0; i <= j; ++i) col[i] = hh[i] + hh[BK + i];
  const double hn = sqrt(hh[2 * BK]);
  col[j + 1] = hn;
  for (int i = 0; i < j; ++i) {
    const double x = a.cs[i] * col[i] + a.sn[i] * col[i + 1];
    col[i + 1] = -a.sn[i] * col[i] + a.cs[i] * col[i + 1];
    col[i] = x;
  }
  const double den = hypot(col[j], col[j + 1]);
  a.cs[j] = den > 0 ? col[j] / den : 1.0, a.sn[j] = den > 0 ? col[j + 1] / den : 0.0;
  col[j] = den;
  a.g[j + 1] = -a.sn[j] * a.g[j];
  a.g[j] = a.cs[j] * a.g[j];
  for (int i = 0; i <= j; ++i) a.H[j * BK + i] = col[i];
  ++a.its;
  a.kk = j + 1;
  if (fabs(a.g[j + 1]) <= a.target || a.its >= a.max_it || !(hn > 0.0) || !isfinite(hn)) {
    a.done = 1;
    coef[t] = 0.0;
  } else {
    coef[t] = 1.0 / hn;
  }
}

// y of the least-squares problem (back substitution over each right-hand side's kk columns) into coef
__global__ void batch_lsq_kernel(int nrhs, BatchArn* __restrict__ arn, double* __restrict__ coef) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nrhs) return;
  BatchArn& a = arn[t];
  double* y = coef + t * BK;
  for (int i = 0; i < BK; ++i) y[i] = 0.0;
  for (int i = a.kk - 1; i >= 0; --i) {
    double s = a.g[i];
    for (int q = i + 1; q < a.kk; ++q) s -= a.H[q * BK + i] * y[q];
    y[i] = a.H[i * BK + i] != 0.0 ? s / a.H[i * BK + i] : 0.0;
  }
}

// r = B - A X, its norm, and the start of a cycle (no host synchronisation)
static fv_status batch_residual(const fv_system* s, BatchWork* bw, int nrhs, const double* B, const double* X,
                                const fv_gmres_opts* o, int first, cudaStream_t st) {
  const long long n = s->n;
  const dim3 gv(bblocks(n), nrhs), gc(rblocks(nrhs), nrhs);
  fv_status rc;
  if ((rc = apply_op_batch(s, nrhs, X, n, bw->r, n, bw->gh, st))) return rc;
  scale_batch_kernel<<<gv, 256, 0, st>>>(n, nullptr, bw->r, n, 1.0, B, bw->r, n);
  cgs_batch_dispatch(0, gc, n, bw->r, n, bw->h, bw->r, bw->part, bw->h, bw->ticket, 2, st,
                     std::make_integer_sequence<int, BK>{});
  batch_start_kernel<<<(nrhs + 31) / 32, 32, 0, st>>>(nrhs, bw->arn, bw->h, bw->coef, first, o->atol, o->rtol,
                                                       o->max_it);
  FV_CUDA(cudaGetLastError());
  return FV_OK;
}

// one restart cycle of m Arnoldi steps for every right-hand side, the update X += Z y, and the next cycle's
// residual: a fixed launch sequence (converged right-hand sides carry zero columns), captured as one graph
static fv_status batch_cycle(const fv_system* s, BatchWork* bw, int nrhs, const double* B, double* X,
                             const fv_gmres_opts* o, cudaStream_t st) {
  const int m = o->restart;
  const long long n = s->n;
  const long long vs = (long long)(m + 1) * n, zs = (long long)m * n;
  const dim3 gv(bblocks(n), nrhs), gc(rblocks(nrhs), nrhs);
  fv_status rc;
  scale_batch_kernel<<<gv, 256, 0, st>>>(n, bw->coef, bw->r, n, 0.0, nullptr, bw->V, vs);
  for (int j = 0; j < m; ++j) {
    double* vj = bw->V + (size_t)j * n;
    double* zj = bw->Z + (size_t)j * n;
    // Z_j = M^{-1} V_j and w = A Z_j for every right-hand side (strided in the bases)
    if ((rc = ras_batch(s, bw, nrhs, vj, vs, zj, zs, st))) return rc;
    if ((rc = apply_op_batch(s, nrhs, zj, zs, bw->w, n, bw->gh, st))) return rc;
    const int nv = j + 1;
    {
      ProfScope ps(FV_K_CGS, st);
      cgs_batch_dispatch(nv, gc, n, bw->V, vs, nullptr, bw->w, bw->part, bw->h, bw->ticket, 0, st,
                         std::make_integer_sequence<int, BK>{});
      cgs_batch_dispatch(nv, gc, n, bw->V, vs, bw->h, bw->w, bw->part, bw->h, bw->ticket, 1, st,
                         std::make_integer_sequence<int, BK>{});
      cgs_batch_dispatch(nv, gc, n, bw->V, vs, bw->h + BK, bw->w, bw->part, bw->h, bw->ticket, 2, st,
                         std::make_integer_sequence<int, BK>{});
      batch_givens_kernel<<<(nrhs + 31) / 32, 32, 0, st>>>(nrhs, j, bw->arn, bw->h, bw->coef);
    }
    FV_CUDA(cudaGetLastError());
    if (j + 1 < m) scale_batch_kernel<<<gv, 256, 0, st>>>(n, bw->coef, bw->w, n, 0.0, nullptr, bw->V + (size_t)(j + 1) * n, vs);
  }
  {
    ProfScope ps(FV_K_VEC, st);
    batch_lsq_kernel<<<(nrhs + 31) / 32, 32, 0, st>>>(nrhs, bw->arn, bw->coef);
    update_batch_kernel<<<gv, 256, 0, st>>>(n, m, bw->Z, zs, bw->coef, X);
  }
  FV_CUDA(cudaGetLastError());
  return batch_residual(s, bw, nrhs, B, X, o, 0, st);
}

fv_status gmres_batch(const fv_system* s, int nrhs, const double* B, double* X, const fv_gmres_opts* o,
                      fv_solve_stats* stats, cudaStream_t st) {
  auto t0 = std::chrono::steady_clock::now();
  const int m = o->restart;
  if (nrhs < 1 || m < 1 || m > BK - 1 || o->max_it < 0)
    return set_error("fv_gmres_solve_batch: nrhs >= 1 and restart in [1, 31] required"), FV_EINVAL;
  if (s->pc.levels != 1) return set_error("fv_gmres_solve_batch: one-level RAS systems only"), FV_EINVAL;
  if (s->subs.bf16) return set_error("fv_gmres_solve_batch: BF16 factors are not supported"), FV_EINVAL;
  fv_status rc = ensure_batch(s, nrhs, m);
  if (rc) return rc;
  BatchWork* bw = s->batch;
  if ((rc = batch_residual(s, bw, nrhs, B, X, o, 1, st))) return rc;
  auto fetch_state = [&]() -> fv_status {
    FV_CUDA(cudaMemcpyAsync(bw->arn_host, bw->arn, nrhs * sizeof(BatchArn), cudaMemcpyDeviceToHost, st));
    FV_CUDA(cudaStreamSynchronize(st));
    return FV_OK;
  };
  if ((rc = fetch_state())) return rc;
  if ((rc = waits_failed(s, "fv_gmres_solve_batch: not begun, in an earlier call ", st))) return rc;
  auto any_active = [&]() {
    for (int t = 0; t < nrhs; ++t)
      if (!bw->arn_host[t].done) return true;
    return false;
  };
  // the cycle runs eagerly on its first use (and while kernel timing is on); afterwards it is captured once
  // for these (B, X, restart) and replayed
  if (bw->cycle && (bw->gB != B || bw->gX != X || bw->gm != m)) {
    cudaGraphExecDestroy(bw->cycle);
    bw->cycle = nullptr;
  }
  while (any_active()) {
    if (prof_enabled() || !bw->warm) {
      if ((rc = batch_cycle(s, bw, nrhs, B, X, o, st))) return rc;
      bw->warm = 1;
    } else {
      if (!bw->cycle) {
        cudaStream_t cs;
        FV_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaGraph_t graph;
        FV_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        rc = batch_cycle(s, bw, nrhs, B, X, o, cs);
        cudaError_t ce = cudaStreamEndCapture(cs, &graph);
        cudaStreamDestroy(cs);
        if (rc) return rc;
        FV_CUDA(ce);
        ce = cudaGraphInstantiate(&bw->cycle, graph, 0);
        cudaGraphDestroy(graph);
        FV_CUDA(ce);
        bw->gB = B, bw->gX = X, bw->gm = m;
      }
      FV_CUDA(cudaGraphLaunch(bw->cycle, st));
    }
    if ((rc = fetch_state())) return rc;
  }
  if ((rc = waits_failed(s, "fv_gmres_solve_batch: ", st))) return rc;
  bool all_conv = true, nan = false;
  for (int t = 0; t < nrhs; ++t) {
    const BatchArn& a = bw->arn_host[t];
    const bool conv = std::isfinite(a.beta) && a.beta <= a.target;
    nan = nan || !std::isfinite(a.beta);
    all_conv = all_conv && conv;
    if (stats) {
      stats[t].iters = a.its;
      stats[t].inner_iters = 0;
      stats[t].converged = conv;
      stats[t].r0 = a.r0;
      stats[t].rfinal = a.beta;
      stats[t].time_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
      stats[t].fallback = 0;
    }
  }
  if (nan) return set_error("fv_gmres_solve_batch: NaN or Inf residual"), FV_ENAN;
  if (!all_conv) return set_error("fv_gmres_solve_batch: max_it reached before the tolerance"), FV_ENOCONV;
  return FV_OK;
}

}  // namespace fv

extern "C" fv_status fv_gmres_solve_batch(const fv_system* s, int nrhs, const double* B, double* X,
                                          const fv_gmres_opts* opts, fv_solve_stats* stats, void* stream) {
  if (!s || !B || !X || !opts || B == X) return fv::set_error("fv_gmres_solve_batch: bad argument"), FV_EINVAL;
  return fv::gmres_batch(s, nrhs, B, X, opts, stats, (cudaStream_t)stream);
}
