// Streamed ILU(0) sweeps of the restricted additive Schwarz preconditioner (paper Sec. 3.3, eqn:onelevel).
//
// One CTA solves one (subdomain, component group) pair, L then U, in one launch.  Off-diagonal couplings are
// component-diagonal, and the diagonal blocks couple only (u, Theta) and B of VTBE and nothing of PPBE, so these
// are independent solves: VTBE runs as groups of 4 and 3 components on different SMs.  P and P_b run as two groups
// in FP64, whose arithmetic bounds a CTA, and as one in FP32, where a step costs its instructions and the second
// component shares the index work.
//
// What bounds it: the wavefronts i + 2 j + k = L of a box are a serial chain of steps.  The mapping keeps the
// chain short and everything else off it:
//  * A thread owns rows of cells along i.  Rows (j, k) are ranked by s = 2 j + k, so the rows active in a step
//    (0 <= L - s < nx) are consecutive ranks: warps are full or idle, and the operands of a step, packed in rank
//    order, sit at rank + offset(L).  Thread t runs the ranks t, t + T, t + 2 T, ..., T at least the widest step: a
//    thread has finished its row before its next one begins.
//  * Of a cell's five neighbours, (i -+ 1, j, k) is the thread's own last value and the three in row (j -+ 1, k)
//    are that row's last three values, of which two are already in registers: a step reads two values from a
//    two-deep ring in shared memory, does two dependent multiply-adds a component, stores one and meets a barrier.
//  * Operands are streamed.  A cell's factors and its grid cell are packed into 16-byte words, chunk by chunk; one
//    thread keeps a ring of chunks filled with cp.async.bulk, ahead of the steps by as much as the ring holds, and a
//    second warp gathers the right-hand side through the cell map (forward) or reads the forward result back
//    (backward) with cp.async, completion counted by mbarriers.
// Positions outside the box have exactly zero factors (assembly writes zero there and the factorization never
// updates them), so every neighbour is read unconditionally from a ring that starts at zero.
#include <cuda_bf16.h>

#include <algorithm>
#include <array>
#include <cstdint>
#include <cstring>
#include <map>
#include <type_traits>
#include <utility>

#include "fv_internal.h"

namespace fv {

namespace {

constexpr int MAX_ROWS = 384;        // cells of the widest step a CTA takes (threads of the solve)
constexpr int PRODUCERS = 64;        // one warp for the operands, one for the right-hand side
constexpr unsigned WAIT_TRIES = 1u << 22;

__device__ __forceinline__ float widen(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float widen(float v) { return v; }
__device__ __forceinline__ double widen(double v) { return v; }
template <class FT>
__device__ __forceinline__ FT narrow(double v) { return (FT)v; }
template <>
__device__ __forceinline__ __nv_bfloat16 narrow<__nv_bfloat16>(double v) { return __double2bfloat16(v); }

// A cell's operands as 4-byte words: the factors (five off-diagonal slots of DG components, then the diagonal
// block's entries the sweep needs), then (backward) the grid cell the result goes to.  P16 planes of 16 bytes a cell
// and a last plane of TAIL words.
template <int DG, class FT, bool FWD>
struct Lay {
  static constexpr int NF = 5 * DG + (FWD ? DG * (DG - 1) / 2 : DG * (DG + 1) / 2);
  static constexpr int NFW = (NF * (int)sizeof(FT) + 3) / 4;
  static constexpr int RAW = NFW + (FWD ? 0 : 1);
  static constexpr int NW = RAW % 4 == 3 ? RAW + 1 : RAW;
  static constexpr int P16 = NW / 4, TAIL = NW % 4;  // TAIL: 0, 1 or 2
  static constexpr int BYTES = NW * 4;
};

// shape tables of the boxes (equal boxes share one): per step {offset of a rank's operands, end of the step's
// cells}, per rank of a row {s, ring positions of its four neighbour rows}
struct Shape {
  int nx, levels, rows, nc;
  int steps, table;  // offsets into the step and row tables
};

struct SweepArgs {
  const Shape* shapes;
  const int* shape_of;    // [count] shape of a box
  const int2* steps;
  const unsigned long long* rows;
  const int* lpt;
  const long long* soff;  // box offsets in the padded streams
  const unsigned char* fw[2];
  const unsigned char* bw[2];
  const int* gather;      // grid cell of a stream's cell, -1: none
  void* loc;              // forward results, [component][sT] per right-hand side
  int* err;
  long long sT, N, rs, zs;  // padded stream length; grid cells; strides of a right-hand side in r and z
  int count, T, table_bytes;
};

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(unsigned bar, int n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned bar, int parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait; a wait that runs out marks the thread dead: it takes part in the remaining barriers but
// touches no staged data and no global memory, and the flag is reported by the host
__device__ __forceinline__ void bar_wait(unsigned bar, int parity, bool& dead, int* err) {
  if (dead) return;
  for (unsigned t = 0; t < WAIT_TRIES; ++t)
    if (bar_try(bar, parity)) return;
  dead = true;
  *err = 1;
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void* src, int bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(bar)
               : "memory");
}
template <int B>
__device__ __forceinline__ void copy_async(unsigned dst, const void* src, bool on) {
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(__cvta_generic_to_global(src)) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(__cvta_generic_to_global(src)), "n"(B),
                 "r"(on ? B : 0)
                 : "memory");
}
// the mbarrier's phase counts this thread once all its earlier cp.async have landed
__device__ __forceinline__ void arrive_on_copies(unsigned bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void step_barrier(int n) {
  if (n == 32) __syncwarp();
  else asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
}

// DG values of one cell in the step ring, one vector access (two for FP64)
template <int DG, class T>
struct RingVec {
  __device__ __forceinline__ static void load(const T* p, T (&v)[DG]) {
    if constexpr (DG == 1) {
      v[0] = *p;
    } else if constexpr (DG == 2) {
      const auto q = *reinterpret_cast<const typename std::conditional<sizeof(T) == 4, float2, double2>::type*>(p);
      v[0] = q.x, v[1] = q.y;
    } else if constexpr (sizeof(T) == 4) {
      const float4 q = *reinterpret_cast<const float4*>(p);
      v[0] = q.x, v[1] = q.y, v[2] = q.z;
      if constexpr (DG == 4) v[3] = q.w;
    } else {
      const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
      v[0] = a.x, v[1] = a.y, v[2] = b.x;
      if constexpr (DG == 4) v[3] = b.y;
    }
  }
  __device__ __forceinline__ static void store(T* p, const T (&v)[DG]) {
    if constexpr (DG == 1) {
      *p = v[0];
    } else if constexpr (DG == 2) {
      typename std::conditional<sizeof(T) == 4, float2, double2>::type q;
      q.x = v[0], q.y = v[1];
      *reinterpret_cast<decltype(q)*>(p) = q;
    } else if constexpr (sizeof(T) == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], DG == 4 ? v[DG - 1] : 0.f);
    } else {
      reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
      reinterpret_cast<double2*>(p)[1] = make_double2(v[2], DG == 4 ? v[DG - 1] : 0.0);
    }
  }
};

// one cell's staged operands in registers
template <int DG, class T, class FT, bool FWD>
struct Cell {
  using L = Lay<DG, FT, FWD>;
  union {
    unsigned w[L::P16 * 4 + 4];
    uint4 q[L::P16 + 1];
    FT f[(L::P16 * 4 + 4) * 4 / sizeof(FT)];
  };
  T y[DG];
  // chunk: the cell's chunk in the operand ring, its planes CH cells long; n: the cell within it
  template <int CH>
  __device__ __forceinline__ void operands(const unsigned char* chunk, int n) {
    const uint4* c = reinterpret_cast<const uint4*>(chunk) + n;
#pragma unroll
    for (int j = 0; j < L::P16; ++j) q[j] = c[j * CH];
    const unsigned char* tail = chunk + L::P16 * 16 * CH;
    if constexpr (L::TAIL == 1) w[L::P16 * 4] = reinterpret_cast<const unsigned*>(tail)[n];
    if constexpr (L::TAIL == 2) {
      const uint2 v = reinterpret_cast<const uint2*>(tail)[n];
      w[L::P16 * 4] = v.x, w[L::P16 * 4 + 1] = v.y;
    }
  }
  __device__ __forceinline__ T fac(int n) const { return (T)widen(f[n]); }
  __device__ __forceinline__ int cell() const { return (int)w[L::NFW]; }
};

// How a system's sweeps run: ring and row table as below, forward results in global memory or (LOCS) shared memory
enum Variant { GLOBAL_LOC, SHARED_LOC, WIDE_ROWS, SMALL_GLOBAL_LOC, SMALL_SHARED_LOC, VARIANTS };
// chunks of the operand ring (log2), cells a chunk (log2)
__host__ __device__ constexpr int slots_log(int kind, bool small) { return small && kind == FV_VTBE ? 2 : 3; }
__host__ __device__ constexpr int chunk_log(int kind, bool small) { return small ? 5 : kind == FV_VTBE ? 6 : 7; }
constexpr int SMALL_STEP = 64;  // widest step of the small ring, which holds two of them (VTBE) or four (PPBE)
constexpr int max_threads(int var) { return (var >= SMALL_GLOBAL_LOC ? 2 * SMALL_STEP : MAX_ROWS) + PRODUCERS; }
constexpr int min_ctas(int var, bool heavy) { return var >= SMALL_GLOBAL_LOC ? (heavy ? 2 : 4) : heavy ? 1 : 2; }

// LOCS: the forward result of the box stays in shared memory.  WIDE: the row table is read from global memory, a row
// ahead, and a row may begin the step after its thread's last one ended (as a test in the common variant that cost 1 to
// 5 % of a step: registers)
template <int DG, int SL, int LG, bool LOCS, bool WIDE, class T, class V, class FT>
__device__ __forceinline__ void sweep_body(const SweepArgs& A, int sd, int g, int c0, T* loc, const V* __restrict__ r,
                                           V* __restrict__ z, unsigned char* smem) {
  using LF = Lay<DG, FT, true>;
  using LB = Lay<DG, FT, false>;
  constexpr int RV = DG == 3 ? 4 : DG;  // values a cell holds in the step ring
  using R = RingVec<DG, T>;
  constexpr int SLOTS = 1 << SL, CH = 1 << LG, CAP = SLOTS << LG;
  const int NC = A.T, tid = threadIdx.x;
  const Shape sh = A.shapes[A.shape_of[sd]];
  const int nx = sh.nx, nc = sh.nc, levels = sh.levels, rows = sh.rows;
  const int nch = (nc + CH - 1) >> LG;
  const long long so = A.soff[sd];
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem);
  const unsigned full = smem_u32(bars), yfull = full + 8 * SLOTS, empty = yfull + 8 * SLOTS, fdone = empty + 8 * SLOTS;
  int2* steps = reinterpret_cast<int2*>(smem + 256);
  unsigned long long* row = reinterpret_cast<unsigned long long*>(steps + levels + 1);
  T* ring = reinterpret_cast<T*>(smem + 256 + A.table_bytes);
  unsigned char* blk = smem + 256 + A.table_bytes + (size_t)2 * NC * RV * sizeof(T);
  // chunk slot k: blk + k BB CH bytes, whichever direction's layout fills it (the two directions overlap in time)
  constexpr int BB = LF::BYTES > LB::BYTES ? LF::BYTES : LB::BYTES;
  constexpr int YB = sizeof(V) > sizeof(T) ? sizeof(V) : sizeof(T);
  unsigned char* ybuf = blk + (size_t)BB * CAP;
  T* sloc = reinterpret_cast<T*>(ybuf + (size_t)DG * YB * CAP);
  loc += so + c0 * A.sT;
  r += c0 * A.N, z += c0 * A.N;
  bool dead = false;
  // step n < nch of the stream: forward chunk n; n >= nch: backward chunk 2 nch - 1 - n
  auto load_chunk = [&](int n) {
    const int slot = n & (SLOTS - 1), c = n < nch ? n : 2 * nch - 1 - n;
    const int bytes = (n < nch ? LF::BYTES : LB::BYTES) * CH;
    const unsigned char* src = n < nch ? (g ? A.fw[1] : A.fw[0]) : (g ? A.bw[1] : A.bw[0]);
    bar_expect(full + 8 * slot, bytes);
    bulk_copy(smem_u32(blk) + (unsigned)(slot * BB * CH), src + ((so >> LG) + c) * bytes, bytes, full + 8 * slot);
  };
  const int first = min(SLOTS, 2 * nch);
  if (tid == NC) {
    for (int s = 0; s < SLOTS; ++s) bar_init(full + 8 * s, 1), bar_init(yfull + 8 * s, 32), bar_init(empty + 8 * s, NC / 32);
    bar_init(fdone, NC);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int n = 0; n < first; ++n) load_chunk(n);
  }
  for (int e = tid; e < 2 * NC * RV; e += blockDim.x) ring[e] = T(0);
  for (int e = tid; e <= levels; e += blockDim.x) steps[e] = A.steps[sh.steps + e];
  if constexpr (!WIDE)
    for (int e = tid; e < rows; e += blockDim.x) row[e] = A.rows[sh.table + e];
  __syncthreads();

  if (tid >= NC + 32) {  // ------------------------------------------------ right-hand side warp
    const int lane = tid - NC - 32;
    const unsigned yb = smem_u32(ybuf);
    constexpr int PL = CH / 32;  // cells of a chunk a lane gathers
    const int* gp = A.gather + so + lane;
    constexpr int AHEAD = 4;    // chunks the cell map is read ahead of its gather
    int gc[AHEAD][PL];
    auto map_of = [&](int n, int (&q)[PL]) {
#pragma unroll
      for (int e = 0; e < PL; ++e) q[e] = n < nch ? __ldg(gp + (n << LG) + 32 * e) : -1;
    };
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) map_of(u, gc[u]);
    for (int n0 = 0; n0 < nch && !dead; n0 += AHEAD) {
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) {
        const int n = n0 + u;
        if (n >= nch || dead) break;
        const int slot = n & (SLOTS - 1), b = (slot << LG) + lane;
        if (n >= SLOTS) bar_wait(empty + 8 * slot, ((n >> SL) - 1) & 1, dead, A.err);
        if (dead) break;
#pragma unroll
        for (int e = 0; e < PL; ++e) {
          const V* src = r + max(gc[u][e], 0);
#pragma unroll
          for (int a = 0; a < DG; ++a)
            copy_async<sizeof(V)>(yb + (unsigned)((a * CAP + b + 32 * e) * sizeof(V)), src + a * A.N, gc[u][e] >= 0);
        }
        arrive_on_copies(yfull + 8 * slot);
        map_of(n + AHEAD, gc[u]);
      }
    }
    if constexpr (!LOCS) {  // read the forward result back
      bar_wait(fdone, 0, dead, A.err);
      for (int n = nch; n < 2 * nch && !dead; ++n) {
        const int slot = n & (SLOTS - 1), b = slot << LG;
        if (n >= SLOTS) bar_wait(empty + 8 * slot, ((n >> SL) - 1) & 1, dead, A.err);
        if (dead) break;
        constexpr int PER = 16 / sizeof(T);
        const T* src = loc + ((2 * nch - 1 - n) << LG);
        for (int e = lane; e < CH / PER; e += 32)
#pragma unroll
          for (int a = 0; a < DG; ++a)
            copy_async<16>(yb + (unsigned)((a * CAP + b + e * PER) * sizeof(T)), src + a * A.sT + e * PER, true);
        arrive_on_copies(yfull + 8 * slot);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // nothing in flight when the shared memory is given back
    return;
  }
  if (tid >= NC) {  // ----------------------------------------------------- operand thread
    if (tid > NC) return;
    int n = first;
    for (; n < 2 * nch; ++n) {
      bar_wait(empty + 8 * (n & (SLOTS - 1)), ((n >> SL) - 1) & 1, dead, A.err);
      if (dead) break;
      load_chunk(n);
    }
    bool late = false;
    for (int q = max(0, n - SLOTS); q < n; ++q) bar_wait(full + 8 * (q & (SLOTS - 1)), (q >> SL) & 1, late, A.err);
    return;
  }

  // ------------------------------------------------------------------ the solve
  int waited = 0;  // chunks that have been waited for
  auto await = [&](int upto, bool y) {
    while (waited < upto) {
      const int slot = waited & (SLOTS - 1), par = (waited >> SL) & 1;
      bar_wait(full + 8 * slot, par, dead, A.err);
      if (y) bar_wait(yfull + 8 * slot, par, dead, A.err);
      ++waited;
    }
  };
  // Chunks go back to the producers warp by warp once the arithmetic has used their operands: a barrier alone
  // does not say that the loads issued before it have returned, and the copies that refill a slot are not
  // ordered with them.
  int freed = 0;  // chunks this warp has released
  const bool lead = (tid & 31) == 0;
  int rank, i;
  const T *jrow, *krow;  // the neighbour rows' places in the ring
  T own[DG], h1[DG], h2[DG];
  constexpr int OFF = -0x10000000;  // i of a thread without a row
  unsigned long long ahead = 0;  // WIDE: the table's entry of the thread's next row
  auto look_ahead = [&](int rk) {
    if constexpr (WIDE) ahead = rk >= 0 && rk < rows ? __ldg(A.rows + sh.table + rk) : 0;
  };
  // row `rk` from step L on (sh0: bit position of the direction's pair of neighbours), the thread's next one after
  // `by` ranks
  auto take_row = [&](int rk, int L, int sh0, int by) {
    rank = rk;
    const bool on = rk >= 0 && rk < rows && !dead;
    const unsigned long long w = WIDE ? ahead : on ? row[rk] : 0;
    look_ahead(rk + by);
    i = on ? L - (int)(w & 0xffff) : OFF;
    jrow = ring + ((int)(w >> sh0) & 0xfff) * RV, krow = ring + ((int)(w >> (sh0 + 12)) & 0xfff) * RV;
#pragma unroll
    for (int a = 0; a < DG; ++a) own[a] = h1[a] = h2[a] = T(0);
  };
  T* const mine = ring + tid * RV;
  const int half = NC * RV;  // ring of two steps: step L in half L & 1
  {
    Cell<DG, T, FT, true> q;
    int ready = 0;  // cells whose operands have landed
    auto fetch = [&](int2 st) {
      if (st.y > ready) {
        await(((st.y - 1) >> LG) + 1, true);
        ready = waited << LG;
        if (dead) i = OFF;
      }
      if ((unsigned)i < (unsigned)nx) {
        const int p = rank + st.x, n = p & (CH - 1), idx = p & (CAP - 1);
        q.template operands<CH>(blk + (idx >> LG) * (BB * CH), n);
#pragma unroll
        for (int a = 0; a < DG; ++a) q.y[a] = (T) reinterpret_cast<const V*>(ybuf)[a * CAP + idx];
      }
    };
    look_ahead(tid);
    take_row(tid, 0, 16, NC);
    int2 cur = steps[0], nxt = steps[1];
    fetch(cur);
    int free_at = min(CH, nc);
    auto step = [&](int L, int now, int last) {  // now, last: ring halves of steps L and L - 1
      if ((unsigned)(i + 1) <= (unsigned)nx) {
        T xj[DG], xk[DG], y[DG];
        R::load(jrow + last, xj);  // (i + 1, j - 1): its two predecessors are in registers
        R::load(krow + last, xk);
        // at i = -1 only xj matters: the arithmetic runs on old operands and is not kept
#pragma unroll
        for (int a = 0; a < DG; ++a) {
          y[a] = q.y[a];
          y[a] -= q.fac(4 * DG + a) * own[a];
          y[a] -= q.fac(2 * DG + a) * h1[a];
          y[a] -= q.fac(1 * DG + a) * h2[a];
          y[a] -= q.fac(0 * DG + a) * xk[a];
          y[a] -= q.fac(3 * DG + a) * xj[a];
#pragma unroll
          for (int c = 0; c < a; ++c) y[a] -= q.fac(5 * DG + a * (a - 1) / 2 + c) * y[c];
        }
        if (i >= 0) {
          R::store(mine + now, y);
          const int p = rank + cur.x;
#pragma unroll
          for (int a = 0; a < DG; ++a) {
            own[a] = y[a];
            if constexpr (LOCS) sloc[a * nc + p] = y[a];
            else loc[a * A.sT + p] = y[a];
          }
        }
#pragma unroll
        for (int a = 0; a < DG; ++a) h2[a] = h1[a], h1[a] = xj[a];
      }
      __syncwarp();
      while (free_at <= cur.y && freed < nch) {
        if (lead) bar_arrive(empty + 8 * (freed & (SLOTS - 1)));
        ++freed;
        free_at = min((freed + 1) << LG, nc);
      }
      cur = nxt;
      if (++i == nx) {
        take_row(rank + NC, L + 1, 16, NC);
        // a row that begins with the next step (a window wider than T) reads (0, j - 1, k) of step L - 1 here; others
        // wait a step at i = -1, which reads it
        if (WIDE && i == 0) R::load(jrow + last, h1);
      }
      nxt = steps[min(L + 2, levels)];
      if (L + 1 < levels) fetch(cur);
      step_barrier(NC);
    };
    int L = 0;
    for (; L + 1 < levels; L += 2) step(L, 0, half), step(L + 1, half, 0);
    if (L < levels) step(L, 0, half);
  }
  if constexpr (!LOCS) {
    __threadfence();  // the forward result is read back by the right-hand side warp's copies
    bar_arrive(fdone);
  }
  {
    Cell<DG, T, FT, false> q;
    int ready = 0x7fffffff;  // first cell whose operands have landed
    auto fetch = [&](int2 st, int begin) {
      if (begin < ready) {
        await(2 * nch - (begin >> LG), !LOCS);
        ready = (2 * nch - waited) << LG;
        if (dead) i = OFF;
      }
      if ((unsigned)i < (unsigned)nx) {
        const int p = rank + st.x, n = p & (CH - 1), slot = (2 * nch - 1 - (p >> LG)) & (SLOTS - 1);
        q.template operands<CH>(blk + slot * (BB * CH), n);
#pragma unroll
        for (int a = 0; a < DG; ++a) q.y[a] = LOCS ? sloc[a * nc + p] : reinterpret_cast<const T*>(ybuf)[a * CAP + (slot << LG) + n];
      }
    };
    // the last rank of this thread
    const int top = tid < rows ? tid + (rows - 1 - tid) / NC * NC : -1;
    look_ahead(top);
    take_row(top, levels - 1, 40, -NC);
    int2 cur = steps[levels - 1], nxt = steps[max(levels - 2, 0)];
    int begin = levels > 1 ? nxt.y : 0;  // first cell of the step whose operands are held
    fetch(cur, begin);
    int free_at = (nch - 1) << LG;
    auto step = [&](int L, int now, int last) {  // last: ring half of step L + 1
      if ((unsigned)i <= (unsigned)nx) {
        T xj[DG], xk[DG], x[DG];
        R::load(jrow + last, xj);  // (i - 1, j + 1)
        R::load(krow + last, xk);
#pragma unroll
        for (int a = DG - 1; a >= 0; --a) {
          x[a] = q.y[a];
          x[a] -= q.fac(0 * DG + a) * own[a];
          x[a] -= q.fac(2 * DG + a) * h1[a];
          x[a] -= q.fac(3 * DG + a) * h2[a];
          x[a] -= q.fac(4 * DG + a) * xk[a];
          x[a] -= q.fac(1 * DG + a) * xj[a];
          // U's diagonal block by rows from the diagonal, the diagonal as its reciprocal
          const int at = 5 * DG + a * DG - a * (a - 1) / 2;
#pragma unroll
          for (int c = a + 1; c < DG; ++c) x[a] -= q.fac(at + c - a) * x[c];
          x[a] *= q.fac(at);
        }
        if (i < nx) {
          R::store(mine + now, x);
          const int go = q.cell();
#pragma unroll
          for (int a = 0; a < DG; ++a) {
            own[a] = x[a];
            if (go >= 0) z[a * A.N + go] = (V)x[a];
          }
        }
#pragma unroll
        for (int a = 0; a < DG; ++a) h2[a] = h1[a], h1[a] = xj[a];
      }
      __syncwarp();
      while (free_at >= begin && freed < 2 * nch) {
        if (lead) bar_arrive(empty + 8 * (freed & (SLOTS - 1)));
        ++freed;
        free_at = (2 * nch - 1 - freed) << LG;
      }
      cur = nxt;
      if (--i == -1) {
        take_row(rank - NC, L - 1, 40, -NC);
        if (WIDE && i == nx - 1) R::load(jrow + last, h1);  // (nx - 1, j + 1, k) of step L + 1
      }
      nxt = steps[max(L - 2, 0)];
      begin = L > 1 ? nxt.y : 0;
      if (L > 0) fetch(cur, begin);
      step_barrier(NC);
    };
    int L = levels - 1;
    for (; L >= 1; L -= 2) step(L, half, 0), step(L - 1, 0, half);
    if (L == 0) step(0, half, 0);
  }
}

// grid: x = component group * boxes + box in decreasing size (the heavier group first), y = right-hand side
template <class T, class V, class FT, int KIND, int VAR>
__global__ void __launch_bounds__(max_threads(VAR), min_ctas(VAR, sizeof(T) == 8 && KIND == FV_VTBE))
    ras_stream_kernel(const __grid_constant__ SweepArgs A, const V* __restrict__ r, V* __restrict__ z) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int rhs = blockIdx.y;
  constexpr int D = KIND == FV_VTBE ? 7 : 2, SL = slots_log(KIND, VAR >= SMALL_GLOBAL_LOC), LG = chunk_log(KIND, VAR >= SMALL_GLOBAL_LOC);
  constexpr bool LOCS = VAR == SHARED_LOC || VAR == SMALL_SHARED_LOC, WIDE = VAR == WIDE_ROWS;
  T* const loc = (T*)A.loc + (size_t)rhs * D * A.sT;
  r += rhs * A.rs, z += rhs * A.zs;
  const int g = (int)blockIdx.x >= A.count, sd = A.lpt[blockIdx.x - g * A.count];
  if constexpr (KIND == FV_VTBE) {
    if (g == 0) sweep_body<4, SL, LG, LOCS, WIDE, T, V, FT>(A, sd, 0, 0, loc, r, z, smem);
    else sweep_body<3, SL, LG, LOCS, WIDE, T, V, FT>(A, sd, 1, 4, loc, r, z, smem);
  } else if constexpr (sizeof(T) == 8) {
    sweep_body<1, SL, LG, LOCS, WIDE, T, V, FT>(A, sd, g, g, loc, r, z, smem);
  } else {
    sweep_body<2, SL, LG, LOCS, WIDE, T, V, FT>(A, sd, 0, 0, loc, r, z, smem);
  }
}

// ------------------------------------------------------------------ packing (setup)
template <class FT, int DG, bool FWD>
__device__ void pack_cell(unsigned char* out, int ch_log, long long at, const double* off, const double* diag, int d, int c0,
                          int cell) {
  using L = Lay<DG, FT, FWD>;
  union {
    unsigned w[L::NW + 2];
    FT f[(L::NW + 2) * 4 / sizeof(FT)];
  };
  for (int t = 0; t < L::NW + 2; ++t) w[t] = 0;
  for (int s = 0; s < 5; ++s)
    for (int a = 0; a < DG; ++a) f[s * DG + a] = narrow<FT>(off[((FWD ? 0 : 6) + s) * d + c0 + a]);
  int n = 5 * DG;
  for (int a = 0; a < DG; ++a)
    for (int c = FWD ? 0 : a; c < (FWD ? a : DG); ++c) {
      const double v = diag[(c0 + a) * d + c0 + c];
      f[n++] = narrow<FT>(!FWD && a == c ? 1.0 / v : v);  // U's pivots as reciprocals, taken in FP64
    }
  if constexpr (!FWD) w[L::NFW] = (unsigned)cell;
  // chunks of CH cells, plane by plane within a chunk
  const int CH = 1 << ch_log, e = (int)(at & (CH - 1));
  unsigned char* chunk = out + (at >> ch_log) * ((long long)L::BYTES << ch_log);
  for (int j = 0; j < L::P16; ++j)
    reinterpret_cast<uint4*>(chunk)[j * CH + e] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  unsigned* tail = reinterpret_cast<unsigned*>(chunk + L::P16 * 16 * CH);
  for (int t = 0; t < L::TAIL; ++t) tail[e * L::TAIL + t] = w[L::P16 * 4 + t];
}

// natural layout off[C][11][d], diag[C][d][d] -> the streams of both groups, both directions.  rank_of: rank of
// a shape's row (j, k) at j + ny k
template <class FT>
__global__ void stream_pack_kernel(int d, int count, const long long* __restrict__ cell_off,
                                   const long long* __restrict__ soff, const int* __restrict__ dims,
                                   const Shape* __restrict__ shapes, const int* __restrict__ shape_of,
                                   const int2* __restrict__ steps, const int* __restrict__ rank_of,
                                   const long long* __restrict__ gmap, const unsigned char* __restrict__ owned,
                                   const double* __restrict__ off, const double* __restrict__ diag, int ch_log,
                                   unsigned char* f0, unsigned char* f1, unsigned char* b0, unsigned char* b1,
                                   int* __restrict__ gather) {
  const long long total = cell_off[count];
  for (long long C = blockIdx.x * (long long)blockDim.x + threadIdx.x; C < total; C += (long long)gridDim.x * blockDim.x) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (cell_off[mid] <= C) lo = mid;
      else hi = mid - 1;
    }
    const int nx = dims[3 * lo], ny = dims[3 * lo + 1];
    const int c = (int)(C - cell_off[lo]);
    const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
    const Shape sh = shapes[shape_of[lo]];
    const long long at = soff[lo] + rank_of[sh.table + j + ny * k] + steps[sh.steps + i + 2 * j + k].x;
    const int cell = (int)gmap[C], own = owned[C] ? cell : -1;
    gather[at] = cell;
    const double *oc = off + C * 11 * d, *dc = diag + C * d * d;
    if (d == 7) {
      pack_cell<FT, 4, true>(f0, ch_log, at, oc, dc, d, 0, cell), pack_cell<FT, 4, false>(b0, ch_log, at, oc, dc, d, 0, own);
      pack_cell<FT, 3, true>(f1, ch_log, at, oc, dc, d, 4, cell), pack_cell<FT, 3, false>(b1, ch_log, at, oc, dc, d, 4, own);
    } else if (sizeof(FT) < 8) {
      pack_cell<FT, 2, true>(f0, ch_log, at, oc, dc, d, 0, cell), pack_cell<FT, 2, false>(b0, ch_log, at, oc, dc, d, 0, own);
    } else {
      pack_cell<FT, 1, true>(f0, ch_log, at, oc, dc, d, 0, cell), pack_cell<FT, 1, false>(b0, ch_log, at, oc, dc, d, 0, own);
      pack_cell<FT, 1, true>(f1, ch_log, at, oc, dc, d, 1, cell), pack_cell<FT, 1, false>(b1, ch_log, at, oc, dc, d, 1, own);
    }
  }
}

template <class FT>
int group_bytes(int d, size_t (&fw)[2], size_t (&bw)[2]) {  // the number of groups, and bytes a cell of each
  if (d == 7) {
    fw[0] = Lay<4, FT, true>::BYTES, bw[0] = Lay<4, FT, false>::BYTES;
    fw[1] = Lay<3, FT, true>::BYTES, bw[1] = Lay<3, FT, false>::BYTES;
    return 2;
  }
  if (sizeof(FT) < 8) {
    fw[0] = Lay<2, FT, true>::BYTES, bw[0] = Lay<2, FT, false>::BYTES, fw[1] = bw[1] = 0;
    return 1;
  }
  fw[0] = fw[1] = Lay<1, FT, true>::BYTES, bw[0] = bw[1] = Lay<1, FT, false>::BYTES;
  return 2;
}

template <class T, class V, class FT, int KIND>
const void* stream_kernel(int var) {
  static const void* const table[VARIANTS] = {
      (const void*)ras_stream_kernel<T, V, FT, KIND, GLOBAL_LOC>, (const void*)ras_stream_kernel<T, V, FT, KIND, SHARED_LOC>,
      (const void*)ras_stream_kernel<T, V, FT, KIND, WIDE_ROWS>, (const void*)ras_stream_kernel<T, V, FT, KIND, SMALL_GLOBAL_LOC>,
      (const void*)ras_stream_kernel<T, V, FT, KIND, SMALL_SHARED_LOC>};
  return table[var];
}

template <class T, class V, class FT>
const void* kernel_of(int d, int var) {
  return d == 7 ? stream_kernel<T, V, FT, FV_VTBE>(var) : stream_kernel<T, V, FT, FV_PPBE>(var);
}

template <class T, class V, class FT, int KIND>
fv_status launch(const fv_system* s, int nrhs, const V* r, long long rs, V* z, long long zs, void* loc, cudaStream_t st) {
  const Subdomains& S = s->subs;
  const SweepStream& q = S.st;
  SweepArgs a{(const Shape*)q.shapes, q.shape_of, (const int2*)q.steps, q.rows, S.lpt, q.soff, {q.fw[0], q.fw[1]},
              {q.bw[0], q.bw[1]}, q.gather, loc, s->words_dev + WORD_SWEEP, q.sT, s->grid->h.N, rs, zs, S.count, q.T, q.table_bytes};
  void* args[] = {&a, &r, &z};
  FV_CUDA(cudaLaunchKernel(stream_kernel<T, V, FT, KIND>(q.variant), dim3(q.groups * S.count, nrhs), dim3(q.T + PRODUCERS), args,
                           q.smem, st));
  return FV_OK;
}

}  // namespace

// Builds the streams of s when every box fits the scheme: its widest step has a thread for every cell (MAX_ROWS), and
// an operand ring that holds a whole step fits in shared memory.  *used = 0: the caller keeps the general sweeps,
// 1.2 to 5 times slower where both can run (us, general against these: PPBE FP32 boxes of 36x36x21 cells 357, 156,
// 48x48x16 516, 205, 4x96x96 1689, 276; VTBE FP32 24x24x32 1067, 322; VTBE FP64 24x24x32 1736, 596).  Rows are held one
// step before they begin where MAX_ROWS threads cover such a window (to 36x36x20 cells: a window of 384); the boxes above
// have steps of 376 to 384 cells and windows to 396, or more rows than shared memory holds a table of, and run WIDE.
fv_status build_stream(fv_system* s, const std::vector<int>& dims, const std::vector<long long>& cell_off, int* used) {
  *used = 0;
  Subdomains& S = s->subs;
  SweepStream& q = S.st;
  const int d = S.d;
  const size_t es = S.fp32 ? 4 : 8;
  if (s->grid->h.N >= (1LL << 31)) return FV_OK;
  // shapes: rows ranked by s = 2 j + k; below(v) = rows with s <= v
  std::map<std::array<int, 3>, int> seen;
  std::vector<Shape> shapes;
  std::vector<int> shape_of(S.count), rank_of;
  std::vector<int2> steps;
  std::vector<unsigned long long> rows;
  std::vector<std::array<int, 3>> boxes;
  int window = 1, widest = 1, max_table = 0, max_steps = 0;
  long long max_nc = 0;
  for (int b = 0; b < S.count; ++b) {
    const std::array<int, 3> box{dims[3 * b], dims[3 * b + 1], dims[3 * b + 2]};
    auto it = seen.find(box);
    if (it == seen.end()) {
      const int nx = box[0], ny = box[1], nz = box[2];
      Shape sh{nx, nx - 1 + 2 * (ny - 1) + nz, ny * nz, nx * ny * nz, (int)steps.size(), (int)rank_of.size()};
      std::vector<int> below(sh.levels + 1, 0);  // below[v + 1]: rows with s <= v
      auto upto = [&](int v) { return v < 0 ? 0 : below[std::min(v, sh.levels - 1) + 1]; };
      for (int j = 0; j < ny; ++j)
        for (int k = 0; k < nz; ++k) below[2 * j + k + 1]++;
      for (int v = 0; v < sh.levels; ++v) below[v + 1] += below[v];
      std::vector<int> next(below.begin(), below.end() - 1);
      rank_of.resize(rank_of.size() + sh.rows);
      for (int j = 0; j < ny; ++j)
        for (int k = 0; k < nz; ++k) rank_of[sh.table + j + ny * k] = next[2 * j + k]++;
      int cells = 0;
      for (int L = 0; L < sh.levels; ++L) {
        const int from = upto(L - nx), n = upto(L) - from;
        steps.push_back(make_int2(cells - from, cells + n));
        cells += n;
        widest = std::max(widest, n);
        // a row held one step longer than it is active (forward: before, backward: after)
        window = std::max(window, std::max(upto(L + 1) - upto(L - nx), upto(L) - upto(L - nx - 1)));
      }
      steps.push_back(make_int2(0, cells));
      it = seen.emplace(box, (int)shapes.size()).first;
      shapes.push_back(sh), boxes.push_back(box);
      max_nc = std::max<long long>(max_nc, sh.nc);
      max_table = std::max(max_table, (sh.levels + 1 + sh.rows) * 8);
      max_steps = std::max(max_steps, (sh.levels + 1) * 8);
    }
    shape_of[b] = it->second;
  }
  if (widest > MAX_ROWS) return FV_OK;
  q.T = (std::min(window, MAX_ROWS) + 31) / 32 * 32;
  for (size_t m = 0; m < shapes.size(); ++m) {
    const Shape& sh = shapes[m];
    const int ny = boxes[m][1], nz = boxes[m][2];
    rows.resize(rank_of.size());
    for (int j = 0; j < ny; ++j)
      for (int k = 0; k < nz; ++k) {
        auto slot = [&](int jj, int kk) -> unsigned long long {  // a row outside the box: any position (zero factor)
          if (jj < 0 || jj >= ny || kk < 0 || kk >= nz) jj = j, kk = k;
          return (unsigned long long)(rank_of[sh.table + jj + ny * kk] % q.T);
        };
        rows[sh.table + rank_of[sh.table + j + ny * k]] = (unsigned long long)(2 * j + k) | slot(j - 1, k) << 16 |
                                                          slot(j, k - 1) << 28 | slot(j + 1, k) << 40 | slot(j, k + 1) << 52;
      }
  }
  size_t fw[2], bw[2];
  q.groups = S.bf16 ? group_bytes<__nv_bfloat16>(d, fw, bw) : S.fp32 ? group_bytes<float>(d, fw, bw) : group_bytes<double>(d, fw, bw);
  int dev = 0, limit = 0, sms = 0;
  FV_CUDA(cudaGetDevice(&dev));
  FV_CUDA(cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  FV_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int dg = d == 7 ? 4 : S.fp32 ? 2 : 1;  // the wider group
  // right-hand sides are staged in the vectors' type; a batch on FP32 factors stages FP64 (one level only)
  const size_t per_cell = std::max(fw[0], bw[0]) + (size_t)dg * (s->pc.levels == 1 && !S.bf16 ? 8 : es);
  const size_t loc = (size_t)dg * max_nc * es;
  const int kind = d == 7 ? FV_VTBE : FV_PPBE, tasks = q.groups * S.count, sm_bytes = limit + 1024;
  const bool heavy = d == 7 && !S.fp32;
  auto ring_smem = [&](bool small) {
    return 256 + q.table_bytes + (size_t)2 * q.T * dg * es + ((size_t)1 << (slots_log(kind, small) + chunk_log(kind, small))) * per_cell;
  };
  // kernels of a variant (FP32 factors: right-hand sides in FP32 and, in a batch, FP64)
  auto kernels = [&](int var) -> std::array<const void*, 2> {
    if (S.bf16) return {kernel_of<float, float, __nv_bfloat16>(d, var), nullptr};
    if (S.fp32) return {kernel_of<float, float, float>(d, var), kernel_of<float, double, float>(d, var)};
    return {kernel_of<double, double, double>(d, var), nullptr};
  };
  auto allow = [&](int var) {
    for (const void* f : kernels(var))
      if (f && cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, limit)) return false;
    return true;
  };
  auto held = [&](int var, size_t smem) {  // CTAs an SM holds
    int n = 0;
    return smem <= (size_t)limit && allow(var) &&
                   !cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernels(var)[0], q.T + PRODUCERS, smem)
               ? n
               : 0;
  };
  q.table_bytes = (max_table + 127) / 128 * 128;
  // A row table above 48 KB is read from global memory where it does not fit or would keep out a CTA that has a task (a row
  // change then waits for its warp's last look ahead: PPBE boxes of 4x96x96 cells, FP32, 144 tasks, 418 us so and 276
  // from shared memory; FP64, 288 tasks, 617 and 767)
  const bool wide = window > MAX_ROWS || ring_smem(false) > (size_t)limit ||
                    (max_table > (48 << 10) && (long long)sms * held(GLOBAL_LOC, ring_smem(false)) < tasks);
  if (wide) q.table_bytes = (max_steps + 127) / 128 * 128;
  // Boxes too many to run at once: a small ring lets an SM hold more of them, where it still holds a step ahead.
  // us, large ring (one CTA an SM for FP64 VTBE, three for PPBE), small: FP64 VTBE 3072 boxes of 6^3 cells 2053, 567, of
  // 10^3 3547, 1391; FP32 VTBE 417, 136 and 786, 337; FP64 PPBE 1296 boxes of 4^3 76, 47; FP32 30, 20
  const bool small = !wide && widest <= SMALL_STEP && window <= 2 * SMALL_STEP && (long long)sms * held(GLOBAL_LOC, ring_smem(false)) < tasks;
  q.ch_log = chunk_log(kind, small);
  q.smem = ring_smem(small);
  if ((((1 << slots_log(kind, small)) - 2) << q.ch_log) < widest || q.smem > (size_t)limit) return FV_OK;
  const long long CH = 1LL << q.ch_log;
  std::vector<long long> so(S.count + 1, 0);
  for (int b = 0; b < S.count; ++b) so[b + 1] = so[b] + (cell_off[b + 1] - cell_off[b] + CH - 1) / CH * CH;
  q.sT = so[S.count];
  // Thousands of boxes of a few cells would be padding for the most part (a box is at least a chunk): general sweeps.  Two
  // by two by two cells are the turn: 24,576 such boxes, general against streamed, FP64 VTBE 781, 1109; FP32 VTBE 296,
  // 256; FP64 PPBE 166, 190; FP32 PPBE 76, 82 us
  if (small && q.sT >= (heavy ? 4 : 5) * S.total_cells) return FV_OK;
  // the forward result stays in shared memory where that costs no CTA an SM would otherwise hold
  const int per_sm = (tasks + sms - 1) / sms;
  const int fit = small ? held(SMALL_GLOBAL_LOC, q.smem) : std::min(sm_bytes / (int)(q.smem + 1024), heavy ? 1 : std::max(2, 1024 / (q.T + PRODUCERS)));
  const bool shared_loc = !wide && q.smem + loc <= (size_t)limit && sm_bytes / (int)(q.smem + loc + 1024) >= std::min(per_sm, fit);
  if (shared_loc) q.smem += loc;
  q.variant = wide ? WIDE_ROWS : small ? (shared_loc ? SMALL_SHARED_LOC : SMALL_GLOBAL_LOC) : shared_loc ? SHARED_LOC : GLOBAL_LOC;
  if (!allow(q.variant)) return cuda_fail(cudaGetLastError(), "fv_assemble_system: shared memory of the sweeps");
  // one allocation for the tables (one copy), one for the streams, the cell map and the forward results
  size_t at = 0;
  auto part = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) / 256 * 256;
    return o;
  };
  const size_t t_soff = part(so.size() * sizeof(long long)), t_shapes = part(shapes.size() * sizeof(Shape)),
               t_steps = part(steps.size() * sizeof(int2)), t_rows = part(rows.size() * sizeof(unsigned long long)),
               t_of = part(shape_of.size() * sizeof(int)), t_ranks = part(rank_of.size() * sizeof(int)), tables = at;
  at = 0;
  const size_t b_fw[2] = {part(fw[0] * q.sT), part(fw[1] * q.sT)}, b_bw[2] = {part(bw[0] * q.sT), part(bw[1] * q.sT)},
               b_loc = part((size_t)d * q.sT * es), b_gather = part(q.sT * sizeof(int)), bytes = at;
  unsigned char *tab = nullptr, *str = nullptr;
  for (auto [p, n] : {std::pair{&tab, tables}, std::pair{&str, bytes}}) {
    if (cudaMalloc(p, n) != cudaSuccess) return set_error("fv_assemble_system: allocation of sweep data failed"), FV_ENOMEM;
    s->allocs.push_back(*p);
  }
  std::vector<unsigned char> host(tables);
  auto put = [&](size_t o, const auto& v) { std::memcpy(host.data() + o, v.data(), v.size() * sizeof(v[0])); };
  put(t_soff, so), put(t_shapes, shapes), put(t_steps, steps), put(t_rows, rows), put(t_of, shape_of), put(t_ranks, rank_of);
  FV_CUDA(cudaMemcpy(tab, host.data(), tables, cudaMemcpyHostToDevice));
  q.soff = (long long*)(tab + t_soff), q.shapes = tab + t_shapes, q.steps = tab + t_steps, q.shape_of = (int*)(tab + t_of);
  q.rows = (unsigned long long*)(tab + t_rows);
  const int* ranks = (const int*)(tab + t_ranks);
  for (int g = 0; g < 2; ++g) q.fw[g] = str + b_fw[g], q.bw[g] = str + b_bw[g];
  q.loc = str + b_loc, q.gather = (int*)(str + b_gather);
  FV_CUDA(cudaMemset(str, 0, b_gather));  // factors, and padding cells of the forward results: copied, never used
  FV_CUDA(cudaMemset(q.gather, 0xff, q.sT * sizeof(int)));  // padding cells gather nothing
  const int blocks = (int)std::min<long long>((S.total_cells + 127) / 128, 152LL * 64);
  auto pack = [&](auto zero) {
    using FT = decltype(zero);
    stream_pack_kernel<FT><<<blocks, 128>>>(d, S.count, S.cell_off, q.soff, S.dims, (const Shape*)q.shapes, q.shape_of,
                                            (const int2*)q.steps, ranks, S.gmap, S.owned, S.off, S.diag, q.ch_log,
                                            q.fw[0], q.fw[1], q.bw[0], q.bw[1], q.gather);
  };
  if (S.bf16) pack(__nv_bfloat16());
  else if (S.fp32) pack(0.f);
  else pack(0.0);
  FV_CUDA(cudaGetLastError());
  FV_CUDA(cudaDeviceSynchronize());
  *used = 1;
  return FV_OK;
}

// z = sum_i (R_i^0)^T (A_i^delta)^{-1} R_i^delta r for nrhs right-hand sides (strides rs, zs).
// One launch against the forward and backward launches of the earlier sweeps (all components of a box in one CTA,
// loads one step ahead in registers for VTBE), us on GB300:
//   FP32 coarse PPBE 6x32^3, boxes 10x10x18: 45 -> 33; 6x64^2x48, boxes 18x18x10: 201 -> 110
//   FP32 PPBE 6x64^3, boxes 36x36x20: 228 -> 147; 6x128^2x96: 875 -> 485
//   FP32 VTBE 6x64^3: 766 -> 674 (the gather of the right-hand side, four bytes a sector, bounds it); 6x128^2x96: 3290 -> 2656
//   FP64 PPBE 6x16^3: 142 -> 71; 6x24^2x36: 140 -> 47; 6x48^2x72: 442 -> 256; VTBE 6x48^2x72: 2520 -> 877
fv_status ras_stream64(const fv_system* s, int nrhs, const double* r, long long rs, double* z, long long zs, void* loc,
                       cudaStream_t st) {
  if (s->subs.fp32)
    return s->subs.d == 7 ? launch<float, double, float, FV_VTBE>(s, nrhs, r, rs, z, zs, loc, st)
                          : launch<float, double, float, FV_PPBE>(s, nrhs, r, rs, z, zs, loc, st);
  return s->subs.d == 7 ? launch<double, double, double, FV_VTBE>(s, nrhs, r, rs, z, zs, loc, st)
                        : launch<double, double, double, FV_PPBE>(s, nrhs, r, rs, z, zs, loc, st);
}

// after a synchronisation: whether a wait of s's sweeps (or of its coarse levels') ran out since the last call
bool sweep_failed(const fv_system* s) {
  bool bad = false;
  for (; s; s = s->coarse)
    if (*(volatile int*)(s->words + WORD_SWEEP)) bad = true, s->words[WORD_SWEEP] = 0;
  return bad;
}

fv_status ras_stream32(const fv_system* s, const float* r, float* z, cudaStream_t st) {
  void* loc = s->subs.st.loc;
  if (s->subs.bf16)
    return s->subs.d == 7 ? launch<float, float, __nv_bfloat16, FV_VTBE>(s, 1, r, 0, z, 0, loc, st)
                          : launch<float, float, __nv_bfloat16, FV_PPBE>(s, 1, r, 0, z, 0, loc, st);
  return s->subs.d == 7 ? launch<float, float, float, FV_VTBE>(s, 1, r, 0, z, 0, loc, st)
                        : launch<float, float, float, FV_PPBE>(s, 1, r, 0, z, 0, loc, st);
}

}  // namespace fv
