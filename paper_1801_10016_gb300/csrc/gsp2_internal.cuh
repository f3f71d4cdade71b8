// Internal data structures shared by the G-SP2 kernels and the host plan code.
//
// Layout in device memory (all inside the caller's workspace):
//   * one "arena" per buffer holds every part's dense s_k x s_k matrix, column-major,
//     padded to ld_k = roundup(s_k, LD_PAD) rows and columns, at element offset off_k;
//     rows/columns in [s_k, ld_k) are zero so padded products stay exact;
//   * part descriptors, the per-part vertex lists S_k (cores ascending, then halo
//     ascending), the scatter permutation, the work lists and the per-step state.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace gsp2 {

constexpr int LD_PAD = 128;      // ld_k multiple (tile edge of every square kernel)
constexpr int SQ_TILE = 64;      // FP32 square tile edge
constexpr int SQ64_TILE = 16;    // FP64 square tile edge
constexpr int TC_TILE = 128;     // tensor-core square tile edge
constexpr int COLS_PER_BLOCK = 8;  // gather/scatter: one warp per column, 8 warps

struct PartDesc {
  int64_t off;   // arena element offset of X_k
  int64_t soff;  // offset of S_k in the vertex-list table
  int32_t s;     // core + halo size
  int32_t c;     // core count
  int32_t ld;    // padded leading dimension
  int32_t nt;    // FP32 square tiles per edge: ceil(s / SQ_TILE)
};

struct Tile {  // one upper-triangular output tile of one part
  int32_t part, ti, tj, slot;  // slot: diagonal-tile trace slot, -1 otherwise
};

struct ColBlock {  // COLS_PER_BLOCK consecutive local columns of one part
  int32_t part, j0;
};

// Per-call device state.  `counter` is the ticket of the last-block-done
// reductions; the block that finishes a reduction sets it back to zero.
struct DevState {
  double eps_min, eps_max;
  double idem_fro;     // idempotency report of the final P (core columns), -1 if not run
  unsigned int counter;
  int32_t tail_left;   // FP64 path: alternating tail steps still to run (0: none)
  int32_t stopped;     // 1: no further purification steps this call (read with the next word)
  int32_t coherent;    // emulated steps: some part was found coherent (OzStepArgs)
  int32_t steps;       // purification steps applied so far
  int32_t status;      // gsp2_status detected on the device
  int32_t nonfinite;   // set by any block that meets NaN/Inf
  int32_t fp64_steps;
  int32_t timeout;     // a bounded device wait gave up
  int32_t pad;
  double inv_hi, inv_lo;  // 1 / (eps_max - eps_min) = inv_hi + inv_lo; inv_hi = 0: to be divided by
};

static_assert(offsetof(DevState, stopped) % 8 == 0, "stopped and coherent are read together");

enum : int32_t { ST_OK = 0, ST_NOT_CONVERGED = 5, ST_TRACE = 6, ST_NONFINITE = 7, ST_TIMEOUT = 9 };
enum : int32_t { MODE_RECORD = 0, MODE_REPLAY = 1 };
enum : int32_t { SQ_FORWARD = 0, SQ_RECOMPUTE = 1, SQ_TAIL_FIRST = 2, SQ_TAIL_NEXT = 3, SQ_RESIDUAL = 4 };

// Exchange slot of a shard plan (a plan over a subset of the parts, one per GPU): the
// last block of a step leaves its partial core traces here instead of deciding, and the
// decision is taken by a separate launch once every shard's partials are summed.
struct ShardSlot {
  double t;      // partial Tr_core[X_step] over this shard's parts
  double y;      // partial Tr_core[X_{step-1}^2]
  int32_t step;  // the step the partials belong to
  int32_t pad;
};

// Which bookkeeping an exchange of a shard plan completes: the gather of X0, a step of
// the purification loop, an alternating tail step in the low precision, an FP64 tail step.
enum : int32_t { SHARD_GATHER = 0, SHARD_LOOP = 1, SHARD_TAIL_LP = 2, SHARD_TAIL_FP64 = 3 };

// Arguments of the per-step trace bookkeeping done by the last block of a step.
struct StepCtl {
  DevState* st;
  int8_t* alpha;     // alpha[i] = branch of step i (1-based), int8
  double* traces;    // traces[i] = T_i (core trace of X_i)
  double* idem;      // idem[i] = e_i = T_i - Tr_core[X_i^2]
  int64_t nocc;
  double idem_tol;
  double trace_tol;
  int32_t mode;
  int32_t last_step;  // max_steps (RECORD) or nsteps (REPLAY)
  int32_t stop_lag;   // stopping test compares e_{i-1} with e_{i-1-stop_lag}
  int32_t tail_steps; // RECORD: alternating steps after the stopping test (last_step includes them)
  ShardSlot* xchg;    // shard plans: export the partial traces here instead of deciding (else NULL)
};

// Arguments of one tensor-core purification step (k_tc.cu).
// Buffers alternate with the step parity: X_{step-1} is read from buffer (step-1)&1 and
// X_step written to buffer step&1.
struct TcStepArgs {
  const PartDesc* parts;
  const Tile* tiles;       // upper tiles: 128x128, or 128 x 128 nb[t] for the wide persistent kernel
  const int8_t* nb;        // wide tiles: 128-column blocks of each tile (1 or 2); NULL: 128x128 tiles
  const void* map_hi[2];   // CUtensorMap[nparts] over each operand arena (hi part)
  const void* map_lo[2];   // CUtensorMap[nparts] over each lo arena (split mode)
  // 16-bit kinds: the persistent kernel keeps only the tiles on or above the diagonal and
  // reads the operand panels right of a tile's block MN-major from them (boxes of 64 rows
  // by one K block), through these maps over the same arenas
  const void* map_mn_hi[2];
  const void* map_mn_lo[2];
  float* master[2];        // FP32 master copies of X
  void* op_hi[2];          // operand arenas
  void* op_lo[2];
  double2* slots;
  int nslots;
  int ntiles;
  StepCtl ctl;
  int step;                // ignored in tail mode (step = steps applied + 1)
  int tail;                // 0: loop step; 1: first alternating tail step; 2: further ones
  // FP32 adjoint of the low-precision plans (FP16 hi + lo operands, explicit buffers):
  // the rebuilt iterate X_step reads the operands of X_{step-1} (xmap_*) and its master
  // xin and writes master xout and operands xo_*; the reverse step `step` reads the
  // operands of X_{step-1} (xmap_*) and Xbar's ping-pong (map_*, master, op_* [2], the
  // roles chosen on the device by step parity).  `step` <= 0 names step n + step (the
  // FP64 tail steps, counted back from the device's step count n); loop steps above
  // n - adj_tail are skipped.
  const void* xmap_hi;
  const void* xmap_lo;
  const void* xmap_mn_hi;
  const void* xmap_mn_lo;
  const float* xin;
  float* xout;
  void* xo_hi;
  void* xo_lo;
  int adj_tail;
  // FP16 operands (KIND 2) of the adjoint: Xbar's are FP16 of Xbar 2^(14 - sig) with one
  // scale exponent per part: xb_sig[k] that of the operands a reverse step reads,
  // xb_sig[nparts + k] that of the operands it writes, chosen before the step from the
  // largest |Xbar| so far plus xb_headroom bits (one step multiplies the largest entry by
  // at most 2 + 2 sqrt(s), Cauchy-Schwarz with ||X||_2 <= 1).  The step records the largest
  // |Xbar_new| of each part (FP32 bits, xb_max) and its last block moves the scales on
  int32_t* xb_sig;
  uint32_t* xb_max;
  int nparts;
  int xb_headroom;
  // the persistent 128x128 kernel's steps and reverse steps: each CTA claims its next tile
  // from this counter (zero between launches; the last block resets it); NULL: static deal
  uint32_t* tile_ctr;
};
constexpr int TC_SIG_MIN = -98, TC_SIG_MAX = 126;  // range of the FP16 adjoint's scale exponents

// Arguments of the graph refresh (k_graph.cu).
struct GraphArgs {
  int64_t n;
  const double* p;  // P in core columns
  double tau;
  const PartDesc* parts;
  const int32_t *S, *perm, *invperm;
  const int64_t *pcolptr, *memptr;
  const int32_t *mempart, *memloc;
  int32_t* deg;     // [n]
  int64_t* rowptr;  // [n + 1]
};

// FP64 products rebuilt from FP16 digits (k_oz.cu)
constexpr int OZ_SLICES = 5;  // digits per entry (11, 8, 11, 8 and 11 bits)
constexpr int OZ_LOW = 2;     // digits the second pass of a tile multiplies
constexpr int OZ_MAX_GRID = 256;  // CTAs of the emulated step (one 128x128 int64 scratch each)
constexpr int OZ_BK = 32;         // K per slice of the emulated step, narrow form (64-byte rows)
constexpr int OZ_BK_WIDE = 64;    // the same, wide form (128-byte rows)

struct OzSlices {
  uint16_t* s[OZ_SLICES];  // FP16 digit arenas (same element indexing as the arenas)
};

// Where the blocks of a launch meet to form coherent parts again.
struct OzAgain {
  int32_t go;    // the launch's place (oz_step_kernel): its items are done, its coherent parts' can be taken again
  int32_t ctr;   // items taken (of all items, those of other parts being passed over)
  int32_t done;  // items done
  int32_t pad;
};

// One emulated step: digits of X_{step-1} are read from buffer (step-1)&1 and the digits
// of X_step written to buffer step&1 (SQ_FORWARD and the tail modes).  SQ_RECOMPUTE (the
// adjoint's rebuilt iterates) reads the digit set `maps` points at and writes digits[0],
// with the recorded branch and no bookkeeping.  The adjoint instantiation reads the digits
// of X (`maps`) and of Xbar / 2^sig (`maps_b`) and writes Xbar's FP64 ping-pong pair
// (xin = Xbar buffer 0, xout = buffer 1, the roles swapped on the device by step parity).
struct OzStepArgs {
  const PartDesc* parts;
  const Tile* tiles;   // 128x128 upper tiles
  int ntiles;
  const void* maps;    // per digit buffer (OZ_SLICES x nparts maps apart): CUtensorMap[3][nparts], K-major
                       // boxes of one digit of a wide tile slice ([0]), of all OZ_SLICES ([1]) or the
                       // first OZ_LOW ([2]) digits of a narrow one
  const void* maps_mn; // the same with MN-major boxes (each tile 128 rows x K columns as two 64-row atoms)
  const void* maps_b;    // adjoint: the same K-major maps over the digits of Xbar / 2^sig
  const void* maps_mn_b; // the same, MN-major
  int32_t* sig;          // adjoint: per-part scale exponent of Xbar's digits (OZ_SIG_NONFINITE: NaN),
                         // replaced by the new Xbar's scale by the last block of the step
  float* normf;          // adjoint: squared row norms of the new Xbar / 2^sig (zero between steps)
  int nparts;
  OzSlices digits[2];
  const double* xin;   // master of X_{step-1}: 64-bit fixed point x 2^56 (the adjoint's Xbar: FP64)
  double* xout;        // master of X_step, the same form
  double2* slots;      // diagonal-tile trace slots
  int nslots;
  long long* acc;      // OZ_MAX_GRID x 128 x 128 fixed-point partial sums, one tile per CTA
  StepCtl ctl;
  int step;            // ignored in tail modes (step = steps applied + 1)
  int mode;            // SQ_FORWARD, SQ_RECOMPUTE, SQ_TAIL_FIRST or SQ_TAIL_NEXT
  // split K: the work item of code 2 t + h is the half h of upper tile t's product (adjoint:
  // h = 0 Xbar X, h = 1 X Xbar; forward: the two halves of each pass's K stages); each writes
  // its 64-bit partial tile to split_acc[2 t + h] and the second of the two to finish
  // (split_cnt[t], left at zero) adds both and forms the tile (X_new, digits, traces)
  int split;
  int pieces;            // column pieces of a tile, each an item of its own (1 or 2; wide: 1)
  int wide;              // K slices of OZ_BK_WIDE in a ring of single digit tiles, not of OZ_BK in units of five
  int halves;            // the plan's items may be split: unsplit ones drain at the same boundary
  // Parts whose digits are coherent (some sum of digit products reached 2^24): coh[part] is the step that
  // found it (adjoint: counted back from the last step), OZ_INCOHERENT if none; coh_new[part] is set by
  // the items of a launch, and cleared by its last block once the part has been formed again in brief rounds
  int32_t *coh, *coh_new;
  OzAgain* again;
  long long* split_acc;  // [2 ntiles][128 x 128], indexed by item code 2 t + h
  uint32_t* split_cnt;   // [ntiles]
  const int32_t* split_items;  // [2 ntiles]: item codes in the order the CTAs take them
  // forward, tail and reverse steps: when set, each CTA claims its next item from this
  // counter (the items are then taken in list order by whichever CTA is free); the step's
  // last block sets it back to zero.  NULL (and the rebuilt iterates): CTA b takes items b,
  // b + gridDim.x, ...
  uint32_t* tile_ctr;
};
constexpr int32_t OZ_INCOHERENT = 0x7FFFFFFF;
constexpr int32_t OZ_SIG_NONFINITE = 0x7FFF;  // scale of a part whose Xbar holds NaN or Inf

// ------------------------------------------------------------------ device helpers

__device__ __forceinline__ double ld_cg(const double* p) { return __ldcg(p); }
// Two consecutive words (8-byte aligned) in one volatile load.
__device__ __forceinline__ uint2 ld_volatile2(const void* p) {
  uint2 v;
  asm volatile("ld.volatile.global.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}

// Programmatic dependent launch: the next launch of the stream may become resident (its blocks
// set up barriers and TMEM while this one drains), and this one waits here until the launch
// before it has completed and its writes are visible.  What that launch writes is read by plain loads: the
// read-only path (__ldg, const __restrict__) is for data that does not change while a kernel runs, and
// these kernels run while it still does.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
template <typename... Params, typename... Args>
cudaError_t launch_pdl(void (*kern)(Params...), int grid, int threads, size_t smem, cudaStream_t s, const Args&... a) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(a)...);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 16-byte asynchronous global->shared copies (both addresses 16-byte aligned).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }
__device__ __forceinline__ void cp_async_wait_1() { asm volatile("cp.async.wait_group 1;\n" ::); }

// Local index of global vertex g in S_k (cores [0, c) ascending, halo [c, s)
// ascending), or -1.
__device__ __forceinline__ int find_local(const int32_t* __restrict__ S, int c, int s, int32_t g) {
  int lo = 0, hi = c;
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (S[m] < g) lo = m + 1; else hi = m;
  }
  if (lo < c && S[lo] == g) return lo;
  lo = c; hi = s;
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (S[m] < g) lo = m + 1; else hi = m;
  }
  if (lo < s && S[lo] == g) return lo;
  return -1;
}

// Last-block-done ticket.  Every block calls it once, after its partial results are
// stored; returns true in exactly one block (the last), which may then read all
// partials.  All threads of the block must call it.
__device__ __forceinline__ bool last_block_ticket(unsigned int* counter) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned int t = atomicAdd(counter, 1u);
    s_last = (t == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// Deterministic block-wide sum of two doubles per thread (fixed tree).  Result valid
// in thread 0.  blockDim.x must be a multiple of 32 and <= 1024.
__device__ __forceinline__ double2 block_sum2(double a, double b) {
  __shared__ double2 red[32];
  a = warp_sum(a);
  b = warp_sum(b);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = make_double2(a, b);
  __syncthreads();
  double2 r = make_double2(0.0, 0.0);
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    for (int i = 0; i < nw; ++i) { r.x += red[i].x; r.y += red[i].y; }
  }
  return r;
}

// The same ticket taken by one warp, after a block barrier that follows the block's partial
// results: the other warps are done, and only this one reads all partials if true.
__device__ __forceinline__ bool last_block_warp(unsigned int* counter) {
  unsigned int t = 0;
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    t = atomicAdd(counter, 1u);
  }
  const bool last = __shfl_sync(0xffffffffu, t, 0) == gridDim.x - 1;
  if (last) __threadfence();
  return last;
}

// Sum of n slots by one warp in a fixed order (every lane gets it).  A block of 640 threads that
// sums them spends its time in FP64 adds of zeros: an FP64 instruction of a warp takes 16 cycles
// of its SM's one FP64 pipe, 200 of them 1.7 us, and the barriers between them as much again
// (from the last tile to the end of an emulated step, n = 512: 6.5 us so; a 22-step density 0.61
// -> 0.54 ms with one warp here and for each diagonal tile's trace).
__device__ __forceinline__ double2 warp_sum_slots(const double2* slots, int n) {
  double a = 0.0, b = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x & 31; k < n; k += 32) {
    const double2 v = __ldcg(slots + k);
    a += v.x;
    b += v.y;
  }
  return make_double2(warp_sum(a), warp_sum(b));
}

// One column of the initial guess, assembled by a warp in shared memory and written once.
// Rows [0, rend) (a multiple of 128) come in chunks: zeros, then the entries t < nq of the row's
// list whose local index lj[t] falls there, put(index, xq[t]) each, then out(first row, the
// chunk's rows).  Zeros written to the arena, entries scattered over them there and the column
// read back for its digits cost a pass over memory more, the arena being larger than L2 in every
// large plan: n = 30000, 256 parts, 0.66 -> 0.49 ms for fixed point and digits (2 GB, 0.29 ms at the
// copy rate; the rest is the chain row -> list -> value, hidden by the warps in flight) and 0.54 ->
// 0.38 ms for FP32 and two FP16 operands.
constexpr int GATHER_BATCH = 4;   // entries per lane in flight (8: 7 % slower for the warps its registers cost)
constexpr int GATHER_ROWS = 512;  // 4 KB of 8-byte words a warp: 6 blocks of 8 warps an SM
template <typename T, typename Put, typename Out>
__device__ __forceinline__ void gather_column(T* buf, int rend, int nq, const int32_t* __restrict__ lj,
                                              const double* xq, int lane, Put put, Out out) {
  for (int r0 = 0; r0 < rend; r0 += GATHER_ROWS) {
    const int m = min(GATHER_ROWS, rend - r0);
    for (int i = lane; i < (int)(m * sizeof(T) / 16); i += 32) reinterpret_cast<uint4*>(buf)[i] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    for (int t0 = lane; t0 < nq; t0 += 32 * GATHER_BATCH) {
      int a[GATHER_BATCH];
      double x[GATHER_BATCH];
#pragma unroll
      for (int u = 0; u < GATHER_BATCH; ++u) a[u] = t0 + 32 * u < nq ? lj[t0 + 32 * u] - r0 : -1;
#pragma unroll
      for (int u = 0; u < GATHER_BATCH; ++u)  // -1 (not in the part) and the other chunks' rows fall outside
        x[u] = a[u] >= 0 && a[u] < m ? xq[t0 + 32 * u] : 0.0;
#pragma unroll
      for (int u = 0; u < GATHER_BATCH; ++u)
        if (a[u] >= 0 && a[u] < m) buf[a[u]] = put(a[u] + r0, x[u]);
    }
    __syncwarp();
    for (int r = 0; r < m; r += 128) out(r0 + r, buf + r);
    __syncwarp();
  }
}

// Sum of one value per warp (zero where a warp has none) in warp order, to slots[blockIdx.x]; then
// the last block forms T_0 from all blocks' slots.  `v` lies in shared memory, one per warp.
__device__ __forceinline__ bool gather_traces(const double* v, double* slots, unsigned int* counter, double& sum) {
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += v[w];
    slots[blockIdx.x] = a;
  }
  if (!last_block_ticket(counter)) return false;
  double a = 0.0;
#pragma unroll 8
  for (unsigned int k = threadIdx.x; k < gridDim.x; k += blockDim.x) a += ld_cg(&slots[k]);
  a = warp_sum(a);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  sum = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
  return threadIdx.x == 0;
}

// Bookkeeping of step `step` (0 = the initial guess X0), run by one thread of the
// last block once the global sums are known:
//   tN = Tr_core[X_step], tY = Tr_core[X_{step-1}^2] (unused for step 0).
// Records T_step and e_{step-1}, applies the stopping test, and in RECORD mode
// chooses the branch of the next step: alpha = +1 iff T_step <= Nocc.
// Stopping test (RECORD): |e| <= idem_tol and (e < 0 or e >= e_{step-1-stop_lag});
// e >= 0 in exact arithmetic and falls once all eigenvalues are near 0 or 1, so a
// small e that is negative or no longer falls leaves only rounding (or the G-SP2
// drift of a core trace that cannot reach Nocc) to iterate on.  Every path uses lag 1
// (the field is kept for experiments with longer lags).
__device__ __forceinline__ void finish_step(const StepCtl& c, int step, double tN, double tY) {
  if (c.xchg) {  // shard plan: the sums over all shards decide, in a later launch
    c.xchg->t = tN;
    c.xchg->y = tY;
    c.xchg->step = step;
    return;
  }
  DevState* st = c.st;
  // everything this reads, in flight together: one thread runs this at the end of every step, and
  // each load that waits for the one before costs the next step 0.4 us
  const bool lagged = step >= 1 + c.stop_lag;
  const double tprev = step > 0 ? c.traces[step - 1] : 0.0;
  const double eprev = step > 0 && lagged ? c.idem[step - 1 - c.stop_lag] : 0.0;
  const int nonfinite = st->nonfinite, status = st->status, tail_left = st->tail_left;
  const int8_t al = c.alpha[step];
  c.traces[step] = tN;
  st->steps = step;
  bool stop = false, fire = false;
  double e = 0.0;
  if (step > 0) {
    e = tprev - tY;
    c.idem[step - 1] = e;
    if (c.mode == MODE_RECORD && lagged && fabs(e) <= c.idem_tol && (e < 0.0 || e >= eprev)) fire = true;
  }
  if (nonfinite || !isfinite(e) || !isfinite(tN)) {
    st->nonfinite = 1;
    st->status = ST_NONFINITE;
    st->stopped = 1;
    return;
  }
  if (c.mode == MODE_RECORD && tail_left > 0) {
    // this step was one of the alternating tail steps
    st->tail_left = tail_left - 1;
    if (tail_left == 1) {
      st->stopped = 1;
    } else {
      c.alpha[step + 1] = (int8_t)(-al);
    }
    return;
  }
  const bool cap = step >= c.last_step - (c.mode == MODE_RECORD ? c.tail_steps : 0);
  if (fire) stop = true;
  if (!stop && cap) {
    stop = true;
    if (c.mode == MODE_RECORD && step > 0 && !(fabs(e) <= c.idem_tol)) st->status = ST_NOT_CONVERGED;
  }
  if (stop && c.mode == MODE_RECORD && c.tail_steps > 0) {
    // start the tail: first branch from the trace rule, then alternating
    st->tail_left = c.tail_steps;
    c.alpha[step + 1] = (tN <= (double)c.nocc) ? (int8_t)1 : (int8_t)-1;
    return;
  }
  if (stop) {
    st->stopped = 1;
    if (c.mode == MODE_REPLAY && status == ST_OK) {
      const double d = tN - (double)c.nocc;
      if (!(fabs(d) <= c.trace_tol)) st->status = ST_TRACE;
    }
  } else if (c.mode == MODE_RECORD) {
    c.alpha[step + 1] = (tN <= (double)c.nocc) ? (int8_t)1 : (int8_t)-1;
  }
}

// Bookkeeping of a tail step of a low-precision run (FP64, or alternating steps in the
// low precision): records T_step, e_{step-1} and the step count; no stopping test and
// no branch choice.
__device__ __forceinline__ void finish_tail(const StepCtl& c, int step, double tN, double tY, bool fp64) {
  if (c.xchg) {
    c.xchg->t = tN;
    c.xchg->y = tY;
    c.xchg->step = step;
    return;
  }
  DevState* st = c.st;
  c.traces[step] = tN;
  c.idem[step - 1] = c.traces[step - 1] - tY;
  st->steps = step;
  if (fp64) st->fp64_steps += 1;
  if (!isfinite(tN) || !isfinite(c.idem[step - 1])) {
    st->nonfinite = 1;
    st->status = ST_NONFINITE;
  }
}

// Conversions between FP64 and the 2^-56 fixed point of x / 2^sig done with integer
// instructions (the FP64 pipe of GB300 is 64x slower than its integer pipe), rounding to
// nearest even.  |x| / 2^sig < 2^7; larger inputs saturate, results below 2^-1022 flush to 0.
__device__ __forceinline__ long long to_fixed(double x, int sig = 0) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  if (ex == 0) return 0;                                    // zero and subnormals (< 2^-1022)
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = ex - 1023 - 52 + 56 - sig;                 // (x / 2^sig) * 2^56 = m * 2^sh
  unsigned long long a;
  if (sh > 10) {
    a = 1ull << 62;                                         // out of range: saturate
  } else if (sh >= 0) {
    a = m << sh;
  } else if (sh > -64) {
    const int k = -sh;
    const unsigned long long q = m >> k, rem = m & ((1ull << k) - 1), half = 1ull << (k - 1);
    a = q + ((rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull);
  } else {
    a = 0;
  }
  return (b >> 63) ? -(long long)a : (long long)a;
}

__device__ __forceinline__ double from_fixed(long long v, int sig = 0) {
  if (v == 0) return 0.0;
  const unsigned long long sgn = v < 0 ? (1ull << 63) : 0ull;
  const unsigned long long a = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int lz = __clzll(a);
  const unsigned long long m = a << lz;                     // top bit at 63
  unsigned long long mant = m >> 11;                        // 53 bits with the leading one
  const unsigned long long rem = m & 0x7FFull;
  int e = 63 - lz - 56 + sig;                               // value = 1.f x 2^e
  if (rem > 0x400ull || (rem == 0x400ull && (mant & 1ull))) {
    mant += 1;
    if (mant >> 53) {
      mant >>= 1;
      e += 1;
    }
  }
  if (e < -1022) return __longlong_as_double((long long)sgn);
  const unsigned long long bits = sgn | ((unsigned long long)(e + 1023) << 52) | (mant & 0xFFFFFFFFFFFFFull);
  return __longlong_as_double((long long)bits);
}

}  // namespace gsp2
