// Dependency graph G_tau from a density matrix (Section 2.2: i and j adjacent when |P_ij| > tau),
// built on the device as a CSR graph with sorted columns.
//
// P is stored in core columns: column g holds the rows S_k of g's part k.  Row i of the graph is
// the union of i itself, the rows of column i above tau, and the columns g whose entry in row i
// is above tau; those are cores of the parts that hold i, and row i sits at the same place of all
// core columns of one part.  A block gathers a row into a bitmap of the n vertices in shared
// memory, which removes duplicates (both P_ij and P_ji stored) and sorts at once; its set bits,
// counted or written in order, are the row.
//
// Per stored value of P the kernel reads 8 B once along its column and one 32-B sector across
// it, and each row scans n / 32 words of its bitmap.  At 4,096 orbitals (1.3 million stored
// values) a graph, sized and then filled, takes 0.63 ms with the copies of the result; sorting the rows on the
// host, after a copy of one flag per stored value, took 61 ms.
#include "gsp2_internal.cuh"
#include "gsp2_kernels.h"

namespace gsp2 {

constexpr int GRAPH_THREADS = 256;
// vertices per bitmap: 1.5 Mbit = 192 KB of shared memory; more vertices take several windows,
// each with its own pass over the row's candidates
constexpr int64_t GRAPH_WINDOW = 1536 * 1024;

template <bool FILL>
__global__ void __launch_bounds__(GRAPH_THREADS) graph_kernel(
    int64_t n, int64_t row0, int64_t rows, const double* __restrict__ p, double tau,
    const PartDesc* __restrict__ parts, const int32_t* __restrict__ Sall, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ invperm, const int64_t* __restrict__ pcolptr, const int64_t* __restrict__ memptr,
    const int32_t* __restrict__ mempart, const int32_t* __restrict__ memloc, int32_t* __restrict__ deg,
    const int64_t* __restrict__ rowptr, int32_t* __restrict__ out) {
  extern __shared__ uint32_t bits[];
  __shared__ int warp_sum_s[GRAPH_THREADS / 32 + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t out0 = FILL ? rowptr[row0] : 0;
  for (int64_t q = blockIdx.x; q < rows; q += gridDim.x) {
    const int64_t i = row0 + q;
    int64_t done = 0;  // entries of the windows before
    for (int64_t w0 = 0; w0 < n; w0 += GRAPH_WINDOW) {
      const int64_t w1 = w0 + GRAPH_WINDOW < n ? w0 + GRAPH_WINDOW : n;
      const int words = (int)((w1 - w0 + 31) >> 5);
      for (int w = tid; w < words; w += GRAPH_THREADS) bits[w] = 0u;
      __syncthreads();
      auto set = [&](int64_t v) {
        if (v >= w0 && v < w1) atomicOr(&bits[(v - w0) >> 5], 1u << ((v - w0) & 31));
      };
      if (tid == 0) set(i);
      for (int64_t m = memptr[i]; m < memptr[i + 1]; ++m) {
        const PartDesc d = parts[mempart[m]];
        const int a = memloc[m];
        const int32_t* S = Sall + d.soff;
        if (a < d.c) {  // i is a core of this part: its stored column
          const double* col = p + pcolptr[i];
          for (int t = tid; t < d.s; t += GRAPH_THREADS)
            if (fabs(col[t]) > tau) set(S[perm[d.soff + t]]);
        }
        const int pos = invperm[d.soff + a];  // row i in each core column of this part
        for (int j = tid; j < d.c; j += GRAPH_THREADS) {
          const int32_t g = S[j];
          if (fabs(p[pcolptr[g] + pos]) > tau) set(g);
        }
      }
      __syncthreads();
      // set bits of this thread's words, and of the words before them
      const int per = (words + GRAPH_THREADS - 1) / GRAPH_THREADS;
      const int b0 = min(tid * per, words), b1 = min(b0 + per, words);
      int cnt = 0;
      for (int w = b0; w < b1; ++w) cnt += __popc(bits[w]);
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) warp_sum_s[warp] = incl;
      __syncthreads();
      if (tid == 0) {
        int s = 0;
        for (int w = 0; w < GRAPH_THREADS / 32; ++w) {
          const int y = warp_sum_s[w];
          warp_sum_s[w] = s;
          s += y;
        }
        warp_sum_s[GRAPH_THREADS / 32] = s;
      }
      __syncthreads();
      if (FILL) {
        int32_t* dst = out + (rowptr[i] - out0) + done + warp_sum_s[warp] + incl - cnt;
        for (int w = b0; w < b1; ++w)
          for (uint32_t b = bits[w]; b; b &= b - 1) *dst++ = (int32_t)(w0 + 32 * (int64_t)w + __ffs((int)b) - 1);
      }
      done += warp_sum_s[GRAPH_THREADS / 32];
      __syncthreads();  // the bitmap and the sums are reused
    }
    if (!FILL && tid == 0) deg[i] = (int32_t)done;
  }
}

// rowptr[0 .. n] from the degrees, one block.
__global__ void __launch_bounds__(1024) graph_scan_kernel(int64_t n, const int32_t* __restrict__ deg,
                                                          int64_t* __restrict__ rowptr) {
  __shared__ int64_t sums[1024];
  const int tid = threadIdx.x;
  const int64_t per = (n + 1023) / 1024, b0 = min(tid * per, n), b1 = min(b0 + per, n);
  int64_t s = 0;
  for (int64_t i = b0; i < b1; ++i) s += deg[i];
  sums[tid] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int64_t y = tid >= o ? sums[tid - o] : 0;
    __syncthreads();
    sums[tid] += y;
    __syncthreads();
  }
  int64_t run = sums[tid] - s;
  for (int64_t i = b0; i < b1; ++i) {
    rowptr[i] = run;
    run += deg[i];
  }
  if (tid == 1023) rowptr[n] = sums[1023];
}

static size_t graph_smem(int64_t n) { return (size_t)(((n < GRAPH_WINDOW ? n : GRAPH_WINDOW) + 31) / 32) * 4; }

template <bool FILL>
static cudaError_t launch_graph(const GraphArgs& g, int64_t row0, int64_t rows, int32_t* out, int nsm, cudaStream_t s) {
  const size_t smem = graph_smem(g.n);
  cudaError_t e = cudaFuncSetAttribute(graph_kernel<FILL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = rows < 16 * (int64_t)nsm ? rows : 16 * (int64_t)nsm;
  graph_kernel<FILL><<<(unsigned)grid, GRAPH_THREADS, smem, s>>>(g.n, row0, rows, g.p, g.tau, g.parts, g.S, g.perm, g.invperm,
                                                                 g.pcolptr, g.memptr, g.mempart, g.memloc, g.deg,
                                                                 g.rowptr, out);
  return cudaGetLastError();
}

cudaError_t launch_graph_rowptr(const GraphArgs& g, int nsm, cudaStream_t s) {
  cudaError_t e = launch_graph<false>(g, 0, g.n, nullptr, nsm, s);
  if (e != cudaSuccess) return e;
  graph_scan_kernel<<<1, 1024, 0, s>>>(g.n, g.deg, g.rowptr);
  return cudaGetLastError();
}

cudaError_t launch_graph_rows(const GraphArgs& g, int64_t row0, int64_t rows, int32_t* out, int nsm, cudaStream_t s) {
  return launch_graph<true>(g, row0, rows, out, nsm, s);
}

}  // namespace gsp2
