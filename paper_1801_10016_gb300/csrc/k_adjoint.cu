// Adjoint of the G-SP2 density matrix: seed (FP64, or FP32 for the low-precision plans),
// the reverse purification steps of the native FP64 plans on the CUDA cores, and the
// scatter-add onto the pattern of H.  (The emulated FP64 plans and the low-precision plans
// run their reverse steps on the tensor cores: k_oz.cu, k_tc.cu.)
//
// With L = sum Pbar .* P and the branch sequence alpha_1..alpha_n fixed:
//   seed:   Xbar_n = sym(M_k), M_k[:, j] = Pbar[S_k, g_j] for core j, 0 for halo columns
//           (X_k is a symmetric function of a symmetric argument);
//   step i: alpha_i = -1 (X_i = X^2):      Xbar <- Xbar X + X Xbar
//           alpha_i = +1 (X_i = 2X - X^2): Xbar <- 2 Xbar - Xbar X - X Xbar
//           with X = X_{i-1};
//   Eq. 1:  dL/dH[S_k, S_k] = -Xbar_0 / (eps_max - eps_min), summed over the parts
//           that hold both indices; the bounds are held fixed.
#include "gsp2_internal.cuh"
#include "gsp2_kernels.h"

namespace gsp2 {

// Seed: one warp per local column b (including the zero padding up to nt*TILE).
template <typename T>
__global__ void __launch_bounds__(256) adj_seed_kernel(const PartDesc* __restrict__ parts,
                                                       const ColBlock* __restrict__ blocks,
                                                       const int32_t* __restrict__ Sall,
                                                       const int32_t* __restrict__ invperm,
                                                       const int64_t* __restrict__ pcolptr,
                                                       const double* __restrict__ pbar, T* __restrict__ xbar) {
  const ColBlock bl = blocks[blockIdx.x];
  const PartDesc p = parts[bl.part];
  const int lane = threadIdx.x & 31;
  const int b = bl.j0 + (threadIdx.x >> 5);
  if (b >= p.nt * SQ_TILE) return;
  const int32_t* S = Sall + p.soff;
  const int32_t* ip = invperm + p.soff;
  T* col = xbar + p.off + (int64_t)b * p.ld;
  const bool bin = b < p.s;
  const int64_t colb = (bin && b < p.c) ? pcolptr[S[b]] : -1;  // column g_b of P if b is a core
  const int ipb = bin ? ip[b] : 0;
  for (int a = lane; a < p.ld; a += 32) {
    double v = 0.0;
    if (bin && a < p.s) {
      const double mab = (colb >= 0) ? pbar[colb + ip[a]] : 0.0;             // M(a, b)
      const double mba = (a < p.c) ? pbar[pcolptr[S[a]] + ipb] : 0.0;       // M(b, a)
      v = 0.5 * (mab + mba);
    }
    col[a] = (T)v;
  }
}

// One reverse step for every part.  Work item = one upper tile (ti <= tj) of edge
// SQ64_TILE, as the forward steps (4,096 orbitals: 68.7 ms per backward with 64-tiles, 50.5 with 16);
// Z_IJ = sum_k Xbar[I,k] X[k,J] + X[I,k] Xbar[k,J] with all four slices streamed from
// columns k of the symmetric Xbar and X.  Result mirrored to (J, I).
// The Xbar buffers alternate with (n - step) so that skipped steps keep the parity: input
// xb[(n - step) & 1], output xb[(n - step + 1) & 1], n the steps applied by the forward;
// steps above n are skipped.
template <typename T>
__global__ void __launch_bounds__(256, 4) adj_step_kernel(const PartDesc* __restrict__ parts,
                                                          const Tile* __restrict__ tiles, const T* __restrict__ Xall,
                                                          T* __restrict__ xb0, T* __restrict__ xb1,
                                                          const int8_t* __restrict__ alpha, const DevState* st,
                                                          int step) {
  static_assert(sizeof(T) == 8, "the native FP64 adjoint");
  constexpr int EDGE = SQ64_TILE, ABK = 16;
  static_assert(EDGE == 16, "one entry of the tile a thread");
  const int n = *(volatile const int32_t*)&st->steps;
  if (step > n) return;
  const T* XBin = ((n - step) & 1) ? xb1 : xb0;
  T* XBout = ((n - step) & 1) ? xb0 : xb1;
  __shared__ __align__(16) T S1[2][ABK][EDGE];  // Xbar rows I
  __shared__ __align__(16) T S2[2][ABK][EDGE];  // X    rows J
  __shared__ __align__(16) T S3[2][ABK][EDGE];  // X    rows I
  __shared__ __align__(16) T S4[2][ABK][EDGE];  // Xbar rows J
  const Tile t = tiles[blockIdx.x];
  const PartDesc p = parts[t.part];
  const T* X = Xall + p.off;
  const T* B = XBin + p.off;
  const int64_t ld = p.ld;
  const int r0 = t.ti * EDGE, c0 = t.tj * EDGE;
  const int kend = (p.s + ABK - 1) / ABK * ABK;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;

  auto load_slice = [&](int buf, int k0) {
    // ABK x EDGE elements per operand: at most 256 16-byte chunks, one per thread per operand
    constexpr int EPC = 16 / (int)sizeof(T);
    static_assert(ABK * EDGE / EPC <= 256, "one chunk per thread");
    const int kr = tid / (EDGE / EPC), c2 = (tid % (EDGE / EPC)) * EPC;
    if (kr < ABK) {
      const int64_t co = (int64_t)(k0 + kr) * ld;
      cp_async16(&S1[buf][kr][c2], B + co + r0 + c2);
      cp_async16(&S2[buf][kr][c2], X + co + c0 + c2);
      cp_async16(&S3[buf][kr][c2], X + co + r0 + c2);
      cp_async16(&S4[buf][kr][c2], B + co + c0 + c2);
    }
    cp_async_commit();
  };

  T acc = T(0);
  const int nk = kend / ABK;
  load_slice(0, 0);
  for (int it = 0; it < nk; ++it) {
    const int buf = it & 1;
    if (it + 1 < nk) {
      load_slice(buf ^ 1, (it + 1) * ABK);
      cp_async_wait_1();
    } else {
      cp_async_wait_all();
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < ABK; ++kk)
      acc = fma(S3[buf][kk][tx], S4[buf][kk][ty], fma(S1[buf][kk][tx], S2[buf][kk][ty], acc));
    __syncthreads();
  }

  const int8_t al = alpha[step];
  T* O = XBout + p.off;
  const int64_t r = r0 + tx, c = c0 + ty;
  const T z = al > 0 ? T(2) * B[c * ld + r] - acc : acc;
  O[c * ld + r] = z;
  if (t.ti != t.tj) O[r * ld + c] = z;
}

// dL/dH on the CSR pattern: for every stored (r, col), the sum over the parts k that
// hold r (membership list of r) and col of -Xbar0_k[col, r] / (eps_max - eps_min), in
// the fixed membership order (ascending part id).  HBAR_WARPS warps per row, lanes over the row's
// entries: the chain entry -> its column's parts -> Xbar0 is all latency (one warp per row: 71 us on
// 4,096 orbitals and 217 us on 8,000, four 35 and 148).  With upper_block > 0 only the tiles of that
// edge on or above the diagonal hold Xbar0 (the emulated adjoint); the symmetric entry is read from there.
constexpr int HBAR_WARPS = 4;
template <typename T>
__global__ void __launch_bounds__(256) adj_hbar_kernel(int64_t n, const int64_t* __restrict__ rowptr,
                                                       const int32_t* __restrict__ colind,
                                                       const int64_t* __restrict__ memptr,
                                                       const int32_t* __restrict__ mempart,
                                                       const int32_t* __restrict__ memloc,
                                                       const PartDesc* __restrict__ parts,
                                                       const int32_t* __restrict__ Sall,
                                                       const T* __restrict__ xb0, const T* __restrict__ xb1,
                                                       double* __restrict__ hbar, const DevState* st,
                                                       int upper_block) {
  const int nsteps = st->steps;
  const T* XB = (nsteps & 1) ? xb1 : xb0;
  // the bounds kernel's 1 / (eps_max - eps_min), correctly rounded; a division in every thread took 7 us
  const double scale = -(st->inv_hi != 0.0 ? st->inv_hi : 1.0 / (st->eps_max - st->eps_min));
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t w = warp; w < n * HBAR_WARPS; w += nwarps) {
    const int64_t r = w / HBAR_WARPS;
    const int64_t m0 = memptr[r], m1 = memptr[r + 1];
    for (int64_t q = rowptr[r] + 32 * (w % HBAR_WARPS) + lane; q < rowptr[r + 1]; q += 32 * HBAR_WARPS) {
      const int32_t col = colind[q];
      // the parts holding both r and col: the intersection of their membership lists, both
      // in ascending part order, walked as a merge (the same parts in the same order as a
      // search of col in every S_k of r's list, so the same sum)
      int64_t mc = memptr[col];
      const int64_t mc1 = memptr[col + 1];
      double sum = 0.0;
      for (int64_t m = m0; m < m1 && mc < mc1; ++m) {
        const int32_t k = mempart[m];
        while (mc < mc1 && mempart[mc] < k) ++mc;
        if (mc == mc1 || mempart[mc] != k) continue;
        const PartDesc p = parts[k];
        const int lc = memloc[mc], lr = memloc[m];
        const bool swap = upper_block > 0 && lc / upper_block > lr / upper_block;
        sum += (double)XB[p.off + (swap ? (int64_t)lc * p.ld + lr : (int64_t)lr * p.ld + lc)];
      }
      hbar[q] = scale * sum;
    }
  }
}

template <typename T>
cudaError_t launch_adj_seed(const PartDesc* parts, const ColBlock* blocks, int nblocks, const int32_t* Sall,
                            const int32_t* invperm, const int64_t* pcolptr, const double* pbar, T* xbar,
                            cudaStream_t s) {
  adj_seed_kernel<T><<<nblocks, 32 * COLS_PER_BLOCK, 0, s>>>(parts, blocks, Sall, invperm, pcolptr, pbar, xbar);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adj_step(const PartDesc* parts, const Tile* tiles, int ntiles, const T* X, T* xb0, T* xb1,
                            const int8_t* alpha, const DevState* st, int step, cudaStream_t s) {
  adj_step_kernel<T><<<ntiles, 256, 0, s>>>(parts, tiles, X, xb0, xb1, alpha, st, step);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adj_hbar(int64_t n, const int64_t* rowptr, const int32_t* colind, const int64_t* memptr,
                            const int32_t* mempart, const int32_t* memloc, const PartDesc* parts,
                            const int32_t* Sall, const T* xb0, const T* xb1, double* hbar, const DevState* st,
                            cudaStream_t s, int upper_block) {
  const int64_t blocks = (n * HBAR_WARPS + 7) / 8;
  adj_hbar_kernel<T><<<(int)(blocks < 1216 ? blocks : 1216), 256, 0, s>>>(n, rowptr, colind, memptr, mempart, memloc, parts, Sall, xb0, xb1, hbar, st,
                                         upper_block);
  return cudaGetLastError();
}

#define GSP2_ADJ_INSTANTIATE(T)                                                                                     \
  template cudaError_t launch_adj_seed<T>(const PartDesc*, const ColBlock*, int, const int32_t*, const int32_t*,   \
                                          const int64_t*, const double*, T*, cudaStream_t);                        \
  template cudaError_t launch_adj_hbar<T>(int64_t, const int64_t*, const int32_t*, const int64_t*, const int32_t*, \
                                          const int32_t*, const PartDesc*, const int32_t*, const T*, const T*,     \
                                          double*, const DevState*, cudaStream_t, int);
GSP2_ADJ_INSTANTIATE(double)
GSP2_ADJ_INSTANTIATE(float)
template cudaError_t launch_adj_step<double>(const PartDesc*, const Tile*, int, const double*, double*, double*,
                                             const int8_t*, const DevState*, int, cudaStream_t);

}  // namespace gsp2
