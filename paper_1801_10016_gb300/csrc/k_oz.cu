// FP64-accurate purification steps on the FP16 tensor cores (sm_103a).
//
// GB300 runs FP64 at 1/1800 of its 16-bit rate, so the FP64 product X X is rebuilt from
// FP16 products, in the spirit of the Ozaki splitting (Ozaki, Ogita, Oishi and Rump, 2012):
//
//   every entry of X (|x| <= 1: the spectrum of X stays in [0, 1]) is written with T = 5
//   balanced digits of 11, 8, 11, 8 and 11 bits, x = sum_t S_t 2^{-e_t} + r with
//   e = 11, 19, 30, 38, 49, |S_0| <= 2^11 |x| + 1, |S_t| at most half of digit t's range
//   (t >= 1), |r| <= 2^-50 (+ 2^-57 from the fixed point); every S_t is an integer that FP16
//   holds exactly (11 significant bits);
//
//   X X = sum_{a+b<T} 2^{-(e_a+e_b)} S_a S_b + (terms of order 2^-47): 15 products.
//
// The products are summed in FP32 in TMEM, in six accumulators.  Five of them hold integers
// (in units of their own scale), which FP32 keeps exactly while they stay below 2^24: (0,0), because
// ||X||_2 <= 1 bounds sum_k |x_ik x_kj| by 1; (0,1) + (1,0) and (0,2) + (2,0), at most 2^19
// and 2^22 times the row 1-norm sum_k |x_ik| (1 to 2 for the localised iterates of a gapped
// system; for rows spread over all K columns whose digits behave like independent values,
// about 2^18 and 2^21); (1,1), whose diagonal is a sum of squares, K 2^12.4 for digits
// spread over their range; and (1,2) + (2,1) + (0,3) + (3,0), about sqrt(K) 2^16 on such rows.
// The width of digit 1 follows from (1,1) staying below 2^24 up to K = 2048 (longer K is
// drained every 2048), that of digit 3 from the fifth accumulator at the same K (with 9 bits its
// largest sums passed 2^24 on dense rows, and the tensor core's truncation left 1.1e-13 at K = 2,049);
// digits 0 and 2 are as wide as FP16 allows, which leaves so little behind them
// that (1,3), (0,4), (2,2) and their mirrors, of order 2^-36 (2^-31 on the diagonal), share
// the sixth accumulator, whose FP32 rounding lies below the dropped products.  Digits of 7
// bits in BF16, whose 8-bit significand caps the width, took 7 digits and 28 products for an
// error per entry of 1.25e-14 at K = 1,184 on dense rows; these give 1.0e-14.
//
// That is how digits behave on most inputs, not a bound.  On coherent rows (entries of one magnitude,
// or slowly varying: the projectors of a Hadamard matrix, of a metallic ring, of rank 1) sums reach
// 2^26 in (0,2) and 2^28 in (1,2) + (0,3), and truncation there left up to 2.4e-11 a step.  So the drains
// look at every sum, and a part of which one has reached 2^24 is formed again, by the last block of the same launch,
// in brief rounds: the accumulators are drained every 32 columns, within which the digits' ranges
// bound every sum by 2^23.8 (rows of 0 <= X <= 1 have off-diagonal 2-norm <= 1/2, and 32 such entries add up to at
// most (1 + sqrt(33)) / 2; the adjoint's operands likewise).  From the next step on the part takes brief rounds at once.
// What a coherent row then loses is the products left out, whose bound is K 2^-49 (4.8e-12 met at K =
// 4,096; the seven digits of 7 bits left out 1.5 times that).  A partial sum that passes 2^24 and comes back in
// every tile of its part would not be seen; (1,1) cannot do so (Cauchy-Schwarz against the diagonal),
// and on the inputs above the largest partial sum lies within 2^0.3 of the largest sum.
// The accumulators are added as integers into a 64-bit fixed point (resolution 2^-56; the
// sixth rounded to it), and a final elementwise pass forms X_new = Y or 2X - Y on that
// grid (the master copy of the iterate stays in this fixed point), the core traces in FP64,
// and the digits of X_new for the next step by integer arithmetic.
//
// The adjoint step Xbar <- Xbar X + X Xbar (or 2 Xbar minus that) runs on the same
// machinery: an upper tile (I, J) of Xbar X + X Xbar is one product over K = 2s, rows I of
// [Xbar | X] times columns J of [X ; Xbar], both symmetric and kept as upper tiles.  Xbar
// has no a-priori bound, so its digits hold Xbar / 2^sig with one power-of-two scale per
// part, chosen from the largest row 2-norm of Xbar so that every row of Xbar / 2^sig has
// 2-norm <= 1/2.  With ||X||_2 <= 1, Cauchy-Schwarz gives
// sum_k |xbar_ik x_kj| + |x_ik xbar_kj| <= 1/2 + 1/2, the bound the forward step rests on,
// so the accumulators behave in the same way and the result carries an error of
// order 2^-47 2^sig.
#include <cuda.h>

#include <type_traits>

#include "gsp2_internal.cuh"
#include "gsp2_kernels.h"
#include "tc_ptx.cuh"

namespace gsp2 {

// Digits of a value held in 64-bit fixed point v = x 2^56 (|x| < 2): rounded to
// w = x 2^49, then written as balanced digits of 8, 11, 8 and 11 bits below S_0, so that
// w = S_0 2^38 + S_1 2^30 + S_2 2^19 + S_3 2^11 + S_4 exactly.  The balanced digits of w are
// the plain bit fields of w + bias less half of each field's range, so each is one
// shift-and-mask.  Digit t is stored as S_t 2^-rho_t with rho = -3, -4, -2, -3, -1: exact in
// FP16, and the products that share an accumulator land at one scale (rho_a + rho_b - e_a -
// e_b is the same for (1,2) and (0,3), and for (1,3), (0,4) and (2,2)).  S_0 beyond 2^11
// (|x| > 1, after low-precision steps) is kept even, which FP16 holds up to 2^12, and S_1
// takes the rest.  Each value is a float whose significand
// holds the field, less the same float of half its range: one AND/OR and one exact subtraction.
__host__ __device__ constexpr int oz_e(int t) {  // x = sum_t S_t 2^-e_t
  return t == 0 ? 11 : (t == 1 ? 19 : (t == 2 ? 30 : (t == 3 ? 38 : 49)));
}
__host__ __device__ constexpr int oz_rho(int t) {  // stored: S_t 2^-rho_t
  return t == 1 ? -4 : (t == 2 ? -2 : (t == 4 ? -1 : -3));
}
// Digit t, found biased by `half` at bit P of m (its field only): no shift is needed where the
// field lies in the float's significand
template <int T, int P>
__device__ __forceinline__ float digit_float(uint32_t m, uint32_t half) {
  constexpr uint32_t e = (uint32_t)(150 - oz_rho(T) - P) << 23;  // bit P weighs 2^-rho
  return __fsub_rn(__uint_as_float(e | m), __uint_as_float(e | (half << P)));
}
// Returns whether |S_0| > 2^11, where FP16 holds even integers only (digits_even).
__device__ __forceinline__ bool digit_floats(long long v, float (&f)[OZ_SLICES]) {
  // the rounding at 2^-49 and every field's bias in one addition; fields: S_4 bits 7-17, S_3
  // 18-25, S_2 26-36, S_1 37-44, S_0 45-58
  constexpr unsigned long long bias =
      (1ull << 6) + (1024ull << 7) + (128ull << 18) + (1024ull << 26) + (128ull << 37) + (8192ull << 45);
  const unsigned long long w = (unsigned long long)v + bias;
  const uint32_t lo = (uint32_t)w, hi = (uint32_t)(w >> 32);
  f[4] = digit_float<4, 7>(lo & (2047u << 7), 1024u);
  f[3] = digit_float<3, 15>((lo >> 3) & (255u << 15), 128u);
  f[2] = digit_float<2, 0>(__funnelshift_r(lo, hi, 26) & 2047u, 1024u);
  f[1] = digit_float<1, 5>(hi & (255u << 5), 128u);
  f[0] = digit_float<0, 9>((hi >> 4) & (16383u << 9), 8192u);
  return hi - ((8192u - 2048u) << 13) >= (4097u << 13);
}
__device__ __forceinline__ void digits_even(float (&f)[OZ_SLICES]) {
  const int s0 = (int)(f[0] * (1.0f / (float)(1 << -oz_rho(0))));
  if ((s0 > 2048 || s0 < -2048) && (s0 & 1)) {
    f[0] -= (float)(1 << -oz_rho(0));
    f[1] += (float)(256 << -oz_rho(1));
  }
}
// two digits as packed FP16 (lo in the lower half)
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;\n" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
// the digits of four values, packed: d[t][0] values 0 and 1, d[t][1] values 2 and 3
__device__ __forceinline__ void digits4(const long long (&v)[4], uint32_t (&d)[OZ_SLICES][2]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float a[OZ_SLICES], b[OZ_SLICES];
    const bool big_a = digit_floats(v[2 * h], a), big_b = digit_floats(v[2 * h + 1], b);
    if (big_a || big_b) {
      digits_even(a);
      digits_even(b);
    }
#pragma unroll
    for (int t = 0; t < OZ_SLICES; ++t) d[t][h] = pack_f16(a[t], b[t]);
  }
}

// The digits of four consecutive elements e .. e + 3 (e a multiple of 4), one 8-byte store
// per digit array (a warp's lanes on consecutive groups of four write 256 B per store).
__device__ __forceinline__ void store_digits4(uint16_t* const* slices, int64_t e, const long long (&v)[4]) {
  uint32_t d[OZ_SLICES][2];
  digits4(v, d);
#pragma unroll
  for (int t = 0; t < OZ_SLICES; ++t) *reinterpret_cast<uint2*>(slices[t] + e) = make_uint2(d[t][0], d[t][1]);
}

// Start of the emulated FP64 tail of a low-precision run: the last FP32 iterate (found on the
// device from the step count) converted to the fixed-point master and written as digits, in one pass
// over the rows on or above each column's diagonal block, the only ones the emulated steps
// read (and the scatter, which reads the upper tiles).  One warp per column up to ld.
__global__ void __launch_bounds__(256) oz_convert_slice_kernel(const PartDesc* __restrict__ parts,
                                                               const ColBlock* __restrict__ blocks,
                                                               const float* const* __restrict__ master_of_step,
                                                               double* __restrict__ X, OzSlices d0, OzSlices d1,
                                                               const DevState* st) {
  long long* __restrict__ xq = reinterpret_cast<long long*>(X);
  const int n = st->steps;
  const OzSlices& sl = (n & 1) ? d1 : d0;
  const float* __restrict__ in = master_of_step[n];
  const ColBlock b = blocks[blockIdx.x];
  const PartDesc p = parts[b.part];
  const int lane = threadIdx.x & 31;
  const int j = b.j0 + (threadIdx.x >> 5);
  if (j >= p.ld) return;
  const int rows = min(p.ld, (j / 128 + 1) * 128);
  const int64_t cbase = p.off + (int64_t)j * p.ld;
  for (int r = 4 * lane; r < rows; r += 128) {  // rows and cbase are multiples of 128
    const float4 f = *reinterpret_cast<const float4*>(in + cbase + r);
    const double x[4] = {(double)f.x, (double)f.y, (double)f.z, (double)f.w};
    long long v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = to_fixed(x[i]);
    longlong2* xo = reinterpret_cast<longlong2*>(xq + cbase + r);
    xo[0] = make_longlong2(v[0], v[1]);
    xo[1] = make_longlong2(v[2], v[3]);
    store_digits4(sl.s, cbase + r, v);
  }
}

// Gather of the emulated path: Eq. 1 and the digits of X0 in one pass.  One warp per column
// j < ld assembles the rows of column j of X0 on or above its diagonal block, the only ones
// the emulated steps read: zeros and the stored entries of row S_j of H that fall there,
// at the local indices of the plan's table (locate_kernel), with the values of Eq. 1 from
// x0_values_kernel, each stored in the 64-bit fixed point x 2^56 of the emulated steps' master
// and as digits.  Blocks store the core-diagonal sum of their columns; the last block forms T_0
// and takes the first branch.
__global__ void __launch_bounds__(32 * COLS_PER_BLOCK, 6) oz_gather_kernel(
    const PartDesc* __restrict__ parts, const ColBlock* __restrict__ blocks, const int32_t* __restrict__ Sall,
    const int64_t* __restrict__ rowptr, const int32_t* __restrict__ loc, const int64_t* __restrict__ locptr,
    const double* x0, double* __restrict__ arena, OzSlices dig, double* __restrict__ slots,
    StepCtl ctl) {
  __shared__ __align__(16) long long cols[COLS_PER_BLOCK][GATHER_ROWS];
  __shared__ double s_tr[COLS_PER_BLOCK];
  pdl_release();
  pdl_wait();
  const ColBlock b = blocks[blockIdx.x];
  const PartDesc p = parts[b.part];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j = b.j0 + w;
  if (lane == 0) s_tr[w] = 0.0;
  __syncwarp();
  if (j < p.ld) {
    const int rend = min(p.ld, (j / 128 + 1) * 128);
    const int64_t cbase = p.off + (int64_t)j * p.ld;  // a multiple of 128, as rend
    long long* const col = reinterpret_cast<long long*>(arena) + cbase;
    int64_t q0 = 0;
    int nq = 0;
    const int32_t* lj = loc;
    if (j < p.s) {
      const int32_t g = Sall[p.soff + j];
      q0 = rowptr[g];
      nq = (int)(rowptr[g + 1] - q0);
      lj = loc + locptr[p.soff + j];
    }
    gather_column(
        cols[w], rend, nq, lj, x0 + q0, lane,
        [&](int a, double x) {
          if (a == j && j < p.c) s_tr[w] = x;
          return to_fixed(x);
        },
        [&](int r, const long long* v) {
          const longlong2* v2 = reinterpret_cast<const longlong2*>(v);
          longlong2* c2 = reinterpret_cast<longlong2*>(col + r);
          c2[lane] = v2[lane];
          c2[32 + lane] = v2[32 + lane];
          const longlong2 a = v2[2 * lane], c = v2[2 * lane + 1];
          store_digits4(dig.s, cbase + r + 4 * lane, {a.x, a.y, c.x, c.y});
        });
  }
  double sum;
  if (gather_traces(s_tr, slots, &ctl.st->counter, sum)) {
    if (ctl.st->nonfinite) ctl.st->status = ST_NONFINITE;
    finish_step(ctl, 0, sum, 0.0);
    ctl.st->counter = 0;
  }
}

// The adjoint's operands.  `after` names the reverse step just run (0: the seed), whose
// Xbar lies in buffer (n - after + 1) & 1 of the pair (x0, x1); kernels for a step that was
// not run (after > n: the forward stopped earlier) return at once.

// Squared row 2-norms of the symmetric Xbar held in its upper 128-tiles (the seed; the
// reverse steps sum theirs in their epilogue), FP64, added into
// norm[soff + r] for rows r < s: the column sums of an upper tile (I, J) give the entries
// of rows J within block I (a diagonal tile holds its whole block), and the row sums of an
// off-diagonal tile the entries of rows I within block J.  One CTA per tile.
__global__ void __launch_bounds__(256) oz_norm_kernel(const PartDesc* __restrict__ parts,
                                                      const Tile* __restrict__ tiles, const double* xb0,
                                                      const double* xb1, int after, double* __restrict__ norm,
                                                      const DevState* st) {
  const int n = *(volatile const int32_t*)&st->steps;
  if (after > n) return;
  const double* X = (after > 0 && ((n - after + 1) & 1)) ? xb1 : xb0;
  const Tile t = tiles[blockIdx.x];
  const PartDesc p = parts[t.part];
  const double* x = X + p.off;
  const int64_t ld = p.ld;
  const int r0 = t.ti * 128, c0 = t.tj * 128;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = 0; q < 16; ++q) {  // warp w: columns c0 + 16 w .. + 15, lanes over the rows
    const int c = c0 + warp * 16 + q;
    if (c >= p.s) break;
    double v = 0.0;
    for (int i = lane; i < 128; i += 32) {
      const int r = r0 + i;
      if (r < p.s) {
        const double d = x[(int64_t)c * ld + r];
        v = fma(d, d, v);
      }
    }
    v = warp_sum(v);
    if (lane == 0) atomicAdd(&norm[p.soff + c], v);
  }
  if (t.ti != t.tj) {  // thread: row r0 + (tid % 128), half of the tile's columns
    const int r = r0 + (threadIdx.x & 127), h = threadIdx.x >> 7;
    if (r < p.s) {
      double v = 0.0;
      for (int q = 0; q < 64; ++q) {
        const int c = c0 + h * 64 + q;
        if (c >= p.s) break;
        const double d = x[(int64_t)c * ld + r];
        v = fma(d, d, v);
      }
      atomicAdd(&norm[p.soff + r], v);
    }
  }
}

// Scale of each part's Xbar digits: the smallest sig with 2^sig >= 2 max_r ||xbar_r||_2
// (with a relative margin of 2^-20 over the rounding of the FP64 sums), 0 for a zero Xbar,
// OZ_SIG_NONFINITE where a row norm is NaN or Inf.  Clears the norms for the next step, and at the
// seed the list of coherent parts coh[2][nparts], again.  One CTA per part.
__global__ void __launch_bounds__(256) oz_scale_kernel(const PartDesc* __restrict__ parts, int after,
                                                       double* __restrict__ norm, int32_t* __restrict__ sig,
                                                       int32_t* __restrict__ coh, const DevState* st) {
  const int n = *(volatile const int32_t*)&st->steps;
  if (after > n) return;
  if (after == 0 && threadIdx.x == 0) {
    coh[blockIdx.x] = OZ_INCOHERENT;
    coh[gridDim.x + blockIdx.x] = 0;
    if (blockIdx.x == 0)
      for (int i = 0; i < (int)(sizeof(OzAgain) / 4); ++i) coh[2 * gridDim.x + i] = 0;
  }
  const PartDesc p = parts[blockIdx.x];
  __shared__ double smax[8];
  double m = 0.0;
  int bad = 0;
  for (int r = threadIdx.x; r < p.s; r += blockDim.x) {
    const double v = norm[p.soff + r];
    norm[p.soff + r] = 0.0;
    if (!(v <= 1.7976931348623157e308)) bad = 1;  // NaN or Inf
    else m = fmax(m, v);
  }
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, smax[w]);
    int e = 0;
    if (bad) e = OZ_SIG_NONFINITE;
    else if (m > 0.0) (void)frexp(2.0 * sqrt(m) * (1.0 + 9.5367431640625e-07), &e);  // 2^(e-1) <= v < 2^e
    sig[blockIdx.x] = e;
  }
}

// Digits of the upper 128-tiles of a symmetric arena, of x / 2^sig[part] from FP64 (an
// adjoint's Xbar), or, with sig NULL, of a forward iterate held in the 64-bit fixed point
// x 2^56, into `out`; entries outside the part (rows or columns >= s) get zero digits.
// One warp per column up to ld.  Skipped where need > n (an iterate the adjoint does not
// reach) or where `after` names a reverse step that was not run.
__global__ void __launch_bounds__(256) oz_digits_kernel(const PartDesc* __restrict__ parts,
                                                        const ColBlock* __restrict__ blocks, const double* x0,
                                                        const double* x1, int after, int need, OzSlices out,
                                                        const int32_t* __restrict__ sig, const DevState* st) {
  const int n = *(volatile const int32_t*)&st->steps;
  if (need > n || after > n) return;
  const double* X = (after > 0 && ((n - after + 1) & 1)) ? x1 : x0;
  const ColBlock b = blocks[blockIdx.x];
  const PartDesc p = parts[b.part];
  const int lane = threadIdx.x & 31;
  const int j = b.j0 + (threadIdx.x >> 5);
  if (j >= p.ld) return;
  const int sg = sig ? sig[b.part] : 0;
  const int rend = min(p.ld, (j / 128 + 1) * 128);
  const int64_t cbase = p.off + (int64_t)j * p.ld;
  for (int r = 4 * lane; r < rend; r += 128) {  // rend and cbase are multiples of 128
    long long v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      v[i] = (r + i >= p.s || j >= p.s || sg == OZ_SIG_NONFINITE) ? 0ll
             : sig ? to_fixed(X[cbase + r + i], sg)
                   : reinterpret_cast<const long long*>(X)[cbase + r + i];
    store_digits4(out.s, cbase + r, v);
  }
}

// One FP64-accurate purification step for every part, in one persistent launch (one CTA
// per SM walks the upper 128x128 tiles: blockIdx.x, then the ones it claims from a counter,
// or blockIdx.x + gridDim.x, ... in the static deal).
//
// The 15 digit products of a tile need six FP32 accumulators of 128 TMEM columns, more than
// the 512 columns of an SM, so a tile takes two passes over K: first the 12 products other
// than (0,0), (0,1) and (1,0) (all five digits, columns 0-511), then those three (digits 0
// and 1, columns 0-255).  Each distinct digit tile is loaded once per K slice and pass and feeds all its
// products (one K = 16 FP16 MMA each); diagonal tiles load rows I only.  The K slices come in one of
// two forms, chosen by the plan (oz_wide in gsp2_api.cu):
//   narrow, K = 32: a unit of the TMA ring holds one operand (rows I or rows J) of the pass, one slice
//   of all five digits in one request, or in the second pass two slices of two digits.  Five units of
//   40 KB keep two and a half slices in flight.
//   wide, K = 64: the ring holds 13 single digit tiles of 16 KB.  A K-major tile then has 128-byte
//   rows, which L2 serves in 0.77 of the time of 64-byte ones (the loads of a step alone, n = 30000: 1.17
//   and 0.90 ms), a tile is given back as soon as its last product is issued, and the MMA warp waits
//   for the tiles in two groups (a wait per tile left the tensor pipe idle: 2.16 ms a step instead of
//   1.59).  Padding of K beyond the next multiple of 16 is not multiplied.
// The epilogue warps turn the passes' sums into 64-bit fixed point (2^-56): narrow, those of the first
// pass are parked in TMEM columns 256-511, which the second pass leaves alone, and the tile's in a
// per-CTA scratch tile (L2-resident); wide, all stay in registers, so that a pass's columns are
// handed back after nothing but their own reads.  The final pass forms X_new = Y or 2X - Y,
// writes the master copy (64-bit fixed point) and the digits of X_new (into the other
// digit buffer) at (I, J) and mirrored at (J, I) (diagonal tiles from their upper
// triangle), and adds the core traces, while the MMAs of the next tile's first pass run.  The new
// iterate is written with evict-first stores: the next step reads it after this launch,
// and keeping it out of L2 leaves room for the digit panels the running tiles share.  The last block
// runs the step bookkeeping, after it has formed again the parts whose sums were found too large (brief
// items, see the top).  K beyond 2048 is taken in rounds of both passes.  n = 30000 (256 parts), per step:
// narrow 1.69, wide 1.59 ms before the drains looked at every sum, 1.62 since; the MMAs at the measured 16-bit
// peak take 1.15, without loads or epilogue 1.29, with loads 1.32, with drains 1.43.
//
// 20 warps: warps 0 and 2 TMA (rows I and rows J: one warp's work per tile would hold
// the ring back), warp 1 TMEM owner and MMA issuer, warps 4..19 epilogue
// (warp w: TMEM lanes 32 (w % 4) .. + 31, columns 32 ((w - 4) / 4) .. + 31 of each group,
// in two chunks of 16), sized so that four epilogue warps per scheduler hide latency.
constexpr int OZ_UNITS = 5;                                      // narrow: operand units of the TMA ring
constexpr uint32_t OZ_UNIT_B = OZ_SLICES * 128u * OZ_BK * 2u;    // one operand's digit tiles
constexpr int OZ_LOW_SUB = 2;                                    // K slices per unit of the second pass
constexpr int OZ_TILES = 13;                                     // wide: digit tiles in the TMA ring
constexpr int OZ_GROUPS = 8;  // wide: barriers of tile groups per operand, more than the ring holds (2 tiles or more)
constexpr int OZ_HEAD = 3;    // wide: steps of the first pass whose tiles come as its first group
constexpr uint32_t OZ_RING_B = OZ_TILES * 128u * OZ_BK_WIDE * 2u;
constexpr int OZ_BARS = 2 * OZ_GROUPS + OZ_TILES + 4 + 1;        // mbarriers of the ring (padded to 16 bytes)
constexpr int OZ_EPI_WARPS = 16;                                 // 4 per TMEM lane quarter
constexpr int OZ_THREADS = 32 * (4 + OZ_EPI_WARPS);
constexpr int OZ_RING = 4;  // dynamic schedule: tiles claimed ahead of the MMA and epilogue warps
// a claimed item as the producer passes it on (code < 0: none)
struct alignas(16) OzItem {
  int64_t off, soff;
  int32_t code, ti, tj, slot;
  int32_t part, s, c, ld;
  int32_t piece, brief;  // brief: rounds of one K = 32 slice
  int32_t rounds, pad;   // rounds of both passes
};
constexpr int OZ_END = -1, OZ_PAUSE = -2;  // codes of no item: the walk ends; it waits for the last block's decision

constexpr int OZ_SMEM = (int)OZ_RING_B + 1024 + 8 * OZ_BARS + 16 + 16 * 128 +
                        8 * 2 * OZ_RING + (int)sizeof(OzItem) * OZ_RING;
static_assert(OZ_UNITS * OZ_UNIT_B <= OZ_RING_B && OZ_UNITS <= OZ_GROUPS, "the narrow ring within the wide one's space");
static_assert(OZ_LOW_SUB * OZ_LOW <= OZ_SLICES, "a unit holds the second pass's slices");
static_assert(OZ_BARS % 2 == 0, "alignment of the reduction slots and items");
static_assert(OZ_SMEM <= 232448, "shared memory of the emulated step");

// Columns of tile column block tj that an MMA must cover: those inside the part, rounded up
// to 16 (N of an M = 128 MMA is a multiple of 16); the rest of the block is zero padding.
__host__ __device__ constexpr int oz_tile_cols(int s, int tj) {
  return s - tj * 128 >= 128 ? 128 : ((s - tj * 128 + 15) & ~15);
}

// Accumulators (first TMEM column): of the first pass, (1,3), (0,4) and (2,2) in columns
// 0-127, (1,2) and (0,3) in 128-255, (0,2) in 256-383 and (1,1) in 384-511; of the second,
// (0,0) in 0-127 and (0,1) in 128-255.  The second pass can start once the columns 0-255 are
// read, and columns 256-511 then hold the first pass's 64-bit sums (narrow: low and high words).
constexpr uint32_t OZ_PARK_LO = 256, OZ_PARK_HI = 384;
__host__ __device__ constexpr bool oz_low_pass(int a, int b) { return a + b <= 1; }
__host__ __device__ constexpr uint32_t oz_col(int a, int b) {
  return a + b == 0 || a + b == 4 ? 0u : (a + b == 2 ? (a == 1 ? 384u : 256u) : 128u);
}
// Narrow slices: products of A digit q in a pass: (q, b) for lo <= b < hi
template <bool LOW>
__host__ __device__ constexpr int oz_q_lo(int q) { return LOW ? 0 : (q < 2 ? 2 - q : 0); }
template <bool LOW>
__host__ __device__ constexpr int oz_q_hi(int q) { return (LOW ? OZ_LOW : OZ_SLICES) - q; }

// Descriptors of one K slice: lower words at the slice's first digit tile, upper words,
// advance of a K = 16 step (16-byte units) and instruction descriptor.
struct OzNarrow {
  uint32_t alo, ahi, blo, bhi, adv_a, adv_b, idesc;
};

// The MMAs of the K = 16 step KK of one slice of a pass, fully unrolled, descriptors formed by adding
// compile-time offsets to the slice's lower words (the 14-bit address field cannot
// carry: shared addresses stay below 2^18).  The products are issued A digit by A digit: the products of
// A digit q follow one another and share their A operand through the
// collector buffer, so each A digit tile is read from shared memory once per K = 16 slice
// instead of once per product (the MMAs' shared-memory reads, A and B, set the pace of the
// tensor pipe otherwise).
template <bool LOW, int KK>
__device__ __forceinline__ void oz_issue_narrow(uint32_t tmem, const OzNarrow& o, bool first_k) {
  constexpr uint32_t step = (128u * OZ_BK * 2u) >> 4;
  const uint32_t alo = o.alo + (KK ? KK * o.adv_a : 0u), blo = o.blo + (KK ? KK * o.adv_b : 0u);
#pragma unroll
  for (int q = 0; q < (LOW ? OZ_LOW : OZ_SLICES); ++q) {
    const int b0 = oz_q_lo<LOW>(q), b1 = oz_q_hi<LOW>(q);
#pragma unroll
    for (int b = b0; b < b1; ++b) {
      const int op = (b1 - b0 == 1) ? 0 : (b == b0 ? 1 : (b == b1 - 1 ? 3 : 2));
      // the first product into each accumulator: (0,0), (0,1); (0,2), (0,3), (0,4), (1,1)
      const bool opens = q == 0 || (q == 1 && b == 1);
      mma_f16_lo(op, tmem + oz_col(q, b), alo + (uint32_t)q * step, o.ahi, blo + (uint32_t)b * step, o.bhi, o.idesc,
                 (KK == 0 && opens && first_k) ? 0u : 1u);
    }
  }
}

// Wide slices: the digit tiles of a K slice come and are used in this order: in step i of a pass over T digits
// digit T - 1 - i of rows I, then digit i of rows J, and the products (T - 1 - i, b), lo <= b <= i, of
// the pass follow.  A tile of rows I is then done, and tiles of rows J not long after they came, so
// that a ring of single tiles refills while the slice is still being multiplied.
template <bool LOW>
__host__ __device__ constexpr int oz_digits() { return LOW ? OZ_LOW : OZ_SLICES; }
template <bool LOW>
__host__ __device__ constexpr int oz_b_lo(int i) {
  const int q = oz_digits<LOW>() - 1 - i;
  return LOW ? 0 : (q < 2 ? 2 - q : 0);
}
// the step after which digit b of rows J is done
template <bool LOW>
__host__ __device__ constexpr int oz_b_last(int b) {
  int last = 0;
  for (int i = 0; i < oz_digits<LOW>(); ++i)
    if (oz_b_lo<LOW>(i) <= b && b <= i) last = i;
  return last;
}

// Descriptors of one K slice: lower words of the digit tiles' descriptors, upper words, advance of a
// K = 16 step (16-byte units), instruction descriptor and K = 16 steps.
struct OzWide {
  uint32_t a[OZ_SLICES], b[OZ_SLICES], ahi, bhi, adv_a, adv_b, idesc;
  int steps;
};

// The MMAs of step I of one slice of a pass, K = 16 steps [K0, K1), fully unrolled.  The products of an
// A digit follow one another and share their A operand through the collector buffer, so each A digit
// tile is read from shared memory once per K = 16 step instead of once per product (the MMAs'
// shared-memory reads, A and B, set the pace of the tensor pipe otherwise).
template <bool LOW, int I, int K0, int K1>
__device__ __forceinline__ void oz_issue_wide(uint32_t tmem, const OzWide& o, bool first) {
  constexpr int q = oz_digits<LOW>() - 1 - I, b0 = oz_b_lo<LOW>(I);
#pragma unroll
  for (int kk = K0; kk < K1; ++kk) {
    if (kk >= o.steps) break;
#pragma unroll
    for (int b = b0; b <= I; ++b) {
      const int op = I == b0 ? 0 : (b == b0 ? 1 : (b == I ? 3 : 2));
      // the first product into each accumulator: (1,0), (0,0); (4,0), (3,0), (2,0), (1,1)
      const bool opens = b == 0 || (!LOW && q == 1 && b == 1);
      mma_f16_lo(op, tmem + oz_col(q, b), o.a[q] + (uint32_t)kk * o.adv_a, o.ahi, o.b[b] + (uint32_t)kk * o.adv_b, o.bhi,
                 o.idesc, (kk == 0 && opens && first) ? 0u : 1u);
    }
  }
}

// The float bits of 1.5 2^(23 - M): a sum v of magnitude below 2^(22 - M) plus this float lies in
// [2^(23 - M), 2^(24 - M)) with spacing 2^-M, so the bits of the sum are these plus v 2^M (rounded).
__host__ __device__ constexpr uint32_t oz_magic(int M) { return ((uint32_t)(150 - M) << 23) | 0x400000u; }

// z[j] += sgn (u[j] + oz_magic(M)) 2^SHIFT for one accumulator of one 16-column chunk, where
// u = v 2^M is the integer its FP32 sums v hold at the scale 2^-M (the sixth accumulator: v 2^M
// rounded); the constants oz_magic(M) 2^SHIFT of all accumulators are taken off once, where z
// starts (kOzOffset; 64-bit arithmetic modulo 2^64).  A chunk whose integers all lie below
// 2^22 in magnitude is converted without the conversion unit, through the float bits, and a 32 x 32 ->
// 64-bit multiply-add (by the power of two, or on the upper word for shifts of 32 and more)
// accumulates it; any other chunk goes through the exact rounding conversion of v 2^M (|u| < 2^31).
// EXACT: mark(largest |u| 2^-24) where FP32 need not have held an integer: from 2^24 on, which only the second
// branch can meet (EVERY: always).
template <int M, int SHIFT, bool EXACT, bool EVERY, typename Mark>
__device__ __forceinline__ void oz_drain_slot(uint32_t taddr, int sgn, const Mark& mark, long long (&z)[16]) {
  uint32_t v[16];
  tmem_ld16(taddr, v);
  const float magic = __uint_as_float(oz_magic(M));
  const float lim = __uint_as_float((uint32_t)(149 - M) << 23);  // 2^(22 - M)
  float mx = 0.0f;
#pragma unroll
  for (int j = 0; j < 16; ++j) mx = fmaxf(mx, fabsf(__uint_as_float(v[j])));
  const float to1 = __uint_as_float((uint32_t)(103 + M) << 23);  // 2^(M - 24)
  if (EXACT && EVERY) mark(mx * to1);
  if (__all_sync(0xffffffffu, mx < lim)) {
    const int32_t mult = sgn * (1 << (SHIFT & 31));
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int32_t g = (int32_t)__float_as_uint(__fadd_rn(__uint_as_float(v[j]), magic));
      if constexpr (SHIFT < 32) {
        asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(z[j]) : "r"(g), "r"(mult));
      } else {
        z[j] += (long long)((unsigned long long)((uint32_t)g * (uint32_t)mult) << 32);
      }
    }
  } else {
    if (EXACT && !EVERY && mx * to1 >= 1.0f) mark(mx * to1);
    const float scale = __uint_as_float((uint32_t)(127 + M) << 23);  // 2^M
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const long long g = (long long)__float2int_rn(__fmul_rn(__uint_as_float(v[j]), scale)) + (long long)oz_magic(M);
      z[j] += (long long)((unsigned long long)(sgn < 0 ? -g : g) << SHIFT);
    }
  }
}

// The drain of the accumulator of product (a, b): stored products carry 2^-(rho_a+rho_b),
// their integers weigh 2^(56-e_a-e_b) on the fixed point's grid.  GRID: the sums are taken as
// multiples of 2^-GRID (the sixth accumulator, not an integer, rounded to 2^-56).
template <int A, int B, int GRID = oz_e(A) + oz_e(B)>
struct OzSlot {
  static constexpr int M = oz_rho(A) + oz_rho(B) - (oz_e(A) + oz_e(B) - GRID);
  static constexpr int SHIFT = 56 - GRID;
  static constexpr unsigned long long offset = (unsigned long long)oz_magic(M) << SHIFT;
  template <bool EVERY, typename Mark>
  static __device__ __forceinline__ void drain(uint32_t taddr, int sgn, const Mark& mark, long long (&z)[16]) {
    oz_drain_slot<M, SHIFT, GRID == oz_e(A) + oz_e(B), EVERY>(taddr + oz_col(A, B), sgn, mark, z);
  }
};
using OzSixth = OzSlot<0, 4, 56>;

// The first pass of one chunk, in two halves: the columns the second pass reuses, then the
// columns that hold the sums from then on, into z (negated for sgn < 0).
template <bool EVERY, typename Mark>
__device__ __forceinline__ void oz_drain_high_a(uint32_t taddr, int sgn, const Mark& mark, long long (&z)[16]) {
  OzSixth::template drain<EVERY>(taddr, sgn, mark, z);
  OzSlot<0, 3>::template drain<EVERY>(taddr, sgn, mark, z);
}
template <bool EVERY, typename Mark>
__device__ __forceinline__ void oz_drain_high_b(uint32_t taddr, int sgn, const Mark& mark, long long (&z)[16]) {
  OzSlot<0, 2>::template drain<EVERY>(taddr, sgn, mark, z);
  OzSlot<1, 1>::template drain<EVERY>(taddr, sgn, mark, z);
}

// The second pass of one chunk into z.
template <bool EVERY, typename Mark>
__device__ __forceinline__ void oz_drain_low(uint32_t taddr, int sgn, const Mark& mark, long long (&z)[16]) {
  OzSlot<0, 0>::template drain<EVERY>(taddr, sgn, mark, z);
  OzSlot<0, 1>::template drain<EVERY>(taddr, sgn, mark, z);
}

// Where z starts: less the constants that the six drains of a round add.
constexpr unsigned long long kOzOffset = OzSixth::offset + OzSlot<0, 3>::offset + OzSlot<0, 2>::offset +
                                         OzSlot<1, 1>::offset + OzSlot<0, 0>::offset + OzSlot<0, 1>::offset;

// |v| 2^-56 as FP32 (integer instructions, truncated: at most 2^-23 below), for the row
// norms of the adjoint's new Xbar on its fixed-point grid.
__device__ __forceinline__ float fixed_to_f32_abs(long long v) {
  const unsigned long long a = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  if (a == 0) return 0.0f;
  const int lz = __clzll(a);
  const uint32_t mant = (uint32_t)((a << lz) >> 40) & 0x7FFFFFu;  // 23 bits below the leading one
  return __uint_as_float(((uint32_t)(63 - lz - 56 + 127) << 23) | mant);
}

// Sum of v[j] (j < 16) over the 32 lanes of a warp in 16 shuffles (each step exchanges half
// of the remaining columns with the partner lane); lanes 2q and 2q + 1 end with the sum of
// column `col` = 8 b4 + 4 b3 + 2 b2 + b1 (b the lane's bits).
__device__ __forceinline__ float warp_colsum16(const float (&v)[16], int lane, int& col) {
  float a8[8], a4[4], a2[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    a8[j] = (h16 ? v[j + 8] : v[j]) + __shfl_xor_sync(0xffffffffu, h16 ? v[j] : v[j + 8], 16);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    a4[j] = (h8 ? a8[j + 4] : a8[j]) + __shfl_xor_sync(0xffffffffu, h8 ? a8[j] : a8[j + 4], 8);
#pragma unroll
  for (int j = 0; j < 2; ++j)
    a2[j] = (h4 ? a4[j + 2] : a4[j]) + __shfl_xor_sync(0xffffffffu, h4 ? a4[j] : a4[j + 2], 4);
  float a1 = (h2 ? a2[1] : a2[0]) + __shfl_xor_sync(0xffffffffu, h2 ? a2[0] : a2[1], 2);
  a1 += __shfl_xor_sync(0xffffffffu, a1, 1);
  col = (h16 ? 8 : 0) + (h8 ? 4 : 0) + (h4 ? 2 : 0) + (h2 ? 1 : 0);
  return a1;
}

// Predicated evict-first stores: the columns of a diagonal tile differ in the lanes that store,
// and a branch per column costs more than the stores.
__device__ __forceinline__ void store_word_if(bool on, long long* q, long long v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @p st.global.cs.b64 [%1], %2;\n}\n" ::"r"((int)on),
               "l"(q), "l"(v)
               : "memory");
}
// the digits of one element: word w (0..3) of the packed digits of four, dstr elements apart
__device__ __forceinline__ void store_digits_if(bool on, uint16_t* d, size_t dstr, const uint32_t (&dw)[OZ_SLICES][2],
                                                int w) {
  static_assert(OZ_SLICES == 5, "five digit arenas");
  unsigned short h[OZ_SLICES];
#pragma unroll
  for (int q = 0; q < OZ_SLICES; ++q) h[q] = (unsigned short)(w & 1 ? dw[q][w >> 1] >> 16 : dw[q][w >> 1]);
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @p st.global.cs.u16 [%1], %6;\n @p st.global.cs.u16 [%2], %7;\n"
      " @p st.global.cs.u16 [%3], %8;\n @p st.global.cs.u16 [%4], %9;\n @p st.global.cs.u16 [%5], %10;\n}\n" ::"r"(
          (int)on),
      "l"(d), "l"(d + dstr), "l"(d + 2 * dstr), "l"(d + 3 * dstr), "l"(d + 4 * dstr), "h"(h[0]), "h"(h[1]), "h"(h[2]),
      "h"(h[3]), "h"(h[4])
      : "memory");
}

// K slices of a part of size sz; brief items count slices of 32 in either form (wide: halves of the
// loaded ones).
template <bool WIDE>
__device__ __forceinline__ int oz_nslices(int sz, bool brief) {
  constexpr int BK = WIDE ? OZ_BK_WIDE : OZ_BK;
  return brief ? (sz + OZ_BK - 1) / OZ_BK : (sz + BK - 1) / BK;
}
// K slices [x, y) of an item: all of them (the adjoint's first ns slices multiply Xbar by X, the rest X
// by Xbar) or one half (0, 1; -1 none), up to or from slice z.
template <bool ADJ, bool WIDE>
__device__ __forceinline__ int3 oz_slices(int sz, int half, bool brief) {
  const int ns = oz_nslices<WIDE>(sz, brief), all = ADJ ? 2 * ns : ns, mid = ADJ ? ns : (ns + 1) / 2;
  return make_int3(half == 1 ? mid : 0, half == 0 ? mid : all, mid);
}
// End of the round of both passes that starts at slice c0: rounds of equal length of at most 2048 columns,
// and (halves: plans whose items may be split) never across the halves, so that a tile's sums are
// rounded alike whether one item forms it or two; one slice of a brief item.
template <bool WIDE>
__device__ __forceinline__ int oz_round_end(int c0, int3 kr, bool halves, bool brief) {
  constexpr int CHUNK = 2048 / (WIDE ? OZ_BK_WIDE : OZ_BK);
  if (brief) return c0 + 1;
  const int left = (halves && c0 < kr.z ? min(kr.z, kr.y) : kr.y) - c0;
  if (left <= CHUNK) return c0 + left;
  const int rounds = (left + CHUNK - 1) / CHUNK;
  return c0 + (left + rounds - 1) / rounds;
}
// How many rounds an item takes.
template <bool WIDE>
__device__ __forceinline__ int oz_rounds(int3 kr, bool halves, bool brief) {
  constexpr int CHUNK = 2048 / (WIDE ? OZ_BK_WIDE : OZ_BK);
  if (brief) return kr.y - kr.x;
  if (halves && kr.x < kr.z && kr.z < kr.y) return (kr.z - kr.x + CHUNK - 1) / CHUNK + (kr.y - kr.z + CHUNK - 1) / CHUNK;
  return (kr.y - kr.x + CHUNK - 1) / CHUNK;
}

// Opens (by a warp) the taking again of coherent parts' items.
__device__ __noinline__ void oz_open_again(OzAgain* again, int place) {
  if ((threadIdx.x & 31) == 0) again->ctr = again->done = 0;
  __threadfence();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) *(volatile int32_t*)&again->go = place;
}
// Item `it` of the launch, with its part's tables; brief where its part was found coherent up to step `brief_to`
// (negative: no part was, or it may not be read yet).
template <bool ADJ, bool WIDE>
__device__ __forceinline__ void oz_read_item(const OzStepArgs& a, int it, int brief_to, OzItem* w) {
  const int code = a.split ? a.split_items[it / a.pieces] : it / a.pieces;
  const Tile t = a.tiles[a.split ? code >> 1 : code];
  // in flight beside the part's tables: the loads of an item wait for this chain
  int32_t coh = OZ_INCOHERENT;
  if (brief_to >= 0) coh = *(volatile int32_t*)&a.coh[t.part];
  const PartDesc p = a.parts[t.part];
  const bool brief = coh <= brief_to;
  w->code = code;
  w->piece = it % a.pieces;
  w->ti = t.ti;
  w->tj = t.tj;
  w->slot = t.slot;
  w->part = t.part;
  w->off = p.off;
  w->soff = p.soff;
  w->s = p.s;
  w->c = p.c;
  w->ld = p.ld;
  w->brief = brief;
  w->rounds = oz_rounds<WIDE>(oz_slices<ADJ, WIDE>(p.s, a.split ? code & 1 : -1, brief), a.halves, brief);
}
// ADJ: the adjoint step (see the top of the file): K runs over [Xbar | X] x [X ; Xbar],
// diagonal tiles load both operands, the epilogue forms Xbar_new in FP64 without digits
// or traces and adds its squared row norms (FP32, on the grid of the input scale); the block that ends the
// launch turns them into each part's new scale.
template <bool ADJ, bool WIDE>
__global__ void __launch_bounds__(OZ_THREADS, 1) oz_step_kernel(const __grid_constant__ OzStepArgs a) {
  constexpr int T = OZ_SLICES;
  constexpr int BK = WIDE ? OZ_BK_WIDE : OZ_BK;  // K per slice
  constexpr uint32_t DTILE = 128u * BK * 2u;     // one digit tile: 128 rows x 64 or 128 B
  // instruction descriptor without N (bits 17..22, N / 8): FP32 accumulate, FP16 A and B, M = 128
  constexpr uint32_t IDESC = (1u << 4) | ((128u >> 4) << 24);

  const bool rec = !ADJ && a.mode == SQ_RECOMPUTE;
  pdl_release();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* sb = smem_raw + (base - raw);
  const uint32_t bars = base + OZ_RING_B;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sb + OZ_RING_B + 8 * OZ_BARS);
  int* s_err = reinterpret_cast<int*>(tmem_slot + 1);
  int* s_half = reinterpret_cast<int*>(tmem_slot + 2);  // split K: halves of the tile done before
  // 1: a sum has reached 2^24.  From the decision at the pause on: 8, and 2 where this block ends the launch, 4 where it
  // forms coherent parts again, 16 while warp 3 waits for that
  __shared__ int s_walk;
  __shared__ int s_taken;  // items taken again
  longlong2* red = reinterpret_cast<longlong2*>(sb + OZ_RING_B + 8 * OZ_BARS + 16);
  // warp 0's producer takes each next tile (claimed from a counter in global memory, or dealt)
  // and passes it on with its part through a ring (full: taken; empty: read by the other
  // producer, the MMA thread and every epilogue warp)
  const uint32_t ring_bars = smem_u32(red + 128);
  OzItem* s_items = reinterpret_cast<OzItem*>(reinterpret_cast<uint8_t*>(red + 128) + 8 * 2 * OZ_RING);
  auto item_full = [&](int q) { return ring_bars + 8u * q; };
  auto item_empty = [&](int q) { return ring_bars + 8u * (OZ_RING + q); };
  auto full = [&](int op, uint32_t g) { return bars + 8u * (op * OZ_GROUPS + g % OZ_GROUPS); };  // rows I 0, rows J 1
  auto empty = [&](int s) { return bars + 8u * (2 * OZ_GROUPS + s); };
  // accumulator barriers: [0] first pass, [1] second
  auto afull = [&](int pass) { return bars + 8u * (2 * OZ_GROUPS + OZ_TILES + pass); };
  auto aempty = [&](int pass) { return bars + 8u * (2 * OZ_GROUPS + OZ_TILES + 2 + pass); };
  auto tile_addr = [&](uint32_t s) { return base + s * DTILE; };                       // wide
  auto unit = [&](int s) { return base + (uint32_t)s * OZ_UNIT_B; };                   // narrow
  int32_t* abort_flag = &a.ctl.st->timeout;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  // work items: the upper tiles, or (split K) each tile's two K halves
  const bool split = a.split != 0;
  // column pieces of a tile, each an item of its own: 1 (128 columns) or 2 (64 columns)
  const int pieces = a.pieces, pcols = 128 / pieces;
  const int nitems = (split ? 2 * a.ntiles : a.ntiles) * pieces;
  // columns of a piece that its MMAs cover
  auto piece_cols = [&](int sz, int tj, int piece) {
    return max(0, min(pcols, oz_tile_cols(sz, tj) - piece * pcols));
  };
  // items claimed at run time (forward, tail and reverse steps; the list order) or dealt in turn
  // (the rebuilt iterates, which may run beside reverse steps and have no last block)
  const bool dyn = a.tile_ctr != nullptr && !rec;

  if (warp == 0) {
    for (int q = lane; q < 2 * OZ_GROUPS + OZ_TILES; q += 32) mbar_init(bars + 8u * q, 1);
    if (lane < 2) {
      mbar_init(afull(lane), 1);
      mbar_init(aempty(lane), OZ_EPI_WARPS);
    }
    if (lane < OZ_RING) {
      mbar_init(item_full(lane), 1);
      mbar_init(item_empty(lane), 2 + OZ_EPI_WARPS);
    }
    if (lane == 0) *s_err = s_walk = s_taken = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  // the first item's tables, which no launch writes, before the launch before this one is done
  if (threadIdx.x == 0) {
    if ((int)blockIdx.x < nitems) oz_read_item<ADJ, WIDE>(a, blockIdx.x, -1, s_items);
    else s_items->code = rec ? OZ_END : OZ_PAUSE;
  }
  pdl_wait();  // everything below reads what the launch before wrote
  int step = a.step;
  bool run, coherent = true;  // whether some part may have been found coherent
  int n = 0;
  if (ADJ || rec) {
    // reverse step `step` exists iff step <= n; a rebuilt X_step is read iff step < n
    n = *(volatile int32_t*)&a.ctl.st->steps;
    run = ADJ ? step <= n : step < n;
  } else if (a.mode == SQ_FORWARD) {
    const uint2 v = ld_volatile2(&a.ctl.st->stopped);
    run = v.x == 0;
    coherent = v.y != 0;
  } else {
    const int32_t stt = *(volatile int32_t*)&a.ctl.st->status;
    run = stt != ST_NONFINITE && stt != ST_TIMEOUT;
    step = *(volatile int32_t*)&a.ctl.st->steps + 1;
  }
  if (!run) {  // the loop has stopped: nothing to do
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    return;
  }
  // a part's items take brief rounds after the step that found it coherent (a rebuilt step: from that one on)
  const int place = ADJ ? n - step + 1 : step, brief_to = !coherent ? -1 : (rec ? place : place - 1);
  if (threadIdx.x == 0 && brief_to >= 0 && s_items->code >= 0 && a.coh[s_items->part] <= brief_to) {
    s_items->brief = 1;
    s_items->rounds =
        oz_rounds<WIDE>(oz_slices<ADJ, WIDE>(s_items->s, split ? s_items->code & 1 : -1, true), false, true);
  }
  // digit buffers read / written (the adjoint's sets are passed explicitly)
  const int dbi = (ADJ || rec) ? 0 : (step - 1) & 1, dbo = (ADJ || rec) ? 0 : step & 1;

  const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(a.maps) + (size_t)dbi * T * a.nparts;
  const CUtensorMap* maps_mn = reinterpret_cast<const CUtensorMap*>(a.maps_mn) + (size_t)dbi * T * a.nparts;
  const CUtensorMap* maps_b = reinterpret_cast<const CUtensorMap*>(a.maps_b);
  const CUtensorMap* maps_mn_b = reinterpret_cast<const CUtensorMap*>(a.maps_mn_b);

  // warp-collective bounded wait (the same outcome in every lane)
  auto wait = [&](uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0;
  };
  // The pause of the walk, passed once by every warp, after its part of this CTA's items: when the last block of
  // the launch has come here, parts found coherent are formed again.
  auto pause = [&]() {
    tc_fence_before();
    asm volatile("bar.sync 2, %0;\n" ::"n"(OZ_THREADS) : "memory");
  };
  auto decision = [&]() {  // (every warp but warp 0, which takes it)
    pause();
    asm volatile("bar.sync 2, %0;\n" ::"n"(OZ_THREADS) : "memory");
    tc_fence_after();
    return (*(volatile int*)&s_walk & 4) != 0;
  };
  auto paused = [&]() { return rec || (*(volatile int*)&s_walk & 8) != 0; };  // (rebuilt steps have no pause)
  if (warp == 0 || warp == 2) {
    // Like the issuing warp below, the whole warp walks the units with warp-uniform values and
    // one elected lane issues the loads.
    const int op = warp >> 1;      // 0: rows I, 1: rows J
    uint32_t su = 0, ph = 0;       // next tile or unit of the ring and its phase
    uint32_t grp = 0;              // wide: groups of tiles this warp has begun
    uint32_t used = 0, phase = 0;  // narrow: units this warp has filled, and the phases of the last fills
    bool bad = false;
    // dynamic: the first item is blockIdx.x, the next ones gridDim.x + the counter's count,
    // each claimed one item ahead so that the atomic's latency hides behind an item's loads
    int nxt = nitems;
    if (op == 0 && lane == 0 && dyn && (int)blockIdx.x < nitems)
      nxt = (int)gridDim.x + (int)atomicAdd(a.tile_ctr, 1u);
    int redo = -1;  // warp 0, after the pause: items taken again
    // Warp 0 takes this CTA's ticket, with a mark in its upper half if a sum has reached 2^24; the last
    // block of the launch to take one knows so whether any has, and all items are done then.  Blocks whose ticket
    // shows such a sum wait a while for that (warp 3: the wait in this loop, even as a call, made every
    // step 1.5 % slower) and help; no block depends on a helper, and none waits in a launch without such a sum.
    // One part of 1,500: 7.3 ms a density with helpers, 29 without; of 4,096 85 and 426.
    auto decide = [&]() {
      if (op != 0) return decision();
      pause();
      redo = 0;
      const unsigned int found = *(volatile int*)&s_walk & 1 ? 0x10000u : 0u;
      unsigned int t = 0;
      if (lane == 0) {
        if (*(volatile int*)s_err) a.ctl.st->timeout = 1;
        __threadfence();
        t = found + atomicAdd(&a.ctl.st->counter, found + 1u);
      }
      t = __shfl_sync(0xffffffffu, t, 0);
      int walk = 8;
      if ((t & 0xFFFFu) == gridDim.x - 1) {
        __threadfence();
        walk = 10;
        if (t >> 16 && *(volatile int32_t*)&a.ctl.st->timeout == 0) {
          walk = 12;
          if constexpr (ADJ) {  // the norms of the rows formed again are summed again too
            for (int k = 0; k < a.nparts; ++k)
              if (__ldcg(a.coh_new + k) && a.coh[k] > brief_to)
                for (int r = lane; r < a.parts[k].s; r += 32) a.normf[a.parts[k].soff + r] = 0.0f;
          }
          oz_open_again(a.again, place);
        }
      } else if (t >> 16) {
        walk = 24;
      }
      if (lane == 0) *(volatile int*)&s_walk = walk;
      __syncwarp();
      asm volatile("bar.arrive 3, 64;\n" ::: "memory");
      asm volatile("bar.sync 2, %0;\n" ::"n"(OZ_THREADS) : "memory");
      return (*(volatile int*)&s_walk & 4) != 0;
    };
    for (int v = 0, it = blockIdx.x; !bad; ++v, it += gridDim.x) {
      const int q = v % OZ_RING;
      if (op == 0) {
        if (v >= OZ_RING && !wait(item_empty(q), ((v / OZ_RING) - 1) & 1)) {
          bad = true;
          break;
        }
        if (lane == 0) {
          if (dyn && v > 0) {
            it = nxt;
            if (it < nitems) nxt = (int)gridDim.x + (int)atomicAdd(a.tile_ctr, 1u);
          }
          if (v > 0) {
            do {  // after the pause: those of parts found coherent by this launch
              if (redo >= 0) it = atomicAdd(&a.again->ctr, 1);
              if (it >= nitems) {
                s_taken = redo;
                s_items[q].code = redo >= 0 || rec ? OZ_END : OZ_PAUSE;
                break;
              }
              if (redo >= 0) ++redo;
              oz_read_item<ADJ, WIDE>(a, it, redo >= 0 ? OZ_INCOHERENT : brief_to, s_items + q);
            } while (redo >= 0 && !(__ldcg(a.coh_new + s_items[q].part) && a.coh[s_items[q].part] > brief_to));
          }
          mbar_arrive(item_full(q));
        }
        __syncwarp();
      } else if (!wait(item_full(q), (v / OZ_RING) & 1)) {
        bad = true;
        break;
      }
      OzItem w;
      w.code = __shfl_sync(0xffffffffu, s_items[q].code, 0);
      w.ti = __shfl_sync(0xffffffffu, s_items[q].ti, 0);
      w.tj = __shfl_sync(0xffffffffu, s_items[q].tj, 0);
      w.part = __shfl_sync(0xffffffffu, s_items[q].part, 0);
      w.s = __shfl_sync(0xffffffffu, s_items[q].s, 0);
      w.piece = __shfl_sync(0xffffffffu, s_items[q].piece, 0);
      const bool brief = __shfl_sync(0xffffffffu, s_items[q].brief, 0) != 0;
      if (op == 1 && lane == 0) mbar_arrive(item_empty(q));
      if (w.code == OZ_PAUSE && decide()) continue;
      if (w.code < 0) break;
      if (piece_cols(w.s, w.tj, w.piece) == 0) continue;
      const int half = split ? w.code & 1 : -1;
      const bool dg = !ADJ && w.ti == w.tj;  // X X on a diagonal tile: B is A
      const int blk = op == 0 ? w.ti : w.tj;
      const int ns = oz_nslices<WIDE>(w.s, brief);
      const int3 kr = oz_slices<ADJ, WIDE>(w.s, half, brief);
      if constexpr (WIDE) {
        const int unit = brief ? OZ_BK : BK;  // brief: a slice's tiles hold its 32 columns and 32 that are not multiplied
        // ring places of this pass over: `by` tiles on
        auto advance = [&](uint32_t by) {
          su += by;
          if (su >= OZ_TILES) {
            su -= OZ_TILES;
            ph ^= 1;
          }
        };
        // The tiles of one slice of a pass over T digits: rows I from the last digit down, rows J from
        // the first up, in turn; on a diagonal tile rows I alone.  The MMA warp waits for them in groups
        // (one barrier each): three and two of the five digits, both of the second pass's, or all of a
        // diagonal tile.  K-major from columns `blk` of the tiles on or above the diagonal (slice
        // block <= blk), else MN-major from rows `blk` of the tile (blk, slice).  The adjoint's first
        // ns slices take Xbar for rows I and X for rows J, the rest X for rows I and Xbar for rows J.
        // A place is waited for when its turn comes, never looked at ahead: 13 being odd, it changes its
        // producer every lap, and this warp knows that the phase before the one it waits for is over only from its
        // last own fill (it lies 11 places before the tile whose release that was).  With a look at all five places
        // at a slice's start, rows J's last could be taken as free one phase early, the release of rows J's third
        // tile becoming visible after that of rows I's last, and a live digit tile was overwritten.
        auto slice = [&](int ks, int T) {
          const bool h2 = ADJ && ks >= ns;
          const bool xb = ADJ && (op == 0) != h2;
          const int k0 = (h2 ? ks - ns : ks) * unit;
          const bool kmajor = k0 / 128 <= blk;
          const CUtensorMap* const map =
              (kmajor ? (xb ? maps_b : maps) : (xb ? maps_mn_b : maps_mn)) + w.part;
          for (int i = 0; i < T; ++i) {
            if (op == 1) advance(1);
            if (!wait(empty(su), ph ^ 1u)) {
              bad = true;
              return;
            }
            const bool head = i == 0 || (i == OZ_HEAD && !dg);
            grp += head;
            const uint32_t bar = full(op, grp - 1u);
            const int dig = op == 0 ? T - 1 - i : i;
            if (elect_one()) {
              if (head) mbar_expect_tx(bar, DTILE * (uint32_t)(T == OZ_LOW || dg ? T : (i == 0 ? OZ_HEAD : T - OZ_HEAD)));
              if (kmajor) tma_load_3d(tile_addr(su), map, k0, blk * 128, dig, bar);
              else tma_load_4d(tile_addr(su), map, 0, k0, 2 * blk, dig, bar);
            }
            advance(op == 0 && !dg ? 2 : 1);
          }
        };
        if (op == 1 && dg) {  // rows I only: this warp's place in the ring moves past them
          const uint32_t by = su + (uint32_t)((kr.y - kr.x) * (OZ_SLICES + OZ_LOW));
          ph ^= (by / OZ_TILES) & 1u;
          su = by % OZ_TILES;
          continue;
        }
        for (int c0 = kr.x, c1; c0 < kr.y && !bad; c0 = c1) {
          c1 = oz_round_end<WIDE>(c0, kr, a.halves, brief);
          for (int kb = c0; kb < c1 && !bad; ++kb) slice(kb, OZ_SLICES);
          for (int kb = c0; kb < c1 && !bad; ++kb) slice(kb, OZ_LOW);
        }
      } else {
        // the next unit of this thread; false if the wait gave up
        auto acquire = [&](uint32_t bytes, uint32_t& u) {
          if (op == 1 && ++su == OZ_UNITS) {
            su = 0;
            ph ^= 1;
          }
          u = su;
          if (!wait(empty(u), ph ^ 1u)) return false;
          if (elect_one()) mbar_expect_tx(full(0, u), bytes);
          used |= 1u << u;
          phase = (phase & ~(1u << u)) | (ph << u);
          if (++su == OZ_UNITS) {
            su = 0;
            ph ^= 1;
          }
          if (op == 0 && !dg && ++su == OZ_UNITS) {
            su = 0;
            ph ^= 1;
          }
          return true;
        };
        // one request brings a slice's digit tiles: K-major from columns `blk` of the tiles on or
        // above the diagonal (slice block <= blk), else MN-major from rows `blk` of the tile (blk,
        // slice).  The adjoint's first ns slices take Xbar for rows I and X for rows J, the rest
        // X for rows I and Xbar for rows J
        auto load = [&](uint32_t dst, uint32_t bar, int ks, size_t at) {
          const bool h2 = ADJ && ks >= ns;
          const bool xb = ADJ && (op == 0) != h2;
          const int k0 = (h2 ? ks - ns : ks) * BK;
          if (elect_one()) {
            if (k0 / 128 <= blk) tma_load_3d(dst, (xb ? maps_b : maps) + at, k0, blk * 128, 0, bar);
            else tma_load_4d(dst, (xb ? maps_mn_b : maps_mn) + at, 0, k0, 2 * blk, 0, bar);  // 64-row atoms x digits
          }
        };
        if (op == 1 && dg) {  // rows I only: this thread's place in the ring moves past them
          for (int c0 = kr.x, c1; c0 < kr.y; c0 = c1) {
            c1 = oz_round_end<WIDE>(c0, kr, a.halves, brief);
            su += (uint32_t)(c1 - c0 + (c1 - c0 + OZ_LOW_SUB - 1) / OZ_LOW_SUB);
          }
          ph ^= (su / OZ_UNITS) & 1u;
          su %= OZ_UNITS;
          continue;
        }
        for (int c0 = kr.x, c1; c0 < kr.y && !bad; c0 = c1) {
          c1 = oz_round_end<WIDE>(c0, kr, a.halves, brief);
          uint32_t u;
          for (int kb = c0; kb < c1; ++kb) {
            if (!acquire(T * DTILE, u)) {
              bad = true;
              break;
            }
            load(unit(u), full(0, u), kb, (size_t)a.nparts + w.part);
          }
          for (int kb = c0; kb < c1 && !bad; kb += OZ_LOW_SUB) {
            const int m = min(OZ_LOW_SUB, c1 - kb);
            if (!acquire((uint32_t)(m * OZ_LOW) * DTILE, u)) {
              bad = true;
              break;
            }
            for (int x = 0; x < m; ++x)
              load(unit(u) + (uint32_t)(x * OZ_LOW) * DTILE, full(0, u), kb + x, (size_t)2 * a.nparts + w.part);
          }
        }
      }
    }
    if (bad) {
      *s_err = 1;
      // loads in flight still write shared memory: wait for them on this warp's own limit
      if (WIDE) {
        for (uint32_t g = grp > OZ_GROUPS - 1 ? grp - (OZ_GROUPS - 1) : 0; g < grp; ++g)
          (void)mbar_wait_own(full(op, g), (g / OZ_GROUPS) & 1);
      } else {
        for (uint32_t u = 0; u < (uint32_t)OZ_UNITS; ++u)
          if (used >> u & 1u) (void)mbar_wait_own(full(0, u), phase >> u & 1u);
      }
      if (!paused()) (void)decide();
    }
  } else if (warp == 1) {
    // The whole warp walks the slices with warp-uniform values (the item's fields through a
    // shuffle), so that descriptors are formed in uniform registers, and one elected lane
    // issues.  A step's MMAs (4 to 12) keep the tensor pipe busy while the next step's tiles are waited for.
    uint32_t su = 0, ph = 0;  // next tile or unit of the ring and its phase
    uint32_t ga = 0, gb = 0;  // wide: groups of tiles of rows I and rows J taken
    int last = -1;            // last tile or unit released by a commit
    uint32_t lastph = 0;
    int v = 0, r = 0;  // items taken, rounds of both passes done by this CTA
    bool bad = false;
    for (; !bad; ++v) {
      const int q = v % OZ_RING;
      if (!wait(item_full(q), (v / OZ_RING) & 1)) {
        bad = true;
        break;
      }
      const int code = __shfl_sync(0xffffffffu, s_items[q].code, 0);
      const int ti = __shfl_sync(0xffffffffu, s_items[q].ti, 0), tj = __shfl_sync(0xffffffffu, s_items[q].tj, 0);
      const int sz = __shfl_sync(0xffffffffu, s_items[q].s, 0);
      const int piece = __shfl_sync(0xffffffffu, s_items[q].piece, 0);
      const bool brief = __shfl_sync(0xffffffffu, s_items[q].brief, 0) != 0;
      if (lane == 0) mbar_arrive(item_empty(q));
      if (code == OZ_PAUSE && decision()) continue;
      if (code < 0) break;
      const int ncols = piece_cols(sz, tj, piece);
      if (ncols == 0) continue;
      const int half = split ? code & 1 : -1;
      const bool dg = !ADJ && ti == tj;
      const int ns = oz_nslices<WIDE>(sz, brief);
      const int3 kr = oz_slices<ADJ, WIDE>(sz, half, brief);
      const uint32_t idesc0 = IDESC | ((uint32_t)(ncols >> 3) << 17);
      if constexpr (WIDE) {
        const int unit = brief ? OZ_BK : BK;
        const uint64_t dk = smem_desc_sw<2 * BK>(0), dm = smem_desc_mn128(0, DTILE / 2);
        // the ring's tile `off` places past s0 (phase p0)
        auto at = [&](uint32_t s0, uint32_t off) { return s0 + off >= OZ_TILES ? s0 + off - OZ_TILES : s0 + off; };
        auto parity = [&](uint32_t s0, uint32_t p0, uint32_t off) { return s0 + off >= OZ_TILES ? p0 ^ 1u : p0; };
        // the next group of tiles of each operand has come (a diagonal tile's serves both)
        auto loaded = [&]() {
          bool in = mbar_wait(full(0, ga), (ga / OZ_GROUPS) & 1, abort_flag);
          ++ga;
          if (!dg) {
            in = in && mbar_wait(full(1, gb), (gb / OZ_GROUPS) & 1, abort_flag);
            ++gb;
          }
          return __all_sync(0xffffffffu, in) != 0;
        };
        // The tiles of a slice lie in the ring in the order the producers fill it (rows I and rows J in
        // turn; on a diagonal tile rows I alone, the tile of a digit serving both).  Descriptors of
        // slice ks, whose first tile is the next of the ring.  Blocks right of the tile's own came in
        // MN-major (transpose bits 15 / 16); a K = 16 step advances 32 B in a K-major row, 2 KB (16 K
        // values) in an MN-major tile
        OzWide o;
        auto prepare = [&](auto low, int ks) {
          constexpr int N = oz_digits<decltype(low)::value>();
          const int k0 = (ADJ && ks >= ns ? ks - ns : ks) * unit, kt = k0 / 128;
          const bool amn = kt > ti, bmn = kt > tj;
          const uint32_t alo = (uint32_t)(amn ? dm : dk) + (base >> 4), blo = (uint32_t)(bmn ? dm : dk) + (base >> 4);
          o.ahi = (uint32_t)((amn ? dm : dk) >> 32);
          o.bhi = (uint32_t)((bmn ? dm : dk) >> 32);
          o.adv_a = amn ? (2048u >> 4) : (32u >> 4);
          o.adv_b = bmn ? (2048u >> 4) : (32u >> 4);
          o.idesc = idesc0 | ((amn ? 1u : 0u) << 15) | ((bmn ? 1u : 0u) << 16);
          o.steps = min(unit / 16, (sz - k0 + 15) / 16);
  #pragma unroll
          for (int q = 0; q < N; ++q) {
            o.a[q] = alo + at(su, dg ? N - 1 - q : 2 * (N - 1 - q)) * (DTILE >> 4);
            o.b[q] = blo + at(su, dg ? N - 1 - q : 2 * q + 1) * (DTILE >> 4);
          }
        };
        // The MMAs of the prepared slice.  Before the last K = 16 step of a group of tiles
        // the next group is waited for, and before that of the slice the next one's descriptors are formed
        // (next()): the tensor pipe has the products issued so far to work on meanwhile.  Every MMA issued is committed, also where a wait gives up.
        auto slice = [&](auto low, bool first, auto next) {
          constexpr bool LOW = decltype(low)::value;
          constexpr int N = oz_digits<LOW>();
          const uint32_t s0 = su, p0 = ph;
          const OzWide c = o;
          su += (uint32_t)(dg ? N : 2 * N);
          if (su >= OZ_TILES) {
            su -= OZ_TILES;
            ph ^= 1;
          }
          bool good = true;
          auto step = [&](auto idx) {
            constexpr int I = decltype(idx)::value;
            constexpr bool ends = I == N - 1 || I == OZ_HEAD - 1;  // of a group
            if (!good) return;
            if (elect_one()) oz_issue_wide<LOW, I, 0, BK / 16 - 1>(tmem, c, first);
            bool more = true;
            if constexpr (I == N - 1) more = next();
            if (ends && more && (I == N - 1 || !dg)) good = loaded();
            if (elect_one()) {
              oz_issue_wide<LOW, I, BK / 16 - 1, BK / 16>(tmem, c, first);
              if (!dg) {
                mma_commit(empty(at(s0, 2 * I)));
  #pragma unroll
                for (int b = 0; b <= I; ++b)
                  if (oz_b_last<LOW>(b) == I) mma_commit(empty(at(s0, 2 * b + 1)));
              } else if (I == N - 1) {
  #pragma unroll
                for (int q = 0; q < N; ++q) mma_commit(empty(at(s0, q)));
              }
            }
            last = (int)at(s0, dg ? 0 : 2 * I);
            lastph = parity(s0, p0, dg ? 0 : 2 * I);
          };
          step(std::integral_constant<int, 0>());
          step(std::integral_constant<int, 1>());
          if constexpr (!LOW) {
            step(std::integral_constant<int, 2>());
            step(std::integral_constant<int, 3>());
            step(std::integral_constant<int, 4>());
          }
          return good;
        };
        prepare(std::false_type(), kr.x);
        bad = !loaded();
        for (int c0 = kr.x, c1; c0 < kr.y && !bad; c0 = c1, ++r) {
          c1 = oz_round_end<WIDE>(c0, kr, a.halves, brief);
          // first pass: it reuses the columns of the previous round's second
          if (r > 0 && !wait(aempty(1), (r - 1) & 1)) {
            bad = true;
            break;
          }
          tc_fence_after();
          for (int kb = c0; kb < c1 && !bad; ++kb)
            bad = !slice(std::false_type(), kb == c0, [&]() {
              if (kb + 1 < c1) prepare(std::false_type(), kb + 1);
              else prepare(std::true_type(), c0);
              return true;
            });
          if (bad) break;
          if (elect_one()) mma_commit(afull(0));
          // second pass: it reuses columns of this round's first
          if (!wait(aempty(0), r & 1)) {
            bad = true;
            break;
          }
          tc_fence_after();
          for (int kb = c0; kb < c1 && !bad; ++kb)
            bad = !slice(std::true_type(), kb == c0, [&]() {
              if (kb + 1 < c1) prepare(std::true_type(), kb + 1);
              else if (c1 < kr.y) prepare(std::false_type(), c1);
              else return false;
              return true;
            });
          if (!bad && elect_one()) mma_commit(afull(1));
        }
      } else {
        // rows J of a piece start 64 rows into each digit tile: 64 B each K-major, one atom MN-major
        const uint32_t poff = (uint32_t)piece * ((64u * BK * 2u) >> 4);
        // operands of slice ks, tile `off` of the units sa (rows I) and sb (rows J): those right of
        // the tile's own block came in MN-major (transpose bits 15 / 16); a K = 16 step advances
        // 32 B in a K-major row, 2 KB (16 K values) in an MN-major tile
        const uint64_t dk = smem_desc_sw<2 * BK>(0), dm = smem_desc_mn128(0, DTILE / 2);
        auto operands = [&](int ks, uint32_t sa, uint32_t sb, int off) {
          const int kt = (ADJ && ks >= ns ? ks - ns : ks) / (128 / BK);
          const bool amn = kt > ti, bmn = kt > tj;
          OzNarrow o;
          o.ahi = (uint32_t)((amn ? dm : dk) >> 32);
          o.alo = (uint32_t)(amn ? dm : dk) + ((unit(sa) + (uint32_t)off * DTILE) >> 4);
          o.adv_a = amn ? (2048u >> 4) : (32u >> 4);
          o.bhi = (uint32_t)((bmn ? dm : dk) >> 32);
          o.blo = (uint32_t)(bmn ? dm : dk) + ((unit(sb) + (uint32_t)off * DTILE) >> 4) + poff;
          o.adv_b = bmn ? (2048u >> 4) : (32u >> 4);
          o.idesc = idesc0 | ((amn ? 1u : 0u) << 15) | ((bmn ? 1u : 0u) << 16);
          return o;
        };
        // the units of the next K step of the ring: rows I, rows J (the same on a diagonal tile)
        uint32_t sa, pa, sb, pb;
        auto take = [&]() {
          sa = su;
          pa = ph;
          if (++su == OZ_UNITS) {
            su = 0;
            ph ^= 1;
          }
          sb = sa;
          pb = pa;
          if (!dg) {
            sb = su;
            pb = ph;
            if (++su == OZ_UNITS) {
              su = 0;
              ph ^= 1;
            }
          }
        };
        auto loaded = [&]() {
          if (!wait(full(0, sa), pa) || (!dg && !wait(full(0, sb), pb))) return false;
          tc_fence_after();
          return true;
        };
        auto release = [&](uint32_t ua, uint32_t ub, uint32_t pub) {
          if (elect_one()) {
            mma_commit(empty(ua));
            if (!dg) mma_commit(empty(ub));
          }
          last = (int)ub;
          lastph = pub;
        };
        for (int c0 = kr.x, c1; c0 < kr.y && !bad; c0 = c1, ++r) {
          c1 = oz_round_end<WIDE>(c0, kr, a.halves, brief);
          // first pass: it reuses the columns of the previous round's second
          take();
          OzNarrow o = operands(c0, sa, sb, 0);
          if (r > 0 && !wait(aempty(1), (r - 1) & 1)) {
            bad = true;
            break;
          }
          tc_fence_after();
          for (int kb = c0; kb < c1; ++kb) {
            if (!loaded()) {
              bad = true;
              break;
            }
            if (elect_one()) oz_issue_narrow<false, 0>(tmem, o, kb == c0);
            const OzNarrow cur = o;
            const uint32_t ua = sa, ub = sb, pub = pb;
            take();  // after the last slice: the first unit of the second pass
            if (kb + 1 < c1) o = operands(kb + 1, sa, sb, 0);
            if (elect_one()) oz_issue_narrow<false, 1>(tmem, cur, false);
            release(ua, ub, pub);
          }
          if (bad) break;
          if (elect_one()) mma_commit(afull(0));
          // second pass: it reuses columns of this round's first
          o = operands(c0, sa, sb, 0);
          if (!wait(aempty(0), r & 1)) {
            bad = true;
            break;
          }
          tc_fence_after();
          for (int kb = c0; kb < c1; kb += OZ_LOW_SUB) {
            const bool two = kb + 1 < c1;
            if (!loaded()) {
              bad = true;
              break;
            }
            if (elect_one()) {
              oz_issue_narrow<true, 0>(tmem, o, kb == c0);
              oz_issue_narrow<true, 1>(tmem, o, false);
            }
            const uint32_t ua = sa, ub = sb, pub = pb;
            if (two) o = operands(kb + 1, sa, sb, OZ_LOW);
            const bool more = kb + OZ_LOW_SUB < c1;
            if (two && elect_one()) oz_issue_narrow<true, 0>(tmem, o, false);
            const OzNarrow cur = o;
            if (more) {
              take();
              o = operands(kb + OZ_LOW_SUB, sa, sb, 0);
            }
            if (two && elect_one()) oz_issue_narrow<true, 1>(tmem, cur, false);
            release(ua, ub, pub);
          }
          if (!bad && elect_one()) mma_commit(afull(1));
        }
      }
    }
    if (bad) {
      *s_err = 1;
      // MMAs already issued keep reading shared memory and writing TMEM: wait (on this
      // warp's own limit) for the last commit, which covers all of them
      if (last >= 0) (void)mbar_wait_own(empty(last), lastph);
    }
  } else if (warp >= 4) {
    const int quarter = warp & 3, colq = (warp - 4) >> 2;
    const int m = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    long long* const cta_acc = a.acc + (size_t)blockIdx.x * (128 * 128);
    int8_t alf;
    if (ADJ || rec) alf = a.ctl.alpha[step];  // the recorded branch of step `step`
    else if (a.mode == SQ_TAIL_FIRST) alf = (a.ctl.traces[step - 1] <= (double)a.ctl.nocc) ? (int8_t)1 : (int8_t)-1;
    else if (a.mode == SQ_TAIL_NEXT) alf = (int8_t)(-a.ctl.alpha[step - 1]);
    else alf = a.ctl.alpha[step];
    // the adjoint's Xbar ping-pong: in = buffer (n - step) & 1, out = the other
    const bool flip = ADJ && ((n - step) & 1);
    auto xin = [&]() { return flip ? (const double*)a.xout : a.xin; };
    auto xq = [&]() { return reinterpret_cast<long long*>(flip ? const_cast<double*>(a.xin) : a.xout); };
    // the sums are formed with the sign the step needs: X_new = 2X + z, z = -Y, or z = Y alone
    const int sgn = alf > 0 ? -1 : 1;
    // the digit arenas of a set lie one arena apart
    const size_t dstr = ADJ ? 0 : (size_t)(a.digits[dbo].s[1] - a.digits[dbo].s[0]);
    int v = 0, rd = 0;  // items taken, rounds of both passes drained
    for (;; ++v) {
      const int iq = v % OZ_RING;
      const bool got = __all_sync(0xffffffffu, mbar_wait(item_full(iq), (v / OZ_RING) & 1, abort_flag));
      if (!got) {
        *s_err = 1;
        break;
      }
      // the item's fields (warp-uniform); wide: read again after the drains, which need the registers
      OzItem t;
      auto fields = [&]() {
        const volatile OzItem& w = s_items[iq];
        t.ti = __shfl_sync(0xffffffffu, w.ti, 0);
        t.tj = __shfl_sync(0xffffffffu, w.tj, 0);
        t.slot = __shfl_sync(0xffffffffu, w.slot, 0);
        t.part = __shfl_sync(0xffffffffu, w.part, 0);
        t.s = __shfl_sync(0xffffffffu, w.s, 0);
        t.c = __shfl_sync(0xffffffffu, w.c, 0);
        t.ld = __shfl_sync(0xffffffffu, w.ld, 0);
        t.off = __shfl_sync(0xffffffffu, w.off, 0);
        t.soff = __shfl_sync(0xffffffffu, w.soff, 0);
        t.piece = __shfl_sync(0xffffffffu, w.piece, 0);
      };
      auto done = [&]() {  // with the item
        __syncwarp();
        if (lane == 0) mbar_arrive(item_empty(iq));
      };
      t.code = __shfl_sync(0xffffffffu, s_items[iq].code, 0);
      const bool brief = __shfl_sync(0xffffffffu, s_items[iq].brief, 0) != 0;
      int rounds = __shfl_sync(0xffffffffu, s_items[iq].rounds, 0);
      fields();
      if (!WIDE || t.code < 0) done();
      if (t.code == OZ_PAUSE && decision()) continue;
      if (t.code < 0) break;
      const int code = t.code;
      const int ti = split ? code >> 1 : code;
      // a split item's 64-bit partial goes to its own tile of split_acc, which the item that
      // finishes the tile reads; otherwise the sums wait in this CTA's scratch tile
      long long* const acc = split ? a.split_acc + (size_t)code * (128 * 128) : cta_acc;
      const OzItem& p = t;
      // columns the MMAs covered; the 16-column chunks beyond them lie in the part's zero
      // padding, which no step writes (the arenas are zeroed when the workspace is bound)
      const int ncols = piece_cols(p.s, t.tj, t.piece);
      if (ncols == 0) {  // a piece in the padding
        if (!ADJ && !rec && t.slot >= 0 && warp == 4 && lane == 0)
          a.slots[t.slot * pieces + t.piece] = make_double2(0.0, 0.0);
        if (WIDE) done();
        continue;
      }
      // a diagonal tile keeps its upper triangle and mirrors it: a chunk wholly left of the
      // warp's first row (all its entries below the diagonal) is neither drained nor formed
      const int cskip = (t.ti == t.tj) ? quarter * 32 : 0;
      bool ok = true;
      // A sum has reached 2^24: the last block of the launch is to form the part again.  (Kept to the end of an item in
      // the wide form, whose registers that suits: marked as in the narrow one it spills 370 bytes and takes 3 %
      // longer; the narrow one, marking at the end, takes 0.7 % longer at n = 512.)
      float top = 0.0f;
      auto mark_part = [&](int part) {  // (a brief item reaches 2^24 only if X has left [0, 1]; it is not formed again)
        a.coh_new[part] = 1;
        atomicOr(&s_walk, 1);  // (brief items come after the decision)
      };
      auto mark = [&](float m) {
        if (WIDE) top = fmaxf(top, m);
        else mark_part(t.part);
      };
      // the warp's chunks of 16 columns (pc0: its first column in the piece)
      const int nch = 2 / pieces, pc0 = colq * 16 * nch, tc0 = t.piece * pcols + pc0;
      const bool on0 = pc0 < ncols && tc0 + 16 > cskip;
      const bool on1 = nch == 2 && pc0 + 16 < ncols && tc0 + 32 > cskip;
      // the previous iterate's lines of this warp (not written by this launch; read from HBM) come
      // to L2 while the MMAs run: lane l, column l of the warp's 32, two lines of 128 B
      if (alf > 0 && (on0 || on1)) {
        const int c = t.tj * 128 + tc0 + lane;
        if (lane < 16 * nch && c < p.s) {
          const double* x = xin() + p.off + (int64_t)c * p.ld + t.ti * 128 + quarter * 32;
          asm volatile("prefetch.global.L2 [%0];\n prefetch.global.L2 [%0 + 128];\n" ::"l"(x));
        }
      }
      // the two passes of every round: read the accumulators' sums (integers at their scales,
      // held exactly in FP32, but for the sixth) and add them as 64-bit integers; each pass hands its
      // columns back
      long long z[16];
      if constexpr (WIDE) {
        // Both chunks' sums stay in registers.  The tensor pipe stands still from a pass's last product
        // until the columns the next pass starts in have been read by every warp, so nothing but that
        // comes first: of the first pass columns 0-255 of both chunks, then the rest while the second
        // pass runs.
        long long z1[16];
        const uint32_t tc = tmem + lane_off + (uint32_t)pc0;
        auto hand_back = [&](int pass) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(aempty(pass));
        };
#pragma unroll
        for (int j = 0; j < 16; ++j) z[j] = z1[j] = 0ll;
        for (; rounds > 0; --rounds, ++rd) {
          const long long less = (long long)(sgn < 0 ? kOzOffset : 0ull - kOzOffset);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            z[j] += less;
            z1[j] += less;
          }
          ok = __all_sync(0xffffffffu, mbar_wait(afull(0), rd & 1, abort_flag)) && ok;
          tc_fence_after();
          if (ok && on0) oz_drain_high_a<WIDE>(tc, sgn, mark, z);
          if (ok && on1) oz_drain_high_a<WIDE>(tc + 16, sgn, mark, z1);
          hand_back(0);
          if (ok && on0) oz_drain_high_b<WIDE>(tc, sgn, mark, z);
          if (ok && on1) oz_drain_high_b<WIDE>(tc + 16, sgn, mark, z1);
          ok = __all_sync(0xffffffffu, mbar_wait(afull(1), rd & 1, abort_flag)) && ok;
          tc_fence_after();
          if (ok && on0) oz_drain_low<WIDE>(tc, sgn, mark, z);
          if (ok && on1) oz_drain_low<WIDE>(tc + 16, sgn, mark, z1);
          hand_back(1);
        }
        // the sums leave the registers for a scratch tile (thread-private entries: column cl, row m):
        // both chunks' of a split item, else the one the final pass takes second
        auto put = [&](int cl, const long long (&v)[16]) {
          long long* zp = acc + (size_t)cl * 128 + m;
#pragma unroll
          for (int j = 0; j < 16; ++j) zp[(size_t)j * 128] = v[j];
        };
        if (on0 && (split || on1)) put(tc0, z);
        if (on1) {
          if (split) put(tc0 + 16, z1);
#pragma unroll
          for (int j = 0; j < 16; ++j) z[j] = z1[j];
        }
      } else {
        const int clast = on1 ? 1 : (on0 ? 0 : -1), cfirst = on1 && on0 ? 0 : -1;
        // one chunk's sums at a time, parked in TMEM between the passes and then in the scratch tile
        // (thread-private entries: column cl, row m) or, the last one's, in registers
        const int all = rounds;
        for (int pass = 0; rounds > 0; pass ^= 1) {
          ok = __all_sync(0xffffffffu, mbar_wait(afull(pass), rd & 1, abort_flag)) && ok;
          tc_fence_after();
          // the first pass hands its columns back as soon as the warp's last chunk has read
          // columns 0-255, which the second reuses
          bool released = false;
#pragma unroll 1
          for (int cc = 0; cc < 2 && ok; ++cc) {
            if (cc != clast && cc != cfirst) continue;
            const int cl = tc0 + cc * 16;  // in the tile
            const uint32_t tc = tmem + lane_off + (uint32_t)(pc0 + cc * 16);
            uint32_t w[16];
            if (pass == 0) {
              // the first pass's sum waits in the columns this warp has just drained (its own
              // columns among 256-511), which the second pass leaves alone
#pragma unroll
              for (int j = 0; j < 16; ++j) z[j] = (long long)(sgn < 0 ? kOzOffset : 0ull - kOzOffset);
              oz_drain_high_a<WIDE>(tc, sgn, mark, z);
              if (cc == clast) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(aempty(0));
                released = true;
              }
              oz_drain_high_b<WIDE>(tc, sgn, mark, z);
#pragma unroll
              for (int j = 0; j < 16; ++j) w[j] = (uint32_t)(unsigned long long)z[j];
              tmem_st16(tc + OZ_PARK_LO, w);
#pragma unroll
              for (int j = 0; j < 16; ++j) w[j] = (uint32_t)((unsigned long long)z[j] >> 32);
              tmem_st16(tc + OZ_PARK_HI, w);
            } else {
              tmem_ld16(tc + OZ_PARK_LO, w);
#pragma unroll
              for (int j = 0; j < 16; ++j) z[j] = (long long)(unsigned long long)w[j];
              tmem_ld16(tc + OZ_PARK_HI, w);
#pragma unroll
              for (int j = 0; j < 16; ++j) z[j] += (long long)((unsigned long long)w[j] << 32);
              oz_drain_low<WIDE>(tc, sgn, mark, z);
              if (cc == clast) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(aempty(1));
                released = true;
              }
              long long* zp = acc + (size_t)cl * 128 + m;
              if (rounds < all) {  // the rounds before
#pragma unroll
                for (int j = 0; j < 16; ++j) z[j] += zp[(size_t)j * 128];
              }
              if (split || cc != clast || rounds > 1) {
#pragma unroll
                for (int j = 0; j < 16; ++j) zp[(size_t)j * 128] = z[j];
              }
            }
          }
          if (pass == 0) tmem_wait_st();
          if (!released) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(aempty(pass));
          }
          if (pass == 1) {
            --rounds;
            ++rd;
          }
        }
      }
      if (!ok) *s_err = 1;
      if constexpr (WIDE)
        if (__any_sync(0xffffffffu, top >= 1.0f) && lane == 0 && !rec && *(volatile int*)&s_items[iq].brief == 0)
          mark_part(*(volatile int*)&s_items[iq].part);
      // split K: the first half to finish leaves its partial; the second adds the first's
      // (64-bit integers: exact, so which one finishes first does not matter) and forms the tile
      const long long* other = nullptr;
      if (split) {
        __threadfence();
        asm volatile("bar.sync 1, %0;\n" ::"n"(32 * OZ_EPI_WARPS) : "memory");
        if (warp == 4 && lane == 0) {
          unsigned int* const cnt = &a.split_cnt[ti * pieces + t.piece];
          const unsigned int before = atomicAdd(cnt, 1u);
          if (before == 1u) *cnt = 0u;  // both halves in: clear for the next launch
          *s_half = (int)before;
        }
        asm volatile("bar.sync 1, %0;\n" ::"n"(32 * OZ_EPI_WARPS) : "memory");
        if (*s_half == 0) {
          if (WIDE) done();
          continue;
        }
        __threadfence();
        other = a.split_acc + (size_t)(code ^ 1) * (128 * 128);
      }
      // final pass of the tile: X_new on the 2^-56 grid, fixed-point master, digits, traces (the
      // adjoint: Xbar_new, FP64 only); column writes are coalesced across the warp.  Only
      // tiles on or above the diagonal are kept (the next step reads the rest MN-major from
      // them); a diagonal tile mirrors its upper triangle, transposed among the lanes so that the
      // mirrored columns are written 128 B (master) and 32 B (each digit) at a time
      if (WIDE) {
        fields();
        done();
      }
      const int64_t ld = p.ld;
      const int r = t.ti * 128 + m;
      const bool diag = t.slot >= 0;
      const int sg = ADJ ? a.sig[t.part] : 0;  // the adjoint's sums hold (Xbar X + X Xbar) / 2^sg
      long long yd = 0ll, xd = 0ll;  // diagonal entry (r, r) of sgn Y and X_new
      float rown = 0.0f;             // adjoint: squared norm of row r over this thread's upper entries
      auto stored = [&](long long xf) {  // adjoint: the FP64 word stored
        return sg == OZ_SIG_NONFINITE ? 0x7FF8000000000000ll : __double_as_longlong(from_fixed(xf, sg));
      };
      const bool dgt = t.ti == t.tj;
      if constexpr (WIDE) {
        // A tile is formed once, so straight-line code for all 16 columns of a chunk would be fetched
        // from L2 as often as it runs (a diagonal tile took 42,000 cycles, most of them waiting
        // for instructions): the columns are stored four at a time in a loop, z turning in registers, and
        // a diagonal tile's mirrored entries go through the same loop a second time.
        auto chunk = [&](int cl) {
          const int cbase = t.tj * 128 + cl;
          // element (row r, column cbase)
          int64_t e = p.off + (int64_t)cbase * ld + r;
          constexpr int B = ADJ ? 8 : 16;  // columns read together
#pragma unroll
          for (int h = 0; h < 16; h += B) {
            long long xn[B];  // the forward iterates are kept in the fixed point itself; the adjoint's Xbar in FP64
#pragma unroll
            for (int j = 0; j < B; ++j)
              xn[j] = alf > 0 ? reinterpret_cast<const long long*>(xin())[e + (int64_t)(h + j) * ld] : 0ll;
#pragma unroll
            for (int j = 0; j < B; ++j) {
              const long long xf = 2 * (ADJ ? to_fixed(__longlong_as_double(xn[j]), sg) : xn[j]) + z[h + j];
              if (!ADJ && dgt && cbase + h + j == r) {  // the thread's one diagonal entry, if it has it
                yd = z[h + j];
                xd = xf;
              }
              z[h + j] = xf;
            }
          }
          if constexpr (ADJ) {
            // every stored entry (r, c) adds to the norm of row r, and of row c unless c = r
            float coln[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int c = cbase + j;
              const float f = (!dgt || c >= r) && r < p.s && c < p.s ? fixed_to_f32_abs(z[j]) : 0.0f;
              rown = fmaf(f, f, rown);
              coln[j] = c != r ? f * f : 0.0f;
            }
            int col;
            const float cs = warp_colsum16(coln, lane, col);
            if (!(lane & 1) && cbase + col < p.s && cs != 0.0f) atomicAdd(&a.normf[p.soff + cbase + col], cs);
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = stored(z[j]);
          }
          // first the thread's own entries: row r, columns cbase + j, those on or above the diagonal.  Then,
          // of a diagonal tile, z transposed: lane l has column c = cbase + l % 16 of rows rb + j, which
          // go to row c of columns rb + j, those below it.  Entry j is stored if at + dir j >= 0.
          int at = dgt ? cbase - r : 128, dir = 1;
#pragma unroll 1
          for (int b = 0;; ++b, e += 4 * ld, at += 4 * dir) {
            if (b == 4) {
              if (!dgt) break;
              transpose16(z, lane);
              const int rb = t.ti * 128 + quarter * 32 + (lane & 16), c = cbase + (lane & 15);
              e = p.off + (int64_t)rb * ld + c;
              at = c - rb - 1;
              dir = -1;
            }
            if (b == 8) break;
#pragma unroll
            for (int j = 0; j < 4; ++j) store_word_if(at + dir * j >= 0, xq() + e + (int64_t)j * ld, z[j]);
            if (!ADJ) {
              uint32_t dw[OZ_SLICES][2];  // four entries' digits, two packed per word
              digits4({z[0], z[1], z[2], z[3]}, dw);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                store_digits_if(at + dir * j >= 0, a.digits[dbo].s[0] + e + (int64_t)j * ld, dstr, dw, j);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const long long w = z[j];
              z[j] = z[4 + j];
              z[4 + j] = z[8 + j];
              z[8 + j] = z[12 + j];
              z[12 + j] = w;
            }
          }
        };
#pragma unroll 1
        for (int cc = 1; cc >= 0 && ok; --cc) {
          if (!(cc ? on1 : on0)) continue;
          const int cl = tc0 + cc * 16;
          if (cc == 0 && on1) {
            const long long* zp = acc + (size_t)cl * 128 + m;
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = zp[(size_t)j * 128];
          }
          if (other) {
            const long long* zo = other + (size_t)cl * 128 + m;
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] += __ldcg(zo + (size_t)j * 128);
          }
          chunk(cl);
        }
      } else {
        // the columns are taken eight at a time in loops, the mirrored entries in one of their own: where
        // a CTA has one or two items, the wide form's loop takes longer (n = 512 density 0.46 against
        // 0.45 ms), its columns being read before any are stored
        const double* const xi = xin();
        long long* const xo = xq();
        const int clast = on1 ? 1 : (on0 ? 0 : -1), cfirst = on1 && on0 ? 0 : -1;
        auto chunk = [&](int cl) {
          const int cbase = t.tj * 128 + cl;
          // element (first row of the warp, column cbase), uniform; the lane's row is added to it
          int64_t e = p.off + (int64_t)cbase * ld + (t.ti * 128 + quarter * 32);
          float coln[16];  // adjoint: squares of the entries (r, c) for the norms of rows c
#pragma unroll 1
          for (int b = 0; b < 2; ++b, e += 8 * ld) {
            const int cb = cbase + 8 * b;
            long long xn[8];  // the forward iterates are kept in the fixed point itself; the adjoint's Xbar in FP64
#pragma unroll
            for (int j = 0; j < 8; ++j)
              xn[j] = alf > 0 ? reinterpret_cast<const long long*>(xi)[(e + (int64_t)j * ld) + lane] : 0ll;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int c = cb + j;
              const bool upper = !dgt || c >= r;
              const long long xf = 2 * (ADJ ? to_fixed(__longlong_as_double(xn[j]), sg) : xn[j]) + z[j];
              if (!ADJ && dgt && c == r) {  // the thread's one diagonal entry, if it has it
                yd = z[j];
                xd = xf;
              }
              if (ADJ) {
                float f = 0.0f;
                if (upper && r < p.s && c < p.s) f = fixed_to_f32_abs(xf);
                // every stored entry (r, c) adds to the norm of row r, and of row c unless c = r
                rown = fmaf(f, f, rown);
                coln[j] = coln[8 + j];
                coln[8 + j] = c != r ? f * f : 0.0f;
              }
              xn[j] = ADJ ? stored(xf) : xf;
              store_word_if(upper, xo + (e + (int64_t)j * ld) + lane, xn[j]);
            }
            if (!ADJ) {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t dw[OZ_SLICES][2];  // four columns' digits, two packed per word
                digits4({xn[4 * h], xn[4 * h + 1], xn[4 * h + 2], xn[4 * h + 3]}, dw);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                  uint16_t* d = a.digits[dbo].s[0] + (e + (int64_t)(4 * h + w) * ld) + lane;
                  store_digits_if(!dgt || cb + 4 * h + w >= r, d, dstr, dw, w);
                }
              }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              z[j] = z[8 + j];
              z[8 + j] = xn[j];
            }
          }
          if (dgt) {
            // the mirrored entries: lane l has column cbase + l % 16 of rows rb + j, which go to row
            // cbase + l % 16 of columns rb + j
            transpose16(z, lane);
            int rb = t.ti * 128 + quarter * 32 + (lane & 16);
            const int c = cbase + (lane & 15);
            int64_t em = p.off + (int64_t)rb * ld + c;
#pragma unroll 1
            for (int b = 0; b < 4; ++b, rb += 4, em += 4 * ld) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                store_word_if(c > rb + j, xo + em + (int64_t)j * ld, z[j]);
              if (!ADJ) {
                uint32_t dw[OZ_SLICES][2];
                digits4({z[0], z[1], z[2], z[3]}, dw);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                  store_digits_if(c > rb + w, a.digits[dbo].s[0] + em + (int64_t)w * ld, dstr, dw, w);
                }
              }
#pragma unroll
              for (int j = 0; j < 12; ++j) z[j] = z[j + 4];
            }
          }
          if constexpr (ADJ) {
            int col;
            const float cs = warp_colsum16(coln, lane, col);
            if (!(lane & 1) && cbase + col < p.s && cs != 0.0f) atomicAdd(&a.normf[p.soff + cbase + col], cs);
          }
        };
#pragma unroll 1
        for (int pc = 0; pc < 2 && ok; ++pc) {
          const int cc = pc == 0 ? clast : cfirst;
          if (cc < 0) continue;
          const int cl = tc0 + cc * 16;
          if (pc == 1) {
            const long long* zp = acc + (size_t)cl * 128 + m;
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = zp[(size_t)j * 128];
          }
          if (other) {
            const long long* zo = other + (size_t)cl * 128 + m;
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] += __ldcg(zo + (size_t)j * 128);
          }
          chunk(cl);
        }
      }
      if (ADJ && ok && r < p.s && rown != 0.0f) atomicAdd(&a.normf[p.soff + r], rown);
      if (!ADJ && !rec && diag) {
        // the thread that has a diagonal entry leaves it (sgn Y, X_new) in shared memory; one warp
        // converts and adds them.  A reduction in every warp would be 160 FP64 instructions, 16
        // cycles each.
        if (m >= tc0 && m < tc0 + 16 * nch) red[m] = make_longlong2(yd, xd);
        asm volatile("bar.sync 1, %0;\n" ::"n"(32 * OZ_EPI_WARPS) : "memory");
        if (warp == 4) {
          double2 sum = make_double2(0.0, 0.0);
          for (int q = t.piece * pcols + lane; q < min(p.c - t.ti * 128, (t.piece + 1) * pcols); q += 32) {
            const longlong2 e = red[q];
            sum.x += from_fixed(sgn < 0 ? -e.x : e.x);
            sum.y += from_fixed(e.y);
          }
          sum.x = warp_sum(sum.x);
          sum.y = warp_sum(sum.y);
          if (lane == 0) a.slots[t.slot * pieces + t.piece] = sum;
        }
        asm volatile("bar.sync 1, %0;\n" ::"n"(32 * OZ_EPI_WARPS) : "memory");
      }
    }
  }
  if (warp == 3) {
    if (!rec) {
      pause();
      asm volatile("bar.sync 3, 64;\n" ::: "memory");  // warp 0's word
      if (*(volatile int*)&s_walk & 16) {
        if (lane == 0) {
          const uint64_t until = global_ns() + 2000000ull;  // no longer than two items take
          bool ready;
          while (!(ready = *(volatile int32_t*)&a.again->go == place) && *(volatile int32_t*)abort_flag == 0 &&
                 global_ns() < until)
            __nanosleep(500);
          __threadfence();
          *(volatile int*)&s_walk = ready ? 12 : 8;
        }
        __syncwarp();
      }
      asm volatile("bar.arrive 2, %0;\n" ::"n"(OZ_THREADS) : "memory");
    }
  } else if (!paused()) {
    (void)decision();
  }
  int walk = *(volatile int*)&s_walk;
  if (rec || walk & 4) {  // else the pause was the end
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (walk & 4) {  // the block whose items are the last to be done ends the launch
      if (threadIdx.x == 0) {
        __threadfence();
        const int taken = s_taken;
        s_walk = taken > 0 && atomicAdd(&a.again->done, taken) + taken == nitems ? 14 : 12;
        __threadfence();
      }
      __syncthreads();
      walk = s_walk;
    }
  }
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
  if (threadIdx.x == 0 && *s_err) {
    a.ctl.st->timeout = 1;
    if (ADJ || rec || walk & 4) a.ctl.st->status = ST_TIMEOUT;  // no step bookkeeping follows
    if (walk & 4) {
      a.ctl.st->stopped = 1;
      a.ctl.st->counter = 0;
      if (dyn) *a.tile_ctr = 0u;
    }
  }
  if (rec || !(walk & 2)) return;
  if (walk & 4 && warp == 3) {
    for (int k = lane; k < a.nparts; k += 32)
      if (a.coh_new[k]) {
        a.coh[k] = min(a.coh[k], place);
        a.coh_new[k] = 0;
      }
    if (!ADJ && lane == 0) a.ctl.st->coherent = 1;
  }
  if (ADJ) {
    __threadfence();
    // the last block: each part's new scale from the largest squared row norm m (on the grid
    // of the old scale sg): the smallest e with 2^e >= 2 sqrt(m) (1 + 2^-10), the margin
    // covering the truncated squares and the FP32 sums; the norms are cleared for the next step
    {
      for (int k = warp; k < a.nparts; k += OZ_THREADS / 32) {
        const PartDesc p = a.parts[k];
        float mx = 0.0f;
        // loads in flight together, eight per lane
        for (int r0 = lane; r0 < p.s; r0 += 32 * 8) {
          float v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = r0 + 32 * q < p.s ? __ldcg(a.normf + p.soff + r0 + 32 * q) : 0.0f;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            mx = fmaxf(mx, v[q]);
            if (r0 + 32 * q < p.s) a.normf[p.soff + r0 + 32 * q] = 0.0f;
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) {
          const int sg = a.sig[k];
          int e = 0;
          if (sg != OZ_SIG_NONFINITE && mx > 0.0f) {
            (void)frexpf(2.0f * sqrtf(mx) * (1.0f + 0.0009765625f), &e);
            a.sig[k] = sg + e;
          }
        }
      }
      if (threadIdx.x == 0) {
        a.ctl.st->counter = 0;
        if (dyn) *a.tile_ctr = 0u;  // every CTA has claimed its last item
      }
    }
    return;
  }

  if (warp == 0) {
    const double2 sum = warp_sum_slots(a.slots, a.nslots * pieces);
    if (threadIdx.x == 0) {
      if (a.ctl.st->timeout) {
        a.ctl.st->status = ST_TIMEOUT;
        a.ctl.st->stopped = 1;
      } else if (a.mode == SQ_FORWARD) {
        finish_step(a.ctl, step, sum.y, sum.x);
      } else {
        int8_t alf;
        if (a.mode == SQ_TAIL_FIRST) alf = (a.ctl.traces[step - 1] <= (double)a.ctl.nocc) ? (int8_t)1 : (int8_t)-1;
        else alf = (int8_t)(-a.ctl.alpha[step - 1]);
        a.ctl.alpha[step] = alf;
        finish_tail(a.ctl, step, sum.y, sum.x, true);
      }
      a.ctl.st->counter = 0;
      if (dyn) *a.tile_ctr = 0u;  // every CTA has claimed its last tile: ready for the next launch
    }
  }
}

cudaError_t launch_oz_convert_slice(const PartDesc* parts, const ColBlock* blocks, int nblocks,
                                    const float* const* master_of_step, double* X, const OzSlices* digits,
                                    const DevState* st, cudaStream_t s) {
  oz_convert_slice_kernel<<<nblocks, 256, 0, s>>>(parts, blocks, master_of_step, X, digits[0], digits[1], st);
  return cudaGetLastError();
}

cudaError_t launch_oz_step(const OzStepArgs& a, int grid, cudaStream_t s, bool adjoint) {
  auto kern = a.wide ? (adjoint ? oz_step_kernel<true, true> : oz_step_kernel<false, true>)
                     : (adjoint ? oz_step_kernel<true, false> : oz_step_kernel<false, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
  if (e != cudaSuccess) return e;
  const int nitems = (a.split ? 2 * a.ntiles : a.ntiles) * a.pieces;
  int gr = grid < nitems ? grid : nitems;
  if (gr > OZ_MAX_GRID) gr = OZ_MAX_GRID;  // one scratch tile per CTA
  return launch_pdl(kern, gr, OZ_THREADS, OZ_SMEM, s, a);
}

cudaError_t launch_oz_gather(const PartDesc* parts, const ColBlock* blocks, int nblocks, const int32_t* Sall,
                             const int64_t* rowptr, const int32_t* loc, const int64_t* locptr, const double* x0,
                             double* arena, const OzSlices& dig, double* slots, const StepCtl& ctl, cudaStream_t s) {
  return launch_pdl(oz_gather_kernel, nblocks, 32 * COLS_PER_BLOCK, 0, s, parts, blocks, Sall, rowptr, loc, locptr, x0,
                    arena, dig, slots, ctl);
}

cudaError_t launch_oz_adj_scale(const PartDesc* parts, int nparts, const Tile* tiles, int ntiles, const double* xb0,
                                const double* xb1, int after, double* norm, int32_t* sig, int32_t* coh,
                                const DevState* st, cudaStream_t s) {
  if (ntiles > 0) oz_norm_kernel<<<ntiles, 256, 0, s>>>(parts, tiles, xb0, xb1, after, norm, st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  oz_scale_kernel<<<nparts, 256, 0, s>>>(parts, after, norm, sig, coh, st);
  return cudaGetLastError();
}

cudaError_t launch_oz_digits(const PartDesc* parts, const ColBlock* blocks, int nblocks, const double* x0,
                             const double* x1, int after, int need, const OzSlices& out, const int32_t* sig,
                             const DevState* st, cudaStream_t s) {
  oz_digits_kernel<<<nblocks, 32 * COLS_PER_BLOCK, 0, s>>>(parts, blocks, x0, x1, after, need, out, sig, st);
  return cudaGetLastError();
}

}  // namespace gsp2
