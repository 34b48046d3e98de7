// CSR sparse kernels: the Newton-step SpMV of the matrix powers kernel
// (Sec. 2, Eq. newtonrecurrence), the residual, the sampled outer product
// of the adjoint gradient and the CSR transpose.
//
// SpMV layout: one thread per row.  One thread per row matters on this
// chip: FP64 warp instructions are expensive (the FP64 pipe is ~1/64 of the
// FP32 rate), so the per-row reduction must not spend shuffles and adds on
// idle lanes; the epilogue multiplies by 1/gamma instead of dividing.
//
// Preferred storage is SELL-32, built at ingest: rows are cut into slices
// of 32 (one warp), and slice q stores entry j of its row l at
// sptr[q] + 32 j + l, padded to the slice's longest row with column -1.
// Lane l of a warp then walks row 32q + l while the warp reads each entry
// index j as one coalesced 256-byte (values) and 128-byte (indices) line,
// with no staging and no barriers; x is gathered through L1 (stencil
// locality gives cache hits).  Up to eight entries per row
// are loaded before the FMAs, so their gathers are in flight together, and
// the chunks follow the slice width exactly (no predicated-off FP64 work).
//
// Rows of uneven length (the transpose of a random pattern, say) would pad
// every slice to its longest row; then the rows are sorted by length within
// windows of 1024 rows first, and a lane's row is looked up (sperm).  The
// entries of a row and their order stay, so the products are the same bits.
// On the transpose of the random band (1M rows, 25 +- 5 entries) the padding
// falls to a few percent and the FP32 product takes 46 us, CSR 108 us.
//
// When the padding would still be large, CSR is used as is: a CTA owns a
// contiguous block of rows and first stages that block's values and
// column indices in shared memory with coalesced streaming loads, then
// each thread walks its own row from shared memory.
#include <cstring>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "k_reduce.cuh"
#include "k_launch.cuh"
#include "sg_internal.h"

namespace sg {

namespace {

constexpr int kThreads = 256;
constexpr int kStage = 2048;   // staged nonzeros per CTA

__device__ __forceinline__ double ld_stream(const double* p) { return __ldcs(p); }
__device__ __forceinline__ float ld_stream(const float* p) { return __ldcs(p); }
__device__ __forceinline__ int ld_stream(const int* p) { return __ldcs(p); }

// MODE 0: y = (A x - theta x + c z) * inv_gamma   (HAS_Z: c z present)
// MODE 1: y = z - A x                              (residual, z = b)
template <int MODE, bool HAS_Z, typename T>
__global__ void __launch_bounds__(kThreads)
spmv_kernel(int n, int rows_per_cta, const int* __restrict__ rowptr,
            const int* __restrict__ colind, const T* __restrict__ val,
            const T* __restrict__ x, const T* __restrict__ z,
            T* __restrict__ y, T theta, T c, T inv_gamma) {
  __shared__ T sval[kStage];
  __shared__ int scol[kStage];
  const int t = threadIdx.x;
  for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * rows_per_cta; r0 < n;
       r0 += static_cast<int64_t>(gridDim.x) * rows_per_cta) {
    const int64_t r1 = (r0 + rows_per_cta < n) ? r0 + rows_per_cta : n;
    const int k0 = rowptr[r0];
    const int len = rowptr[r1] - k0;
    const bool staged = len <= kStage;
    if (staged) {
      for (int e = t; e < len; e += kThreads) {
        sval[e] = ld_stream(val + k0 + e);
        scol[e] = ld_stream(colind + k0 + e);
      }
    }
    __syncthreads();
    for (int64_t row = r0 + t; row < r1; row += kThreads) {
      const int a = rowptr[row], b = rowptr[row + 1];
      T sum = T(0);
      if (staged) {
        for (int k = a - k0; k < b - k0; ++k) sum = fma(sval[k], __ldg(x + scol[k]), sum);
      } else {
        for (int k = a; k < b; ++k) sum = fma(ld_stream(val + k), __ldg(x + ld_stream(colind + k)), sum);
      }
      if (MODE == 1) {
        y[row] = z[row] - sum;
      } else {
        T v = fma(-theta, x[row], sum);
        if (HAS_Z) v = fma(c, z[row], v);
        y[row] = v * inv_gamma;
      }
    }
    __syncthreads();
  }
}

// U consecutive entries (j .. j+U-1) of a SELL-32 row starting at k: the
// indices and values are loaded first, then the gathers, then the FMAs, so
// all of the chunk's loads are in flight together.  Padding (column -1)
// is skipped per lane.
template <int U, typename T>
__device__ __forceinline__ void sell_chunk(const int* __restrict__ scol,
                                           const T* __restrict__ sval, const T* x, int k,
                                           T& sum) {
  int c[U];
  T v[U], xv[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    c[u] = ld_stream(scol + k + 32 * u);
    v[u] = ld_stream(sval + k + 32 * u);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) xv[u] = c[u] >= 0 ? x[c[u]] : T(0);
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (c[u] >= 0) sum = fma(v[u], xv[u], sum);
}

// Sum over the SELL-32 row `row` (entries in column order, padding
// skipped), the same FMA sequence as the CSR walk of that row.  The slice
// width is the same for the whole warp, so the chunking below is uniform
// and issues exactly one FMA instruction per stored entry index.
template <typename T>
__device__ __forceinline__ T sell_row(const int* __restrict__ sptr,
                                      const int* __restrict__ scol,
                                      const T* __restrict__ sval, const T* x, int64_t row) {
  const int64_t q = row >> 5;
  const int a = sptr[q], e = sptr[q + 1];
  const int w = (e - a) >> 5;
  int k = a + static_cast<int>(row & 31);
  T sum = T(0);
  int j = 0;
  for (; j + 8 <= w; j += 8, k += 256) sell_chunk<8>(scol, sval, x, k, sum);
  switch (w - j) {
    case 7: sell_chunk<7>(scol, sval, x, k, sum); break;
    case 6: sell_chunk<6>(scol, sval, x, k, sum); break;
    case 5: sell_chunk<5>(scol, sval, x, k, sum); break;
    case 4: sell_chunk<4>(scol, sval, x, k, sum); break;
    case 3: sell_chunk<3>(scol, sval, x, k, sum); break;
    case 2: sell_chunk<2>(scol, sval, x, k, sum); break;
    case 1: sell_chunk<1>(scol, sval, x, k, sum); break;
    default: break;
  }
  return sum;
}

// The same chunk with the columns as 16-bit offsets from the slice's base
// (0xFFFF: padding).
template <int U, typename T>
__device__ __forceinline__ void sell_chunk16(int base, const uint16_t* __restrict__ soff,
                                             const T* __restrict__ sval, const T* x, int k,
                                             T& sum) {
  unsigned o[U];
  T v[U], xv[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    o[u] = __ldcs(soff + k + 32 * u);
    v[u] = ld_stream(sval + k + 32 * u);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) xv[u] = o[u] != 0xFFFFu ? x[base + static_cast<int>(o[u])] : T(0);
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (o[u] != 0xFFFFu) sum = fma(v[u], xv[u], sum);
}

template <typename T>
__device__ __forceinline__ T sell_row16(const int* __restrict__ sptr, const int* __restrict__ sbase,
                                        const uint16_t* __restrict__ soff,
                                        const T* __restrict__ sval, const T* x, int64_t row) {
  const int64_t q = row >> 5;
  const int a = sptr[q], e = sptr[q + 1];
  const int w = (e - a) >> 5;
  const int base = sbase[q];
  int k = a + static_cast<int>(row & 31);
  T sum = T(0);
  int j = 0;
  for (; j + 8 <= w; j += 8, k += 256) sell_chunk16<8>(base, soff, sval, x, k, sum);
  switch (w - j) {
    case 7: sell_chunk16<7>(base, soff, sval, x, k, sum); break;
    case 6: sell_chunk16<6>(base, soff, sval, x, k, sum); break;
    case 5: sell_chunk16<5>(base, soff, sval, x, k, sum); break;
    case 4: sell_chunk16<4>(base, soff, sval, x, k, sum); break;
    case 3: sell_chunk16<3>(base, soff, sval, x, k, sum); break;
    case 2: sell_chunk16<2>(base, soff, sval, x, k, sum); break;
    case 1: sell_chunk16<1>(base, soff, sval, x, k, sum); break;
    default: break;
  }
  return sum;
}

// OFF16: columns from (sbase, soff) instead of scol.  PERM: row pos of the
// slices is the matrix's row sperm[pos] (negative: none).
template <int MODE, bool HAS_Z, bool OFF16, bool PERM, typename T>
__global__ void __launch_bounds__(kThreads)
sell_kernel(int n, int64_t rows32, const int* __restrict__ sptr,
            const int* __restrict__ scol, const int* __restrict__ sbase,
            const uint16_t* __restrict__ soff, const int* __restrict__ sperm,
            const T* sval, const T* x, const T* z, T* __restrict__ y, T theta, T c, T inv_gamma) {
  sval += wait_previous();
  release_next();
  for (int64_t pos = blockIdx.x * static_cast<int64_t>(kThreads) + threadIdx.x; pos < rows32;
       pos += static_cast<int64_t>(gridDim.x) * kThreads) {
    const int64_t row = PERM ? static_cast<int64_t>(__ldg(sperm + pos)) : pos;
    const T sum = OFF16 ? sell_row16(sptr, sbase, soff, sval, x, pos)
                        : sell_row(sptr, scol, sval, x, pos);
    if (PERM ? row >= 0 : row < n) {
      if (MODE == 1) {
        y[row] = z[row] - sum;
      } else {
        T v = fma(-theta, x[row], sum);
        if (HAS_Z) v = fma(c, z[row], v);
        y[row] = v * inv_gamma;
      }
    }
  }
}

int rows_per_cta(const DevCsr& A) {
  // as many rows as keep the CTA's nonzeros within the staging buffer,
  // with 25% slack for row-length variation; at most one row per thread
  const double per = A.mean_row > 0 ? A.mean_row * 1.25 : 1.0;
  int r = static_cast<int>(kStage / per);
  if (r > kThreads) r = kThreads;
  if (r < 32) r = 32;
  return r;
}

int grid_for(const DevCsr& A, int rpc) {
  int64_t blocks = (static_cast<int64_t>(A.n) + rpc - 1) / rpc;
  const int64_t cap = static_cast<int64_t>(device_sm_count()) * 16;
  if (blocks > cap) blocks = cap;
  return static_cast<int>(blocks < 1 ? 1 : blocks);
}

template <int MODE, bool HAS_Z, typename T>
void dispatch(const DevCsr& A, const T* val, const T* sval, const T* x, const T* z, T* y,
              T theta, T c, T gamma, cudaStream_t st) {
  if (A.sptr && sval) {
    const int64_t rows32 = static_cast<int64_t>(A.nslices) * 32;
    int64_t blocks = (rows32 + kThreads - 1) / kThreads;
    const int64_t cap = static_cast<int64_t>(device_sm_count()) * 64;
    if (blocks > cap) blocks = cap;
    const int g = static_cast<int>(blocks < 1 ? 1 : blocks);
    const T ig = T(1) / gamma;
    auto go = [&](auto kernel) {
      launch_early(true, kernel, g, kThreads, 0, st, A.n, rows32, A.sptr, A.scol, A.sbase, A.soff,
                   A.sperm, sval, x, z, y, theta, c, ig);
    };
    if (A.soff && A.sperm) go(sell_kernel<MODE, HAS_Z, true, true, T>);
    else if (A.soff) go(sell_kernel<MODE, HAS_Z, true, false, T>);
    else if (A.sperm) go(sell_kernel<MODE, HAS_Z, false, true, T>);
    else go(sell_kernel<MODE, HAS_Z, false, false, T>);
    SG_LAUNCH_CHECK();
    return;
  }
  const int rpc = rows_per_cta(A);
  spmv_kernel<MODE, HAS_Z, T><<<grid_for(A, rpc), kThreads, 0, st>>>(
      A.n, rpc, A.rowptr, A.colind, val, x, z, y, theta, c, T(1) / gamma);
  SG_LAUNCH_CHECK();
}

// ------------------------------------------------------------------------
// One Arnoldi step of the Ritz pre-pass (Sec. 3.4) in a single cooperative
// launch: w = A v_j with the partial sums of w.w and v_0.w fused into the
// SpMV, then the j+1 modified Gram-Schmidt phases (h_l = v_l.w from the
// previous phase's partials, w -= h_l v_l, partials of v_{l+1}.w), then
// w /= ||w||.  Phases are separated by a grid barrier on a global arrival
// counter and generation word; every block is resident (cooperative
// launch), and each wait is time-bounded: on timeout the kernel records
// an error and runs to completion with whatever it has.  bar: 64 zeroed
// words (arrival counter and generation on separate 128-byte lines).
constexpr uint64_t kBarrierNs = 2000000000ull;

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// bar[0]: arrivals; bar[32]: generation (a separate 128-byte line, so the
// pollers do not contend with the arrivals)
__device__ void grid_barrier(unsigned* bar, unsigned nblocks, int* err,
                             uint64_t limit_ns = kBarrierNs) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 32;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) == nblocks - 1) {
      bar[0] = 0;
      __threadfence();
      atomicAdd(bar + 32, 1u);
    } else if (*reinterpret_cast<volatile int*>(err) == 0) {
      // (after an earlier timeout every barrier is skipped, so a broken
      // barrier costs one time limit, not one per phase)
      const uint64_t t0 = now_ns();
      unsigned spins = 0;
      while (*gen == g) {
        __nanosleep(32);
        if ((++spins & 255u) == 0 && now_ns() - t0 > limit_ns) {
          atomicExch(err, 1);
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
}

// Grid barrier on a counter that only grows: every CTA adds one per
// barrier, and barrier number k of the launch (counting from 0) is passed
// once the counter reaches base + G (k + 1), base being the counter's value
// when the launch started (known to the host, which zeroes the counter at
// the start of a pre-pass).  No reset and no generation word: the last
// arrival releases the waiters directly, one L2 round trip sooner than
// grid_barrier.  The wait is time-bounded like grid_barrier's.
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ void grid_barrier_count(unsigned* ctr, unsigned target, int* err,
                                   uint64_t limit_ns = kBarrierNs) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    if (*reinterpret_cast<volatile int*>(err) == 0) {
      const uint64_t t0 = now_ns();
      unsigned spins = 0;
      while (static_cast<int>(ld_acquire_u32(ctr) - target) < 0) {
        if ((++spins & 255u) == 0 && now_ns() - t0 > limit_ns) {
          atomicExch(err, 1);
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
}

constexpr int kCoopThreads = 1024;  // one CTA per SM, 32 warps in flight
constexpr int kCoopStage = 8192;    // staged nonzeros per CTA tile

// SELL: the SpMV phase walks the SELL-32 arrays (rowptr = sptr, colind =
// scol, val = sval, rows_per_cta unused) instead of staging CSR tiles.
template <typename T, bool SELL>
__global__ void __launch_bounds__(kCoopThreads, 1)
arnoldi_step_kernel(int n, int rows_per_cta, const int* __restrict__ rowptr,
                    const int* __restrict__ colind, const T* __restrict__ val,
                    T* __restrict__ V, int64_t ld, int j, double* __restrict__ H,
                    int ldh, double* __restrict__ wn, double* __restrict__ red,
                    unsigned* bar, int* err, int64_t rows32) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  T* sval = reinterpret_cast<T*>(coop_smem);
  int* scol = reinterpret_cast<int*>(coop_smem + sizeof(T) * kCoopStage);
  const int G = gridDim.x;
  const int t = threadIdx.x;
  const T* vj = V + static_cast<int64_t>(j) * ld;
  const T* v0 = V;
  T* w = V + static_cast<int64_t>(j + 1) * ld;
  double* pWW = red;
  double* pA = red + G;
  double* pB = red + 2 * G;
  // phase 0: w = A v_j, partials of w.w and v_0.w
  T accw = T(0), accv = T(0);
  if (SELL) {
    for (int64_t row = blockIdx.x * static_cast<int64_t>(kCoopThreads) + t; row < rows32;
         row += static_cast<int64_t>(G) * kCoopThreads) {
      const T sum = sell_row(rowptr, colind, val, vj, row);
      if (row < n) {
        w[row] = sum;
        accw = fma(sum, sum, accw);
        accv = fma(v0[row], sum, accv);
      }
    }
  } else
  for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * rows_per_cta; r0 < n;
       r0 += static_cast<int64_t>(G) * rows_per_cta) {
    const int64_t r1 = (r0 + rows_per_cta < n) ? r0 + rows_per_cta : n;
    const int k0 = rowptr[r0];
    const int len = rowptr[r1] - k0;
    const bool staged = len <= kCoopStage;
    if (staged) {
      for (int e = t; e < len; e += kCoopThreads) {
        sval[e] = ld_stream(val + k0 + e);
        scol[e] = ld_stream(colind + k0 + e);
      }
    }
    __syncthreads();
    for (int64_t row = r0 + t; row < r1; row += kCoopThreads) {
      const int a = rowptr[row], b = rowptr[row + 1];
      T sum = T(0);
      if (staged) {
        for (int k = a - k0; k < b - k0; ++k) sum = fma(sval[k], __ldg(vj + scol[k]), sum);
      } else {
        for (int k = a; k < b; ++k) sum = fma(ld_stream(val + k), __ldg(vj + ld_stream(colind + k)), sum);
      }
      w[row] = sum;
      accw = fma(sum, sum, accw);
      accv = fma(v0[row], sum, accv);
    }
    __syncthreads();
  }
  {
    const double sw = block_sum_few_d<kCoopThreads>(static_cast<double>(accw));
    const double sv = block_sum_few_d<kCoopThreads>(static_cast<double>(accv));
    if (t == 0) { pWW[blockIdx.x] = sw; pA[blockIdx.x] = sv; }
  }
  grid_barrier(bar, G, err);
  if (blockIdx.x == 0) {
    const double ww = sum_partials_few_d<kCoopThreads>(pWW, G);
    if (t == 0) wn[j] = sqrt(ww);
  }
  // MGS phases l = 0..j (four independent element streams per thread)
  const int64_t stride = static_cast<int64_t>(G) * kCoopThreads;
  const int64_t i0 = blockIdx.x * static_cast<int64_t>(kCoopThreads) + t;
  double* pin = pA;
  double* pout = pB;
  for (int l = 0; l <= j; ++l) {
    const double h = sum_partials_few_d<kCoopThreads>(pin, G);
    if (blockIdx.x == 0 && t == 0) H[l + static_cast<int64_t>(j) * ldh] = h;
    const T ht = static_cast<T>(h);
    const T* vl = V + static_cast<int64_t>(l) * ld;
    const T* vn = (l < j) ? V + static_cast<int64_t>(l + 1) * ld : w;
    T acc = T(0);
    int64_t i = i0;
    for (; i + 3 * stride < n; i += 4 * stride) {
      T wv[4], vv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) { wv[u] = w[i + u * stride]; vv[u] = vl[i + u * stride]; }
      T nv[4];
      if (l < j) {
#pragma unroll
        for (int u = 0; u < 4; ++u) nv[u] = vn[i + u * stride];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const T wi = fma(-ht, vv[u], wv[u]);
        w[i + u * stride] = wi;
        acc = fma(l < j ? nv[u] : wi, wi, acc);
      }
    }
    for (; i < n; i += stride) {
      const T wi = fma(-ht, vl[i], w[i]);
      w[i] = wi;
      acc = fma(l < j ? vn[i] : wi, wi, acc);
    }
    const double tot = block_sum_few_d<kCoopThreads>(static_cast<double>(acc));
    if (t == 0) pout[blockIdx.x] = tot;
    grid_barrier(bar, G, err);
    double* tmp = pin; pin = pout; pout = tmp;
  }
  // normalise
  const double nrm = sqrt(sum_partials_few_d<kCoopThreads>(pin, G));
  if (blockIdx.x == 0 && t == 0) H[(j + 1) + static_cast<int64_t>(j) * ldh] = nrm;
  const double inv = 1.0 / nrm;
  for (int64_t i = i0; i < n; i += stride)
    w[i] = static_cast<T>(static_cast<double>(w[i]) * inv);
}

// The FP64 step with w resident on chip.  w = A v_j is first formed in V's
// column j+1 by the SpMV kernel (full occupancy, and the whole L1 for the
// gathers of v_j); then CTA b of this cooperative kernel loads its rows
// [b R, (b+1) R) of w into shared memory and keeps them there through the
// MGS phases to the final normalisation.  A thread always touches the same
// rows, so w needs no barrier of its own; each phase streams only v_l (just
// read as the previous phase's v_{l+1}, an L2 hit) and v_{l+1}, instead of
// reading and writing w through HBM as well.  Phase order, fused next-vector
// dot and per-CTA partials are those of arnoldi_step_kernel; only the rows a
// CTA owns differ.  It runs for the matrices that the fixed-point step below
// is not for (rows_even): whole pre-pass with its products, 60 steps at 149K
// rows 10.9 ms (fixed point 4.66), at 2.10M rows 25.2 ms (14.1), 40 steps at
// 400K rows in CSR 9.4 ms (6.5; arnoldi_step_kernel 10.6).  The FP64 pipe
// bounds it.
__global__ void __launch_bounds__(kCoopThreads, 1)
arnoldi_mgs_resident64_kernel(int n, int rows_cta, double* __restrict__ V, int64_t ld, int j,
                              double* __restrict__ H, int ldh, double* __restrict__ wn,
                              double* __restrict__ red, unsigned* ctr, unsigned base, int* err) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  double* ws = reinterpret_cast<double*>(coop_smem);
  const int G = gridDim.x;
  const int t = threadIdx.x;
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * rows_cta;
  const int64_t r1 = (r0 + rows_cta < n) ? r0 + rows_cta : n;
  const int nr = r1 > r0 ? static_cast<int>(r1 - r0) : 0;
  const double* v0 = V + r0;
  double* w = V + static_cast<int64_t>(j + 1) * ld + r0;
  double* pWW = red;
  double* pA = red + G;
  double* pB = red + 2 * G;
  // this CTA's rows of w = A v_j, partials of w.w and v_0.w
  double accw = 0.0, accv = 0.0;
  for (int i = t; i < nr; i += kCoopThreads) {
    const double wi = w[i];
    ws[i] = wi;
    accw = fma(wi, wi, accw);
    accv = fma(v0[i], wi, accv);
  }
  {
    const double sw = block_sum_few_d<kCoopThreads>(accw);
    const double sv = block_sum_few_d<kCoopThreads>(accv);
    if (t == 0) { pWW[blockIdx.x] = sw; pA[blockIdx.x] = sv; }
  }
  unsigned target = base + static_cast<unsigned>(G);
  grid_barrier_count(ctr, target, err);
  if (blockIdx.x == 0) {
    const double ww = sum_partials_few_d<kCoopThreads>(pWW, G);
    if (t == 0) wn[j] = sqrt(ww);
  }
  // MGS phases l = 0..j: h_l from the previous phase's partials, w -= h_l
  // v_l, partials of v_{l+1}.w (of w.w in the last phase)
  double* pin = pA;
  double* pout = pB;
  for (int l = 0; l <= j; ++l) {
    const double h = sum_partials_few_d<kCoopThreads>(pin, G);
    if (blockIdx.x == 0 && t == 0) H[l + static_cast<int64_t>(j) * ldh] = h;
    const double* vl = V + static_cast<int64_t>(l) * ld + r0;
    const double* vn = V + static_cast<int64_t>(l + 1) * ld + r0;
    double acc = 0.0;
    int i = t;
    if (l < j) {
      for (; i + 3 * kCoopThreads < nr; i += 4 * kCoopThreads) {
        double wv[4], vv[4], nv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          wv[u] = ws[i + u * kCoopThreads];
          vv[u] = vl[i + u * kCoopThreads];
          nv[u] = vn[i + u * kCoopThreads];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const double wi = fma(-h, vv[u], wv[u]);
          ws[i + u * kCoopThreads] = wi;
          acc = fma(nv[u], wi, acc);
        }
      }
      for (; i < nr; i += kCoopThreads) {
        const double wi = fma(-h, vl[i], ws[i]);
        ws[i] = wi;
        acc = fma(vn[i], wi, acc);
      }
    } else {
      for (; i < nr; i += kCoopThreads) {
        const double wi = fma(-h, vl[i], ws[i]);
        ws[i] = wi;
        acc = fma(wi, wi, acc);
      }
    }
    const double tot = block_sum_few_d<kCoopThreads>(acc);
    if (t == 0) pout[blockIdx.x] = tot;
    target += static_cast<unsigned>(G);
    grid_barrier_count(ctr, target, err);
    double* tmp = pin; pin = pout; pout = tmp;
  }
  // normalise into V's column j+1
  const double nrm = sqrt(sum_partials_few_d<kCoopThreads>(pin, G));
  if (blockIdx.x == 0 && t == 0) H[(j + 1) + static_cast<int64_t>(j) * ldh] = nrm;
  const double inv = 1.0 / nrm;
  for (int i = t; i < nr; i += kCoopThreads) w[i] = ws[i] * inv;
}

// The same step in fixed point: w resident as above, the vectors streamed
// past it, for matrices whose rows are of like size (rows_even).
//
// In FP64 the FP64 pipe bounds a projection (two FMAs a row at 2 a clock and
// SM: 13 of 20 us at 4.19M rows, where the vector takes 5 us from HBM), then
// the exchange of the partial sums between the CTAs (4 us).  So:
//   * v_l is kept as signed 60-bit integers relative to the largest
//     magnitude of the CTA's rows of it (|v| < 2^ev), w as integers of at
//     most 61 bits relative to a bound on its rows (unit 2^(ew - 62)); both
//     are cut into two signed 32-bit halves, and a row costs seven 32 x 32
//     bit multiply-adds instead of two FP64 FMAs:
//       dot:  sum vh wh 2^64 + (vh wl + vl wh) 2^32 + vl wl, exact but for the
//             low half of vl wl;
//       w -= h v:  h 2^ev in units of w, rounded to an integer, times v 2^-60,
//             rounded to w's unit.
//     The unit of v is 2^-58 of the CTA's largest entry or less, that of w
//     2^-60 or less at the start: relative to the vectors' norms the
//     projections round less than FP64 ones do, but an entry far below its
//     CTA's largest keeps fewer bits than FP64's 53 (below 2^-60 of it,
//     none).  That matters where the next product with A multiplies small
//     entries by large ones, and rows_even leaves those matrices to FP64.
//     Since |w| can grow while it is projected, its bound grows by
//     |h| 2^ev per projection and w is shifted down when the bound reaches
//     2^61 units.
//   * the CTAs' partial sums are added with integer atomics on a common grid
//     of 2^-70 ||A v_j|| (no partial sum exceeds ||A v_j||): any order gives
//     the same total.  Each of the two words of a sum counts its arrivals in
//     its low byte, so the sum, its completeness and the release of the
//     waiters are one L2 round trip (1.2 us, the counter barrier with 152
//     partial sums read back 3.6 us); no fence is needed, the CTAs share
//     nothing else.
//   * the exchange overlaps the next pass over the rows: pass q takes h_q v_q
//     out of w and sums d_{q+2} = v_{q+2}.w, in which h_{q+1} v_{q+1} is
//     still present, and h_{q+2} = d_{q+2} - (v_{q+2}.v_{q+1}) h_{q+1}: the
//     coefficient MGS computes, in another rounding order.  The products of
//     neighbouring vectors are formed once, when a vector is made.
// The new vector is w scaled in fixed point, and rounded once to FP64 for the
// next product with A.  When ||A v_j||^2 is not a normal number well inside FP64's range (zero, an
// overflow, a NaN in the matrix) the step runs in FP64 on the decoded
// vectors, one projection per barrier.
//
// Measured, whole pre-pass with its products, FP64 pipe -> here: 120 steps
// at 4.19M rows (25 entries) 172 -> 98 ms (a projection 19.9 -> 8.9 us, 3.8
// TB/s of the vector's bytes), at 2.10M (7 entries) 93 -> 45 ms; 60 steps at
// 152K rows 11.1 -> 4.6 ms (5.4 -> 1.9 us: the exchange's latency).  What is
// left at 4.19M rows is reading v_{q+2} from HBM and, for the rows past the
// four batches that tensor memory holds, v_q once more through L2.  1024
// threads (64 registers) were slower at every size (152K rows: 6.0 ms), a
// ring of four smaller batches as well (144 ms at 4.19M rows), and neither
// prefetch into L2 (lines or bulk, one to six batches ahead) changed
// anything.
constexpr int kFxThreads = 512;   // one CTA per SM; 128 registers hold two batches of loads
constexpr int kFxBatch = 4;       // pairs of rows per thread and batch of loads
constexpr int kFxTmem = 4;        // batches that tensor memory keeps, of two vectors
constexpr int kFxV = 60;          // bits of v below 2^ev
constexpr int kFxW = 62;          // bits of w below 2^ew (at most 2^61 used)
constexpr int kFxGrid = 70;       // bits of a partial sum below ||A v_j||

__device__ __forceinline__ double pow2d(int e) {   // 2^e, |e| < 1022
  return __longlong_as_double(static_cast<long long>(e + 1023) << 52);
}

// x 2^(bits - e) rounded to the nearest integer, |x| < 2^e, bits <= 62
// (0 for a non-finite x)
__device__ __forceinline__ long long to_fixed(double x, int e, int bits) {
  const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
  const int E = static_cast<int>((u >> 52) & 0x7FF);
  unsigned long long m = 0;
  if (E != 0 && E != 0x7FF) {
    const unsigned long long mant = (u & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = E - 1075 + bits - e;   // <= bits - 53
    if (sh >= 0) m = mant << (sh > 9 ? 9 : sh);
    else if (sh > -60) m = (mant + (1ull << (-sh - 1))) >> (-sh);
  }
  return (u >> 63) ? -static_cast<long long>(m) : static_cast<long long>(m);
}

// the least e with |x| < 2^e for the bit pattern of a finite |x| > 0
// (subnormals: -1021)
__device__ __forceinline__ int exponent_above(unsigned long long bits) {
  const int E = static_cast<int>((bits >> 52) & 0x7FF);
  return (E == 0 ? 1 : E) - 1022;
}

// a signed integer as (high word, signed low word): x = hi 2^32 + lo with
// |lo| <= 2^31, stored with the high word already corrected
__device__ __forceinline__ long long fx_code(long long x) {
  return x + ((x << 1) & 0x100000000ll);
}
__device__ __forceinline__ double fx_decode(long long code, double unit) {
  const long long x = (static_cast<long long>(static_cast<int>(code >> 32)) << 32) +
                      static_cast<int>(code);
  return static_cast<double>(x) * unit;
}

// a b + c as the one multiply-add it is (with the C++ expression in its place
// a 60-step pre-pass takes 14.97 ms instead of 14.15 at 2.10M rows, 4.67
// instead of 4.66 at 149K).
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// one row's product, v = (vh, vl), w = (wh, wl):
// hh += vh wh, c += vh wl + vl wh + the high half of vl wl
__device__ __forceinline__ void fx_mul(int vl, int vh, int wl, int wh, long long& hh, long long& c) {
  hh = fx_mad(vh, wh, hh);
  c = fx_mad(vh, wl, c);
  c = fx_mad(vl, wh, c);
  c += __mulhi(vl, wl);
}
// (high word, signed low word) of x
__device__ __forceinline__ void fx_split(long long x, int& lo, int& hi) {
  lo = static_cast<int>(x);
  hi = static_cast<int>(x >> 32) + static_cast<int>(static_cast<unsigned>(lo) >> 31);
}
__device__ __forceinline__ void fx_dot(int vl, int vh, long long w, long long& hh, long long& c) {
  int wl, wh;
  fx_split(w, wl, wh);
  fx_mul(vl, vh, wl, wh, hh, c);
}
// c's high half into hh (exact: c keeps the low half); at least every four
// rows (each adds less than 2^60.6 to |c|)
__device__ __forceinline__ void fx_flush(long long& hh, long long& c) {
  hh += c >> 32;
  c &= 0xFFFFFFFFll;
}

// w + v (nh 2^32 + nl) 2^-60, rounded (vl nl, at most four units, left out)
__device__ __forceinline__ long long fx_axpy(int vl, int vh, int nh, int nl, long long w) {
  const long long c = fx_mad(vl, nh, fx_mad(vh, nl, 1ll << 27));
  const long long m = fx_mad(vh, nh, 0);
  return w + (m << 4) + (c >> 28);
}
// x (nh 2^32 + nl) 2^-64, rounded, |x| < 2^62
__device__ __forceinline__ long long fx_scale(long long x, int nh, int nl) {
  int xl, xh;
  fx_split(x, xl, xh);
  long long c = fx_mad(xl, nh, fx_mad(xh, nl, 1ll << 31));
  c += __mulhi(xl, nl);
  return fx_mad(xh, nh, c >> 32);
}

// Tensor memory as storage: this thread's lane, four pairs of rows in 16
// consecutive columns.  These instructions are .aligned: the whole warp has
// to execute them converged, and their callers branch per lane at the ragged
// end of a CTA's rows, so each of the three converges the warp itself.
__device__ __forceinline__ void fx_tmem_st(uint32_t addr, const int4* v) {
  __syncwarp();
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16};" ::"r"(addr),
      "r"(v[0].x), "r"(v[0].y), "r"(v[0].z), "r"(v[0].w), "r"(v[1].x), "r"(v[1].y), "r"(v[1].z),
      "r"(v[1].w), "r"(v[2].x), "r"(v[2].y), "r"(v[2].z), "r"(v[2].w), "r"(v[3].x), "r"(v[3].y),
      "r"(v[3].z), "r"(v[3].w)
      : "memory");
}
// (the wait is in the same statement: no use of the registers can move
// before it)
__device__ __forceinline__ void fx_tmem_ld(uint32_t addr, int4* v) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0].x), "=r"(v[0].y), "=r"(v[0].z), "=r"(v[0].w), "=r"(v[1].x), "=r"(v[1].y),
        "=r"(v[1].z), "=r"(v[1].w), "=r"(v[2].x), "=r"(v[2].y), "=r"(v[2].z), "=r"(v[2].w),
        "=r"(v[3].x), "=r"(v[3].y), "=r"(v[3].z), "=r"(v[3].w)
      : "r"(addr)
      : "memory");
}
__device__ __forceinline__ void fx_tmem_wait_st() {
  __syncwarp();
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// T 2^s; rounded to the nearest integer for s < 0
__device__ __forceinline__ __int128 fx_shift(__int128 T, int s) {
  if (s >= 0) return T << (s > 64 ? 64 : s);
  const int r = -s > 120 ? 120 : -s;
  return (T + (static_cast<__int128>(1) << (r - 1))) >> r;
}

// A coefficient on the common grid: (hi 2^36 + lo) 2^(e0 - 70), 0 <= lo < 2^36
struct FxCoef {
  long long hi, lo;
  __device__ __forceinline__ void carry() {
    hi += lo >> 36;
    lo &= (1ll << 36) - 1;
  }
  // (hi 2^36 + lo) 2^s rounded, for results below 2^62
  __device__ __forceinline__ long long scaled(int s) const {
    if (s >= 0) return s > 26 ? 0 : (hi << (36 + s)) + (lo << s);
    int r = -s;
    if (r <= 36) return (hi << (36 - r)) + ((lo + (1ll << (r - 1))) >> r);
    r -= 36;
    return (hi + (1ll << ((r > 62 ? 62 : r) - 1))) >> (r > 62 ? 62 : r);
  }
  // bits that scaled(s) takes at most
  __device__ __forceinline__ int bits(int s) const {
    if (hi == 0 && lo == 0) return 0;
    const unsigned long long m = static_cast<unsigned long long>(hi < 0 ? -hi : hi) + 1;
    return 64 - __clzll(static_cast<long long>(m)) + 36 + s;
  }
  __device__ __forceinline__ double in_grid() const {
    return fma(static_cast<double>(hi), 68719476736.0, static_cast<double>(lo));
  }
};

// words of one step's exchanges: [0] the full barriers' counter, then a
// (low, high) pair per coefficient
__host__ __device__ constexpr int64_t fx_set_words(int k) { return 2 + 2 * (static_cast<int64_t>(k) + 1); }

// What a pre-pass keeps between its steps beside V: exps, per vector and
// CTA, the exponents ev; gram[l] = v_{l+1}.v_l of the steps before the last
// one, whose CTA partials are gpart; two sets of exchange words, used in turn
// (each step clears the next one's).
struct FxState {
  double* red;                 // 2 G partial sums
  double* gpart;               // G
  double* gram;
  int* exps;
  unsigned long long* set;
  unsigned long long* next_set;
  int set_words;
};

__global__ void __launch_bounds__(kFxThreads, 1)
arnoldi_mgs_resident_kernel(int n, int rows_cta, double* V, int64_t ld, int j, double* xv,
                            double* __restrict__ H, int ldh, double* __restrict__ wn,
                            FxState fs, int* err) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  constexpr int T = kFxThreads, W = kFxThreads / 32;
  __shared__ unsigned wsum[2][4][W];           // a pass's sums, four limbs per warp
  __shared__ unsigned long long wmax[W];
  __shared__ uint32_t tmem_base;
  __shared__ int bc[2][5];                     // of a pass: -h (nl, nh), w's shift; last pass: two
  long long* ws = reinterpret_cast<long long*>(coop_smem);      // w, fixed point
  double* wd = reinterpret_cast<double*>(coop_smem);            // w, FP64 (before and after)
  const int G = gridDim.x, cta = blockIdx.x;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int64_t r0 = static_cast<int64_t>(cta) * rows_cta;
  const int64_t r1 = (r0 + rows_cta < n) ? r0 + rows_cta : n;
  const int nr = r1 > r0 ? static_cast<int>(r1 - r0) : 0;
  const int np = (nr + 1) >> 1;                // pairs of rows (the last may be half)
  double* w = V + static_cast<int64_t>(j + 1) * ld + r0;
  auto col = [&](int l) { return reinterpret_cast<int4*>(V + static_cast<int64_t>(l) * ld + r0); };
  unsigned* ctr = reinterpret_cast<unsigned*>(fs.set);
  unsigned target = 0;
  double* pWW = fs.red;
  double* pNN = fs.red + G;
  constexpr unsigned long long kMag = 0x7FFFFFFFFFFFFFFFull;
  // largest of the threads' values; every thread receives it
  auto block_max = [&](unsigned long long m) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
      m = o > m ? o : m;
    }
    __syncthreads();
    if (lane == 0) wmax[warp] = m;
    __syncthreads();
    m = wmax[lane % W];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
      m = o > m ? o : m;
    }
    return m;
  };
  // the warp's sum of the threads' hh 2^64 + c 2^32 (0 <= c < 2^32) into
  // wsum[b], in units of 2^40: limbs of 22 bits, the last one signed
  auto warp_sums = [&](long long hh, long long c, int b) {
    const unsigned long long lo = (static_cast<unsigned long long>(hh) << 24) |
                                  static_cast<unsigned long long>(c >> 8);
    const long long hi = hh >> 40;
    const unsigned s0 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(lo & 0x3FFFFF));
    const unsigned s1 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>((lo >> 22) & 0x3FFFFF));
    const unsigned s2 = __reduce_add_sync(
        0xffffffffu, static_cast<unsigned>((lo >> 44) | (static_cast<unsigned long long>(hi) << 20)) & 0x3FFFFF);
    const int s3 = __reduce_add_sync(0xffffffffu, static_cast<int>(hi >> 2));
    if (lane == 0) {
      wsum[b][0][warp] = s0;
      wsum[b][1][warp] = s1;
      wsum[b][2][warp] = s2;
      wsum[b][3][warp] = static_cast<unsigned>(s3);
    }
  };
  // the CTA's sum of wsum[b] (by one warp, every lane receives it)
  auto cta_sum = [&](int b) -> __int128 {
    const unsigned s0 = __reduce_add_sync(0xffffffffu, lane < W ? wsum[b][0][lane] : 0u);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, lane < W ? wsum[b][1][lane] : 0u);
    const unsigned s2 = __reduce_add_sync(0xffffffffu, lane < W ? wsum[b][2][lane] : 0u);
    const int s3 = __reduce_add_sync(0xffffffffu, lane < W ? static_cast<int>(wsum[b][3][lane]) : 0);
    const __int128 top = static_cast<__int128>((static_cast<long long>(s3) << 22) + s2) << 44;
    return top + static_cast<long long>((static_cast<unsigned long long>(s1) << 22) + s0);
  };
  auto to_double = [](__int128 x) {
    return fma(static_cast<double>(static_cast<long long>(x >> 48)), 281474976710656.0,
               static_cast<double>(static_cast<long long>(x & ((static_cast<__int128>(1) << 48) - 1))));
  };

  // Pair p = (k U + u) T + t of the CTA's rows is thread t's, batch k.  The
  // first four batches of v_q stay in tensor memory from the pass that reads
  // it (as v_{q+2} two passes before) to the one that takes it out of w:
  // the thread's lane, columns 128 (warp / 4) + 32 k + 16 (q % 2) + 4 u.
  // (The kernel's registers fill an SM, so no other kernel's allocation can
  // be in the way there.)
  constexpr int U = kFxBatch;
  const int nb = np / (U * T);                 // whole batches
  const int tail = nb * U * T;                 // first pair of the rest
  const int nbt = (np + U * T - 1) / (U * T);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(&tmem_base))), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tm = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) +
                      static_cast<uint32_t>((warp >> 2) * 128);

  if (cta == 0)   // the words of the next step (used two launches ago)
    for (int i = t; i < fs.set_words; i += T) fs.next_set[i] = 0;
  if (j == 0) {
    // v_0 arrives in FP64: to fixed point in place
    double* q = V + r0;
    unsigned long long mx = 0;
    for (int i = t; i < nr; i += T) {
      const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(q[i])) & kMag;
      mx = b > mx ? b : mx;
    }
    mx = block_max(mx);
    int ev = mx == 0 ? -100 : exponent_above(mx);
    if (ev < -100) ev = -100;
    if (t == 0) fs.exps[cta] = ev;
    long long* qc = reinterpret_cast<long long*>(q);
    for (int p = t; p < np; p += T)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = 2 * p + u;
        qc[i] = i < nr ? fx_code(to_fixed(q[i], ev, kFxV)) : 0;
      }
    __syncthreads();
  }
  // this CTA's rows of w = A v_j, partial of w.w, largest magnitude
  double accw = 0.0;
  unsigned long long mx = 0;
  for (int p0 = t; p0 < np; p0 += 4 * T) {
    double2 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int p = p0 + u * T;
      x[u] = make_double2(0.0, 0.0);
      if (2 * p + 1 < nr) x[u] = __ldcg(reinterpret_cast<const double2*>(w) + p);
      else if (2 * p < nr) x[u].x = w[2 * p];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int p = p0 + u * T;
      if (p < np) *reinterpret_cast<double2*>(wd + 2 * p) = x[u];
      accw = fma(x[u].x, x[u].x, accw);
      accw = fma(x[u].y, x[u].y, accw);
      unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x[u].x)) & kMag;
      mx = b > mx ? b : mx;
      b = static_cast<unsigned long long>(__double_as_longlong(x[u].y)) & kMag;
      mx = b > mx ? b : mx;
    }
  }
  {
    const double sw = block_sum_few_d<T>(accw);
    if (t == 0) pWW[cta] = sw;
  }
  mx = block_max(mx);
  // v_j.v_{j-1}, from the partial sums the previous step left
  const double gnew = j > 0 ? sum_partials_few_d<T>(fs.gpart, G) : 0.0;
  if (cta == 0 && t == 0 && j > 0) fs.gram[j - 1] = gnew;
  target += static_cast<unsigned>(G);
  grid_barrier_count(ctr, target, err);
  const double ww = sum_partials_few_d<T>(pWW, G);
  const double wnorm = sqrt(ww);
  if (cta == 0 && t == 0) wn[j] = wnorm;

  double acc = 0.0;         // FP64 form: thread partial of ||w||^2 after the projections
  double unit = 0.0;        // fixed point: w's unit then (0: FP64 form)
  const int evj = fs.exps[static_cast<int64_t>(j) * G + cta];
  if (ww > 1e-280 && ww < 1e280) {
    // ------------------------------------------------- fixed point
    const int e0 = exponent_above(static_cast<unsigned long long>(__double_as_longlong(wnorm)));
    int ew = mx == 0 ? e0 - 100 : exponent_above(mx) + 2;
    if (ew < e0 - 100) ew = e0 - 100;
    long long bound = mx == 0 ? 0 : 1ll << 60;   // |w| <= bound <= 2^61, in units (warp 1 keeps it)
    auto ev_of = [&](int l) { return fs.exps[static_cast<int64_t>(l) * G + cta]; };
    // warp 0: adds the CTA's sum of v_l.w in wsum[b] to coefficient l
    auto post = [&](int l, int b, int evl) {
      const __int128 P = fx_shift(cta_sum(b), 40 + (ew - kFxW) + (evl - kFxV) + kFxGrid - e0);
      if (lane < 2) {
        const unsigned long long part = lane == 0
            ? static_cast<unsigned long long>(P) & ((1ull << 36) - 1)
            : static_cast<unsigned long long>(static_cast<long long>(P >> 36));
        atomicAdd(fs.set + 2 + 2 * l + lane, (part << 8) + 1ull);
      }
    };
    // warp 1: coefficient l once every CTA has posted it
    auto fetch = [&](int l) -> FxCoef {
      unsigned long long word = 0;
      if (lane < 2) {
        const unsigned long long* slot = fs.set + 2 + 2 * l + lane;
        const uint64_t t0 = now_ns();
        unsigned spins = 0;
        for (;;) {
          asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(word) : "l"(slot) : "memory");
          if (static_cast<unsigned>(word & 0xFF) == static_cast<unsigned>(G)) break;
          if ((++spins & 255u) == 0) {
            // (after a timeout anywhere every wait is left at once)
            if (*reinterpret_cast<volatile int*>(err) != 0) break;
            if (now_ns() - t0 > kBarrierNs) {
              atomicExch(err, 1);
              break;
            }
          }
        }
      }
      __syncwarp();
      FxCoef c;
      c.lo = static_cast<long long>(__shfl_sync(0xffffffffu, word, 0)) >> 8;
      c.hi = static_cast<long long>(__shfl_sync(0xffffffffu, word, 1)) >> 8;
      return c;
    };
    // g h: the neighbour's part of a coefficient
    auto neighbour = [&](double g, const FxCoef& h) -> FxCoef {
      const double d = g * h.in_grid();
      const double dh = floor(d * pow2d(-36));
      FxCoef c;
      c.hi = static_cast<long long>(dh);
      c.lo = __double2ll_rn(fma(dh, -68719476736.0, d));
      return c;
    };
    auto minus = [&](const FxCoef& c, const FxCoef& d) -> FxCoef {
      FxCoef r;
      r.hi = c.hi - d.hi;
      r.lo = c.lo - d.lo;
      r.carry();
      return r;
    };
    // the shift of w that h v needs room for (into ew and bound)
    auto make_room = [&](const FxCoef& h, int ev, int& e, long long& bd) -> int {
      const int s = e0 + ev - e + kFxW - kFxGrid;
      int up = h.bits(s) - 61;
      long long grow = 0;
      if (up <= 0) {
        const long long q = h.scaled(s);
        grow = q < 0 ? -q : q;                  // |h| 2^ev in units of w
        up = bd + grow + 8 > (1ll << 61) ? 2 : 0;
      } else {
        up += 2;
      }
      if (up > 0) {
        bd = up < 62 ? (bd >> up) + 1 : 1;
        const long long q = h.scaled(s - up);
        grow = q < 0 ? -q : q;
        e += up;
      }
      bd += grow + 8;
      return up;
    };
    // -h 2^ev in units of w, as (nl, nh)
    auto factor = [&](const FxCoef& h, int ev, int e, int* out) {
      const long long q = -h.scaled(e0 + ev - e + kFxW - kFxGrid);
      const int nl = static_cast<int>(q);
      out[0] = nl;
      out[1] = static_cast<int>((q - nl) >> 32);
    };
    auto shift_w = [&](int up) {
      const int sh = up > 62 ? 62 : up;
      for (int p = t; p < np; p += T) {
        longlong2 f = *reinterpret_cast<longlong2*>(ws + 2 * p);
        f.x = (f.x + (1ll << (sh - 1))) >> sh;
        f.y = (f.y + (1ll << (sh - 1))) >> sh;
        *reinterpret_cast<longlong2*>(ws + 2 * p) = f;
      }
    };
    auto put_h = [&](int l, const FxCoef& h) {
      if (cta == 0 && lane == 0) H[l + static_cast<int64_t>(j) * ldh] = h.in_grid() * pow2d(e0 - kFxGrid);
    };

    // w to fixed point; v_0.w and v_1.w
    {
      long long h0 = 0, h1 = 0, c = 0, d = 0;
      const int4* v0 = col(0);
      const int4* v1 = col(j > 0 ? 1 : 0);
      for (int k = 0; k < nbt; ++k) {
        int4 a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int p = (k * U + u) * T + t;
          a[u] = b[u] = make_int4(0, 0, 0, 0);
          if (p < np) {
            a[u] = __ldcg(v0 + p);
            b[u] = __ldcg(v1 + p);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int p = (k * U + u) * T + t;
          if (p < np) {
            const double2 x = *reinterpret_cast<const double2*>(wd + 2 * p);
            longlong2 f;
            f.x = to_fixed(x.x, ew, kFxW);
            f.y = to_fixed(x.y, ew, kFxW);
            *reinterpret_cast<longlong2*>(ws + 2 * p) = f;
            fx_dot(a[u].x, a[u].y, f.x, h0, c);
            fx_dot(a[u].z, a[u].w, f.y, h0, c);
            fx_dot(b[u].x, b[u].y, f.x, h1, d);
            fx_dot(b[u].z, b[u].w, f.y, h1, d);
            fx_flush(h0, c);
            fx_flush(h1, d);
          }
        }
        if (k < kFxTmem) {
          fx_tmem_st(tm + 32 * k, a);
          fx_tmem_st(tm + 32 * k + 16, b);
        }
      }
      fx_tmem_wait_st();
      warp_sums(h0, c, 0);
      warp_sums(h1, d, 1);
    }
    int4 a[U], v[U];                   // the next batch of v_q (past tensor memory's) and v_{q+2}
    const int4* va = nullptr;
    const int4* vb = nullptr;
    auto load = [&](int k) {
      if (k < nb) {
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldcg(vb + (k * U + u) * T);
        if (k >= kFxTmem) {
#pragma unroll
          for (int u = 0; u < U; ++u) a[u] = __ldcg(va + (k * U + u) * T);
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          a[u] = v[u] = make_int4(0, 0, 0, 0);
          if (tail + u * T + t < np) {
            v[u] = __ldcg(vb + tail + u * T);
            if (k >= kFxTmem) a[u] = __ldcg(va + tail + u * T);
          }
        }
      }
    };
    // the first batch of pass q: in flight during the exchange before it
    auto load_first = [&](int q) {
      va = col(q) + t;
      vb = col(q + 2) + t;
      load(0);
    };
    if (j >= 2) load_first(0);
    __syncthreads();
    FxCoef hp{}, hc{};                 // warp 1: the last coefficients, h_{q} and h_{q+1}
    int evp = 0, evc = 0;
    if (warp == 0) {
      post(0, 0, ev_of(0));
      if (j > 0) post(1, 1, ev_of(1));
    } else if (warp == 1) {
      evc = ev_of(0);
      hc = fetch(0);
      hc.carry();
      if (j > 1) {
        const int up = make_room(hc, evc, ew, bound);
        if (lane == 0) bc[0][2] = up;
        int f[2];
        factor(hc, evc, ew, f);
        if (lane == 0) { bc[0][0] = f[0]; bc[0][1] = f[1]; }
        ew -= up;                      // (every thread adds it at the pass)
      }
    }
    __syncthreads();

    // pass q = 0..j-2: w -= h_q v_q, and the sum of v_{q+2}.w
    for (int q = 0; q + 2 <= j; ++q) {
      const int b = q & 1;
      const uint32_t tq = tm + 16 * b;
      int evn = 0;
      FxCoef near{};
      if (warp == 0) {
        if (q > 0) post(q + 1, b ^ 1, ev_of(q + 1));
      } else if (warp == 1) {
        // (FP64, a few hundred cycles: here, not while the others wait)
        evn = ev_of(q + 1);
        near = neighbour(fs.gram[q], hc);
        put_h(q, hc);
      }
      const int nl = bc[b][0], nh = bc[b][1], up = bc[b][2];
      if (up > 0) {
        shift_w(up);
        ew += up;
      }
      long long hh = 0, c = 0;
      for (int k = 0; k < nb; ++k) {
        int4 x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) { x[u] = a[u]; y[u] = v[u]; }
        load(k + 1);
        if (k < kFxTmem) fx_tmem_ld(tq + 32 * k, x);
        longlong2* wp = reinterpret_cast<longlong2*>(ws) + k * U * T + t;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          longlong2 f = wp[u * T];
          f.x = fx_axpy(x[u].x, x[u].y, nh, nl, f.x);
          f.y = fx_axpy(x[u].z, x[u].w, nh, nl, f.y);
          wp[u * T] = f;
          fx_dot(y[u].x, y[u].y, f.x, hh, c);
          fx_dot(y[u].z, y[u].w, f.y, hh, c);
          if (u & 1) fx_flush(hh, c);
        }
        if (k < kFxTmem) fx_tmem_st(tq + 32 * k, y);
      }
      if (nb < nbt && nb < kFxTmem) fx_tmem_ld(tq + 32 * nb, a);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int p = tail + u * T + t;
        if (p < np) {
          longlong2 f = *reinterpret_cast<const longlong2*>(ws + 2 * p);
          f.x = fx_axpy(a[u].x, a[u].y, nh, nl, f.x);
          f.y = fx_axpy(a[u].z, a[u].w, nh, nl, f.y);
          *reinterpret_cast<longlong2*>(ws + 2 * p) = f;
          fx_dot(v[u].x, v[u].y, f.x, hh, c);
          fx_dot(v[u].z, v[u].w, f.y, hh, c);
          fx_flush(hh, c);
        }
      }
      if (nb < nbt && nb < kFxTmem) fx_tmem_st(tq + 32 * nb, v);
      fx_tmem_wait_st();
      if (q + 3 <= j) load_first(q + 1);
      warp_sums(hh, c, b);
      if (warp == 1) {
        // h_{q+1}, posted a pass ago, and what the next pass needs of it
        hp = hc;
        evp = evc;
        hc = minus(fetch(q + 1), near);
        evc = evn;
        if (q + 3 <= j) {
          const int up2 = make_room(hc, evc, ew, bound);
          int f[2];
          factor(hc, evc, ew, f);
          if (lane == 0) { bc[b ^ 1][0] = f[0]; bc[b ^ 1][1] = f[1]; bc[b ^ 1][2] = up2; }
          ew -= up2;
        }
      }
      __syncthreads();
    }
    // the last coefficient, then the last two projections together
    if (warp == 0) {
      if (j > 1) post(j, j & 1, evj);
    } else if (warp == 1) {
      int f[4] = {0, 0, 0, 0}, up = 0;
      if (j > 0) {
        const FxCoef near = neighbour(gnew, hc);
        hp = hc;
        evp = evc;
        hc = minus(fetch(j), near);
        evc = evj;
        up = make_room(hp, evp, ew, bound);
      }
      up += make_room(hc, evc, ew, bound);
      if (j > 0) factor(hp, evp, ew, f);
      factor(hc, evc, ew, f + 2);
      ew -= up;
      if (lane == 0) {
        for (int i = 0; i < 4; ++i) bc[0][i] = f[i];
        bc[0][4] = up;
      }
      if (j > 0) put_h(j - 1, hp);
      put_h(j, hc);
    }
    __syncthreads();
    {
      const int nl = bc[0][0], nh = bc[0][1], ml = bc[0][2], mh = bc[0][3], up = bc[0][4];
      if (up > 0) {
        shift_w(up);
        ew += up;
      }
      const int4* va = col(j > 0 ? j - 1 : 0);
      const int4* vb = col(j);
      unit = pow2d(ew - kFxW);
      long long hh = 0, c = 0;
      unsigned long long m = 0;
      for (int k = 0; k < nbt; ++k) {
        int4 x[U], y[U];
        if (k < kFxTmem) {
          fx_tmem_ld(tm + 32 * k + 16 * ((j + 1) & 1), x);
          fx_tmem_ld(tm + 32 * k + 16 * (j & 1), y);
        } else {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int p = (k * U + u) * T + t;
            x[u] = y[u] = make_int4(0, 0, 0, 0);
            if (p < np) {
              x[u] = __ldcg(va + p);
              y[u] = __ldcg(vb + p);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int p = (k * U + u) * T + t;
          if (p < np) {
            longlong2 f = *reinterpret_cast<const longlong2*>(ws + 2 * p);
            f.x = fx_axpy(x[u].x, x[u].y, nh, nl, f.x);
            f.y = fx_axpy(x[u].z, x[u].w, nh, nl, f.y);
            f.x = fx_axpy(y[u].x, y[u].y, mh, ml, f.x);
            f.y = fx_axpy(y[u].z, y[u].w, mh, ml, f.y);
            *reinterpret_cast<longlong2*>(ws + 2 * p) = f;
            // w.w in units of 16 unit^2 (|w| may reach 2^61), the largest |w|
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const long long z = i == 0 ? f.x : f.y;
              int zl, zh;
              fx_split((z + 2) >> 2, zl, zh);
              hh = fx_mad(zh, zh, hh);
              c = fx_mad(2 * zh, zl, c);
              c += __mulhi(zl, zl);
              const unsigned long long az = static_cast<unsigned long long>(z < 0 ? -z : z);
              m = az > m ? az : m;
            }
            fx_flush(hh, c);
          }
        }
      }
      warp_sums(hh, c, 0);
      mx = block_max(m);               // (its barriers cover wsum)
    }
  } else {
    // -------------------------------------------------- FP64, decoded vectors
    double* pA = fs.red;            // (free again once every CTA has read pWW)
    double* pB = fs.red + G;
    auto unit_of = [&](int l) { return pow2d(fs.exps[static_cast<int64_t>(l) * G + cta] - kFxV); };
    __syncthreads();
    const long long* v0 = reinterpret_cast<const long long*>(col(0));
    double part = 0.0, ul = unit_of(0);
    for (int i = t; i < nr; i += T) part = fma(fx_decode(v0[i], ul), wd[i], part);
    target += static_cast<unsigned>(G);
    grid_barrier_count(ctr, target, err);
    for (int l = 0; l <= j; ++l) {
      const double tot = block_sum_few_d<T>(part);
      if (t == 0) pA[cta] = tot;
      target += static_cast<unsigned>(G);
      grid_barrier_count(ctr, target, err);
      const double h = sum_partials_few_d<T>(pA, G);
      if (cta == 0 && t == 0) H[l + static_cast<int64_t>(j) * ldh] = h;
      const long long* vl = reinterpret_cast<const long long*>(col(l));
      const long long* vn = reinterpret_cast<const long long*>(col(l < j ? l + 1 : l));
      const double un = unit_of(l < j ? l + 1 : l);
      part = 0.0;
      for (int i = t; i < nr; i += T) {
        const double wi = fma(-h, fx_decode(vl[i], ul), wd[i]);
        wd[i] = wi;
        part = fma(l < j ? fx_decode(vn[i], un) : wi, wi, part);
      }
      ul = un;
      double* tmp = pA; pA = pB; pB = tmp;
    }
    acc = part;
    pNN = pA;                       // (the other one may still be being read)
  }
  if (unit != 0.0) {
    if (warp == 0) {
      const __int128 x = cta_sum(0);
      if (lane == 0) pNN[cta] = to_double(x) * pow2d(40 + 4) * unit * unit;
    }
  } else {
    const double tot = block_sum_few_d<T>(acc);
    if (t == 0) pNN[cta] = tot;
  }
  target += static_cast<unsigned>(G);
  grid_barrier_count(ctr, target, err);
  // normalise: fixed point into column j+1, FP64 for the next product with A
  const double nrm = sqrt(sum_partials_few_d<T>(pNN, G));
  if (cta == 0 && t == 0) H[(j + 1) + static_cast<int64_t>(j) * ldh] = nrm;
  const double inv = 1.0 / nrm;
  int ev = -100, sh = 0, nl = 0, nh = 0;
  if (unit != 0.0) {
    if (mx != 0) {
      // v = w unit inv: w shifted left to 62 bits times a 62-bit factor,
      // |v| < 2^ev with ev as small as the factor's range allows
      sh = __clzll(static_cast<long long>(mx)) - 2;      // 2^61 <= |w| 2^sh < 2^62 for the largest
      const double f = unit * inv;                       // v per unit of w
      ev = exponent_above(static_cast<unsigned long long>(__double_as_longlong(f))) + 62 - sh;
      if (ev < -100) ev = -100;
      if (ev > 100) ev = 100;                            // (breakdown: f is not finite)
      // the factor is f 2^-sh 2^(60 - ev) 2^64 < 2^62
      const long long q = __double2ll_rn(f * pow2d(64 + kFxV - ev - sh));
      nl = static_cast<int>(q);
      nh = static_cast<int>((q - nl) >> 32);
    }
  } else {
    mx = 0;
    for (int p = t; p < np; p += T) {
      double2 x = *reinterpret_cast<const double2*>(wd + 2 * p);
      x.x *= inv;
      x.y = 2 * p + 1 < nr ? x.y * inv : 0.0;
      *reinterpret_cast<double2*>(wd + 2 * p) = x;
      unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x.x)) & kMag;
      mx = b > mx ? b : mx;
      b = static_cast<unsigned long long>(__double_as_longlong(x.y)) & kMag;
      mx = b > mx ? b : mx;
    }
    mx = block_max(mx);
    if (mx != 0) ev = exponent_above(mx);
    if (ev < -100) ev = -100;
    if (ev > 100) ev = 100;     // (not a unit vector: the step broke down)
  }
  if (t == 0) fs.exps[static_cast<int64_t>(j + 1) * G + cta] = ev;
  // the new vector, and its product with v_j
  long long hh = 0, c = 0;
  longlong2* wc = reinterpret_cast<longlong2*>(w);
  double* xr = xv + r0;
  const int4* vj = col(j);
  const double uv = pow2d(ev - kFxV);
#pragma unroll 4
  for (int p = t; p < np; p += T) {
    const int4 y = __ldcg(vj + p);
    longlong2 f;
    double2 x;
    if (unit != 0.0) {
      f = *reinterpret_cast<const longlong2*>(ws + 2 * p);
      f.x = fx_scale(f.x << sh, nh, nl);
      f.y = fx_scale(f.y << sh, nh, nl);
      x.x = static_cast<double>(f.x) * uv;
      x.y = static_cast<double>(f.y) * uv;
      if (!(inv < HUGE_VAL)) x.x = x.y = inv * 0.0;   // (w vanished: NaN, as 0 / 0)
    } else {
      x = *reinterpret_cast<const double2*>(wd + 2 * p);
      f.x = to_fixed(x.x, ev, kFxV);
      f.y = to_fixed(x.y, ev, kFxV);
    }
    if (2 * p + 1 < nr) *reinterpret_cast<double2*>(xr + 2 * p) = x;
    else xr[2 * p] = x.x;
    f.x = fx_code(f.x);
    f.y = fx_code(f.y);
    wc[p] = f;
    fx_mul(y.x, y.y, static_cast<int>(f.x), static_cast<int>(f.x >> 32), hh, c);
    fx_mul(y.z, y.w, static_cast<int>(f.y), static_cast<int>(f.y >> 32), hh, c);
    fx_flush(hh, c);
  }
  warp_sums(hh, c, 1);
  __syncthreads();
  if (warp == 0) {
    const __int128 x = cta_sum(1);
    if (lane == 0) fs.gpart[cta] = to_double(x) * pow2d(40 + ev - kFxV + evj - kFxV);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512)
                 : "memory");
  }
}

// FP32 form of the same step with grouped lookahead (used for the steps
// past the two-barrier step's basis limit, kIcMaxCols vectors): the MGS
// projections are taken kGrp basis vectors per grid barrier.  With d_k = v_k.w and the
// group's Gram entries G_kq = v_k.v_q (q < k), all summed in the pass that
// precedes the group, the MGS coefficients follow exactly by forward
// substitution, h_k = d_k - sum_{q<k} G_kq h_q (what MGS computes, in
// another rounding order); w then loses the group in MGS order,
// w -= h_0 v_0, w -= h_1 v_1, ...  One barrier per group instead of one
// per vector: the FP32 step is barrier-bound, not bandwidth-bound, and
// reads every basis vector twice either way.
constexpr int kGrp = 4;
// per block, kNP sums: d_k = v_k.w at k (k < kGrp), then the Gram entry
// v_k.v_q (q < k) at kGrp + k(k-1)/2 + q; the norm pass uses slot 0
constexpr int kNP = kGrp + kGrp * (kGrp - 1) / 2;

__device__ __forceinline__ void group_sums(const float* __restrict__ V, int64_t ld, int64_t row,
                                           int l, int g, float wi, float* acc) {
  float v[kGrp];
#pragma unroll
  for (int k = 0; k < kGrp; ++k) v[k] = k < g ? V[row + static_cast<int64_t>(l + k) * ld] : 0.0f;
#pragma unroll
  for (int k = 0; k < kGrp; ++k) {
    acc[k] = fmaf(v[k], wi, acc[k]);
#pragma unroll
    for (int q = 0; q < k; ++q) acc[kGrp + k * (k - 1) / 2 + q] = fmaf(v[k], v[q], acc[kGrp + k * (k - 1) / 2 + q]);
  }
}

template <bool SELL>
__global__ void __launch_bounds__(kCoopThreads, 1)
arnoldi_step_grouped_kernel(int n, int rows_per_cta, const int* __restrict__ rowptr,
                            const int* __restrict__ colind, const float* __restrict__ val,
                            float* __restrict__ V, int64_t ld, int j,
                            double* __restrict__ H, int ldh, double* __restrict__ wn,
                            double* __restrict__ red, unsigned* bar, int* err,
                            int64_t rows32) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  __shared__ double swarp[kCoopThreads / 32][kNP];
  __shared__ double ssum[kNP];
  __shared__ double hs[kGrp];
  const int G = gridDim.x;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const float* vj = V + static_cast<int64_t>(j) * ld;
  float* w = V + static_cast<int64_t>(j + 1) * ld;
  double* pin = red;
  double* pout = red + static_cast<int64_t>(G) * kNP;
  double* pW = red + 2 * static_cast<int64_t>(G) * kNP;
  const int64_t stride = static_cast<int64_t>(G) * kCoopThreads;
  const int64_t i0 = blockIdx.x * static_cast<int64_t>(kCoopThreads) + t;

  // block sums of acc[0..np) -> dst[blockIdx.x * dstride + p]: FP32
  // shuffles within each warp, FP64 only in the one warp that combines
  // the 32 warp sums (FP64 instructions in every warp made the FP64 pipe
  // the limit of this FP32 kernel)
  auto block_partials = [&](const float* acc, int np, double* dst, int dstride) {
    for (int p = 0; p < np; ++p) {
      const float v = warp_sum_f(acc[p]);
      if (lane == 0) swarp[warp][p] = static_cast<double>(v);
    }
    __syncthreads();
    if (warp == 0) {
      for (int p = 0; p < np; ++p) {
        const double v = warp_sum_d<kCoopThreads>(swarp[lane][p]);
        if (lane == 0) dst[static_cast<int64_t>(blockIdx.x) * dstride + p] = v;
      }
    }
    __syncthreads();
  };
  // fixed-order sums over the G blocks' partials -> ssum[0..np)
  auto gather = [&](const double* src, int np) {
    if (warp < np) {
      double v = 0.0;
      for (int c = lane; c < G; c += 32) v += src[static_cast<int64_t>(c) * kNP + warp];
      v = warp_sum_d<kCoopThreads>(v);
      if (lane == 0) ssum[warp] = v;
    }
    __syncthreads();
  };

  const int ncols = j + 1;  // basis vectors v_0 .. v_j to project out
  int g1 = ncols < kGrp ? ncols : kGrp;
  // phase 0: w = A v_j; partials of w.w and of group 0's dots and Gram
  {
    float acc[kNP];
#pragma unroll
    for (int p = 0; p < kNP; ++p) acc[p] = 0.0f;
    float accw[1] = {0.0f};
    if (SELL) {
      for (int64_t row = i0; row < rows32; row += stride) {
        const float sum = sell_row(rowptr, colind, val, vj, row);
        if (row < n) {
          w[row] = sum;
          accw[0] = fmaf(sum, sum, accw[0]);
          group_sums(V, ld, row, 0, g1, sum, acc);
        }
      }
    } else {
      float* sval = reinterpret_cast<float*>(coop_smem);
      int* scol = reinterpret_cast<int*>(coop_smem + sizeof(float) * kCoopStage);
      for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * rows_per_cta; r0 < n;
           r0 += static_cast<int64_t>(G) * rows_per_cta) {
        const int64_t r1 = (r0 + rows_per_cta < n) ? r0 + rows_per_cta : n;
        const int k0 = rowptr[r0];
        const int len = rowptr[r1] - k0;
        const bool staged = len <= kCoopStage;
        if (staged) {
          for (int e = t; e < len; e += kCoopThreads) {
            sval[e] = ld_stream(val + k0 + e);
            scol[e] = ld_stream(colind + k0 + e);
          }
        }
        __syncthreads();
        for (int64_t row = r0 + t; row < r1; row += kCoopThreads) {
          const int a = rowptr[row], b = rowptr[row + 1];
          float sum = 0.0f;
          if (staged) {
            for (int k = a - k0; k < b - k0; ++k) sum = fmaf(sval[k], __ldg(vj + scol[k]), sum);
          } else {
            for (int k = a; k < b; ++k)
              sum = fmaf(ld_stream(val + k), __ldg(vj + ld_stream(colind + k)), sum);
          }
          w[row] = sum;
          accw[0] = fmaf(sum, sum, accw[0]);
          group_sums(V, ld, row, 0, g1, sum, acc);
        }
        __syncthreads();
      }
    }
    block_partials(accw, 1, pW, 1);
    block_partials(acc, kNP, pin, kNP);
  }
  grid_barrier(bar, G, err);
  if (blockIdx.x == 0 && warp == 0) {
    double ww = 0.0;
    for (int c = lane; c < G; c += 32) ww += pW[c];
    ww = warp_sum_d<kCoopThreads>(ww);
    if (lane == 0) wn[j] = sqrt(ww);
  }
  // groups of kGrp basis vectors
  for (int l0 = 0; l0 < ncols; l0 += kGrp) {
    const int gs = g1;
    const int l1 = l0 + gs;
    const int gn = (ncols - l1) < kGrp ? (ncols - l1) : kGrp;  // next group (0: none)
    gather(pin, kNP);
    if (t == 0) {
      for (int k = 0; k < gs; ++k) {
        double hk = ssum[k];
        for (int q = 0; q < k; ++q) hk -= ssum[kGrp + k * (k - 1) / 2 + q] * hs[q];
        hs[k] = hk;
        if (blockIdx.x == 0) H[(l0 + k) + static_cast<int64_t>(j) * ldh] = hk;
      }
    }
    __syncthreads();
    float hf[kGrp];
#pragma unroll
    for (int k = 0; k < kGrp; ++k) hf[k] = k < gs ? static_cast<float>(hs[k]) : 0.0f;
    float acc[kNP];
#pragma unroll
    for (int p = 0; p < kNP; ++p) acc[p] = 0.0f;
    // two elements per iteration, so both elements' loads are in flight
    // together (one element at a time left each thread waiting on memory)
    int64_t i = i0;
    for (; i + stride < n; i += 2 * stride) {
      float wi[2], vu[2][kGrp];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        wi[e] = w[i + e * stride];
#pragma unroll
        for (int k = 0; k < kGrp; ++k)
          vu[e][k] = k < gs ? V[i + e * stride + static_cast<int64_t>(l0 + k) * ld] : 0.0f;
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int k = 0; k < kGrp; ++k)
          if (k < gs) wi[e] = fmaf(-hf[k], vu[e][k], wi[e]);
        w[i + e * stride] = wi[e];
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (gn > 0) group_sums(V, ld, i + e * stride, l1, gn, wi[e], acc);
        else acc[0] = fmaf(wi[e], wi[e], acc[0]);
      }
    }
    for (; i < n; i += stride) {
      float wi = w[i];
#pragma unroll
      for (int k = 0; k < kGrp; ++k)
        if (k < gs) wi = fmaf(-hf[k], V[i + static_cast<int64_t>(l0 + k) * ld], wi);
      w[i] = wi;
      if (gn > 0) group_sums(V, ld, i, l1, gn, wi, acc);
      else acc[0] = fmaf(wi, wi, acc[0]);
    }
    block_partials(acc, kNP, pout, kNP);
    grid_barrier(bar, G, err);
    double* tmp = pin; pin = pout; pout = tmp;
    g1 = gn;
  }
  // normalise: the last pass left the partials of ||w||^2 in slot 0
  gather(pin, 1);
  const double nrm = sqrt(ssum[0]);
  if (blockIdx.x == 0 && t == 0) H[(j + 1) + static_cast<int64_t>(j) * ldh] = nrm;
  const float inv = static_cast<float>(1.0 / nrm);
  for (int64_t i = i0; i < n; i += stride) w[i] *= inv;
}

// FP32 step with two grid barriers (the inverse compact WY form of MGS):
// for the basis v_0..v_j, the MGS coefficients of w = A v_j satisfy
//   h_k = d_k - sum_{q<k} G_kq h_q,  d_k = v_k.w,  G_kq = v_k.v_q,
// so with the lower triangle L of V^T V, h = (I + L)^{-1} d: the
// projections MGS takes one after another, in another rounding order
// (low-synchronisation MGS of Swirydowicz, Langou, Ananthan, Yang and
// Thomas).  Each step then reads the basis twice at full bandwidth:
//   pass A: w = A v_j chunk by chunk (a CTA's own rows, staged with v_j in
//           shared memory), and for every column q of the chunk the
//           partials of v_q.w and v_q.v_j (the new Gram row);
//   barrier; every CTA sums the partials in the same fixed order, keeps
//           row j of the Gram matrix, and solves (I + L) h = d;
//   pass B: w -= sum_q h_q v_q for the CTA's rows (q ascending, the MGS
//           order per element) with the partials of ||w||^2;
//   barrier; w /= ||w||.
// The Gram matrix is stored packed by rows (row k at k(k-1)/2) in global
// memory for the later steps and staged in shared memory before pass A.
constexpr int kIcChunk = 4096;                 // rows per staged chunk
constexpr int kIcMaxCols = 161;                // basis vectors v_0..v_j per step

__host__ __device__ constexpr int ic_tri(int ncols) { return ncols * (ncols - 1) / 2; }

// dynamic shared memory: sw, sv (chunk), column sums, Gram triangle, d, h,
// two scalars, -h in FP32
__host__ __device__ constexpr size_t ic_smem_bytes(int ncols) {
  return sizeof(float) * 2 * kIcChunk + sizeof(double) * 2 * ncols +
         sizeof(double) * (ic_tri(ncols) + 2 * ncols + 8) + sizeof(float) * ncols;
}

// partials: (2 ncols + 1) per CTA for pass A, then G for the norm, then the
// packed Gram matrix of up to kIcMaxCols vectors
int64_t ic_red_doubles(int G) {
  return static_cast<int64_t>(2 * kIcMaxCols + 2) * G + ic_tri(kIcMaxCols);
}

template <bool SELL>
__global__ void __launch_bounds__(kCoopThreads, 1)
arnoldi_step_icwy_kernel(int n, const int* __restrict__ rowptr,
                         const int* __restrict__ colind, const float* __restrict__ val,
                         float* __restrict__ V, int64_t ld, int j, double* __restrict__ H,
                         int ldh, double* __restrict__ wn, double* __restrict__ red,
                         unsigned* bar, int* err) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  __shared__ double swarp[kCoopThreads / 32];
  const int ncols = j + 1;
  const int G = gridDim.x;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  float* sw = reinterpret_cast<float*>(coop_smem);
  float* sv = sw + kIcChunk;
  double* slots = reinterpret_cast<double*>(sv + kIcChunk);  // [q][2]: v_q.w, v_q.v_j
  double* tri = slots + 2 * ncols;
  double* dk = tri + ic_tri(ncols);
  double* hk = dk + ncols;
  double* misc = hk + ncols;  // [0]: ||A v_j||^2, [1]: ||w||^2 after projection
  float* nh = reinterpret_cast<float*>(misc + 8);  // -h_q in FP32 for pass B

  const int P = 2 * ncols + 1;
  double* pA = red;                                                   // G x P
  double* pN = red + static_cast<int64_t>(2 * kIcMaxCols + 1) * G;    // G
  double* gram = red + static_cast<int64_t>(2 * kIcMaxCols + 2) * G;  // packed rows

  const float* vj = V + static_cast<int64_t>(j) * ld;
  float* w = V + static_cast<int64_t>(j + 1) * ld;
  // this CTA's rows: whole 32-row slices, as even as possible
  const int64_t nsl = (static_cast<int64_t>(n) + 31) / 32;
  const int64_t r0 = 32 * (nsl * blockIdx.x / G);
  int64_t r1 = 32 * (nsl * (blockIdx.x + 1) / G);
  if (r1 > n) r1 = n;

  // the Gram rows of the earlier steps (read during pass A's latency)
  for (int e = t; e < ic_tri(j); e += kCoopThreads) tri[e] = gram[e];
  for (int e = t; e < 2 * ncols; e += kCoopThreads) slots[e] = 0.0;

  // ------------------------------------------------------------ pass A
  float accww = 0.0f;
  for (int64_t c0 = r0; c0 < r1; c0 += kIcChunk) {
    const int len = static_cast<int>((r1 - c0) < kIcChunk ? (r1 - c0) : kIcChunk);
    __syncthreads();  // the previous chunk's readers are done with sw / sv
    for (int r = t; r < len; r += kCoopThreads) {
      const int64_t row = c0 + r;
      float sum;
      if (SELL) {
        sum = sell_row(rowptr, colind, val, vj, row);
      } else {
        sum = 0.0f;
        const int a = rowptr[row], b = rowptr[row + 1];
        for (int k = a; k < b; ++k) sum = fmaf(ld_stream(val + k), __ldg(vj + ld_stream(colind + k)), sum);
      }
      w[row] = sum;
      sw[r] = sum;
      sv[r] = vj[row];
      accww = fmaf(sum, sum, accww);
    }
    __syncthreads();
    // column q of the chunk belongs to warp q % 32: lane l adds the rows
    // 4 l + 128 it in FP32 (eight float4 loads in flight), the lanes are
    // combined by shuffles, and the chunk's sum is added in FP64 in chunk
    // order
    for (int q = warp; q < ncols; q += 32) {
      const float* vq = V + static_cast<int64_t>(q) * ld + c0;
      float d = 0.0f, gm = 0.0f;
      if (len == kIcChunk) {
#pragma unroll 1
        for (int it0 = 0; it0 < kIcChunk / 128; it0 += 8) {
          float4 a[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            a[u] = *reinterpret_cast<const float4*>(vq + (it0 + u) * 128 + lane * 4);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int r = (it0 + u) * 128 + lane * 4;
            const float4 x = *reinterpret_cast<const float4*>(sw + r);
            const float4 y = *reinterpret_cast<const float4*>(sv + r);
            d = fmaf(a[u].x, x.x, d); d = fmaf(a[u].y, x.y, d);
            d = fmaf(a[u].z, x.z, d); d = fmaf(a[u].w, x.w, d);
            gm = fmaf(a[u].x, y.x, gm); gm = fmaf(a[u].y, y.y, gm);
            gm = fmaf(a[u].z, y.z, gm); gm = fmaf(a[u].w, y.w, gm);
          }
        }
      } else {
        for (int r = lane; r < len; r += 32) {
          const float a = vq[r];
          d = fmaf(a, sw[r], d);
          gm = fmaf(a, sv[r], gm);
        }
      }
      d = warp_sum_f(d);
      gm = warp_sum_f(gm);
      if (lane == 0) {
        slots[2 * q] += static_cast<double>(d);
        slots[2 * q + 1] += static_cast<double>(gm);
      }
    }
  }
  // CTA partials: per column; ||A v_j||^2
  __syncthreads();
  for (int q = t; q < ncols; q += kCoopThreads) {
    pA[static_cast<int64_t>(blockIdx.x) * P + 2 * q] = slots[2 * q];
    pA[static_cast<int64_t>(blockIdx.x) * P + 2 * q + 1] = slots[2 * q + 1];
  }
  {
    const float v = warp_sum_f(accww);
    if (lane == 0) swarp[warp] = static_cast<double>(v);
    __syncthreads();
    if (warp == 0) {
      const double s = warp_sum_d<kCoopThreads>(swarp[lane]);
      if (lane == 0) pA[static_cast<int64_t>(blockIdx.x) * P + 2 * ncols] = s;
    }
  }
  grid_barrier(bar, G, err);

  // ------------------------------------------- sums and the coefficients
  // every CTA adds the G partials of each sum in the same fixed order
  for (int p = warp; p < P; p += 32) {
    double v = 0.0;
    for (int c = lane; c < G; c += 32) v += pA[static_cast<int64_t>(c) * P + p];
    v = warp_sum_d<kCoopThreads>(v);
    if (lane == 0) {
      if (p == 2 * ncols) misc[0] = v;
      else if (p & 1) { if ((p >> 1) < j) tri[ic_tri(j) + (p >> 1)] = v; }  // Gram row j
      else dk[p >> 1] = v;
    }
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int q = t; q < j; q += kCoopThreads) gram[ic_tri(j) + q] = tri[ic_tri(j) + q];
    if (t == 0) wn[j] = sqrt(misc[0]);
  }
  // forward substitution (I + L) h = d by one warp: lanes own rows
  // k = lane + 32 m; column q's h_q is final once columns < q are applied
  if (warp == 0) {
    constexpr int kM = (kIcMaxCols + 31) / 32;
    double dr[kM];
#pragma unroll
    for (int m = 0; m < kM; ++m) {
      const int k = lane + 32 * m;
      dr[m] = k < ncols ? dk[k] : 0.0;
    }
    // the row groups m past the basis are left by a warp-uniform break:
    // predicated FP64 instructions would still take their pipe time
    const int mused = (ncols + 31) / 32;
    for (int q = 0; q < ncols; ++q) {
      double mine = dr[0];
#pragma unroll
      for (int m = 1; m < kM; ++m)
        if (m == (q >> 5)) mine = dr[m];
      const double hq = __shfl_sync(0xffffffffu, mine, q & 31);
      if (lane == 0) hk[q] = hq;
#pragma unroll
      for (int m = 0; m < kM; ++m) {
        if (m >= mused) break;
        const int k = lane + 32 * m;
        if (k > q && k < ncols) dr[m] = fma(-tri[ic_tri(k) + q], hq, dr[m]);
      }
    }
  }
  __syncthreads();
  for (int q = t; q < ncols; q += kCoopThreads) {
    nh[q] = -static_cast<float>(hk[q]);
    if (blockIdx.x == 0) H[q + static_cast<int64_t>(j) * ldh] = hk[q];
  }
  __syncthreads();

  // ------------------------------------------------------------ pass B
  float accn = 0.0f;
  for (int64_t r = r0 + 4 * static_cast<int64_t>(t); r < r1; r += 4 * kCoopThreads) {
    if (r + 3 < r1) {
      float4 wv = *reinterpret_cast<const float4*>(w + r);
      int q = 0;
      for (; q + 8 <= ncols; q += 8) {
        float4 vv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          vv[u] = *reinterpret_cast<const float4*>(V + static_cast<int64_t>(q + u) * ld + r);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float h = nh[q + u];
          wv.x = fmaf(h, vv[u].x, wv.x); wv.y = fmaf(h, vv[u].y, wv.y);
          wv.z = fmaf(h, vv[u].z, wv.z); wv.w = fmaf(h, vv[u].w, wv.w);
        }
      }
      for (; q < ncols; ++q) {
        const float4 vv = *reinterpret_cast<const float4*>(V + static_cast<int64_t>(q) * ld + r);
        const float h = nh[q];
        wv.x = fmaf(h, vv.x, wv.x); wv.y = fmaf(h, vv.y, wv.y);
        wv.z = fmaf(h, vv.z, wv.z); wv.w = fmaf(h, vv.w, wv.w);
      }
      *reinterpret_cast<float4*>(w + r) = wv;
      accn = fmaf(wv.x, wv.x, accn); accn = fmaf(wv.y, wv.y, accn);
      accn = fmaf(wv.z, wv.z, accn); accn = fmaf(wv.w, wv.w, accn);
    } else {
      for (int64_t rr = r; rr < r1; ++rr) {
        float wi = w[rr];
        for (int q = 0; q < ncols; ++q) wi = fmaf(nh[q], V[static_cast<int64_t>(q) * ld + rr], wi);
        w[rr] = wi;
        accn = fmaf(wi, wi, accn);
      }
    }
  }
  {
    const float v = warp_sum_f(accn);
    __syncthreads();  // swarp is free again
    if (lane == 0) swarp[warp] = static_cast<double>(v);
    __syncthreads();
    if (warp == 0) {
      const double s = warp_sum_d<kCoopThreads>(swarp[lane]);
      if (lane == 0) pN[blockIdx.x] = s;
    }
  }
  grid_barrier(bar, G, err);
  if (warp == 0) {
    double v = 0.0;
    for (int c = lane; c < G; c += 32) v += pN[c];
    v = warp_sum_d<kCoopThreads>(v);
    if (lane == 0) misc[1] = v;
  }
  __syncthreads();
  const double nrm = sqrt(misc[1]);
  if (blockIdx.x == 0 && t == 0) H[(j + 1) + static_cast<int64_t>(j) * ldh] = nrm;
  const float inv = static_cast<float>(1.0 / nrm);
  for (int64_t r = r0 + t; r < r1; r += kCoopThreads) w[r] *= inv;
}

// The two-barrier FP32 step while the basis has at most kIcMaxCols
// vectors and the partials buffer holds its sums; false: not launched.
template <bool SELL>
bool launch_arnoldi_icwy(const DevCsr& A, const float* val, float* V, int64_t ld, int j,
                         double* H, int ldh, double* wn, double* red, int red_cap,
                         unsigned* bar, int* err, cudaStream_t st) {
  if (j + 1 > kIcMaxCols) return false;
  const void* fn = reinterpret_cast<const void*>(arnoldi_step_icwy_kernel<SELL>);
  const int smax = static_cast<int>(ic_smem_bytes(kIcMaxCols));
  ensure_dynamic_smem(fn, smax);
  int per_sm = 0;
  SG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kCoopThreads, smax));
  const int mb = per_sm * device_sm_count();
  SG_REQUIRE(mb > 0, SG_ECUDA, "arnoldi step: no resident blocks");
  int G = device_sm_count();
  if (G > mb) G = mb;
  if (ic_red_doubles(G) > red_cap) return false;
  int n = A.n;
  const int* rp = SELL ? A.sptr : A.rowptr;
  const int* ci = SELL ? A.scol : A.colind;
  void* args[] = {&n, const_cast<int**>(&rp), const_cast<int**>(&ci), const_cast<float**>(&val),
                  &V, &ld, &j, &H, const_cast<int*>(&ldh), &wn, &red, &bar, &err};
  SG_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kCoopThreads), args,
                                      ic_smem_bytes(j + 1), st));
  count_launch();
  return true;
}

// Rows per CTA of a resident FP64 step's kernel fn for n rows, or 0 when a
// CTA's slice of w would not fit in shared memory next to the kernel's static
// reduction buffers (then the streaming step runs).  One CTA per SM, at
// least min_rows rows per CTA (fewer CTAs, cheaper exchanges, on small
// systems).
int resident_rows_per_cta(int64_t n, const void* fn, int min_rows, int* grid) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> limit;   // dynamic bytes available
  const int dev = current_device();
  int avail;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = limit.find({dev, fn});
    if (it == limit.end()) {
      int optin = 0;
      SG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
      cudaFuncAttributes fa{};
      SG_CUDA(cudaFuncGetAttributes(&fa, fn));
      it = limit.emplace(std::make_pair(dev, fn),
                         optin - static_cast<int>(fa.sharedSizeBytes) - 1024).first;
    }
    avail = it->second;
  }
  const int64_t sms = device_sm_count();
  int64_t R = (n + sms - 1) / sms;
  if (R < min_rows) R = min_rows;
  R = (R + 31) / 32 * 32;
  if (R * static_cast<int64_t>(sizeof(double)) > avail) return 0;
  *grid = static_cast<int>((n + R - 1) / R);
  return static_cast<int>(R);
}

// doubles of `red` that the resident FP64 step takes in a pre-pass of k steps
int64_t fixed_red_doubles(int G, int k) {
  return 3 * static_cast<int64_t>(G) + (k + 1) + (static_cast<int64_t>(k) + 2) / 2 * G +
         2 * fx_set_words(k);
}

template <typename T, bool SELL>
void launch_arnoldi_step(const DevCsr& A, const T* val, T* V, int64_t ld, int j,
                         int k, T* xv, double* H, int ldh, double* wn, double* red, int red_cap,
                         unsigned* bar, int* err, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    int G = 0;
    const void* fn = reinterpret_cast<const void*>(arnoldi_mgs_resident_kernel);
    int R = A.rows_even == 1 && xv ? resident_rows_per_cta(A.n, fn, 1024, &G) : 0;
    if (R > 0 && G <= device_sm_count() && G < 256 && fixed_red_doubles(G, k) <= red_cap) {
      const int smem = R * static_cast<int>(sizeof(double));
      ensure_dynamic_smem(fn, smem);
      int per_sm = 0;
      SG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kFxThreads, smem));
      if (per_sm >= 1) {
        const int64_t sw = fx_set_words(k);
        unsigned long long* sets =
            reinterpret_cast<unsigned long long*>(red + fixed_red_doubles(G, k) - 2 * sw);
        FxState fs{};
        fs.red = red;
        fs.gpart = red + 2 * G;
        fs.gram = red + 3 * G;
        fs.exps = reinterpret_cast<int*>(fs.gram + (k + 1));
        fs.set = sets + (j & 1) * sw;
        fs.next_set = sets + ((j + 1) & 1) * sw;
        fs.set_words = static_cast<int>(sw);
        if (j == 0) SG_CUDA(cudaMemsetAsync(sets, 0, sizeof(unsigned long long) * 2 * sw, st));
        // w = A v_j into V's column j+1 (v_j in FP64: V's column 0, then xv),
        // in whatever storage A has, then the projections on chip
        dispatch<0, false, T>(A, A.val, A.sval, j == 0 ? V : xv, nullptr,
                              V + static_cast<int64_t>(j + 1) * ld, T(0), T(0), T(1), st);
        int n = A.n;
        int rc = R;
        void* args[] = {&n, &rc, &V, &ld, &j, &xv, &H, const_cast<int*>(&ldh), &wn, &fs, &err};
        SG_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kFxThreads), args, smem, st));
        count_launch();
        return;
      }
    }
    fn = reinterpret_cast<const void*>(arnoldi_mgs_resident64_kernel);
    R = A.rows_even != 1 ? resident_rows_per_cta(A.n, fn, 2048, &G) : 0;
    if (R > 0 && G <= device_sm_count() && 3 * G <= red_cap) {
      const int smem = R * static_cast<int>(sizeof(double));
      ensure_dynamic_smem(fn, smem);
      int per_sm = 0;
      SG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kCoopThreads, smem));
      if (per_sm >= 1) {
        // w = A v_j into V's column j+1, then the MGS phases on chip
        dispatch<0, false, T>(A, A.val, A.sval, V + static_cast<int64_t>(j) * ld, nullptr,
                              V + static_cast<int64_t>(j + 1) * ld, T(0), T(0), T(1), st);
        // barriers per step j: one after the w partials, one per MGS phase
        // (j + 1); the counter (word 16 of the barrier block, zeroed at the
        // start of the pre-pass) has seen G (j' + 2) arrivals per earlier step
        int n = A.n;
        int rc = R;
        unsigned* ctr = bar + 16;
        unsigned base = static_cast<unsigned>(G) * static_cast<unsigned>(j) *
                        static_cast<unsigned>(j + 3) / 2u;
        void* args[] = {&n, &rc, &V, &ld, &j, &H, const_cast<int*>(&ldh), &wn, &red, &ctr,
                        &base, &err};
        SG_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kCoopThreads), args, smem, st));
        count_launch();
        return;
      }
    }
  }
  const int smem = SELL ? 0 : kCoopStage * static_cast<int>(sizeof(T) + sizeof(int));
  // FP32: the two-barrier step while the basis fits it, then the grouped-
  // lookahead step; FP64 keeps one projection per phase, the rounding order
  // of the MGS oracle
  if constexpr (sizeof(T) == 4) {
    if (launch_arnoldi_icwy<SELL>(A, val, V, ld, j, H, ldh, wn, red, red_cap, bar, err, st))
      return;
  }
  const void* fn = reinterpret_cast<const void*>(arnoldi_step_kernel<T, SELL>);
  if constexpr (sizeof(T) == 4) fn = reinterpret_cast<const void*>(arnoldi_step_grouped_kernel<SELL>);
  ensure_dynamic_smem(fn, smem);
  int per_sm = 0;
  SG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kCoopThreads, smem));
  const int mb = per_sm * device_sm_count();
  SG_REQUIRE(mb > 0, SG_ECUDA, "arnoldi step: no resident blocks");
  int G = device_sm_count();  // one CTA per SM: fewer arrivals and partials
  if (G > mb) G = mb;
  const int need = sizeof(T) == 4 ? (2 * kNP + 1) * G : 3 * G;
  SG_REQUIRE(need <= red_cap, SG_EINVAL, "arnoldi step: partials buffer too small");
  // rows per tile: the staged nonzeros fit with 25% slack, <= one per thread
  const double per = A.mean_row > 0 ? A.mean_row * 1.25 : 1.0;
  int rpc = static_cast<int>(kCoopStage / per);
  if (rpc > kCoopThreads) rpc = kCoopThreads;
  if (rpc < 32) rpc = 32;
  int n = A.n;
  int64_t rows32 = static_cast<int64_t>(A.nslices) * 32;
  const int* rp = SELL ? A.sptr : A.rowptr;
  const int* ci = SELL ? A.scol : A.colind;
  void* args[] = {&n, &rpc, const_cast<int**>(&rp), const_cast<int**>(&ci),
                  const_cast<T**>(&val), &V, &ld, &j, &H, const_cast<int*>(&ldh), &wn, &red,
                  &bar, &err, &rows32};
  SG_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kCoopThreads), args, smem, st));
  count_launch();
}

__global__ void sampled_outer_kernel(int n, const int* __restrict__ rowptr,
                                     const int* __restrict__ colind,
                                     const double* __restrict__ lam,
                                     const double* __restrict__ x,
                                     double* __restrict__ dval) {
  // one warp per 32/8 rows, 8 lanes per row, like the SpMV
  constexpr int VEC = 8, RPW = 32 / VEC;
  const int lane = threadIdx.x & 31;
  const int sub = lane / VEC, l = lane % VEC;
  const int64_t warp = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t base = warp * RPW; base < n; base += nwarps * RPW) {
    const int64_t row = base + sub;
    if (row >= n) continue;
    const double li = -lam[row];
    const int s = rowptr[row], e = rowptr[row + 1];
    for (int k = s + l; k < e; k += VEC) dval[k] = li * __ldg(x + colind[k]);
  }
}

// Largest magnitudes of the rows (eight lanes per row), as bit patterns: of
// those, out[0] the largest and out[1] the complement of the smallest (both 0
// before).  An infinity or NaN has the largest pattern.
__global__ void __launch_bounds__(kThreads)
row_extent_kernel(int n, const int* __restrict__ rowptr, const double* __restrict__ val,
                  unsigned long long* out) {
  constexpr int VEC = 8;
  __shared__ unsigned long long sh[2][kThreads / 32];
  const int l = threadIdx.x % VEC;
  unsigned long long hi = 0, lo = 0;
  // (every lane of a warp takes the same number of turns)
  for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * kThreads / VEC; r0 < n;
       r0 += static_cast<int64_t>(gridDim.x) * kThreads / VEC) {
    const int64_t r = r0 + threadIdx.x / VEC;
    unsigned long long m = 0;
    if (r < n) {
      const int e = rowptr[r + 1];
      for (int k = rowptr[r] + l; k < e; k += VEC) {
        const unsigned long long b =
            static_cast<unsigned long long>(__double_as_longlong(val[k])) & 0x7FFFFFFFFFFFFFFFull;
        m = b > m ? b : m;
      }
    }
#pragma unroll
    for (int off = VEC / 2; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
      m = o > m ? o : m;
    }
    if (r < n) {
      hi = m > hi ? m : hi;
      lo = ~m > lo ? ~m : lo;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    unsigned long long o = __shfl_xor_sync(0xffffffffu, hi, off);
    hi = o > hi ? o : hi;
    o = __shfl_xor_sync(0xffffffffu, lo, off);
    lo = o > lo ? o : lo;
  }
  if (threadIdx.x % 32 == 0) {
    sh[0][threadIdx.x / 32] = hi;
    sh[1][threadIdx.x / 32] = lo;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    unsigned long long m = 0;
    for (int w = 0; w < kThreads / 32; ++w) m = sh[threadIdx.x][w] > m ? sh[threadIdx.x][w] : m;
    atomicMax(out + threadIdx.x, m);
  }
}

// --- transpose: places of the entries in their columns, scan of the column
// lengths, scatter of (row, entry), sort within the new rows; the values are
// gathered afterwards, so new values on the same pattern cost one gather
// (1M rows, 25M entries: 8.3 ms with the values carried along, a single-block
// scan and a thread sorting each row in global memory; new values now take
// 0.15 ms, and 0.1 ms more for the SELL copy) ---
__global__ void count_cols_kernel(int64_t nnz, const int* __restrict__ colind,
                                  int* __restrict__ counts, int* __restrict__ place) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
       k += 4 * stride) {
    // four atomics in flight per thread
    int p[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      p[u] = k + u * stride < nnz ? atomicAdd(counts + colind[k + u * stride], 1) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k + u * stride < nnz) place[k + u * stride] = p[u];
  }
}

// exclusive scan of n counters in three steps: sums of blocks of kScanBlock
// counters, the scan of those sums by one block, the blocks' own scans
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanBlock = kScanThreads * kScanItems;

__device__ __forceinline__ int scan_block_sum(int v, int* sh, int* before) {
  // sum over the block; *before: over the threads before this one
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += o;
  }
  if (lane == 31) sh[warp] = inc;
  __syncthreads();
  int base = 0, tot = 0;
  for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) {
    if (w < warp) base += sh[w];
    tot += sh[w];
  }
  __syncthreads();
  *before = base + inc - v;
  return tot;
}

__global__ void __launch_bounds__(kScanThreads)
scan_sums_kernel(int n, const int* __restrict__ counts, int* __restrict__ sums) {
  __shared__ int sh[kScanThreads / 32];
  const int64_t a = static_cast<int64_t>(blockIdx.x) * kScanBlock;
  int v = 0, before = 0;
  for (int i = threadIdx.x; i < kScanBlock; i += kScanThreads)
    if (a + i < n) v += counts[a + i];
  const int tot = scan_block_sum(v, sh, &before);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024)
scan_sums_scan_kernel(int nb, int* __restrict__ sums) {
  __shared__ int sh[32];
  int run = 0;
  for (int a = 0; a < nb; a += 1024) {
    const int i = a + threadIdx.x;
    const int v = i < nb ? sums[i] : 0;
    int before = 0;
    const int tot = scan_block_sum(v, sh, &before);
    if (i < nb) sums[i] = run + before;
    run += tot;
  }
}

__global__ void __launch_bounds__(kScanThreads)
scan_apply_kernel(int n, int total, const int* __restrict__ counts, const int* __restrict__ sums,
                  int* __restrict__ rowptr) {
  __shared__ int sh[kScanThreads / 32];
  const int64_t a = static_cast<int64_t>(blockIdx.x) * kScanBlock + threadIdx.x * kScanItems;
  int c[kScanItems], v = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    c[i] = a + i < n ? counts[a + i] : 0;
    v += c[i];
  }
  int before = 0;
  scan_block_sum(v, sh, &before);
  int run = sums[blockIdx.x] + before;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (a + i < n) rowptr[a + i] = run;
    run += c[i];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) rowptr[n] = total;
}

// eight lanes per row of the original
__global__ void scatter_kernel(int n, const int* __restrict__ rowptr,
                               const int* __restrict__ colind, const int* __restrict__ place,
                               const int* __restrict__ trowptr, int* __restrict__ tcol,
                               int* __restrict__ tsrc) {
  constexpr int VEC = 8;
  const int l = threadIdx.x % VEC;
  for (int64_t r = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) / VEC; r < n;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x / VEC) {
    const int e = rowptr[r + 1];
    for (int k = rowptr[r] + l; k < e; k += VEC) {
      const int pos = trowptr[colind[k]] + place[k];
      tcol[pos] = static_cast<int>(r);
      tsrc[pos] = k;
    }
  }
}

// Each row by column index, one warp per row: an entry's place is the number
// of smaller ones.  That makes the transpose independent of the atomics'
// order.  The entries' original numbers are in the same order as their
// columns, so long rows sort those (through tmp) and look the columns up.
__global__ void sort_rows_kernel(int n, const int* __restrict__ rowptr, int* col, int* src,
                                 int* tmp, int n0, const int* __restrict__ rowptr0) {
  constexpr int M = 4;    // up to 128 entries in registers
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; r < n;
       r += (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5) {
    const int a = rowptr[r], len = rowptr[r + 1] - a;
    if (len <= 32 * M) {
      int c[M], k[M], place[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int i = lane + 32 * m;
        c[m] = i < len ? col[a + i] : 0x7FFFFFFF;
        k[m] = i < len ? src[a + i] : 0;
        place[m] = 0;
      }
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (32 * m >= len) break;
        const int cnt = len - 32 * m < 32 ? len - 32 * m : 32;
        for (int i = 0; i < cnt; ++i) {
          const int o = __shfl_sync(0xffffffffu, c[m], i);
#pragma unroll
          for (int z = 0; z < M; ++z) place[z] += o < c[z];
        }
      }
      __syncwarp();
#pragma unroll
      for (int m = 0; m < M; ++m)
        if (lane + 32 * m < len) {
          col[a + place[m]] = c[m];
          src[a + place[m]] = k[m];
        }
    } else {
      for (int i = lane; i < len; i += 32) {
        const int k = src[a + i];
        int place = 0;
        for (int z = 0; z < len; ++z) place += src[a + z] < k;
        tmp[a + place] = k;
      }
      __syncwarp();
      for (int i = lane; i < len; i += 32) {
        const int k = tmp[a + i];
        int lo = 0, hi = n0 - 1;       // the row that holds entry k: the last with rowptr0 <= k
        while (lo < hi) {
          const int mid = lo + (hi - lo + 1) / 2;
          if (rowptr0[mid] <= k) lo = mid;
          else hi = mid - 1;
        }
        src[a + i] = k;
        col[a + i] = lo;
      }
    }
    __syncwarp();
  }
}

__global__ void gather_values_kernel(int64_t nnz, const int* __restrict__ src,
                                     const double* __restrict__ val, double* __restrict__ out) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
       k += 4 * stride) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = k + u * stride < nnz ? __ldg(val + src[k + u * stride]) : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k + u * stride < nnz) out[k + u * stride] = v[u];
  }
}

}  // namespace

void spmv_newton(const DevCsr& A, const double* x, const double* z,
                 double* y, double theta, double c, double gamma,
                 cudaStream_t st) {
  if (c != 0.0 && z)
    dispatch<0, true, double>(A, A.val, A.sval, x, z, y, theta, c, gamma, st);
  else
    dispatch<0, false, double>(A, A.val, A.sval, x, nullptr, y, theta, 0.0, gamma, st);
}

void spmv_newton32(const DevCsr& A, const float* x, const float* z, float* y,
                   float theta, float c, float gamma, cudaStream_t st) {
  if (c != 0.0f && z)
    dispatch<0, true, float>(A, A.val32, A.sval32, x, z, y, theta, c, gamma, st);
  else
    dispatch<0, false, float>(A, A.val32, A.sval32, x, nullptr, y, theta, 0.0f, gamma, st);
}

void residual(const DevCsr& A, const double* b, const double* x, double* r,
              cudaStream_t st) {
  dispatch<1, false, double>(A, A.val, A.sval, x, b, r, 0.0, 0.0, 1.0, st);
}

void sampled_outer(const DevCsr& A, const double* lam, const double* x,
                   double* dval, cudaStream_t st) {
  int64_t gb = (static_cast<int64_t>(A.n) + 31) / 32;
  const int64_t cap = static_cast<int64_t>(device_sm_count()) * 16;
  const int g = static_cast<int>(gb > cap ? cap : (gb < 1 ? 1 : gb));
  sampled_outer_kernel<<<g, kThreads, 0, st>>>(A.n, A.rowptr, A.colind, lam, x,
                                               dval);
  SG_LAUNCH_CHECK();
}

int64_t transpose_work_ints(const DevCsr& A) {
  const int64_t nb = (static_cast<int64_t>(A.n) + kScanBlock - 1) / kScanBlock;
  return A.n + nb + A.nnz;
}

void csr_transpose(const DevCsr& A, DevCsr& T, int32_t* work, cudaStream_t st) {
  const int nb = static_cast<int>((static_cast<int64_t>(A.n) + kScanBlock - 1) / kScanBlock);
  int* counts = work;
  int* sums = counts + A.n;
  int* place = sums + nb;
  SG_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * A.n, st));
  const int g = device_sm_count() * 8;
  if (A.nnz) {
    count_cols_kernel<<<g, kThreads, 0, st>>>(A.nnz, A.colind, counts, place);
    SG_LAUNCH_CHECK();
  }
  scan_sums_kernel<<<nb, kScanThreads, 0, st>>>(A.n, counts, sums);
  SG_LAUNCH_CHECK();
  scan_sums_scan_kernel<<<1, 1024, 0, st>>>(nb, sums);
  SG_LAUNCH_CHECK();
  scan_apply_kernel<<<nb, kScanThreads, 0, st>>>(A.n, static_cast<int>(A.nnz), counts, sums,
                                                 T.rowptr);
  SG_LAUNCH_CHECK();
  scatter_kernel<<<g, kThreads, 0, st>>>(A.n, A.rowptr, A.colind, place, T.rowptr, T.colind, T.src);
  SG_LAUNCH_CHECK();
  sort_rows_kernel<<<g, kThreads, 0, st>>>(A.n, T.rowptr, T.colind, T.src, place, A.n, A.rowptr);
  SG_LAUNCH_CHECK();
}

void transpose_values(const DevCsr& A, const DevCsr& T, cudaStream_t st) {
  if (!A.nnz) return;
  gather_values_kernel<<<device_sm_count() * 8, kThreads, 0, st>>>(A.nnz, T.src, A.val, T.val);
  SG_LAUNCH_CHECK();
}

namespace {

// slice widths: width[q] = 32 * (longest row of slice q), rows in perm's order
__global__ void sell_width_kernel(int nslices, const int* __restrict__ rowptr,
                                  const int* __restrict__ perm, int* __restrict__ width) {
  const int lane = threadIdx.x & 31;
  for (int64_t q = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; q < nslices;
       q += (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5) {
    const int r = perm[q * 32 + lane];
    const int w = __reduce_max_sync(0xffffffffu, r >= 0 ? rowptr[r + 1] - rowptr[r] : 0);
    if (lane == 0) width[q] = 32 * w;
  }
}

constexpr int kSellWindow = 1024;

// The same with the rows in order (a CTA per window of kSellWindow rows), and
// into *sorted the entries that the slices would hold with the rows of every
// window sorted by length, without sorting them: the slice that holds ranks
// 32 t .. 32 t + 31 is as wide as the row of rank 32 t, so the widths of a
// window add up to sum over l >= 1 of ceil(N_l / 32), N_l the rows of length
// l or more.  N_l comes from a histogram of the lengths up to 1023; what
// longer rows have beyond that is added by their ranks among themselves.
// (A pattern that does not fit either way used to pay for the sort: an
// allocation, kernel, copy and synchronisation more, 0.66 ms at 4.2M rows
// and 0.04 ms at 4096.)
__global__ void __launch_bounds__(kSellWindow)
sell_extent_kernel(int n, int nslices, const int* __restrict__ rowptr, int* __restrict__ width,
                   unsigned long long* sorted) {
  __shared__ int count[kSellWindow];
  __shared__ int longer[kSellWindow];   // lengths above 1023
  __shared__ int nlong;
  __shared__ int above[kSellWindow / 32];
  __shared__ unsigned long long sum[kSellWindow / 32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * kSellWindow + t;
  const int len = r < n ? rowptr[r + 1] - rowptr[r] : 0;
  const int64_t q = r >> 5;
  const int w = __reduce_max_sync(0xffffffffu, len);
  if (lane == 0 && q < nslices) width[q] = 32 * w;
  count[t] = 0;
  if (t == 0) nlong = 0;
  __syncthreads();
  const int bin = min(len, kSellWindow - 1);
  const unsigned same = __match_any_sync(0xffffffffu, bin);
  if (lane == __ffs(same) - 1) atomicAdd(&count[bin], __popc(same));
  if (len >= kSellWindow) longer[atomicAdd(&nlong, 1)] = len;
  __syncthreads();
  // N_t: rows of length t or more
  int v = count[t];
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_down_sync(0xffffffffu, v, off);
    if (lane + off < 32) v += o;
  }
  if (lane == 0) above[warp] = v;
  __syncthreads();
  for (int k = warp + 1; k < kSellWindow / 32; ++k) v += above[k];
  unsigned long long s = t >= 1 ? static_cast<unsigned long long>((v + 31) / 32) : 0;
  if (t < nlong) {
    const int mine = longer[t];
    int rank = 0;
    for (int k = 0; k < nlong; ++k) rank += longer[k] > mine || (longer[k] == mine && k < t);
    if (rank % 32 == 0) s += static_cast<unsigned long long>(mine - (kSellWindow - 1));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) sum[warp] = s;
  __syncthreads();
  if (t == 0) {
    unsigned long long total = 0;
    for (int k = 0; k < kSellWindow / 32; ++k) total += sum[k];
    atomicAdd(sorted, 32 * total);
  }
}

// Rows of every window of kSellWindow sorted by length, longest first, equal
// ones in row order: a row's place is the number of rows before it.
// Positions past the last row hold -1.

__global__ void __launch_bounds__(kSellWindow)
sell_sort_kernel(int n, const int* __restrict__ rowptr, int64_t positions,
                 int* __restrict__ perm) {
  __shared__ int key[kSellWindow];
  const int64_t w0 = static_cast<int64_t>(blockIdx.x) * kSellWindow;
  const int t = threadIdx.x;
  const int64_t r = w0 + t;
  // longer rows and, among equal ones, earlier rows have the larger key;
  // lengths beyond 2^20 are taken as equal
  int mine = -1 - t;
  if (r < n) mine = min(rowptr[r + 1] - rowptr[r], 1 << 20) * kSellWindow + (kSellWindow - 1 - t);
  key[t] = mine;
  __syncthreads();
  int place = 0;
#pragma unroll 8
  for (int i = 0; i < kSellWindow; ++i) place += key[i] > mine;
  if (w0 + place < positions) perm[w0 + place] = r < n ? static_cast<int>(r) : -1;
}

// one thread per (padded) row: entry j of the row at position 32q + l ->
// sptr[q] + 32 j + l
template <bool COLS>
__global__ void sell_fill_kernel(int n, int64_t rows32, const int* __restrict__ rowptr,
                                 const int* __restrict__ colind,
                                 const double* __restrict__ val, const int* __restrict__ perm,
                                 const int* __restrict__ sptr, int* __restrict__ scol,
                                 double* __restrict__ sval) {
  for (int64_t pos = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; pos < rows32;
       pos += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t q = pos >> 5;
    const int base = sptr[q] + static_cast<int>(pos & 31);
    const int w = (sptr[q + 1] - sptr[q]) >> 5;
    const int64_t r = perm ? perm[pos] : (pos < n ? pos : -1);
    const int a = r >= 0 ? rowptr[r] : 0;
    const int len = r >= 0 ? rowptr[r + 1] - a : 0;
    for (int j = 0; j < w; ++j) {
      const int k = base + 32 * j;
      if (j < len) {
        if (COLS) scol[k] = colind[a + j];
        sval[k] = val[a + j];
      } else {
        if (COLS) scol[k] = -1;
        sval[k] = 0.0;
      }
    }
  }
}

// per slice (one warp): the smallest stored column (0 for an all-padding
// slice), and a flag when the slice's columns span 65535 or more
__global__ void sell_base_kernel(int nslices, const int* __restrict__ sptr,
                                 const int* __restrict__ scol, int* __restrict__ sbase,
                                 int* __restrict__ wide) {
  const int lane = threadIdx.x & 31;
  for (int64_t q = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; q < nslices;
       q += (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5) {
    int lo = 0x7FFFFFFF, hi = -1;
    const int e = sptr[q + 1];
    for (int k = sptr[q] + lane; k < e; k += 32) {
      const int c = scol[k];
      if (c >= 0) {
        lo = min(lo, c);
        hi = max(hi, c);
      }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (hi < 0) lo = hi = 0;
    if (lane == 0) {
      sbase[q] = lo;
      if (hi - lo >= 0xFFFF) atomicOr(wide, 1);
    }
  }
}

// 16-bit offsets of every stored entry from its slice's base
__global__ void sell_off_kernel(int64_t rows32, const int* __restrict__ sptr,
                                const int* __restrict__ scol, const int* __restrict__ sbase,
                                uint16_t* __restrict__ soff) {
  for (int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; r < rows32;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t q = r >> 5;
    const int w = (sptr[q + 1] - sptr[q]) >> 5;
    const int b = sbase[q];
    for (int j = 0; j < w; ++j) {
      const int k = sptr[q] + static_cast<int>(r & 31) + 32 * j;
      const int c = scol[k];
      soff[k] = c >= 0 ? static_cast<uint16_t>(c - b) : static_cast<uint16_t>(0xFFFF);
    }
  }
}

void free_sell(DevCsr& A) {
  if (A.sptr) cudaFree(A.sptr);
  if (A.scol) cudaFree(A.scol);
  if (A.sval) cudaFree(A.sval);
  if (A.sval32) cudaFree(A.sval32);
  if (A.sbase) cudaFree(A.sbase);
  if (A.soff) cudaFree(A.soff);
  if (A.sperm) cudaFree(A.sperm);
  A.sptr = A.scol = A.sbase = A.sperm = nullptr;
  A.soff = nullptr;
  A.sval = nullptr;
  A.sval32 = nullptr;
  A.nslices = 0;
  A.sell_nnz = 0;
}

// The 16-bit column offsets when every slice fits them; left null otherwise.
void build_sell_offsets(DevCsr& A, cudaStream_t st) {
  int* wide = nullptr;
  SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&wide), sizeof(int)));
  int hwide = 0;
  try {
    SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&A.sbase), sizeof(int) * A.nslices));
    SG_CUDA(cudaMemsetAsync(wide, 0, sizeof(int), st));
    sell_base_kernel<<<device_sm_count() * 8, kThreads, 0, st>>>(A.nslices, A.sptr, A.scol,
                                                                 A.sbase, wide);
    SG_LAUNCH_CHECK();
    SG_CUDA(cudaMemcpyAsync(&hwide, wide, sizeof(int), cudaMemcpyDeviceToHost, st));
    SG_CUDA(cudaStreamSynchronize(st));
    if (!hwide) {
      SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&A.soff), sizeof(uint16_t) * A.sell_nnz));
      sell_off_kernel<<<device_sm_count() * 8, kThreads, 0, st>>>(
          static_cast<int64_t>(A.nslices) * 32, A.sptr, A.scol, A.sbase, A.soff);
      SG_LAUNCH_CHECK();
      SG_CUDA(cudaStreamSynchronize(st));
    }
  } catch (...) {
    cudaFree(wide);
    throw;
  }
  cudaFree(wide);
  if (!A.soff) {
    cudaFree(A.sbase);
    A.sbase = nullptr;
  }
}

}  // namespace

void build_sell(DevCsr& A, cudaStream_t st) {
  free_sell(A);
  if (A.n <= 0 || A.nnz <= 0) return;
  const int nsl = static_cast<int>((static_cast<int64_t>(A.n) + 31) / 32);
  const int64_t pos = static_cast<int64_t>(nsl) * 32;
  const unsigned windows = static_cast<unsigned>((pos + kSellWindow - 1) / kSellWindow);
  // on the device and the host: the entries with sorted rows (64 bits), widths
  const size_t words = 2 + static_cast<size_t>(nsl);
  std::vector<int> hw(words);
  std::vector<int> hp(static_cast<size_t>(nsl) + 1);
  int64_t tot = 0;
  int* buf = nullptr;
  // keep SELL only when the padding is modest and the offsets fit int32
  auto fits = [&](int64_t entries) {
    return entries < (int64_t(1) << 31) - 1 &&
           entries <= A.nnz + A.nnz / 5 + 32 * static_cast<int64_t>(nsl);
  };
  auto take_widths = [&] {
    SG_CUDA(cudaMemcpyAsync(hw.data(), buf, sizeof(int) * words, cudaMemcpyDeviceToHost, st));
    SG_CUDA(cudaStreamSynchronize(st));
    tot = 0;
    for (int q = 0; q < nsl; ++q) {
      hp[q] = static_cast<int>(tot < (int64_t(1) << 31) ? tot : 0);
      tot += hw[2 + q];
    }
  };
  SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&buf), sizeof(int) * words));
  bool keep = false;
  try {
    SG_CUDA(cudaMemsetAsync(buf, 0, sizeof(unsigned long long), st));
    sell_extent_kernel<<<windows, kSellWindow, 0, st>>>(A.n, nsl, A.rowptr, buf + 2,
                                                        reinterpret_cast<unsigned long long*>(buf));
    SG_LAUNCH_CHECK();
    take_widths();
    keep = fits(tot);
    int64_t sorted = 0;
    std::memcpy(&sorted, hw.data(), sizeof(sorted));
    if (!keep && fits(sorted)) {
      SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&A.sperm), sizeof(int) * pos));
      sell_sort_kernel<<<windows, kSellWindow, 0, st>>>(A.n, A.rowptr, pos, A.sperm);
      SG_LAUNCH_CHECK();
      sell_width_kernel<<<device_sm_count() * 8, kThreads, 0, st>>>(nsl, A.rowptr, A.sperm, buf + 2);
      SG_LAUNCH_CHECK();
      take_widths();
      keep = fits(tot);
    }
  } catch (...) {
    cudaFree(buf);
    free_sell(A);
    throw;
  }
  cudaFree(buf);
  if (!keep) {
    free_sell(A);
    return;
  }
  hp[nsl] = static_cast<int>(tot);
  try {
    SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&A.sptr), sizeof(int) * (nsl + 1)));
    SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&A.scol), sizeof(int) * tot));
    SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&A.sval), sizeof(double) * tot));
    SG_CUDA(cudaMemcpyAsync(A.sptr, hp.data(), sizeof(int) * (nsl + 1), cudaMemcpyHostToDevice, st));
    A.nslices = nsl;
    A.sell_nnz = tot;
    const int64_t rows32 = static_cast<int64_t>(nsl) * 32;
    sell_fill_kernel<true><<<device_sm_count() * 8, kThreads, 0, st>>>(
        A.n, rows32, A.rowptr, A.colind, A.val, A.sperm, A.sptr, A.scol, A.sval);
    SG_LAUNCH_CHECK();
    SG_CUDA(cudaStreamSynchronize(st));  // the host offsets go out of scope
    build_sell_offsets(A, st);
  } catch (...) {
    free_sell(A);
    throw;
  }
}

void sell_refill_values(const DevCsr& A, cudaStream_t st) {
  if (!A.sptr) return;
  const int64_t rows32 = static_cast<int64_t>(A.nslices) * 32;
  sell_fill_kernel<false><<<device_sm_count() * 8, kThreads, 0, st>>>(
      A.n, rows32, A.rowptr, A.colind, A.val, A.sperm, A.sptr, nullptr, A.sval);
  SG_LAUNCH_CHECK();
}

namespace {

__global__ void colnorm_kernel(int n, const int* __restrict__ rowptr,
                               const double* __restrict__ val, double* __restrict__ d) {
  for (int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; r < n;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    double ss = 0.0;
    for (int k = rowptr[r]; k < rowptr[r + 1]; ++k) ss = fma(val[k], val[k], ss);
    d[r] = ss > 0.0 ? 1.0 / sqrt(ss) : 1.0;
  }
}

__global__ void scale_cols_kernel(int64_t cnt, const int* __restrict__ col,
                                  const double* __restrict__ val,
                                  const double* __restrict__ d, double* __restrict__ out) {
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < cnt;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = col[k];
    out[k] = c >= 0 ? val[k] * d[c] : 0.0;
  }
}

__global__ void diag_kernel(int64_t n, const double* __restrict__ d,
                            const double* x, double* y, int div) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    y[i] = div ? x[i] / d[i] : x[i] * d[i];
}

}  // namespace

namespace {

// A grid barrier that cannot complete: it expects one block more than the
// grid has, so every block's bounded wait runs out and sets err.
__global__ void barrier_probe_kernel(unsigned* bar, int* err, uint64_t limit_ns) {
  grid_barrier(bar, gridDim.x + 1, err, limit_ns);
}

}  // namespace

bool probe_grid_barrier_timeout(uint64_t limit_ns, cudaStream_t st) {
  unsigned* bar = nullptr;
  SG_CUDA(cudaMalloc(reinterpret_cast<void**>(&bar), 256));
  bool timed_out = false;
  try {
    SG_CUDA(cudaMemsetAsync(bar, 0, 256, st));
    int* err = reinterpret_cast<int*>(bar + 48);
    barrier_probe_kernel<<<2, 32, 0, st>>>(bar, err, limit_ns);
    SG_LAUNCH_CHECK();
    int host = 0;
    SG_CUDA(cudaMemcpyAsync(&host, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    SG_CUDA(cudaStreamSynchronize(st));
    timed_out = host != 0;
  } catch (...) {
    cudaFree(bar);
    throw;
  }
  SG_CUDA(cudaFree(bar));
  return timed_out;
}

void column_scale_factors(const DevCsr& AT, double* d, cudaStream_t st) {
  colnorm_kernel<<<device_sm_count() * 8, kThreads, 0, st>>>(AT.n, AT.rowptr, AT.val, d);
  SG_LAUNCH_CHECK();
}

void scale_columns(const DevCsr& A, const double* d, DevCsr& E, cudaStream_t st) {
  const int g = device_sm_count() * 8;
  if (A.nnz) {
    scale_cols_kernel<<<g, kThreads, 0, st>>>(A.nnz, A.colind, A.val, d, E.val);
    SG_LAUNCH_CHECK();
  }
  if (A.sptr && E.sval) {
    scale_cols_kernel<<<g, kThreads, 0, st>>>(A.sell_nnz, A.scol, A.sval, d, E.sval);
    SG_LAUNCH_CHECK();
  }
}

void row_extent(const DevCsr& A, unsigned long long* out, cudaStream_t st) {
  SG_CUDA(cudaMemsetAsync(out, 0, 2 * sizeof(unsigned long long), st));
  int64_t blocks = (static_cast<int64_t>(A.n) * 8 + kThreads - 1) / kThreads;
  const int64_t cap = static_cast<int64_t>(device_sm_count()) * 8;
  if (blocks > cap) blocks = cap;
  row_extent_kernel<<<static_cast<unsigned>(blocks), kThreads, 0, st>>>(A.n, A.rowptr, A.val, out);
  SG_LAUNCH_CHECK();
}

// The fixed-point pre-pass step holds an entry of a vector to about 2^-58 of
// its CTA's largest one, FP64 to 2^-53 of itself.  The loss in v_j comes back
// multiplied by A's entries, so it shows in H where an entry of A is large
// against the product's size.  If the largest magnitudes of all rows lie
// within a factor f, that cannot be: following each row's largest entry from
// row to row ends in a cycle, so |A| restricted to any set of rows that is
// closed under it has a spectral radius of at least max|a| / f.  D B D^-1
// with random powers of two in D, the 32^2 and 150 x 101 stencils, 20 and 8
// steps, the largest error of H relative to its column's largest entry,
// fixed point against FP64, by f:
//   1: 5e-15, 5e-15     2^2: 5e-15, 1e-14    2^4: 5e-15, 5e-15
//   2^6: 1e-14, 7e-15   2^8: 5e-14, 1e-14    2^18: 4e-11, 9e-15
// so the line lies at 16 (a matrix of zero rows, infinities or NaN is beyond
// it too).  Rows or columns scaled alone lose nothing in fixed point up to
// 2^50; they go to FP64 by this rule all the same.
bool rows_are_even(const unsigned long long* out) {
  const unsigned long long hi = out[0], lo = ~out[1];
  if (lo == 0 || hi >= 0x7FF0000000000000ull) return false;
  double a, b;
  std::memcpy(&a, &hi, sizeof(a));
  std::memcpy(&b, &lo, sizeof(b));
  return a <= 16.0 * b;
}

void diag_apply(int64_t n, const double* d, const double* x, double* y, bool div,
                cudaStream_t st) {
  if (n <= 0) return;
  diag_kernel<<<device_sm_count() * 8, kThreads, 0, st>>>(n, d, x, y, div ? 1 : 0);
  SG_LAUNCH_CHECK();
}

int64_t prepass_red_doubles(int k) {
  const int64_t a = ic_red_doubles(device_sm_count());
  const int64_t b = fixed_red_doubles(device_sm_count(), k);
  return a > b ? a : b;
}

void arnoldi_step(const DevCsr& A, double* V, int64_t ld, int j, int k, double* xv, double* H,
                  int ldh, double* wn, double* red, int red_cap, unsigned* bar,
                  int* err, cudaStream_t st) {
  if (A.sptr && A.sval && !A.sperm)   // (the fused steps walk the slices in row order)
    launch_arnoldi_step<double, true>(A, A.sval, V, ld, j, k, xv, H, ldh, wn, red, red_cap, bar, err, st);
  else
    launch_arnoldi_step<double, false>(A, A.val, V, ld, j, k, xv, H, ldh, wn, red, red_cap, bar, err, st);
}

void arnoldi_step32(const DevCsr& A, float* V, int64_t ld, int j, double* H,
                    int ldh, double* wn, double* red, int red_cap, unsigned* bar,
                    int* err, cudaStream_t st) {
  float* none = nullptr;
  if (A.sptr && A.sval32 && !A.sperm)
    launch_arnoldi_step<float, true>(A, A.sval32, V, ld, j, 0, none, H, ldh, wn, red, red_cap, bar, err, st);
  else
    launch_arnoldi_step<float, false>(A, A.val32, V, ld, j, 0, none, H, ldh, wn, red, red_cap, bar, err, st);
}

}  // namespace sg
