// MinSR Gram matrix T = Obar Obar^T at FP64 accuracy on the 5th-generation tensor cores (tcgen05,
// sm_103a) by error-free slicing (Ootomo, Ozaki and Yokota, "DGEMM on integer matrix
// multiplication unit", 2024; Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication", 2012): GB300's FP64 pipes run at 1/64 of the FP32 rate, its BF16 tensor
// cores at 2000 times the FP64 rate.
//
// Slices.  Row i of Obar is scaled by a power of two 2^-e_i, above its largest modulus and such that
// its squared norm is below 2^8, and written in fixed point with NS = 7 signed 8-bit digits,
//   x = 2^e_i sum_p d_p 2^(-7 - 8 p) + err,   |d_p| <= 128,   |err| <= 2^(e_i - 56),
// each digit an integer that BF16 holds exactly.  T_ij = 2^(e_i + e_j) sum_d 2^(-14 - 8 d) v_d with
// v_d = sum_{p + q = d} sum_k d_p(i, k) d_q(j, k); the terms with d >= NS (below 2^-56) are dropped.
//
// Exactness.  Over a chunk of CK = 32 columns |v_d| <= 7 * 32 * 2^14 < 2^22: every partial sum the
// FP32 accumulators in tensor memory ever hold is an integer below 2^24, so the products and sums
// are exact.  After every chunk the epilogue warps read the seven v_d, turn them into integers
// (one FP32 add of 1.5 * 2^23 puts the integer in the low mantissa bits) and add them to 64-bit
// fixed-point sums in registers with lsb 2^-54 of the scaled rows; |T_ij| 2^(54 - e_i - e_j) < 2^62 by
// Cauchy-Schwarz.  Only the digits below that lsb round, once a chunk (half up and half down on alternate
// chunks of the columns).  Integer addition is associative: the partial sums of tiles that are split
// over several CTAs along K, or of panels of columns, are added with 64-bit integer atomics and give the
// same bits in any order and for any split.
//
// Scale.  With one lsb for the whole matrix taken from the largest row norm, a row of equal entries
// beside rows with one large entry (norms 300 times apart at 80 000 columns) left those rows' products
// 37 bits.  Now the norms are at most 16 to 32 apart (one large entry is at least 1/2): what is lost is the
// low end of a flat row's digits, 2^-56 of its scale.  Rows of norm 8 to 16 also keep the dropped products
// (1e-15 at 21 632 columns for a norm of 1) below the rounding of the result.  Largest error over |a||b| of
// 16 x 16 entries against long double at 21 632 columns, before -> now: one flat row among spiky ones
// 2.4e-13 -> 5.1e-15, spiky rows 8.4e-15 -> 5.1e-15, Gaussian rows 0.9e-16 -> 1.2e-16, the rounding of the
// result (an FP64 multiply-add sum in order: 8.2e-15, 8.2e-15, 1.1e-14).
//
// Measured on the whole MinSR step (one GB300): 4096 x 21 632 from 118.4 ms with the float-float
// FP32 Gram (85.2 ms of it) to 44.2 ms, 1000 x 3528 from 8.28 ms with the FP64 FMA Gram (3.9 ms)
// to 4.71 ms (the Gram matrix itself 10.9 and 0.18 ms); dtheta against 64-bit linear algebra 3.0e-13 -> 3.0e-15 and 4.8e-15 -> 1.7e-15.
// tests/test_gpu_gram_slices.py holds the error bound against an extended-precision sum.
#include <cuda_bf16.h>

#include "peps_kernels.cuh"
#include "peps_slices.cuh"

namespace peps {
namespace {

constexpr int FL = 54;  // fixed-point sums: lsb 2^-FL of the scaled rows (that of d = 4, 5)
constexpr int NL = 8;   // squared norms of the scaled rows are below 2^NL: |T_ij| 2^FL < 2^62

// a += w 2^32 and a += w m, one instruction each (written as 64-bit shifts and sums the 64 sums of a
// thread spill: 11.8 -> 15.9 ms for the Gram matrix of 4096 x 21 632)
static_assert(FL == 54, "the weights of the digit products");
__device__ __forceinline__ void add_high(long long& a, int w) {
  asm("{\n .reg .b32 l, h;\n mov.b64 {l, h}, %0;\n add.s32 h, h, %1;\n mov.b64 %0, {l, h};\n}\n" : "+l"(a) : "r"(w));
}
__device__ __forceinline__ void mad_wide(long long& a, int w, int m) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(w), "r"(m));
}

// Row scales: rowE[r] = the largest biased exponent of the row (at least 1: the exponent of a
// subnormal), raised until the scaled squared norm is below 2^NL, or ROW_NONFINITE when an entry is Inf
// or NaN.  One CTA per row; the second pass finds the row in L2.
__global__ void __launch_bounds__(256) k_slice_rows(const double* __restrict__ A, long long K, int* rowE) {
  __shared__ int sE[8];
  __shared__ float sN[8];
  const unsigned long long* x = reinterpret_cast<const unsigned long long*>(A) + (size_t)blockIdx.x * K;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int e = 1;
#pragma unroll 8
  for (long long k = threadIdx.x; k < K; k += 256) e = max(e, (int)(x[k] >> 52) & 0x7ff);
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) sE[warp] = e;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) e = max(e, sE[w]);
  float n = 0.f;
  if (e < 2047) {
#pragma unroll 8
    for (long long k = threadIdx.x; k < K; k += 256) {
      const unsigned long long b = x[k];
      const int sh = e - max((int)(b >> 52) & 0x7ff, 1);
      // |x| / 2^(e - 1022) with 23 mantissa bits; entries below 2^-60 of the scale are left out
      const float v = (sh < 60 && (b << 1)) ? __int_as_float(((126 - sh) << 23) | (int)((b >> 29) & 0x7fffff)) : 0.f;
      n = fmaf(v, v, n);
    }
  }
  n = warp_sum(n);
  if (lane == 0) sN[warp] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) n += sN[w];
    int ex = 0;
    frexpf(n * 1.001f, &ex);  // the squared norm is below 2^ex (1.001: the truncated mantissas and the sum's rounding)
    rowE[blockIdx.x] = e < 2047 ? e + (ex > NL ? (ex - NL + 1) / 2 : 0) : ROW_NONFINITE;
  }
}

// Digits of the columns [k0, k0 + kw) of A into D[p][row][k] (rows padded with zeros to Npad,
// columns to Kpad).  A thread takes eight columns of one row: integer arithmetic on the bits of
// the doubles (the FP64 pipes would be the limit), one 16-byte store per digit.
__global__ void __launch_bounds__(256) k_slice_digits(const double* __restrict__ A, int Ns, long long K, long long k0,
                                                      int kw, int Npad, int Kpad, const int* __restrict__ rowE,
                                                      __nv_bfloat16* __restrict__ D) {
  const int nv = Kpad / 8;
  const long long total = (long long)Npad * nv;
  const size_t plane = (size_t)Npad * Kpad;
  for (long long o = blockIdx.x * 256ll + threadIdx.x; o < total; o += gridDim.x * 256ll) {
    const int r = (int)(o / nv), kb = (int)(o - (long long)r * nv) * 8;
    const int E = r < Ns ? rowE[r] : ROW_NONFINITE;
    const unsigned long long* x = reinterpret_cast<const unsigned long long*>(A) + (size_t)(r < Ns ? r : 0) * K + k0 + kb;
    uint32_t w[NS][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const unsigned long long b = (E >= 0 && kb + j < kw) ? x[j] : 0ull;
      put_digits(fixed_point(b, E), j, w);
    }
#pragma unroll
    for (int p = 0; p < NS; ++p)
      *reinterpret_cast<uint4*>(D + p * plane + (size_t)r * Kpad + kb) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
  }
}

// One CTA per (tile, K part): a 128 x 128 tile on or below the diagonal over the chunks [c0, c1).
// Warp 8 loads (two TMA boxes of 32 columns x 128 rows x 7 digits per chunk, double buffered),
// warp 9 issues the 28 digit products of a chunk as four units (d = 0..1, 2..3, 4..5, 6), each
// unit into one of two pairs of 128-column accumulators, so that warps 0..7 drain one unit while
// the tensor cores run the next.  256 threads hold 64 sums each (warp w: tensor-memory lanes
// 32 (w mod 4).., columns 64 (w / 4)..).
//   The MMAs of a chunk take 56 x 64 = 3584 tensor cycles and its epilogue about 22 instructions
// per element = 2800 issue cycles on the four schedulers: the tile shape balances the two, and
// shared memory feeds both operands of a 128 x 128 x 16 MMA at its full 128 bytes per cycle.  Measured, the
// tensor pipe is active 42 % of the time (1024 x 21 632; 50 % of the measured BF16 peak at 4096 rows): the
// epilogue's eight warps wait for their tensor-memory loads.
// cb: the chunk of the matrix's columns that the map's first one is.
__global__ void __launch_bounds__(SL_THREADS, 1) k_gram_sl(const __grid_constant__ CUtensorMap map, int full, int ks,
                                                           int nchunk, int cb, int Ns, unsigned long long* Tm, int ld,
                                                           int* err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* ring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar[SSTAGES], empty_bar[SSTAGES], ufull[2], uempty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int t, c0 = 0, c1 = nchunk;
  if ((int)blockIdx.x < full) {
    t = blockIdx.x;
  } else {
    const int r = blockIdx.x - full, part = r % ks;
    t = full + r / ks;
    c0 = (int)((long long)nchunk * part / ks);
    c1 = (int)((long long)nchunk * (part + 1) / ks);
  }
  int ti = 0;
  while (t >= ti + 1) { t -= ti + 1; ++ti; }
  const int tj = t;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
      mbar_init(&ufull[s], 1);
      mbar_init(&uempty[s], EPI_WARPS);
    }
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == EPI_WARPS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  const int nc = c1 - c0;
  if (warp == EPI_WARPS) {
    if (lane == 0) {
      int issued = 0;
      for (int c = 0; c < nc; ++c) {
        const int s = c & 1;
        if (c >= SSTAGES && !wait_ok(&empty_bar[s], ((c >> 1) - 1) & 1, &failed)) break;
        uint8_t* st = ring + (size_t)s * SSTAGE;
        mbar_expect_tx(&full_bar[s], SSTAGE);
        tma_load_3d(st, &map, (c0 + c) * CK, ti * SM_, 0, &full_bar[s]);
        tma_load_3d(st + SOPND, &map, (c0 + c) * CK, tj * SM_, 0, &full_bar[s]);
        issued = c + 1;
      }
      // the loads of the last stages have landed before the CTA may leave (bounded)
      for (int c = issued > SSTAGES ? issued - SSTAGES : 0; c < issued; ++c)
        for (int i = 0; i < (1 << 16) && !mbar_try(&full_bar[c & 1], (c >> 1) & 1); ++i) {}
    }
  } else if (warp == EPI_WARPS + 1) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int c = 0; c < nc && ok; ++c) {
        const int s = c & 1;
        if (!wait_ok(&full_bar[s], (c >> 1) & 1, &failed)) break;
        const uint32_t a0 = smem_u32(ring + (size_t)s * SSTAGE), b0 = a0 + SOPND;
        for (int u = 0; u < 4; ++u, ++g) {
          const int slot = g & 1;
          if (g >= 2 && !wait_ok(&uempty[slot], ((g >> 1) - 1) & 1, &failed)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;");
          for (int d = 2 * u; d < 2 * u + 2 && d < NS; ++d) {
            const uint32_t acc = tmem + slot * 256 + (d & 1) * 128;
            for (int p = 0; p <= d; ++p) {
              const uint64_t da = desc64(a0 + p * STILE), db = desc64(b0 + (d - p) * STILE);
              mma_sl(acc, da, db, p > 0);
              mma_sl(acc, da + 2, db + 2, 1u);  // 16 bf16 = 32 bytes further along K
            }
          }
          mma_commit(&ufull[slot]);
        }
        // (only where the loader waits for it: nothing may arrive on a barrier after the CTA has left)
        if (ok && c + SSTAGES < nc) mma_commit(&empty_bar[s]);
      }
    }
  } else {
    const uint32_t tw = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 64;
    long long acc[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0;
    bool ok = true;
    for (int c = 0; c < nc; ++c) {
      const int half = (1 << (61 - FL)) - ((cb + c0 + c) & 1);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t slot = u & 1, par = (2 * c + (u >> 1)) & 1;
        ok = ok && wait_ok(&ufull[slot], par, &failed);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t ta = tw + slot * 256;
#pragma unroll
        for (int cc = 0; cc < 64; cc += 16) {
          float va[16], vb[16];
          tmem_ld16(ta + cc, va);
          if (u < 3) tmem_ld16(ta + 128 + cc, vb);
          tmem_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int a = f2i_exact(va[j]);  // of weight 2^(-14 - 16 u)
            if (u < 3) {
              const int w = a * 256 + f2i_exact(vb[j]);  // |w| < 2^31
              if (u == 0) add_high(acc[cc + j], w);
              if (u == 1) mad_wide(acc[cc + j], w, 1 << (FL - 38));
              if (u == 2) mad_wide(acc[cc + j], w, 1);
            } else {
              mad_wide(acc[cc + j], (a + half) >> (62 - FL), 1);
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) mbar_arrive(&uempty[slot]);
      }
      if (!ok) break;
    }
    if (ok && !failed) {
      const int row = ti * SM_ + (warp & 3) * 32 + lane, col0 = tj * SM_ + (warp >> 2) * 64;
      if (row < Ns) {
#pragma unroll
        for (int j = 0; j < 64; ++j)
          if (col0 + j <= row) atomicAdd(Tm + (size_t)row * ld + col0 + j, (unsigned long long)acc[j]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (failed && threadIdx.x == 0) atomicExch(err, 1);
  if (warp == EPI_WARPS) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// The fixed-point sums of the lower triangle, in place, to T_ij = sum 2^(e_i + e_j - FL) in double,
// and the upper triangle mirrored from it (32 x 32 tiles through shared memory).  Rows with a
// non-finite entry give NaN.
__global__ void __launch_bounds__(256) k_slice_finish(double* T, int Ns, int ld, const int* __restrict__ rowE) {
  __shared__ double tile[32][33];
  int t = blockIdx.x, bi = 0;
  bi = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((long long)(bi + 1) * (bi + 2) / 2 <= t) ++bi;
  while ((long long)bi * (bi + 1) / 2 > t) --bi;
  const int bj = t - (int)((long long)bi * (bi + 1) / 2);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int c = bj * 32 + tx;
  const int ec = c < Ns ? rowE[c] : 0;
  for (int k = ty; k < 32; k += 8) {
    const int r = bi * 32 + k;
    double v = 0.0;
    if (r < Ns && c <= r) {
      const int er = rowE[r];
      v = scalbn((double)__double_as_longlong(T[(size_t)r * ld + c]), er + ec - FL - 2044);
      if (er < 0 || ec < 0) v = __longlong_as_double(0x7ff8000000000000ll);
      T[(size_t)r * ld + c] = v;
    }
    tile[k][tx] = v;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    const int r = bj * 32 + k, cu = bi * 32 + tx;  // transposed position (upper triangle)
    if (cu < Ns && r < cu) T[(size_t)r * ld + cu] = tile[tx][k];
  }
}

long long round_up(long long x, long long a) { return (x + a - 1) / a * a; }

// Most bytes of digits held at once: above it the columns are sliced and multiplied in panels
// (16384 rows x 80 000 columns would need 18 GB; a 2 GB panel of 9152 columns costs one more
// round of atomics per panel, 0.1 % of its products).
constexpr size_t SLICE_CAP = 2ull << 30;

}  // namespace

size_t gram_sl_bytes(int Ns, long long K) {
  const size_t rows = (size_t)round_up(Ns, SM_), head = (size_t)round_up(4ll * Ns, 1024);
  const size_t all = rows * (size_t)round_up(K > 0 ? K : 1, CK) * 2 * NS;
  const size_t least = rows * CK * 2 * NS;
  return head + (all < SLICE_CAP ? all : (SLICE_CAP > least ? SLICE_CAP : least));
}

cudaError_t launch_gram_sl(const double* A, int Ns, long long K, void* ws, size_t ws_bytes, double* Tm, int ld, int* err,
                           cudaStream_t s, long long* launches) {
  EncodeTiled enc = get_encode();
  if (!enc) return cudaErrorNotSupported;
  const int Npad = (int)round_up(Ns, SM_);
  const size_t head = (size_t)round_up(4ll * Ns, 1024);
  int* rowE = (int*)ws;
  __nv_bfloat16* D = (__nv_bfloat16*)((char*)ws + head);
  const long long fit = (long long)((ws_bytes - head) / ((size_t)Npad * 2 * NS)) / CK * CK;  // columns of a panel
  if (fit < CK) return cudaErrorInvalidValue;
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  k_slice_rows<<<Ns, 256, 0, s>>>(A, K, rowE);
  const size_t smem = (size_t)SSTAGES * SSTAGE + 1024;
  if ((e = cudaFuncSetAttribute(k_gram_sl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  const int nt = Npad / SM_, tiles = nt * (nt + 1) / 2;
  long long nl = 1;
  for (long long k0 = 0; k0 < K; k0 += fit) {
    const int kw = (int)(K - k0 < fit ? K - k0 : fit), Kpad = (int)round_up(kw, CK), nchunk = Kpad / CK;
    const long long vecs = (long long)Npad * (Kpad / 8);
    k_slice_digits<<<(int)(vecs / 256 < 16 * nsm ? vecs / 256 + 1 : 16 * nsm), 256, 0, s>>>(A, Ns, K, k0, kw, Npad, Kpad,
                                                                                        rowE, D);
    CUtensorMap map;
    const cuuint64_t dims[3] = {(cuuint64_t)Kpad, (cuuint64_t)Npad, NS};
    const cuuint64_t strides[2] = {(cuuint64_t)Kpad * 2, (cuuint64_t)Kpad * 2 * Npad};
    const cuuint32_t box[3] = {CK, SM_, NS}, estr[3] = {1, 1, 1};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, D, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    // whole waves of tiles take all of K (the CTAs of a wave walk K together and share the
    // operands through L2); the tiles of the last, partial wave are split along K into the
    // number of parts that fills the SMs best
    const int full = tiles / nsm * nsm, rest = tiles - full;
    int ks = 1;
    if (rest) {
      const int kmax = nchunk < 4 ? 1 : (nchunk / 4 < 32 ? nchunk / 4 : 32);
      double best = 1e30;
      for (int q = 1; q <= kmax; ++q) {
        const double waves = (double)((rest * q + nsm - 1) / nsm) / q + 0.002 * q;
        if (waves < best) { best = waves; ks = q; }
      }
    }
    k_gram_sl<<<full + rest * ks, SL_THREADS, smem, s>>>(map, full, ks, nchunk, (int)(k0 / CK), Ns,
                                                         (unsigned long long*)Tm, ld, err);
    nl += 2;
  }
  const long long nb = (Ns + 31) / 32;
  k_slice_finish<<<(int)(nb * (nb + 1) / 2), 256, 0, s>>>(Tm, Ns, ld, rowE);
  *launches = nl + 1;
  return cudaGetLastError();
}

}  // namespace peps
