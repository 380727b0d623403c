// (T + lambda I)^-1 ebar by a blocked right-looking Cholesky factorisation in FP64 (rcond == 0; solve
// modes 0 and 2, and the fallback of mode 1).  GB300's FP64 pipes issue one warp instruction per
// 64 cycles on each SM sub-partition, so the n^3 / 3 of the trailing updates go to the tensor
// cores (digit products of peps_slices.cuh, exact up to 2^-55 of the scaled rows), and what stays
// in FP64 is spread over the sub-partitions:
//   k_chol_diag    the 64 x 64 diagonal block, one CTA, a ninth warp working one pivot ahead;
//   k_chol_panel   the rows below it by substitution (4 to 16 lanes share a row, so that every
//                  sub-partition of the GPU has rows), and the digits of the solved rows;
//   k_chol_update  A_ij -= X_i X_j^T on 128 x 128 tiles, one kernel per panel.
// The triangular solves multiply by the inverses of the diagonal blocks (formed once): a 64-step
// substitution on one warp was most of each of their 2 n / 64 dependent launches.
// Measured (one GB300, whole MinSR step): 4096 x 21 632 with refinement (solve = 2) 44.2 -> 27.8 ms
// against a float-float factor on the FP32 pipes, 1000 x 3528 (solve = 0) 4.71 -> 2.68 ms against
// FP64 FMA tiles; dtheta's error against 64-bit linear algebra is unchanged (3.0e-15, 1.7e-15).
// The diagonal blocks are now the longest part, 38 % of a 4096-row solve (100 us each, cold, under a
// profiler): one SM's FP64 pipes, barriers and instruction fetches.
#include "peps_kernels.cuh"
#include "peps_slices.cuh"

namespace peps {
namespace {

constexpr int CB = 64;

// sqrt(d)^-1 of a pivot d > 0: the single-precision reciprocal square root and two Newton steps
// y <- y (3 - d y^2) / 2 (23 -> 46 -> beyond 53 bits), a shorter chain of FP64 operations than sqrt
// and a division; outside the float range the plain ones.
__device__ __forceinline__ double pivot_rsqrt(double d) {
  if (d > 1e-30 && d < 1e30) {
    double y = (double)rsqrtf((float)d);
    y = y * fma(-0.5 * d, y * y, 1.5);
    return y * fma(-0.5 * d, y * y, 1.5);
  }
  return 1.0 / sqrt(d);
}

// Factor the diagonal block at (k0, k0) in place (lower triangle; nb = min(64, n - k0) rows) and
// write the reciprocals of its diagonal to rd[k0 ..].  Threads 0..255: row i = t / 4 holds the
// columns 4 m + t % 4 in registers.  Step j: the pivot's reciprocal root comes from warp 8, the
// rows subtract column j from column j + 1 first and publish it, and the rest of step j's update
// runs while warp 8 takes the next root.  gate (may be NULL): nothing happens while *gate is 0.
__global__ void __launch_bounds__(288) k_chol_diag64(double* A, int n, int k0, double* rd, int* bad, const int* gate) {
  if (gate && !*gate) return;
  __shared__ double col[2][CB], piv[2];
  const int nb = min(CB, n - k0), t = threadIdx.x, i = t >> 2, q = t & 3;
  const bool data = t < 256;
  double a[16];
  if (data) {
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int c = 4 * m + q;
      a[m] = (i < nb && c <= i) ? A[(size_t)(k0 + i) * n + k0 + c] : 0.0;
    }
    if (q == 0) col[0][i] = a[0];
  }
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int m = 0; m < 16; ++m) {
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int j = 4 * m + jj;
      if (j >= nb) break;
      if (!data) {
        const double d = col[j & 1][j];
        const bool ok = d > 0.0;  // false for NaN too
        const double r = pivot_rsqrt(ok ? d : 1.0);
        if ((t & 31) == 0) {
          piv[j & 1] = r;
          rd[k0 + j] = r;
          if (!ok) *bad = 1;
        }
      } else if (j > 0 && i >= j + 1) {
        // the rest of step j - 1: columns from j + 1 on
        const double* cp = col[(j - 1) & 1];
#pragma unroll
        for (int mm = m; mm < 16; ++mm) {
          const int c = 4 * mm + q;
          if (4 * mm + 3 > j && c > j && c <= i) a[mm] = fma(-s, cp[c], a[mm]);
        }
      }
      __syncthreads();
      if (data && i >= j) {
        const double r = piv[j & 1], cij = col[j & 1][i];
        s = cij * r * r;
        if (q == jj) a[m] = cij * r;  // L_ij (the pivot too: d / sqrt(d))
        if (j + 1 < nb && i >= j + 1 && q == ((jj + 1) & 3)) {
          const int mn = m + (jj == 3 ? 1 : 0);
          if (mn < 16) {
            a[mn] = fma(-s, col[j & 1][j + 1], a[mn]);
            col[(j + 1) & 1][i] = a[mn];
          }
        }
      }
      __syncthreads();
    }
  }
  if (data && i < nb) {
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int c = 4 * m + q;
      if (c < nb) A[(size_t)(k0 + i) * n + k0 + c] = c <= i ? a[m] : 0.0;
    }
  }
}

// Rows below the diagonal block (full: 64 columns): A_ik <- A_ik L_kk^-T by substitution, and the
// digits of the solved rows (D[p][row][64], rowE).  A row is shared by LPR lanes (columns
// m LPR + lane), a warp holds 32 / LPR rows, a CTA four warps (one per sub-partition); the host
// takes the smallest LPR whose rows still leave no sub-partition idle.
template <int LPR>
__global__ void __launch_bounds__(128) k_chol_panel(double* A, int n, int k0, const double* __restrict__ rd,
                                                    __nv_bfloat16* D, int* rowE, const int* gate) {
  if (gate && !*gate) return;
  constexpr int R = 32 / LPR, NC = CB / LPR;
  __shared__ __align__(16) double Lc[CB][CB + 1];  // Lc[j][i] = L_ij below the diagonal, 0 elsewhere
  __shared__ double rs[CB];
  for (int o = threadIdx.x; o < CB * CB; o += 128) {
    const int i = o / CB, j = o % CB;
    Lc[j][i] = j < i ? A[(size_t)(k0 + i) * n + k0 + j] : 0.0;
  }
  if (threadIdx.x < CB) rs[threadIdx.x] = rd[k0 + threadIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % LPR, g = lane / LPR;
  const int row0 = k0 + CB + (blockIdx.x * 4 + warp) * R, row = row0 + g;
  double a[NC];
#pragma unroll
  for (int m = 0; m < NC; ++m) a[m] = row < n ? A[(size_t)row * n + k0 + m * LPR + sub] : 0.0;
#pragma unroll
  for (int m = 0; m < NC; ++m) {
#pragma unroll
    for (int sj = 0; sj < LPR; ++sj) {
      const int j = m * LPR + sj;
      const double x = __shfl_sync(0xffffffffu, a[m] * rs[j], g * LPR + sj);
      if (sub == sj) a[m] = x;
#pragma unroll
      for (int mm = m; mm < NC; ++mm) a[mm] = fma(-x, Lc[j][mm * LPR + sub], a[mm]);
    }
  }
  __syncthreads();  // the block of L is no longer needed: its memory stages the solved rows
  double(*xs)[R][CB] = reinterpret_cast<double(*)[R][CB]>(&Lc[0][0]);
#pragma unroll
  for (int m = 0; m < NC; ++m) xs[warp][g][m * LPR + sub] = a[m];
  __syncwarp();
  for (int rr = 0; rr < R && row0 + rr < n; ++rr) {
    const double2 v = reinterpret_cast<const double2*>(xs[warp][rr])[lane];
    reinterpret_cast<double2*>(A + (size_t)(row0 + rr) * n + k0)[lane] = v;  // n and k0 are even
    const unsigned long long bx = (unsigned long long)__double_as_longlong(v.x), by = (unsigned long long)__double_as_longlong(v.y);
    int e = max(max((int)(bx >> 52) & 0x7ff, (int)(by >> 52) & 0x7ff), 1);
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) rowE[row0 + rr] = e < 2047 ? e : ROW_NONFINITE;
    uint32_t w[NS][4];
    put_digits(e < 2047 ? fixed_point(bx, e) : 0, 0, w);
    put_digits(e < 2047 ? fixed_point(by, e) : 0, 1, w);
#pragma unroll
    for (int p = 0; p < NS; ++p)
      reinterpret_cast<uint32_t*>(D + ((size_t)p * n + row0 + rr) * CB)[lane] = w[p][0];
  }
}

// a 2^e, rounded to nearest even, by integer operations (the FP64 pipe would need three of its
// slow instructions); e such that the result is normal, else scalbn
__device__ __forceinline__ double fix_to_double(long long a, int e) {
  if (a == 0) return 0.0;
  unsigned long long m = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
  const int z = __clzll((long long)m);
  m <<= z;
  const int ex = 63 - z + e + 1022;  // biased exponent minus one (the mantissa's leading one adds it)
  if (ex < 1 || ex > 2043) return scalbn((double)a, e);
  unsigned long long k = m >> 11;
  const unsigned rem = (unsigned)m & 0x7ffu;
  k += (rem > 0x400u || (rem == 0x400u && (k & 1))) ? 1 : 0;
  return __longlong_as_double((long long)((((unsigned long long)ex) << 52) + k | (a < 0 ? 0x8000000000000000ull : 0ull)));
}

// A_ij -= X_i X_j^T for the lower-triangle tiles right of and below the panel: as k_gram_sl with
// the panel's 64 columns as two chunks, both loaded at once, and lsb 2^-54 of the scaled rows
// (64 2^54 < 2^61; only the last digit products round).  The sums go straight to doubles.
__global__ void __launch_bounds__(SL_THREADS, 1) k_chol_update(const __grid_constant__ CUtensorMap map, double* A, int n,
                                                               int k0, const int* __restrict__ rowE, int* bad,
                                                               const int* gate) {
  if (gate && !*gate) return;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* ring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar[2], ufull[2], uempty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int t = blockIdx.x, ti = 0;
  while (t >= ti + 1) { t -= ti + 1; ++ti; }
  const int r0 = k0 + CB + ti * SM_, c0 = k0 + CB + t * SM_;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&ufull[s], 1);
      mbar_init(&uempty[s], EPI_WARPS);
    }
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int s = 0; s < 2; ++s) {
      uint8_t* st = ring + (size_t)s * SSTAGE;
      mbar_expect_tx(&full_bar[s], SSTAGE);
      tma_load_3d(st, &map, s * CK, r0, 0, &full_bar[s]);
      tma_load_3d(st + SOPND, &map, s * CK, c0, 0, &full_bar[s]);
    }
  }
  if (warp == EPI_WARPS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  if (warp == EPI_WARPS + 1) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int c = 0; c < 2 && ok; ++c) {
        if (!wait_ok(&full_bar[c], 0, &failed)) break;
        const uint32_t a0 = smem_u32(ring + (size_t)c * SSTAGE), b0 = a0 + SOPND;
        for (int u = 0; u < 4; ++u, ++g) {
          const int slot = g & 1;
          if (g >= 2 && !wait_ok(&uempty[slot], ((g >> 1) - 1) & 1, &failed)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;");
          for (int d = 2 * u; d < 2 * u + 2 && d < NS; ++d) {
            const uint32_t acc = tmem + slot * 256 + (d & 1) * 128;
            for (int p = 0; p <= d; ++p) {
              const uint64_t da = desc64(a0 + p * STILE), db = desc64(b0 + (d - p) * STILE);
              mma_sl(acc, da, db, p > 0);
              mma_sl(acc, da + 2, db + 2, 1u);
            }
          }
          mma_commit(&ufull[slot]);
        }
      }
    }
  } else if (warp < EPI_WARPS) {
    const uint32_t tw = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 64;
    long long acc[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0;
    bool ok = true;
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t slot = u & 1, par = (u >> 1) & 1;  // two uses of each slot per chunk
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
            const int a = f2i_exact(va[j]);
            if (u < 3) {
              const int w = a * 256 + f2i_exact(vb[j]);
              if (u == 0) acc[cc + j] += (long long)w << 32;
              if (u == 1) acc[cc + j] += (long long)w * 65536;
              if (u == 2) acc[cc + j] += w;
            } else {
              acc[cc + j] += (a + 128 - c) >> 8;
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) mbar_arrive(&uempty[slot]);
      }
      if (!ok) break;
    }
    const int row = r0 + (warp & 3) * 32 + lane, cb = c0 + (warp >> 2) * 64;
    if (ok && row < n) {
      const int er = rowE[row];
      double* Ar = A + (size_t)row * n;
#pragma unroll
      for (int j = 0; j < 64; j += 2) {
        const int cj = cb + j;
        if (cj <= row) {  // n, cj even: cj + 1 < n, and an entry right of the diagonal is not read again
          double2 v = *reinterpret_cast<double2*>(Ar + cj);
          const int e0 = rowE[cj], e1 = rowE[cj + 1];
          const double nan = __longlong_as_double(0x7ff8000000000000ll);
          v.x -= (er < 0 || e0 < 0) ? nan : fix_to_double(acc[j], er + e0 - 2044 - 54);
          v.y -= (er < 0 || e1 < 0) ? nan : fix_to_double(acc[j + 1], er + e1 - 2044 - 54);
          *reinterpret_cast<double2*>(Ar + cj) = v;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (failed && threadIdx.x == 0) {
    *bad = 1;
    for (int s = 0; s < 2; ++s)
      for (int i = 0; i < (1 << 16) && !mbar_try(&full_bar[s], 0); ++i) {}
  }
  if (warp == EPI_WARPS) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

__global__ void k_add_diag(double* A, int n, int nreal, double lambda, const int* gate) {
  if (gate && !*gate) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    A[(size_t)i * n + i] += (i < nreal) ? lambda : 1.0;  // a padding index gets 1 (its rhs is 0)
}

// F (lower) = A + d with d_i = lambda (i < nreal) or 1 (padding); A is kept
__global__ void k_lower_copy(const double* __restrict__ A, double* __restrict__ F, int n, int nreal, double lambda) {
  const int i = blockIdx.y * 8 + (threadIdx.x >> 5), j = blockIdx.x * 32 + (threadIdx.x & 31);
  if (i >= n || j > i) return;
  double v = A[(size_t)i * n + j];
  if (i == j) v += (i < nreal) ? lambda : 1.0;
  F[(size_t)i * n + j] = v;
}

// Inverses X of the 64 x 64 diagonal blocks of the factor, Li[block][i][c] (zero outside the lower
// triangle and the block's rows): four threads per column c, each a quarter of the sum
// x_i = -rd_i sum_{k = c}^{i - 1} L_ik x_k.  L sits below the diagonal of S, X transposed above it.
__global__ void __launch_bounds__(256) k_tri_inv(const double* __restrict__ L, int n, const double* __restrict__ rd,
                                                 double* Li, const int* gate) {
  if (gate && !*gate) return;
  __shared__ double S[CB][CB + 2];
  __shared__ double rs[CB];
  const int k0 = blockIdx.x * CB, nb = min(CB, n - k0);
  for (int o = threadIdx.x; o < CB * CB; o += 256) {
    const int i = o / CB, j = o % CB;
    if (j < i) S[i][j] = i < nb ? L[(size_t)(k0 + i) * n + k0 + j] : 0.0;
    else S[i][j + 1] = 0.0;
  }
  if (threadIdx.x < CB) rs[threadIdx.x] = threadIdx.x < nb ? rd[k0 + threadIdx.x] : 0.0;
  __syncthreads();
  const int c = threadIdx.x >> 2, q = threadIdx.x & 3;
  double* X = S[c] + 1;  // X[i], i >= c
  if (q == 0) X[c] = rs[c];
  __syncwarp();
  const int c0 = (threadIdx.x >> 5) * 8;  // first column of this warp
  for (int i = c0 + 1; i < nb; ++i) {
    double s = 0.0;
    for (int k = c0 + q; k < i; k += 4)
      if (k >= c) s = fma(S[i][k], X[k], s);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (q == 0 && i > c) X[i] = -s * rs[i];
    __syncwarp();
  }
  __syncthreads();
  for (int o = threadIdx.x; o < CB * CB; o += 256) {
    const int i = o / CB, j = o % CB;
    Li[(size_t)blockIdx.x * CB * CB + o] = (j <= i && i < nb) ? S[j][i + 1] : 0.0;
  }
}

// One block of L y = v: y_k = Li_k v_k in every CTA (CTA 0 stores it), then v -= L y_k on the rows
// below, four threads per row.  One launch per block.
__global__ void __launch_bounds__(256) k_trsv64_fwd(const double* __restrict__ L, const double* __restrict__ Li, int n,
                                                    int k0, double* v, double* y, const int* gate) {
  if (gate && !*gate) return;
  __shared__ double vs[CB], ys[CB];
  const int t = threadIdx.x, i = t >> 2, q = t & 3;
  if (t < CB) vs[t] = k0 + t < n ? v[k0 + t] : 0.0;
  __syncthreads();
  const double* Lb = Li + (size_t)(k0 / CB) * CB * CB + i * CB + 16 * q;
  double s = 0.0;
#pragma unroll
  for (int l = 0; l < 16; ++l) s = fma(Lb[l], vs[16 * q + l], s);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  if (q == 0) {
    ys[i] = s;
    if (blockIdx.x == 0 && k0 + i < n) y[k0 + i] = s;
  }
  __syncthreads();
  const int r = k0 + CB + blockIdx.x * 64 + i;
  double u = 0.0;
  if (r < n) {
    const double2* Lr = reinterpret_cast<const double2*>(L + (size_t)r * n + k0 + 16 * q);  // n is even
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      const double2 w = Lr[l];
      u = fma(w.x, ys[16 * q + 2 * l], u);
      u = fma(w.y, ys[16 * q + 2 * l + 1], u);
    }
  }
  u += __shfl_xor_sync(0xffffffffu, u, 1);
  u += __shfl_xor_sync(0xffffffffu, u, 2);
  if (r < n && q == 0) v[r] -= u;
}

// One block of L^T z = y: z_k = Li_k^T y_k, then y -= L^T z_k on the rows above (a CTA takes 64 of
// them, four groups of 64 threads a quarter of the block's rows each).
__global__ void __launch_bounds__(256) k_trsv64_bwd(const double* __restrict__ L, const double* __restrict__ Li, int n,
                                                    int k0, double* y, double* z, const int* gate) {
  if (gate && !*gate) return;
  __shared__ double ys[CB], zs[CB], part[4][CB];
  const int t = threadIdx.x, i = t & 63, q = t >> 6;
  if (t < CB) ys[t] = k0 + t < n ? y[k0 + t] : 0.0;
  __syncthreads();
  const double* Lb = Li + (size_t)(k0 / CB) * CB * CB + i;
  double s = 0.0;
#pragma unroll
  for (int l = 0; l < 16; ++l) s = fma(Lb[(16 * q + l) * CB], ys[16 * q + l], s);
  part[q][i] = s;
  __syncthreads();
  if (t < CB) {
    const double x = (part[0][t] + part[1][t]) + (part[2][t] + part[3][t]);
    zs[t] = x;
    if (blockIdx.x == 0 && k0 + t < n) z[k0 + t] = x;
  }
  __syncthreads();
  const int c = blockIdx.x * 64 + i;  // rows above the block: columns c < k0 of the block's rows of L
  double u = 0.0;
  if (c < k0) {
#pragma unroll
    for (int l = 0; l < 16; ++l)
      if (k0 + 16 * q + l < n) u = fma(L[(size_t)(k0 + 16 * q + l) * n + c], zs[16 * q + l], u);
  }
  part[q][i] = u;
  __syncthreads();
  if (t < CB && c < k0) y[c] -= (part[0][t] + part[1][t]) + (part[2][t] + part[3][t]);
}

// Workspace carved from `ws` (chol64_ws_bytes(n)): the inverted diagonal blocks, the reciprocal
// pivots, the panel's digits and row exponents.
struct CholWs {
  double *Li, *rd;
  __nv_bfloat16* D;
  int* rowE;
};
CholWs carve_chol(void* ws, int n) {
  CholWs w;
  const size_t nb = (size_t)(n + CB - 1) / CB;
  w.D = (__nv_bfloat16*)ws;  // first: 16-byte aligned rows for the tensor map
  w.Li = (double*)((char*)ws + ((size_t)NS * n * CB * 2 + 255) / 256 * 256);
  w.rd = w.Li + nb * CB * CB;
  w.rowE = (int*)(w.rd + nb * CB);
  return w;
}

// Factor the lower triangle of A in place; *launches counts kernels.
cudaError_t factor64(double* A, int n, const CholWs& w, int* bad, const int* gate, cudaStream_t s, long long* launches) {
  EncodeTiled enc = get_encode();
  if (!enc) return cudaErrorNotSupported;
  CUtensorMap map;
  const cuuint64_t dims[3] = {CB, (cuuint64_t)n, NS};
  const cuuint64_t strides[2] = {CB * 2, (cuuint64_t)n * CB * 2};
  const cuuint32_t box[3] = {CK, SM_, NS}, estr[3] = {1, 1, 1};
  // rows past n read as zeros
  if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, w.D, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const size_t smem = (size_t)2 * SSTAGE + 1024;
  cudaError_t e = cudaFuncSetAttribute(k_chol_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  for (int k0 = 0; k0 < n; k0 += CB) {
    k_chol_diag64<<<1, 288, 0, s>>>(A, n, k0, w.rd, bad, gate);
    ++*launches;
    const int rest = n - k0 - CB;
    if (rest <= 0) break;
    if (rest > 16 * nsm) k_chol_panel<4><<<(rest + 31) / 32, 128, 0, s>>>(A, n, k0, w.rd, w.D, w.rowE, gate);
    else if (rest > 8 * nsm) k_chol_panel<8><<<(rest + 15) / 16, 128, 0, s>>>(A, n, k0, w.rd, w.D, w.rowE, gate);
    else k_chol_panel<16><<<(rest + 7) / 8, 128, 0, s>>>(A, n, k0, w.rd, w.D, w.rowE, gate);
    const int nt = (rest + SM_ - 1) / SM_;
    k_chol_update<<<nt * (nt + 1) / 2, SL_THREADS, smem, s>>>(map, A, n, k0, w.rowE, bad, gate);
    *launches += 2;
  }
  k_tri_inv<<<(n + CB - 1) / CB, 256, 0, s>>>(A, n, w.rd, w.Li, gate);
  ++*launches;
  return cudaGetLastError();
}

__global__ void k_vcopy64(const double* src, double* dst, int n, const int* gate) {
  if (gate && !*gate) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
__global__ void k_vadd64(const double* src, double* dst, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] += src[i];
}

// v <- (L L^T)^-1 v (y: n doubles of scratch)
void apply64(const double* L, int n, const CholWs& w, double* v, double* y, const int* gate, cudaStream_t s,
             long long* launches) {
  for (int k0 = 0; k0 < n; k0 += CB) {
    const int rows = n - k0 - CB;
    k_trsv64_fwd<<<rows > 0 ? (rows + 63) / 64 : 1, 256, 0, s>>>(L, w.Li, n, k0, v, y, gate);
  }
  for (int k0 = ((n - 1) / CB) * CB; k0 >= 0; k0 -= CB)
    k_trsv64_bwd<<<k0 > 0 ? (k0 + 63) / 64 : 1, 256, 0, s>>>(L, w.Li, n, k0, y, v, gate);
  *launches += 2 * ((n + CB - 1) / CB);
}

// gate (may be NULL): the fallback flag of the mixed solve; a factorisation it gates marks the
// fallback in info[2] = 0
__global__ void k_chol_info(int* bad, int nreal, double* info, const int* gate) {
  if (gate && !*gate) return;
  info[0] = *bad ? -1.0 : (double)nreal;
  info[1] = NAN;
  info[2] = gate ? 0.0 : NAN;
}
__global__ void k_zero_int(int* p, const int* gate) {
  if (gate && !*gate) return;
  *p = 0;
}
__global__ void k_refined_info(const int* bad, int nreal, const double* rn, int iters, double* info) {
  info[0] = *bad ? -1.0 : (double)nreal;
  info[1] = (rn[1] > 0.0) ? sqrt(rn[0] / rn[1]) : 0.0;
  info[2] = (double)iters;
}

}  // namespace

size_t chol64_ws_bytes(int n) {
  const size_t nb = (size_t)(n + CB - 1) / CB;
  return ((size_t)NS * n * CB * 2 + 255) / 256 * 256 + nb * CB * (CB + 1) * 8 + (size_t)n * 4 + 256;
}

// Returns launches issued; *err for a CUDA error.  info[0] = Ns (-1 if T + lambda was not
// positive definite in floating point), info[1..2] = NaN (no eigenvalues computed).  With a gate,
// every launch does nothing unless *gate != 0 when it runs.
long long chol_solve(double* A, int n, int nreal, double lambda, const double* ebar, double* x, int* bad,
                     double* info, const int* gate, double* scratch, void* ws, cudaStream_t s, cudaError_t* err) {
  long long launches = 4;
  const CholWs w = carve_chol(ws, n);
  k_zero_int<<<1, 1, 0, s>>>(bad, gate);
  k_add_diag<<<(n + 255) / 256, 256, 0, s>>>(A, n, nreal, lambda, gate);
  if ((*err = factor64(A, n, w, bad, gate, s, &launches)) != cudaSuccess) return launches;
  k_vcopy64<<<(n + 255) / 256, 256, 0, s>>>(ebar, x, n, gate);
  apply64(A, n, w, x, scratch, gate, s, &launches);
  k_chol_info<<<1, 1, 0, s>>>(bad, nreal, info, gate);
  *err = cudaGetLastError();
  return launches;
}

// solve = 2: the FP64 factor of a copy F of T + lambda, then `iters` steps of refinement with FP64
// residuals against T.  info = (Ns or -1, relative residual after refinement, iters, -).
long long chol_solve_refined(double* A, double* F, int n, int nreal, double lambda, const double* ebar, double* x,
                             double* r, double* rn, double* part, int iters, int* bad, double* info, double* scratch,
                             void* ws, cudaStream_t s, cudaError_t* err) {
  long long launches = 4;
  const CholWs w = carve_chol(ws, n);
  k_zero_int<<<1, 1, 0, s>>>(bad, nullptr);
  k_lower_copy<<<dim3((n + 31) / 32, (n + 7) / 8), 256, 0, s>>>(A, F, n, nreal, lambda);
  if ((*err = factor64(F, n, w, bad, nullptr, s, &launches)) != cudaSuccess) return launches;
  k_vcopy64<<<(n + 255) / 256, 256, 0, s>>>(ebar, x, n, nullptr);
  apply64(F, n, w, x, scratch, nullptr, s, &launches);
  for (int it = 0; it <= iters; ++it) {
    launches += launch_residual(A, n, nreal, lambda, ebar, x, r, part, it == iters ? rn : nullptr, s);
    if (it == iters) break;
    apply64(F, n, w, r, scratch, nullptr, s, &launches);
    k_vadd64<<<(n + 255) / 256, 256, 0, s>>>(r, x, n);
    ++launches;
  }
  k_refined_info<<<1, 1, 0, s>>>(bad, nreal, rn, iters, info);
  *err = cudaGetLastError();
  return launches;
}

}  // namespace peps
