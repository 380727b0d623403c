// Contraction kernels of the finite-PEPS hot path (sm_103a): environment pass, one- and two-row
// sandwiches (amplitudes, local-energy ratios, log-derivatives), per-sample combine, and the
// Metropolis sweep.  All kernels are persistent: each CTA loops over work items
// (blockIdx.x, blockIdx.x + gridDim.x, ...) and owns one slice of the global scratch arena.
// Included by peps_kernels_f64.cu and peps_kernels_f32.cu, which instantiate it for one real
// type each (two translation units compile in parallel).
#pragma once
#include "peps_kernels.cuh"

namespace peps {

// ------------------------------------------------------------------------------------------
// environment store: per sample 2*Lx rows of Ly sites; slot x+1 holds E^u[x] (x = -1..Lx-2),
// slot Lx+x-1 holds E^l[x] (x = 1..Lx).  logs: cumulative log factor of every slot.
template <typename G>
__host__ __device__ inline size_t env_sample_elems(const G& g) { return (size_t)2 * g.Lx * g.Ly * g.se; }
template <typename G>
__device__ inline int slot_up(const G& g, int x) { return x + 1; }
template <typename G>
__device__ inline int slot_lo(const G& g, int x) { return g.Lx + x - 1; }

template <typename T>
__device__ RowWork<T> carve_row(const Plan& p, char* smem, char* gbase) {
  RowWork<T> w;
  w.R = (T*)buf_ptr(p, B_R, smem, gbase);
  w.Rhist = (T*)buf_ptr(p, B_RHIST, smem, gbase);
  w.E = (T*)buf_ptr(p, B_E, smem, gbase);
  w.A = (T*)buf_ptr(p, B_A, smem, gbase);
  w.Z = (T*)buf_ptr(p, B_Z, smem, gbase);
  w.ZS = (T*)buf_ptr(p, B_ZS, smem, gbase);
  w.W = (T*)buf_ptr(p, B_W, smem, gbase);
  w.C = (T*)buf_ptr(p, B_C, smem, gbase);
  w.sig = (T*)buf_ptr(p, B_SIG, smem, gbase);
  w.sel = (int*)buf_ptr(p, B_SEL, smem, gbase);
  w.red = (double*)buf_ptr(p, B_RED, smem, gbase);
  w.ci = p.ci;
  w.ctr = p.ctr;
  return w;
}

// One side of configuration Ss's environments into env (one sample's store): the upper ones
// E^u[-1..Lx-2] (and the trivial E^l[Lx] that closes psi_top = E^u[Lx-2] . T_proj[Lx-1]) or the lower
// ones E^l[1..Lx].  One row step for both sides: its code is large, and a second copy in a kernel whose
// CTAs work on either side costs instruction fetches.
template <typename T, typename G>
__device__ __forceinline__ void build_side(const G& g, int lower, const T* Tpad, const uint8_t* Ss, T* env, double* logs,
                                           const RowWork<T>& w, int* st, int* flag) {
  const size_t row = (size_t)g.Ly * g.se;
  T* trivial_lo = env + (size_t)slot_lo(g, g.Lx) * row;
  for (int k = 0; k < g.Ly; ++k) {
    if (!lower) blk_unit(env + (size_t)slot_up(g, -1) * row + (size_t)k * g.se, g.se);
    blk_unit(trivial_lo + (size_t)k * g.se, g.se);
  }
  if (threadIdx.x == 0) {
    if (!lower) logs[slot_up(g, -1)] = 0.0;
    logs[slot_lo(g, g.Lx)] = 0.0;
  }
  __syncthreads();
  double lg = 0.0;
  for (int i = 0; i < g.Lx - 1; ++i) {
    const int x = lower ? g.Lx - 1 - i : i, slot = lower ? slot_lo(g, x) : slot_up(g, x);
    const uint8_t* Srow = Ss + (size_t)x * g.Ly;
    T* out = env + (size_t)slot * row;
    Scaled f;
    if (i == 0) f = env_first_row(g, out, Tpad, x, Srow, lower != 0, w.A, w.Z, w.red, st);
    else f = env_row_step_inl(g, env + (size_t)(lower ? slot_lo(g, x + 1) : slot_up(g, x - 1)) * row, out, Tpad, x, Srow,
                              lower != 0, w, st, flag);
    if (threadIdx.x == 0) logs[slot] = lg += sc_log(f);
  }
  __syncthreads();
}
template <typename T, typename G>
__device__ __noinline__ void build_side_call(const G g, int lower, const T* Tpad, const uint8_t* Ss, T* env, double* logs,
                                             const RowWork<T> w, int* st, int* flag) {
  build_side(g, lower, Tpad, Ss, env, logs, w, st, flag);
}

// One side (0 upper, 1 lower) of sample smp's environments, with the whole CTA.
template <typename T, typename G>
__device__ __forceinline__ void env_item(const G g, const RowWork<T>& w, const T* __restrict__ Tpad,
                                         const uint8_t* __restrict__ S,
                         int smp, int side, T* envs, double* logs, int* status) {
  __shared__ int st, flag;
  const int N = g.Lx * g.Ly;
  if (threadIdx.x == 0) st = 0;
  __syncthreads();
  T* env = envs + (size_t)smp * env_sample_elems(g);
  double* lg = logs + (size_t)smp * 2 * g.Lx;
  const uint8_t* Ss = S + (size_t)smp * N;
  build_side(g, side, Tpad, Ss, env, lg, w, &st, &flag);
  if (threadIdx.x == 0) {
    if (st) atomicOr(status + smp, st);
  }
  __syncthreads();
}

template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, EnvBlocks<T>::value) k_env(G g, Plan plan, const T* __restrict__ Tpad,
                                                  const uint8_t* __restrict__ S, int Ns, int sides, T* envs,
                                                  double* logs, int* status) {
  extern __shared__ __align__(16) char smem[];
  RowWork<T> w = carve_row<T>(plan, smem, plan.gbase);
  const int nside = (sides == 3) ? 2 : 1;
  for (int item = blockIdx.x; item < Ns * nside; item += gridDim.x) {
    const int smp = item / nside;
    const int side = (sides == 3) ? (item % nside) : (sides == 1 ? 0 : 1);
    env_item(g, w, Tpad, S, smp, side, envs, logs, status);
  }
}

// ------------------------------------------------------------------------------------------
// Sandwich bookkeeping shared by the row and pair kernels.
template <typename G>
__device__ inline void site_dims(const G& g, int x, int y, int* Dl, int* Du, int* Dr, int* Dd) {
  *Dl = (y == 0) ? 1 : g.D;
  *Du = (x == 0) ? 1 : g.D;
  *Dr = (y == g.Ly - 1) ? 1 : g.D;
  *Dd = (x == g.Lx - 1) ? 1 : g.D;
}

// local state of `site` in configuration Ss after replacing the term's sites by the digits of b
__device__ inline int state_after(const int* ti, int site, const uint8_t* Ss, int b, int d) {
  const int k = ti[TI_K];
  int pw = 1;
  for (int t = k - 1; t >= 0; --t) {
    if (ti[TI_S0 + t] == site) return (b / pw) % d;
    pw *= d;
  }
  return Ss[site];
}

__device__ inline int local_index(const int* ti, const uint8_t* Ss, int d) {
  int a = 0;
  for (int t = 0; t < ti[TI_K]; ++t) a = a * d + Ss[ti[TI_S0 + t]];
  return a;
}

// ------------------------------------------------------------------------------------------
// One-row sandwich at row x of sample smp: psi_x, O of row x, E_loc terms inside row x.
// One-row sandwich at row x of sample smp, with the whole CTA.
template <typename T, typename G>
__device__ __forceinline__ void row_item(const G g, const Plan plan, char* smem, const T* __restrict__ Tpad,
                                         const uint8_t* __restrict__ S, int smp, int x, const T* envs,
                                         const double* logs, T* O, const long long* site_off, long long Np,
                                         const TermTab tt, double* rowout, int* status) {
  char* gbase = plan.gbase;
  T* LP = (T*)buf_ptr(plan, B_LP, smem, gbase);   // (Ly+1) x se
  T* RP = (T*)buf_ptr(plan, B_RP, smem, gbase);   // (Ly+1) x se
  T* t1 = (T*)buf_ptr(plan, B_T1, smem, gbase);
  T* t2 = (T*)buf_ptr(plan, B_T2, smem, gbase);
  T* eu = (T*)buf_ptr(plan, B_EU, smem, gbase);
  T* el = (T*)buf_ptr(plan, B_EL, smem, gbase);
  T* A = (T*)buf_ptr(plan, B_A, smem, gbase);
  T* LW = (T*)buf_ptr(plan, B_LW, smem, gbase);
  T* LW2 = (T*)buf_ptr(plan, B_LW2, smem, gbase);
  double* red = (double*)buf_ptr(plan, B_RED, smem, gbase);
  __shared__ Scaled logL[MAX_LY + 1], logR[MAX_LY + 1];  // factors taken out of the partials
  __shared__ dz fO;
  __shared__ int st;
  const int N = g.Lx * g.Ly, Ly = g.Ly, se = g.se;
  const size_t rowsz = (size_t)Ly * se;
  const uint8_t* Ss = S + (size_t)smp * N;
  const T* env = envs + (size_t)smp * env_sample_elems(g);
  const double* lg = logs + (size_t)smp * 2 * g.Lx;
  const T* EU = env + (size_t)slot_up(g, x - 1) * rowsz;
  const T* EL = env + (size_t)slot_lo(g, x + 1) * rowsz;
  if (threadIdx.x == 0) st = 0;
  // right partials R[Ly] = unit, R[y] = R[y+1] absorbed over column y
  __shared__ int bu[MAX_LY + 1], bl[MAX_LY + 1], sl_[MAX_LY], sr_[MAX_LY];
  mps_bonds(g, EU, bu, sl_, sr_);
  mps_bonds(g, EL, bl, sl_, sr_);
  const int D = g.D, chi = g.chi, cd = g.chi * g.D;
  auto ext = [&](int y) { return BondExt{bu[y], bu[y + 1], bl[y], bl[y + 1]}; };
  blk_unit(RP + (size_t)Ly * se, cd);
  if (threadIdx.x == 0) logR[Ly] = sc_one();
  for (int y = Ly - 1; y >= 0; --y) {
    blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
    blk_copy(el, EL + (size_t)y * se, bl[y] * cd);
    load_A(A, Tpad, g, x * Ly + y, Ss[x * Ly + y], false);
    __syncthreads();
    absorb1_right(g, ext(y), RP + (size_t)(y + 1) * se, eu, A, el, t1, t2, RP + (size_t)y * se);
    const double l = (double)blk_normalize(RP + (size_t)y * se, bu[y] * D, chi, bl[y], red, &st);
    if (threadIdx.x == 0) logR[y] = sc_mul(logR[y + 1], l);
  }
  // left partials
  blk_unit(LP, cd);
  if (threadIdx.x == 0) logL[0] = sc_one();
  __syncthreads();
  for (int y = 0; y < Ly; ++y) {
    blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
    blk_copy(el, EL + (size_t)y * se, bl[y] * cd);
    load_A(A, Tpad, g, x * Ly + y, Ss[x * Ly + y], false);
    __syncthreads();
    absorb1(g, ext(y), LP + (size_t)y * se, eu, A, el, t1, t2, LP + (size_t)(y + 1) * se);
    const double l = (double)blk_normalize(LP + (size_t)(y + 1) * se, bu[y + 1] * D, chi, bl[y + 1], red, &st);
    if (threadIdx.x == 0) logL[y + 1] = sc_mul(logL[y], l);
  }
  __syncthreads();
  const T val = LP[(size_t)Ly * se];
  // 1 / psi_x without its scale, in thread 0
  const dz ival = threadIdx.x == 0 ? dz_div(dz{1.0, 0.0}, to_dz(val)) : dz{0.0, 0.0};
  // ---- log-derivatives of row x
  if (O != nullptr) {
    for (int y = 0; y < Ly; ++y) {
      const int site = x * Ly + y;
      blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
      {
        // the lower environment site transposed, elT[z][b][d] = el[b][d][z] (into LW2)
        const T* ely = EL + (size_t)y * se;
        const int nb = bl[y] * D;  // (b, d) for b below the bond
        const FDiv fz = fdiv_of(bl[y + 1]);
        for (int o = threadIdx.x; o < nb * fz.k; o += blockDim.x) {
          const int bd = fdiv_q(o, fz), z = o - bd * fz.k;
          LW2[z * cd + bd] = ely[(size_t)bd * chi + z];
        }
      }
      __syncthreads();
      site_env1(g, ext(y), LP + (size_t)y * se, eu, LW2, RP + (size_t)(y + 1) * se, t1, t2, A);
      if (threadIdx.x == 0) {
        const double sc = sc_ratio(sc_mul(logL[y], logR[y + 1]), logL[Ly]);
        fO = dz{ival.re * sc, ival.im * sc};
      }
      int Dl, Du, Dr, Dd;
      site_dims(g, x, y, &Dl, &Du, &Dr, &Dd);
      const int blk = Dl * Du * Dr * Dd;
      const int s_here = Ss[site];
      T* Orow = O + (size_t)smp * Np + site_off[site];
      __syncthreads();
      const dz f = fO;
      for (int s = 0; s < g.d; ++s)
        for (int c = threadIdx.x; c < blk; c += blockDim.x) {
          T v = T(0);
          if (s == s_here) {
            const int dd = c % Dd, r = (c / Dd) % Dr, u = (c / (Dd * Dr)) % Du, l = c / (Dd * Dr * Du);
            const T a = A[((l * D + u) * D + r) * D + dd];
            if constexpr (Scal<T>::complex) v = from_dz<T>(dz_mul(to_dz(a), f));
            else v = (T)((double)a * f.re);
          }
          Orow[s * blk + c] = v;
        }
      __syncthreads();
    }
  }
  // ---- local-energy terms inside row x
  double ere = 0.0, eim = 0.0;
  if (tt.nterm > 0) {
    for (int ti_ = tt.row_off[x]; ti_ < tt.row_off[x + 1]; ++ti_) {
      const int* ti = tt.tinfo + (size_t)ti_ * TI_N;
      const int a = local_index(ti, Ss, g.d);
      for (int e = ti[TI_EOFF]; e < ti[TI_EOFF] + ti[TI_ECNT]; ++e) {
        if (tt.ent_ab[2 * e] != a) continue;
        const int b = tt.ent_ab[2 * e + 1];
        const double hr = tt.ent_h[2 * e], hi = tt.ent_h[2 * e + 1];
        if (b == a) { ere += hr; eim += hi; continue; }
        const int y0 = ti[TI_Y0], w = ti[TI_W];
        const T* cur = LP + (size_t)y0 * se;
        T* nxt = LW;
        Scaled lw = logL[y0];  // carried in thread 0
        for (int c = y0; c < y0 + w; ++c) {
          const int site = x * Ly + c;
          blk_copy(eu, EU + (size_t)c * se, bu[c] * cd);
          blk_copy(el, EL + (size_t)c * se, bl[c] * cd);
          load_A(A, Tpad, g, site, state_after(ti, site, Ss, b, g.d), false);
          __syncthreads();
          absorb1(g, ext(c), cur, eu, A, el, t1, t2, nxt);
          const double l = (double)blk_normalize(nxt, bu[c + 1] * D, chi, bl[c + 1], red, &st);
          if (threadIdx.x == 0) lw = sc_mul(lw, l);
          cur = nxt;
          nxt = nxt == LW ? LW2 : LW;
        }
        const T v = blk_dot(cur, RP + (size_t)(y0 + w) * se, bu[y0 + w] * D, chi, bl[y0 + w], red);
        if (threadIdx.x == 0) {
          const dz q = dz_mul(to_dz(v), ival);
          const double f = sc_ratio(sc_mul(lw, logR[y0 + w]), logL[Ly]);
          ere += (hr * q.re - hi * q.im) * f;
          eim += (hr * q.im + hi * q.re) * f;
        }
      }
    }
  }
  if (threadIdx.x == 0) {
    double* out = rowout + ((size_t)smp * g.Lx + x) * 4;
    const dz vz = to_dz(val);
    const double av = dz_abs(vz);
    out[0] = (av > 0.0) ? sc_log(sc_mul(logL[Ly], av)) + lg[slot_up(g, x - 1)] + lg[slot_lo(g, x + 1)] : -INFINITY;
    out[1] = (vz.im == 0.0) ? ((vz.re < 0.0) ? 3.141592653589793 : 0.0) : atan2(vz.im, vz.re);
    out[2] = ere;
    out[3] = eim;
    int s = st;
    if (!(av > 0.0) || !isfinite(out[0]) || !isfinite(ere) || !isfinite(eim)) s |= ST_NONFINITE;
    if (s) atomicOr(status + smp, s);
  }
  __syncthreads();
}

template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, EnvBlocks<T>::value) k_row(G g, Plan plan, const T* __restrict__ Tpad,
                                                  const uint8_t* __restrict__ S, int Ns, int x_lo, int x_hi,
                                                  const T* envs, const double* logs, T* O, const long long* site_off,
                                                  long long Np, TermTab tt, double* rowout, int* status) {
  extern __shared__ __align__(16) char smem[];
  const int nx = x_hi - x_lo;
  for (int item = blockIdx.x; item < Ns * nx; item += gridDim.x)
    row_item(g, plan, smem, Tpad, S, item / nx, x_lo + item % nx, envs, logs, O, site_off, Np, tt, rowout, status);
}

// ------------------------------------------------------------------------------------------
// Two-row sandwich at rows x, x+1: psi_{x,x+1} and the E_loc terms spanning the two rows.
// Two-row sandwich at rows x, x+1 of sample smp, with the whole CTA.
template <typename T, typename G>
__device__ __forceinline__ void pair_item(const G g, const Plan plan, char* smem, const T* __restrict__ Tpad,
                                          const uint8_t* __restrict__ S, int smp, int x, const T* envs,
                                          const double* logs, const TermTab tt, double* pairout, int* status) {
  char* gbase = plan.gbase;
  T* LP = (T*)buf_ptr(plan, B_LP, smem, gbase);   // (Ly+1) x s2
  T* RP = (T*)buf_ptr(plan, B_RP, smem, gbase);   // (Ly+1) x s2
  T* t1 = (T*)buf_ptr(plan, B_T1, smem, gbase);
  T* t2 = (T*)buf_ptr(plan, B_T2, smem, gbase);
  T* eu = (T*)buf_ptr(plan, B_EU, smem, gbase);
  T* el = (T*)buf_ptr(plan, B_EL, smem, gbase);
  T* A1 = (T*)buf_ptr(plan, B_A, smem, gbase);
  T* A2 = (T*)buf_ptr(plan, B_A2, smem, gbase);
  T* LW = (T*)buf_ptr(plan, B_LW, smem, gbase);
  T* LW2 = (T*)buf_ptr(plan, B_LW2, smem, gbase);
  double* red = (double*)buf_ptr(plan, B_RED, smem, gbase);
  __shared__ Scaled logL[MAX_LY + 1], logR[MAX_LY + 1];  // factors taken out of the partials
  __shared__ int st;
  const int N = g.Lx * g.Ly, Ly = g.Ly, se = g.se, s2 = g.s2;
  const size_t rowsz = (size_t)Ly * se;
  // skip row pairs without terms
  if (tt.nterm == 0 || tt.pair_off[x] == tt.pair_off[x + 1]) {
    if (threadIdx.x == 0) {
      double* out = pairout + ((size_t)smp * g.Lx + x) * 4;
      out[0] = 0.0; out[1] = 0.0; out[2] = 0.0; out[3] = 0.0;
    }
    return;
  }
  const uint8_t* Ss = S + (size_t)smp * N;
  const T* env = envs + (size_t)smp * env_sample_elems(g);
  const T* EU = env + (size_t)slot_up(g, x - 1) * rowsz;
  const T* EL = env + (size_t)slot_lo(g, x + 2) * rowsz;
  if (threadIdx.x == 0) st = 0;
  __shared__ int bu[MAX_LY + 1], bl[MAX_LY + 1], sl_[MAX_LY], sr_[MAX_LY];
  mps_bonds(g, EU, bu, sl_, sr_);
  mps_bonds(g, EL, bl, sl_, sr_);
  const int D2 = g.D * g.D, chi = g.chi, cd = g.chi * g.D;
  auto ext = [&](int y) { return BondExt{bu[y], bu[y + 1], bl[y], bl[y + 1]}; };
  blk_unit(RP + (size_t)Ly * s2, D2 * chi);
  if (threadIdx.x == 0) logR[Ly] = sc_one();
  for (int y = Ly - 1; y >= 0; --y) {
    blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
    blk_copy(el, EL + (size_t)y * se, bl[y] * cd);
    load_A(A1, Tpad, g, x * Ly + y, Ss[x * Ly + y], false);
    load_A(A2, Tpad, g, (x + 1) * Ly + y, Ss[(x + 1) * Ly + y], false);
    __syncthreads();
    absorb2_right(g, ext(y), RP + (size_t)(y + 1) * s2, eu, A1, A2, el, t1, t2, RP + (size_t)y * s2, plan.cx);
    const double l = (double)blk_normalize(RP + (size_t)y * s2, bu[y] * D2, chi, bl[y], red, &st);
    if (threadIdx.x == 0) logR[y] = sc_mul(logR[y + 1], l);
  }
  blk_unit(LP, D2 * chi);
  if (threadIdx.x == 0) logL[0] = sc_one();
  __syncthreads();
  // the left partials are only needed up to the last window start; build them all
  for (int y = 0; y < Ly; ++y) {
    blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
    blk_copy(el, EL + (size_t)y * se, bl[y] * cd);
    load_A(A1, Tpad, g, x * Ly + y, Ss[x * Ly + y], false);
    load_A(A2, Tpad, g, (x + 1) * Ly + y, Ss[(x + 1) * Ly + y], false);
    __syncthreads();
    absorb2(g, ext(y), LP + (size_t)y * s2, eu, A1, A2, el, t1, t2, LP + (size_t)(y + 1) * s2, plan.cx);
    const double l = (double)blk_normalize(LP + (size_t)(y + 1) * s2, bu[y + 1] * D2, chi, bl[y + 1], red, &st);
    if (threadIdx.x == 0) logL[y + 1] = sc_mul(logL[y], l);
  }
  __syncthreads();
  const T val = LP[(size_t)Ly * s2];
  const dz ival = threadIdx.x == 0 ? dz_div(dz{1.0, 0.0}, to_dz(val)) : dz{0.0, 0.0};
  double ere = 0.0, eim = 0.0;
  for (int ti_ = tt.pair_off[x]; ti_ < tt.pair_off[x + 1]; ++ti_) {
    const int* ti = tt.tinfo + (size_t)ti_ * TI_N;
    const int a = local_index(ti, Ss, g.d);
    for (int e = ti[TI_EOFF]; e < ti[TI_EOFF] + ti[TI_ECNT]; ++e) {
      if (tt.ent_ab[2 * e] != a) continue;
      const int b = tt.ent_ab[2 * e + 1];
      const double hr = tt.ent_h[2 * e], hi = tt.ent_h[2 * e + 1];
      if (b == a) { ere += hr; eim += hi; continue; }
      const int y0 = ti[TI_Y0], w = ti[TI_W];
      const T* cur = LP + (size_t)y0 * s2;
      T* nxt = LW;
      Scaled lw = logL[y0];  // carried in thread 0
      for (int c = y0; c < y0 + w; ++c) {
        blk_copy(eu, EU + (size_t)c * se, bu[c] * cd);
        blk_copy(el, EL + (size_t)c * se, bl[c] * cd);
        load_A(A1, Tpad, g, x * Ly + c, state_after(ti, x * Ly + c, Ss, b, g.d), false);
        load_A(A2, Tpad, g, (x + 1) * Ly + c, state_after(ti, (x + 1) * Ly + c, Ss, b, g.d), false);
        __syncthreads();
        absorb2(g, ext(c), cur, eu, A1, A2, el, t1, t2, nxt, plan.cx);
        const double l = (double)blk_normalize(nxt, bu[c + 1] * D2, chi, bl[c + 1], red, &st);
        if (threadIdx.x == 0) lw = sc_mul(lw, l);
        cur = nxt;
        nxt = nxt == LW ? LW2 : LW;
      }
      const T v = blk_dot(cur, RP + (size_t)(y0 + w) * s2, bu[y0 + w] * D2, chi, bl[y0 + w], red);
      if (threadIdx.x == 0) {
        const dz q = dz_mul(to_dz(v), ival);
        const double f = sc_ratio(sc_mul(lw, logR[y0 + w]), logL[Ly]);
        ere += (hr * q.re - hi * q.im) * f;
        eim += (hr * q.im + hi * q.re) * f;
      }
    }
  }
  if (threadIdx.x == 0) {
    double* out = pairout + ((size_t)smp * g.Lx + x) * 4;
    out[0] = 0.0;
    out[1] = 0.0;
    out[2] = ere;
    out[3] = eim;
    int s = st;
    if (!(dz_abs(to_dz(val)) != 0.0) || !isfinite(ere) || !isfinite(eim)) s |= ST_NONFINITE;
    if (s) atomicOr(status + smp, s);
  }
  __syncthreads();
}

template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, MinBlocks<T>::value) k_pair(G g, Plan plan, const T* __restrict__ Tpad,
                                                   const uint8_t* __restrict__ S, int Ns, const T* envs,
                                                   const double* logs, TermTab tt, double* pairout, int* status) {
  extern __shared__ __align__(16) char smem[];
  const int nx = g.Lx - 1;
  for (int item = blockIdx.x; item < Ns * nx; item += gridDim.x)
    pair_item(g, plan, smem, Tpad, S, item / nx, item % nx, envs, logs, tt, pairout, status);
}

// ------------------------------------------------------------------------------------------
// Per-sample combine: ln psi_top from row Lx-1, E_loc = diagonal + row terms + pair terms.
// One warp (all 32 lanes) per sample.
__device__ __forceinline__ void combine_sample(const Geo g, int smp, const uint8_t* __restrict__ S,
                                               const double* rowout, const double* pairout, int use_rows_all,
                                               int use_pairs, const DiagTab dg, double* logabs, double* phase,
                                               double* eloc) {
  const int lane = threadIdx.x & 31;
  const int N = g.Lx * g.Ly;
  const uint8_t* Ss = S + (size_t)smp * N;
  double re = 0.0, im = 0.0;
  if (eloc) {
    for (int p = lane; p < dg.npairs; p += 32) re += dg.pair_v[p] * (double)Ss[dg.pair_ij[2 * p]] * (double)Ss[dg.pair_ij[2 * p + 1]];
    if (dg.onsite)
      for (int i = lane; i < N; i += 32) re += dg.onsite[(size_t)i * g.d + (Ss[i] < g.d ? Ss[i] : 0)];
    if (use_rows_all)
      for (int x = lane; x < g.Lx; x += 32) {
        re += rowout[((size_t)smp * g.Lx + x) * 4 + 2];
        im += rowout[((size_t)smp * g.Lx + x) * 4 + 3];
      }
    if (use_pairs)
      for (int x = lane; x < g.Lx - 1; x += 32) {
        re += pairout[((size_t)smp * g.Lx + x) * 4 + 2];
        im += pairout[((size_t)smp * g.Lx + x) * 4 + 3];
      }
    re = warp_sum(re);
    im = warp_sum(im);
  }
  if (lane == 0) {
    const double* top = rowout + ((size_t)smp * g.Lx + (g.Lx - 1)) * 4;
    if (logabs) logabs[smp] = top[0];
    if (phase) phase[smp] = top[1];
    if (eloc) { eloc[2 * smp] = re; eloc[2 * smp + 1] = im; }
  }
}

#ifdef PEPS_DEFINE_COMMON
__global__ void k_combine(Geo g, int Ns, const uint8_t* __restrict__ S, const double* rowout, const double* pairout,
                          int use_rows_all, int use_pairs, DiagTab dg, double* logabs, double* phase, double* eloc) {
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarp = (gridDim.x * blockDim.x) >> 5;
  for (int smp = wid; smp < Ns; smp += nwarp)
    combine_sample(g, smp, S, rowout, pairout, use_rows_all, use_pairs, dg, logabs, phase, eloc);
}
// Global rotation of the physical index: out[site][s][c] = sum_t M[s][t] in[site][t][c] for the
// compact parameter layout (site blocks [s][l][u][r][d]); in: real or (re, im) pairs, out:
// (re, im) pairs.  One CTA per site (persistent over sites).
__global__ void k_rotate_theta(int N, int d, const long long* __restrict__ site_off, RotM M,
                               const double* __restrict__ in, int in_cplx, double* __restrict__ out) {
  for (int site = blockIdx.x; site < N; site += gridDim.x) {
    const long long off = site_off[site];
    const long long blk = (site_off[site + 1] - off) / d;
    for (long long o = threadIdx.x; o < d * blk; o += blockDim.x) {
      const int s = (int)(o / blk);
      const long long c = o % blk;
      double re = 0.0, im = 0.0;
      for (int t = 0; t < d; ++t) {
        const long long k = off + t * blk + c;
        const double xr = in_cplx ? in[2 * k] : in[k], xi = in_cplx ? in[2 * k + 1] : 0.0;
        const double mr = M.m[2 * (s * d + t)], mi = M.m[2 * (s * d + t) + 1];
        re += mr * xr - mi * xi;
        im += mr * xi + mi * xr;
      }
      out[2 * (off + o)] = re;
      out[2 * (off + o) + 1] = im;
    }
  }
}

// E_loc^bound = diagonal pairs + on-site terms + the per-term sums of k_bound.  One warp per sample.
__global__ void k_bound_combine(Geo g, int Ns, int nt, const uint8_t* __restrict__ S, const double* bout, DiagTab dg,
                                double* eloc) {
  const int lane = threadIdx.x & 31;
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarp = (gridDim.x * blockDim.x) >> 5;
  const int N = g.Lx * g.Ly;
  for (int smp = wid; smp < Ns; smp += nwarp) {
    const uint8_t* Ss = S + (size_t)smp * N;
    double re = 0.0, im = 0.0;
    for (int p = lane; p < dg.npairs; p += 32) re += dg.pair_v[p] * (double)Ss[dg.pair_ij[2 * p]] * (double)Ss[dg.pair_ij[2 * p + 1]];
    if (dg.onsite)
      for (int i = lane; i < N; i += 32) re += dg.onsite[(size_t)i * g.d + (Ss[i] < g.d ? Ss[i] : 0)];
    for (int t = lane; t < nt; t += 32) {
      re += bout[((size_t)smp * nt + t) * 2];
      im += bout[((size_t)smp * nt + t) * 2 + 1];
    }
    re = warp_sum(re);
    im = warp_sum(im);
    if (lane == 0) { eloc[2 * smp] = re; eloc[2 * smp + 1] = im; }
  }
}
#endif

// ------------------------------------------------------------------------------------------
// Buffers of the moves of one row, carved from the sampler's plan.
template <typename T>
struct MoveBufs {
  T *RP, *t1, *t2, *eu, *el, *A1, *A2, *LW, *LW2, *LC;
  double* red;
};
template <typename T>
__device__ MoveBufs<T> carve_moves(const Plan& plan, char* smem, char* gbase) {
  MoveBufs<T> b;
  b.RP = (T*)buf_ptr(plan, B_RP, smem, gbase);
  b.t1 = (T*)buf_ptr(plan, B_T1, smem, gbase);
  b.t2 = (T*)buf_ptr(plan, B_T2, smem, gbase);
  b.eu = (T*)buf_ptr(plan, B_EU, smem, gbase);
  b.el = (T*)buf_ptr(plan, B_EL, smem, gbase);
  b.A1 = (T*)buf_ptr(plan, B_A, smem, gbase);
  b.A2 = (T*)buf_ptr(plan, B_A2, smem, gbase);
  b.LW = (T*)buf_ptr(plan, B_LW, smem, gbase);
  b.LW2 = (T*)buf_ptr(plan, B_LW2, smem, gbase);
  b.LC = (T*)buf_ptr(plan, B_LP, smem, gbase);
  b.red = (double*)buf_ptr(plan, B_RED, smem, gbase);
  return b;
}

// Random slots before row x in a sweep: the rows already visited (x of them going down,
// Lx-1-x going up) times the moves of a row (in-row moves plus, for exchanges, Ly vertical ones).
template <typename G>
__device__ inline unsigned sweep_slot0(const G& g, int x, int up, int move) {
  const unsigned per = (unsigned)(((move == 0) ? g.Ly - 1 : g.Ly) + ((move == 0) ? g.Ly : 0));
  return (unsigned)(up ? (g.Lx - 1 - x) : x) * per;
}

// The moves of row x of one chain in a sweep going down (up = 0) or up (up = 1): the in-row
// moves (exchange (x,y)<->(x,y+1), flip (x,y), y in order) judged with
// psi_x = E^u[x-1] . T[x] . E^l[x+1], then the vertical exchanges of the rows (xt, xt+1), with
// xt = x going down (x < Lx-1) and xt = x-1 going up (x > 0), judged with
// psi_{xt,xt+1} = E^u[xt-1] . T[xt] . T[xt+1] . E^l[xt+2].  Slots from slot0 on; Sl (shared) is
// updated in place; *acc counts the accepted moves (the same value in every thread).
template <typename T, typename G>
__device__ __noinline__ void row_moves(const G g, const Plan plan, const MoveBufs<T> b, const T* Tpad, uint8_t* Sl,
                          const T* env, int x, int up, int move, unsigned slot0, unsigned long long sweep_id, int c,
                          unsigned long long seed, long long* acc, int* st) {
  __shared__ Scaled logR[MAX_LY + 1];   // factors taken out of the partials
  __shared__ Scaled logLc, lcur;        // of the running left partial; |psi| of the configuration
  __shared__ int accept_flag;
  __shared__ int bu[MAX_LY + 1], bl[MAX_LY + 1], sl_[MAX_LY], sr_[MAX_LY];
  auto ext = [&](int y) { return BondExt{bu[y], bu[y + 1], bl[y], bl[y + 1]}; };
  const int D = g.D, D2 = g.D * g.D, chi = g.chi, cd = g.chi * g.D;
  const int Ly = g.Ly, Lx = g.Lx, se = g.se, s2 = g.s2;
  const size_t rowsz = (size_t)Ly * se;
  const int nmv = (move == 0) ? Ly - 1 : Ly;
  unsigned slot = slot0;
  T *RP = b.RP, *t1 = b.t1, *t2 = b.t2, *eu = b.eu, *el = b.el, *A1 = b.A1, *A2 = b.A2, *LW = b.LW, *LW2 = b.LW2,
    *LC = b.LC;
  double* red = b.red;
  // ---- moves inside row x with psi_x (E^u[x-1], E^l[x+1])
  {
    const T* EU = env + (size_t)slot_up(g, x - 1) * rowsz;
    const T* EL = env + (size_t)slot_lo(g, x + 1) * rowsz;
    mps_bonds(g, EU, bu, sl_, sr_);
    mps_bonds(g, EL, bl, sl_, sr_);
    blk_unit(RP + (size_t)Ly * se, cd);
    if (threadIdx.x == 0) logR[Ly] = sc_one();
    for (int y = Ly - 1; y >= 0; --y) {
      blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
      blk_copy(el, EL + (size_t)y * se, bl[y] * cd);
      load_A(A1, Tpad, g, x * Ly + y, Sl[x * Ly + y], false);
      __syncthreads();
      absorb1_right(g, ext(y), RP + (size_t)(y + 1) * se, eu, A1, el, t1, t2, RP + (size_t)y * se);
      const double l = (double)blk_normalize(RP + (size_t)y * se, bu[y] * D, chi, bl[y], red, st);
      if (threadIdx.x == 0) logR[y] = sc_mul(logR[y + 1], l);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      lcur = sc_amplitude(logR[0], dz_abs(to_dz(RP[0])));
      logLc = sc_one();
    }
    blk_unit(LC, cd);
    __syncthreads();
    for (int y = 0; y < nmv; ++y) {
      const unsigned my_slot = slot++;
      const int i0 = x * Ly + y, i1 = i0 + 1;
      const bool possible = (move == 0) ? (Sl[i0] != Sl[i1]) : true;
      int taken = 0;
      if (possible) {
        // the window: LC with column y in its proposed state (LW2, kept: it is the next LC if
        // the move is accepted), then for an exchange column y+1 as well (LW)
        const int w_ = (move == 0) ? 2 : 1;
        Scaled lw = sc_one();  // in thread 0
        double l0 = 0.0;
        for (int cc = 0; cc < w_; ++cc) {
          const int site = i0 + cc;
          int s_new;
          if (move == 0) s_new = (cc == 0) ? Sl[i1] : Sl[i0];
          else s_new = g.d - 1 - Sl[site];
          blk_copy(eu, EU + (size_t)(y + cc) * se, bu[y + cc] * cd);
          blk_copy(el, EL + (size_t)(y + cc) * se, bl[y + cc] * cd);
          load_A(A1, Tpad, g, site, s_new, false);
          __syncthreads();
          if (cc == 0) {
            absorb1(g, ext(y), LC, eu, A1, el, t1, t2, LW2);
            l0 = (double)blk_normalize(LW2, bu[y + 1] * D, chi, bl[y + 1], red, st);
            if (threadIdx.x == 0) lw = sc_mul(logLc, l0);
          } else {
            absorb1(g, ext(y + 1), LW2, eu, A1, el, t1, t2, LW);
            const double l = (double)blk_normalize(LW, bu[y + 2] * D, chi, bl[y + 2], red, st);
            if (threadIdx.x == 0) lw = sc_mul(lw, l);
          }
          __syncthreads();
        }
        const T v = blk_dot(w_ == 2 ? LW : LW2, RP + (size_t)(y + w_) * se, bu[y + w_] * D, chi, bl[y + w_], red);
        if (threadIdx.x == 0) {
          const double u = uniform53(my_slot, (uint32_t)sweep_id, (uint32_t)c, 0u, seed);
          const Scaled l1 = sc_mul(sc_mul(lw, logR[y + w_]), dz_abs(to_dz(v)));
          accept_flag = sc_accept(u, l1, lcur) ? 1 : 0;
          if (accept_flag) {
            lcur = l1;
            if (move == 0) { const uint8_t tmp = Sl[i0]; Sl[i0] = Sl[i1]; Sl[i1] = tmp; }
            else Sl[i0] = (uint8_t)(g.d - 1 - Sl[i0]);
          }
        }
        __syncthreads();
        *acc += accept_flag;
        taken = accept_flag;
        if (taken) {
          // column y now holds the proposed state: the new LC is the window's first column
          T* const tmp = LC;
          LC = LW2;
          LW2 = tmp;
          if (threadIdx.x == 0) logLc = sc_mul(logLc, l0);
        }
      }
      if (!taken) {
        blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
        blk_copy(el, EL + (size_t)y * se, bl[y] * cd);
        load_A(A1, Tpad, g, x * Ly + y, Sl[x * Ly + y], false);
        __syncthreads();
        absorb1(g, ext(y), LC, eu, A1, el, t1, t2, LW2);
        const double l = (double)blk_normalize(LW2, bu[y + 1] * D, chi, bl[y + 1], red, st);
        T* const tmp = LC;
        LC = LW2;
        LW2 = tmp;
        if (threadIdx.x == 0) logLc = sc_mul(logLc, l);
      }
    }
  }
  // ---- vertical moves (xt, y) <-> (xt+1, y) with psi_{xt,xt+1} (E^u[xt-1], E^l[xt+2])
  const int xt = up ? x - 1 : x;
  if (move == 0 && xt >= 0 && xt < Lx - 1) {
    const T* EU = env + (size_t)slot_up(g, xt - 1) * rowsz;
    const T* EL2 = env + (size_t)slot_lo(g, xt + 2) * rowsz;
    mps_bonds(g, EU, bu, sl_, sr_);
    mps_bonds(g, EL2, bl, sl_, sr_);
    blk_unit(RP + (size_t)Ly * s2, D2 * chi);
    if (threadIdx.x == 0) logR[Ly] = sc_one();
    for (int y = Ly - 1; y >= 0; --y) {
      blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
      blk_copy(el, EL2 + (size_t)y * se, bl[y] * cd);
      load_A(A1, Tpad, g, xt * Ly + y, Sl[xt * Ly + y], false);
      load_A(A2, Tpad, g, (xt + 1) * Ly + y, Sl[(xt + 1) * Ly + y], false);
      __syncthreads();
      absorb2_right(g, ext(y), RP + (size_t)(y + 1) * s2, eu, A1, A2, el, t1, t2, RP + (size_t)y * s2, plan.cx);
      const double l = (double)blk_normalize(RP + (size_t)y * s2, bu[y] * D2, chi, bl[y], red, st);
      if (threadIdx.x == 0) logR[y] = sc_mul(logR[y + 1], l);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      lcur = sc_amplitude(logR[0], dz_abs(to_dz(RP[0])));
      logLc = sc_one();
    }
    blk_unit(LC, D2 * chi);
    __syncthreads();
    for (int y = 0; y < Ly; ++y) {
      const unsigned my_slot = slot++;
      const int i0 = xt * Ly + y, i1 = (xt + 1) * Ly + y;
      blk_copy(eu, EU + (size_t)y * se, bu[y] * cd);
      blk_copy(el, EL2 + (size_t)y * se, bl[y] * cd);
      int taken = 0;
      if (Sl[i0] != Sl[i1]) {
        load_A(A1, Tpad, g, i0, Sl[i1], false);
        load_A(A2, Tpad, g, i1, Sl[i0], false);
        __syncthreads();
        absorb2(g, ext(y), LC, eu, A1, A2, el, t1, t2, LW2, plan.cx);
        const double l0 = (double)blk_normalize(LW2, bu[y + 1] * D2, chi, bl[y + 1], red, st);
        const T v = blk_dot(LW2, RP + (size_t)(y + 1) * s2, bu[y + 1] * D2, chi, bl[y + 1], red);
        if (threadIdx.x == 0) {
          const double u = uniform53(my_slot, (uint32_t)sweep_id, (uint32_t)c, 0u, seed);
          const Scaled l1 = sc_mul(sc_mul(sc_mul(logLc, l0), logR[y + 1]), dz_abs(to_dz(v)));
          accept_flag = sc_accept(u, l1, lcur) ? 1 : 0;
          if (accept_flag) {
            lcur = l1;
            const uint8_t tmp = Sl[i0]; Sl[i0] = Sl[i1]; Sl[i1] = tmp;
          }
        }
        __syncthreads();
        *acc += accept_flag;
        taken = accept_flag;
        if (taken) {
          // the proposal's window is the new LC
          T* const tmp = LC;
          LC = LW2;
          LW2 = tmp;
          if (threadIdx.x == 0) logLc = sc_mul(logLc, l0);
        }
      }
      if (!taken) {
        load_A(A1, Tpad, g, i0, Sl[i0], false);
        load_A(A2, Tpad, g, i1, Sl[i1], false);
        __syncthreads();
        absorb2(g, ext(y), LC, eu, A1, A2, el, t1, t2, LW2, plan.cx);
        const double l = (double)blk_normalize(LW2, bu[y + 1] * D2, chi, bl[y + 1], red, st);
        T* const tmp = LC;
        LC = LW2;
        LW2 = tmp;
        if (threadIdx.x == 0) logLc = sc_mul(logLc, l);
      }
    }
  }
}

// Trivial boundary rows of a sweep: E^u[-1] (going down) or E^l[Lx] (going up), log 0.
template <typename T, typename G>
__device__ void sweep_trivial_row(const G& g, T* env, double* lg, int up) {
  const size_t rowsz = (size_t)g.Ly * g.se;
  const int slot = up ? slot_lo(g, g.Lx) : slot_up(g, -1);
  for (int k = 0; k < g.Ly; ++k) blk_unit(env + (size_t)slot * rowsz + (size_t)k * g.se, g.se);
  if (threadIdx.x == 0) lg[slot] = 0.0;
}

// ------------------------------------------------------------------------------------------
// The Metropolis sweep split by rows (FP32: the row steps then run at the environment kernel's
// occupancy).  A downward sweep = k_env (lower environments of every chain), then for
// x = 0 .. Lx-1: k_sweep_moves(x) and k_env_row(x) (E^u[x] from the updated row); an upward
// sweep starts from the upper environments (the previous sweep's, or k_env's at the start of a
// call) and runs x = Lx-1 .. 0 with k_env_row building E^l[x].
template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, EnvBlocks<T>::value) k_sweep_moves(G g, Plan plan,
                                                        const T* __restrict__ Tpad, uint8_t* S, int Ns, int move,
                                                        int x, int up, unsigned long long seed,
                                                        unsigned long long sweep_id, T* envs, double* logs,
                                                        long long* accepted, int* status) {
  extern __shared__ __align__(16) char smem[];
  char* gbase = plan.gbase;
  const MoveBufs<T> b = carve_moves<T>(plan, smem, gbase);
  uint8_t* Sl = (uint8_t*)buf_ptr(plan, B_S, smem, gbase);
  __shared__ int st;
  const int N = g.Lx * g.Ly;
  const unsigned slot0 = sweep_slot0(g, x, up, move);
  for (int c = blockIdx.x; c < Ns; c += gridDim.x) {
    uint8_t* Sg = S + (size_t)c * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) Sl[i] = Sg[i];
    if (threadIdx.x == 0) st = 0;
    long long acc = 0;
    T* env = envs + (size_t)c * env_sample_elems(g);
    double* lg = logs + (size_t)c * 2 * g.Lx;
    if ((!up && x == 0) || (up && x == g.Lx - 1)) sweep_trivial_row(g, env, lg, up);
    __syncthreads();
    row_moves(g, plan, b, Tpad, Sl, env, x, up, move, slot0, sweep_id, c, seed, &acc, &st);
    for (int i = threadIdx.x; i < N; i += blockDim.x) Sg[i] = Sl[i];
    if (threadIdx.x == 0) {
      if (accepted) accepted[c] += acc;
      if (st) atomicOr(status + c, st);
    }
    __syncthreads();
  }
}

// One environment row of every chain from its (updated) row x, for the sweep's direction:
// going down E^u[x] (the first row for x = 0, else one row step from E^u[x-1]), going up E^l[x]
// (the last row for x = Lx-1, else one row step from E^l[x+1]); compiled for the environment
// kernel's occupancy.  ustat (may be null): also collects the row steps' status bits (the last
// sweep's, for a later evaluation that reuses these environments).
template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, EnvBlocks<T>::value) k_env_row(G g, Plan plan, const T* __restrict__ Tpad,
                                                      const uint8_t* __restrict__ S, int Ns, int x, int lower,
                                                      T* envs, double* logs, int* status, int* ustat) {
  extern __shared__ __align__(16) char smem[];
  char* gbase = plan.gbase;
  RowWork<T> w = carve_row<T>(plan, smem, gbase);
  __shared__ int st, flag;
  const int N = g.Lx * g.Ly;
  const size_t rowsz = (size_t)g.Ly * g.se;
  for (int c = blockIdx.x; c < Ns; c += gridDim.x) {
    if (threadIdx.x == 0) st = 0;
    __syncthreads();
    T* env = envs + (size_t)c * env_sample_elems(g);
    double* lg = logs + (size_t)c * 2 * g.Lx;
    const uint8_t* Ss = S + (size_t)c * N;
    const int slot = lower ? slot_lo(g, x) : slot_up(g, x), prev = lower ? slot_lo(g, x + 1) : slot_up(g, x - 1);
    const bool first = lower ? x == g.Lx - 1 : x == 0;
    double l0 = 0.0;  // the row before's logarithm, in thread 0
    if (threadIdx.x == 0 && !first) l0 = lg[prev];
    Scaled l;
    if (first)
      l = env_first_row(g, env + (size_t)slot * rowsz, Tpad, x, Ss + (size_t)x * g.Ly, lower != 0, w.A, w.Z, w.red, &st);
    else
      l = env_row_step_inl(g, env + (size_t)prev * rowsz, env + (size_t)slot * rowsz, Tpad, x, Ss + (size_t)x * g.Ly,
                           lower != 0, w, &st, &flag);
    if (threadIdx.x == 0) {
      lg[slot] = l0 + sc_log(l);
      if (st) atomicOr(status + c, st);
      if (st && ustat) atomicOr(ustat + c, st);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// Metropolis sweeps in one launch: one CTA per chain (persistent over chains); the FP64 and
// complex path.  Sweeps alternate direction with the sweep id (even: down the rows, odd: up),
// each starting from the environments the previous one left: going down, the lower
// environments of the current configuration (built at the sweep's start) and E^u rebuilt row
// by row; going up, the upper ones (the previous sweep's, or built at the start of the launch)
// and E^l rebuilt row by row.  Same moves, slots and decisions as the split FP32 sweep.
template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, MinBlocks<T>::value) k_sample(G g, Plan plan, const T* __restrict__ Tpad, uint8_t* S,
                                                     int Ns, int move, int nsweeps, unsigned long long seed,
                                                     unsigned long long sweep0, T* envs, double* logs,
                                                     long long* accepted, int* status) {
  extern __shared__ __align__(16) char smem[];
  char* gbase = plan.gbase;
  RowWork<T> w = carve_row<T>(plan, smem, gbase);
  const MoveBufs<T> b = carve_moves<T>(plan, smem, gbase);
  uint8_t* Sl = (uint8_t*)buf_ptr(plan, B_S, smem, gbase);
  __shared__ int st, flag;
  const int N = g.Lx * g.Ly, Ly = g.Ly, Lx = g.Lx;
  const size_t rowsz = (size_t)Ly * g.se;
  for (int c = blockIdx.x; c < Ns; c += gridDim.x) {
    uint8_t* Sg = S + (size_t)c * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) Sl[i] = Sg[i];
    if (threadIdx.x == 0) st = 0;
    long long acc = 0;
    T* env = envs + (size_t)c * env_sample_elems(g);
    double* lg = logs + (size_t)c * 2 * Lx;
    __syncthreads();
    for (int t = 0; t < nsweeps; ++t) {
      const unsigned long long sweep_id = sweep0 + (unsigned long long)t;
      const int up = (int)(sweep_id & 1ull);
      if (!up) {
        build_side_call(g, 1, Tpad, Sl, env, lg, w, &st, &flag);
        sweep_trivial_row(g, env, lg, 0);
        __syncthreads();
        for (int x = 0; x < Lx; ++x) {
          row_moves(g, plan, b, Tpad, Sl, env, x, 0, move, sweep_slot0(g, x, 0, move), sweep_id, c, seed, &acc, &st);
          if (x < Lx - 1) {
            const size_t sl = (size_t)slot_up(g, x) * rowsz;
            Scaled l;
            if (x == 0) l = env_first_row(g, env + sl, Tpad, 0, Sl, false, w.A, w.Z, w.red, &st);
            else l = env_row_step(g, env + (size_t)slot_up(g, x - 1) * rowsz, env + sl, Tpad, x,
                                  Sl + (size_t)x * Ly, false, w, &st, &flag);
            if (threadIdx.x == 0) lg[slot_up(g, x)] = (x == 0 ? 0.0 : lg[slot_up(g, x - 1)]) + sc_log(l);
            __syncthreads();
          }
        }
      } else {
        if (t == 0) build_side_call(g, 0, Tpad, Sl, env, lg, w, &st, &flag);
        sweep_trivial_row(g, env, lg, 1);
        __syncthreads();
        for (int x = Lx - 1; x >= 0; --x) {
          row_moves(g, plan, b, Tpad, Sl, env, x, 1, move, sweep_slot0(g, x, 1, move), sweep_id, c, seed, &acc, &st);
          if (x > 0) {
            const size_t sl = (size_t)slot_lo(g, x) * rowsz;
            Scaled l;
            if (x == Lx - 1) l = env_first_row(g, env + sl, Tpad, x, Sl + (size_t)x * Ly, true, w.A, w.Z, w.red, &st);
            else l = env_row_step(g, env + (size_t)slot_lo(g, x + 1) * rowsz, env + sl, Tpad, x,
                                  Sl + (size_t)x * Ly, true, w, &st, &flag);
            if (threadIdx.x == 0) lg[slot_lo(g, x)] = (x == Lx - 1 ? 0.0 : lg[slot_lo(g, x + 1)]) + sc_log(l);
            __syncthreads();
          }
        }
      }
    }
    for (int i = threadIdx.x; i < N; i += blockDim.x) Sg[i] = Sl[i];
    if (threadIdx.x == 0) {
      if (accepted) accepted[c] += acc;
      if (st) atomicOr(status + c, st);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// Variational-bound local energy with one fixed cut: every amplitude is
// psi_i(S) = E^u[i-1](S) . E^l[i](S) (0-based rows; the upper MPS holds rows 0..i-1).  One work
// item per (sample, term): for every off-diagonal entry h[a][b] of the term the environments of
// S' (the term's sites set to the digits of b) are rebuilt only on the rows between the first
// changed row and the cut, starting from S's stored environments (rows farther from the cut
// are identical for S and S'), then overlapped.  bout[(smp nt + t)]: the term's sum
// h[a][b] psi_i(S') / psi_i(S) (diagonal entries included) as (re, im); item t = 0 also writes
// ln|psi_i(S)| and its phase.
template <typename T, typename G>
__global__ void __launch_bounds__(NTHREADS, MinBlocks<T>::value) k_bound(G g, Plan plan, const T* __restrict__ Tpad,
                                                    const uint8_t* __restrict__ S, int Ns, int cut,
                                                    const T* envs, const double* logs, TermTab tt, double* bout,
                                                    double* logabs, double* phase, int* status) {
  extern __shared__ __align__(16) char smem[];
  char* gbase = plan.gbase;
  RowWork<T> w = carve_row<T>(plan, smem, gbase);
  uint8_t* Sl = (uint8_t*)buf_ptr(plan, B_S, smem, gbase);
  T* EUb = (T*)buf_ptr(plan, B_LP, smem, gbase);   // 2 rows: rebuilt upper environments
  T* ELb = (T*)buf_ptr(plan, B_RP, smem, gbase);   // 2 rows: rebuilt lower environments
  T* Lb = (T*)buf_ptr(plan, B_LW, smem, gbase);    // 2 chi^2: overlap partials
  T* tb = (T*)buf_ptr(plan, B_LW2, smem, gbase);   // chi D chi
  T* Lb2 = Lb + (size_t)g.chi * g.chi;
  __shared__ int st, flag;
  const int N = g.Lx * g.Ly, Ly = g.Ly, Lx = g.Lx;
  const size_t rowsz = (size_t)Ly * g.se;
  const int nt = tt.nterm > 0 ? tt.nterm : 1;
  const int su = slot_up(g, cut - 1), sl = slot_lo(g, cut);
  for (int item = blockIdx.x; item < Ns * nt; item += gridDim.x) {
    const int smp = item / nt, t = item % nt;
    const uint8_t* Ss = S + (size_t)smp * N;
    const T* env = envs + (size_t)smp * env_sample_elems(g);
    const double* lg = logs + (size_t)smp * 2 * Lx;
    if (threadIdx.x == 0) st = 0;
    __syncthreads();
    Scaled f0 = sc_one();
    const dz z0 = to_dz(mps_overlap(g, env + (size_t)su * rowsz, env + (size_t)sl * rowsz, Lb, Lb2, tb, w.red, &st, &f0));
    const double l0 = threadIdx.x == 0 ? lg[su] + lg[sl] + sc_log(f0) : 0.0;
    double ere = 0.0, eim = 0.0;
    if (t < tt.nterm) {
      const int* ti = tt.tinfo + (size_t)t * TI_N;
      const int a = local_index(ti, Ss, g.d);
      for (int e = ti[TI_EOFF]; e < ti[TI_EOFF] + ti[TI_ECNT]; ++e) {
        if (tt.ent_ab[2 * e] != a) continue;
        const int b = tt.ent_ab[2 * e + 1];
        const double hr = tt.ent_h[2 * e], hi = tt.ent_h[2 * e + 1];
        if (b == a) { ere += hr; eim += hi; continue; }
        // S' and the rows it changes on each side of the cut
        for (int i = threadIdx.x; i < N; i += blockDim.x) Sl[i] = (uint8_t)state_after(ti, i, Ss, b, g.d);
        int rlo = Lx, rhi = -1;
        for (int k = 0; k < ti[TI_K]; ++k) {
          const int site = ti[TI_S0 + k], r = site / Ly;
          if (state_after(ti, site, Ss, b, g.d) == Ss[site]) continue;
          if (r < cut) rlo = min(rlo, r);
          else rhi = max(rhi, r);
        }
        __syncthreads();
        const T* EU = env + (size_t)su * rowsz;
        double lu = lg[su];
        if (rlo < cut) {
          const T* prev = env + (size_t)slot_up(g, rlo - 1) * rowsz;
          lu = lg[slot_up(g, rlo - 1)];
          for (int r = rlo; r < cut; ++r) {
            T* out = EUb + (size_t)((r - rlo) & 1) * rowsz;
            Scaled f;
            if (r == 0) f = env_first_row(g, out, Tpad, 0, Sl, false, w.A, w.Z, w.red, &st);
            else f = env_row_step(g, prev, out, Tpad, r, Sl + (size_t)r * Ly, false, w, &st, &flag);
            if (threadIdx.x == 0) lu = (r == 0 ? 0.0 : lu) + sc_log(f);
            prev = out;
          }
          EU = prev;
        }
        const T* EL = env + (size_t)sl * rowsz;
        double ll = lg[sl];
        if (rhi >= cut) {
          const T* prev = env + (size_t)slot_lo(g, rhi + 1) * rowsz;
          ll = lg[slot_lo(g, rhi + 1)];
          for (int r = rhi; r >= cut; --r) {
            T* out = ELb + (size_t)((rhi - r) & 1) * rowsz;
            Scaled f;
            if (r == Lx - 1) f = env_first_row(g, out, Tpad, Lx - 1, Sl + (size_t)(Lx - 1) * Ly, true, w.A, w.Z, w.red, &st);
            else f = env_row_step(g, prev, out, Tpad, r, Sl + (size_t)r * Ly, true, w, &st, &flag);
            if (threadIdx.x == 0) ll = (r == Lx - 1 ? 0.0 : ll) + sc_log(f);
            prev = out;
          }
          EL = prev;
        }
        Scaled f1 = sc_one();
        const dz z1 = to_dz(mps_overlap(g, EU, EL, Lb, Lb2, tb, w.red, &st, &f1));
        if (threadIdx.x == 0 && (z1.re != 0.0 || z1.im != 0.0)) {
          const double l1 = lu + ll + sc_log(f1);
          const dz q = dz_div(z1, z0);
          const double f = exp(l1 - l0);
          ere += (hr * q.re - hi * q.im) * f;
          eim += (hr * q.im + hi * q.re) * f;
        }
      }
    }
    if (threadIdx.x == 0) {
      double* o = bout + ((size_t)smp * nt + t) * 2;
      o[0] = ere;
      o[1] = eim;
      const double av = dz_abs(z0);
      int s = st;
      if (t == 0) {
        const double la = (av > 0.0) ? log(av) + l0 : -INFINITY;
        if (logabs) logabs[smp] = la;
        if (phase) phase[smp] = (z0.im == 0.0) ? ((z0.re < 0.0) ? 3.141592653589793 : 0.0) : atan2(z0.im, z0.re);
      }
      if (!(av > 0.0) || !isfinite(ere) || !isfinite(eim)) s |= ST_NONFINITE;
      if (s) atomicOr(status + smp, s);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// theta (compact, double) -> padded kernel layout [site][s][l][u][r][d] in T
template <typename T>
__global__ void k_pad_theta(Geo g, const double* __restrict__ theta, const long long* site_off, T* Tpad) {
  const long long total = (long long)g.Lx * g.Ly * g.d * g.sT;
  const int D = g.D;
  for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < total; o += (long long)gridDim.x * blockDim.x) {
    const int dd = o % D, r = (o / D) % D, u = (o / (D * D)) % D, l = (o / (D * D * D)) % D;
    const int s = (o / g.sT) % g.d;
    const int site = (int)(o / ((long long)g.sT * g.d));
    const int x = site / g.Ly, y = site % g.Ly;
    int Dl, Du, Dr, Dd;
    site_dims(g, x, y, &Dl, &Du, &Dr, &Dd);
    T v = T(0);
    if (l < Dl && u < Du && r < Dr && dd < Dd) {
      const long long k = site_off[site] + (((long long)s * Dl + l) * Du + u) * Dr * Dd + (long long)r * Dd + dd;
      if constexpr (Scal<T>::complex) v = from_dz<T>(dz{theta[2 * k], theta[2 * k + 1]});  // (re, im) pairs
      else v = (T)theta[k];
    }
    Tpad[o] = v;
  }
}

// ------------------------------------------------------------------------------------------
// host-side launch wrappers (explicit instantiations for double and float).  Every launch goes
// to the kernel instantiated for the handle's (chi, D) when one exists, else to the runtime-
// geometry kernel.
template <typename F>
static cudaError_t with_geo(const Geo& g, F&& f) {
  if (g.chi == 16 && g.D == 4) return f(GeoS<16, 4>{g.Lx, g.Ly, g.d, g.cut});
  if (g.chi == 24 && g.D == 4) return f(GeoS<24, 4>{g.Lx, g.Ly, g.d, g.cut});
  return f(g);
}
// complex PEPS run the runtime-shape kernels only
template <typename T, typename F>
static cudaError_t with_geo_for(const Geo& g, F&& f) {
  if constexpr (Scal<T>::complex) return f(g);
  else return with_geo(g, f);
}

// Each translation unit defines PEPS_PART_ENV, PEPS_PART_ROW (k_row, k_pair, parameter padding)
// or PEPS_PART_SAMPLE and instantiates its kernels with PEPS_INST_<part>(T).
// (the occupancy at the fewest threads a launch may take, which gives the most CTAs)
#define PEPS_KATTR(NAME, KERNEL, MINT)                                                                             \
  template <typename T>                                                                                          \
  cudaError_t NAME(const Geo& g, size_t set_bytes, int* occ, size_t occ_smem) {                                  \
    return with_geo_for<T>(g, [&](auto gg) {                                                                            \
      using GG = decltype(gg);                                                                                   \
      cudaError_t e = cudaSuccess;                                                                               \
      if (set_bytes) e = cudaFuncSetAttribute(KERNEL<T, GG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)set_bytes); \
      if (e == cudaSuccess && occ) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, KERNEL<T, GG>, MINT, occ_smem); \
      return e;                                                                                                  \
    });                                                                                                          \
  }

#ifdef PEPS_PART_BATCH
// ------------------------------------------------------------------------------------------
// Ragged multi-instance batch in one persistent launch (runtime-shape kernels: every instance
// has its own lattice, D and chi).  The work queue lists (instance, sample) items, the costliest
// instances first; each CTA takes the next item with one atomic and runs that sample's whole
// evaluation with the same device functions as the per-handle kernels (so the results are bit
// for bit theirs): the environment sides, the one-row sandwiches of every row needed, the two-row
// sandwiches, and the combine.  The caller zeroes *next and every instance's status.
// the three phases as separate functions: their register allocations stay separate instead of
// one inlined body holding every phase's live ranges
// (an instance whose (chi, D) has a compiled specialisation runs it, as the per-handle kernels do)
template <typename T, typename G>
__device__ __noinline__ void batch_env(const BatchInst<T>& b, G g, char* smem, int smp) {
  RowWork<T> w = carve_row<T>(b.pe, smem, b.pe.gbase);
  env_item(g, w, b.Tpad, b.S, smp, 0, b.envs, b.logs, b.status);
  if (b.sides == 3) env_item(g, w, b.Tpad, b.S, smp, 1, b.envs, b.logs, b.status);
}
template <typename T, typename G>
__device__ __noinline__ void batch_row(const BatchInst<T>& b, G g, char* smem, int smp, int x) {
  row_item(g, b.pr, smem, b.Tpad, b.S, smp, x, b.envs, b.logs, b.O, b.site_off, b.Np, b.tt, b.rowout, b.status);
}
template <typename T, typename G>
__device__ __noinline__ void batch_pair(const BatchInst<T>& b, G g, char* smem, int smp, int x) {
  pair_item(g, b.pq, smem, b.Tpad, b.S, smp, x, b.envs, b.logs, b.tt, b.pairout, b.status);
}
template <typename T, typename G>
__device__ __forceinline__ void batch_sample(const BatchInst<T>& b, G g, char* smem, int smp) {
  batch_env<T, G>(b, g, smem, smp);
  const int x_lo = (b.sides == 3) ? 0 : g.Lx - 1;
  for (int x = x_lo; x < g.Lx; ++x) batch_row<T, G>(b, g, smem, smp, x);
  if (b.pairs)
    for (int x = 0; x + 1 < g.Lx; ++x) batch_pair<T, G>(b, g, smem, smp, x);
}

template <typename T>
__global__ void __launch_bounds__(NTHREADS, EnvBlocks<T>::value) k_batch(const BatchInst<T>* __restrict__ inst, int ninst, long long nitems,
                                                    unsigned long long* next) {
  extern __shared__ __align__(16) char smem[];
  __shared__ long long item_s;
  for (;;) {
    if (threadIdx.x == 0) item_s = (long long)atomicAdd(next, 1ull);
    __syncthreads();
    const long long item = item_s;
    if (item >= nitems) break;
    int i = 0;
    while (i + 1 < ninst && inst[i + 1].item0 <= item) ++i;
    const BatchInst<T>& b = inst[i];
    const int smp = (int)(item - b.item0);
    const Geo g = b.g;
    if constexpr (!Scal<T>::complex) {
      if (g.chi == 16 && g.D == 4) batch_sample<T>(b, GeoS<16, 4>{g.Lx, g.Ly, g.d, g.cut}, smem, smp);
      else if (g.chi == 24 && g.D == 4) batch_sample<T>(b, GeoS<24, 4>{g.Lx, g.Ly, g.d, g.cut}, smem, smp);
      else batch_sample<T>(b, g, smem, smp);
    } else {
      batch_sample<T>(b, g, smem, smp);
    }
    __syncthreads();
    if (threadIdx.x < 32)
      combine_sample(g, smp, b.S, b.rowout, b.pairout, b.want_e, b.pairs, b.dg, b.logabs, b.phase, b.eloc);
    __syncthreads();
  }
}

template <typename T>
cudaError_t launch_batch(const BatchInst<T>* inst, int ninst, long long nitems, unsigned long long* next, int grid,
                         size_t smem, cudaStream_t s) {
  k_batch<T><<<grid, NTHREADS, smem, s>>>(inst, ninst, nitems, next);
  return cudaGetLastError();
}
template <typename T>
cudaError_t kattr_batch(size_t set_bytes, int* occ, size_t occ_smem) {
  cudaError_t e = cudaSuccess;
  if (set_bytes) e = cudaFuncSetAttribute(k_batch<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)set_bytes);
  if (e == cudaSuccess && occ) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k_batch<T>, NTHREADS, occ_smem);
  return e;
}
#define PEPS_INST_BATCH(T)                                                                                       \
  template cudaError_t launch_batch<T>(const BatchInst<T>*, int, long long, unsigned long long*, int, size_t,     \
                                       cudaStream_t);                                                             \
  template cudaError_t kattr_batch<T>(size_t, int*, size_t);
#endif

#ifdef PEPS_PART_ENV
template <typename T>
cudaError_t launch_env(const Geo& g, const Plan& p, int grid, size_t smem, const T* Tpad, const uint8_t* S, int Ns,
                       int sides, T* envs, double* logs, int* status, cudaStream_t s) {
  return with_geo_for<T>(g, [&](auto gg) {
    k_env<T, decltype(gg)><<<grid, cta_threads(sizeof(typename Scal<T>::R), g.n, grid), smem, s>>>(gg, p, Tpad, S, Ns, sides, envs, logs, status);
    return cudaGetLastError();
  });
}
template <typename T>
cudaError_t launch_env_row(const Geo& g, const Plan& p, int grid, size_t smem, const T* Tpad, const uint8_t* S, int Ns,
                           int x, int lower, T* envs, double* logs, int* status, int* ustat, cudaStream_t s) {
  return with_geo_for<T>(g, [&](auto gg) {
    k_env_row<T, decltype(gg)><<<grid, cta_threads(sizeof(typename Scal<T>::R), g.n, grid), smem, s>>>(
        gg, p, Tpad, S, Ns, x, lower, envs, logs, status, ustat);
    return cudaGetLastError();
  });
}
PEPS_KATTR(kattr_env_only, k_env, cta_threads(sizeof(typename Scal<T>::R), g.n, 1 << 30))
PEPS_KATTR(kattr_env_row, k_env_row, cta_threads(sizeof(typename Scal<T>::R), g.n, 1 << 30))
// k_env and, in FP32, the sampler's k_env_row, which runs on the same plan
template <typename T>
cudaError_t kattr_env(const Geo& g, size_t set_bytes, int* occ, size_t occ_smem) {
  cudaError_t e = cudaSuccess;
  if constexpr (sizeof(T) == 4)
    if (set_bytes) e = kattr_env_row<T>(g, set_bytes, nullptr, 0);
  return e == cudaSuccess ? kattr_env_only<T>(g, set_bytes, occ, occ_smem) : e;
}
#define PEPS_INST_ENV_ROW(T)                                                                                      \
  template cudaError_t launch_env_row<T>(const Geo&, const Plan&, int, size_t, const T*, const uint8_t*, int, int, int, T*, \
                                         double*, int*, int*, cudaStream_t);
#define PEPS_INST_ENV(T)                                                                                          \
  template cudaError_t launch_env<T>(const Geo&, const Plan&, int, size_t, const T*, const uint8_t*, int, int, T*, \
                                     double*, int*, cudaStream_t);                                        \
  template cudaError_t kattr_env<T>(const Geo&, size_t, int*, size_t);
#endif

#ifdef PEPS_PART_ROW
template <typename T>
cudaError_t launch_row(const Geo& g, const Plan& p, int grid, size_t smem, const T* Tpad, const uint8_t* S, int Ns,
                       int x_lo, int x_hi, const T* envs, const double* logs, T* O, const long long* site_off,
                       long long Np, const TermTab& tt, double* rowout, int* status, cudaStream_t s) {
  return with_geo_for<T>(g, [&](auto gg) {
    k_row<T, decltype(gg)><<<grid, cta_threads(sizeof(typename Scal<T>::R), g.n, grid), smem, s>>>(gg, p, Tpad, S, Ns, x_lo, x_hi, envs, logs, O, site_off, Np,
                                                        tt, rowout, status);
    return cudaGetLastError();
  });
}
template <typename T>
cudaError_t launch_pair(const Geo& g, const Plan& p, int grid, size_t smem, const T* Tpad, const uint8_t* S, int Ns,
                        const T* envs, const double* logs, const TermTab& tt, double* pairout, int* status, cudaStream_t s) {
  return with_geo_for<T>(g, [&](auto gg) {
    k_pair<T, decltype(gg)><<<grid, cta_threads(sizeof(typename Scal<T>::R), g.n, grid), smem, s>>>(gg, p, Tpad, S, Ns, envs, logs, tt, pairout, status);
    return cudaGetLastError();
  });
}
template <typename T>
cudaError_t launch_pad(const Geo& g, const double* theta, const long long* site_off, T* Tpad, cudaStream_t s) {
  k_pad_theta<T><<<304, 256, 0, s>>>(g, theta, site_off, Tpad);
  return cudaGetLastError();
}
PEPS_KATTR(kattr_row, k_row, cta_threads(sizeof(typename Scal<T>::R), g.n, 1 << 30))
PEPS_KATTR(kattr_pair, k_pair, cta_threads(sizeof(typename Scal<T>::R), g.n, 1 << 30))
#define PEPS_INST_ROW(T)                                                                                          \
  template cudaError_t launch_row<T>(const Geo&, const Plan&, int, size_t, const T*, const uint8_t*, int, int, int, \
                                     const T*, const double*, T*, const long long*, long long, const TermTab&,    \
                                     double*, int*, cudaStream_t);                                                \
  template cudaError_t launch_pair<T>(const Geo&, const Plan&, int, size_t, const T*, const uint8_t*, int, const T*, \
                                      const double*, const TermTab&, double*, int*, cudaStream_t);                \
  template cudaError_t launch_pad<T>(const Geo&, const double*, const long long*, T*, cudaStream_t);              \
  template cudaError_t kattr_row<T>(const Geo&, size_t, int*, size_t);                                           \
  template cudaError_t kattr_pair<T>(const Geo&, size_t, int*, size_t);
#endif

#ifdef PEPS_PART_SAMPLE
// The FP32 moves take 64 threads beyond six CTAs per SM: they are sandwiches of one sample after the
// other, with a barrier per product (4096 chains, 8x8, D = 4, chi = 16: 41.6 -> 36.4 ms; the row step's
// kernels lose, 61.3 -> 65.2 ms).
template <typename T>
static int sample_threads(int n, int grid) {
  const int nt = cta_threads(sizeof(typename Scal<T>::R), n, grid);
  return sizeof(T) == 4 && grid > 6 * N_SM ? 64 : nt;
}
// FP32 runs the sweep split by rows (k_env for the lower environments, then k_sweep_moves and
// k_env_row per row; the environment plan pe / grid_e / smem_e for the row steps); the other
// precisions run the single-launch k_sample.
template <typename T>
cudaError_t launch_sample(const Geo& g, const Plan& p, int grid, size_t smem, const Plan& pe, int grid_e,
                          size_t smem_e, const T* Tpad, uint8_t* S, int Ns, int move, int nsweeps,
                          unsigned long long seed, unsigned long long sweep0, T* envs, double* logs,
                          long long* accepted, int* status, int* ustat, cudaStream_t s) {
  const int nt = sample_threads<T>(g.n, grid);
  return with_geo_for<T>(g, [&](auto gg) {
    using GG = decltype(gg);
    if constexpr (sizeof(T) == 4) {
      cudaError_t e = cudaSuccess;
      for (int t = 0; t < nsweeps; ++t) {
        const unsigned long long sid = sweep0 + t;
        const int up = (int)(sid & 1ull);
        int* us = (t == nsweeps - 1) ? ustat : nullptr;
        // a downward sweep starts from the lower environments of its configurations; an upward one
        // from the upper ones, which the previous sweep of this call left
        if (!up || t == 0) {
          if ((e = launch_env<T>(g, pe, grid_e, smem_e, Tpad, S, Ns, up ? 1 : 2, envs, logs, status, s)) != cudaSuccess) return e;
        }
        for (int i = 0; i < g.Lx; ++i) {
          const int x = up ? g.Lx - 1 - i : i;
          k_sweep_moves<T, GG><<<grid, nt, smem, s>>>(gg, p, Tpad, S, Ns, move, x, up, seed, sid, envs, logs, accepted,
                                                      status);
          if (i < g.Lx - 1 &&
              (e = launch_env_row<T>(g, pe, grid_e, smem_e, Tpad, S, Ns, x, up, envs, logs, status, us, s)) != cudaSuccess)
            return e;
        }
      }
    } else {
      k_sample<T, GG><<<grid, nt, smem, s>>>(gg, p, Tpad, S, Ns, move, nsweeps, seed, sweep0, envs, logs, accepted, status);
    }
    return cudaGetLastError();
  });
}
template <typename T>
cudaError_t kattr_sample(const Geo& g, size_t set_bytes, int* occ, size_t occ_smem) {
  const int nt = sample_threads<T>(g.n, 1 << 30);
  return with_geo_for<T>(g, [&](auto gg) {
    using GG = decltype(gg);
    auto kernel = [&](auto* k) {
      cudaError_t e = cudaSuccess;
      if (set_bytes) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)set_bytes);
      if (e == cudaSuccess && occ) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, nt, occ_smem);
      return e;
    };
    if constexpr (sizeof(T) == 4) return kernel(&k_sweep_moves<T, GG>);
    else return kernel(&k_sample<T, GG>);
  });
}
#define PEPS_INST_SAMPLE(T)                                                                                       \
  template cudaError_t launch_sample<T>(const Geo&, const Plan&, int, size_t, const Plan&, int, size_t, const T*, \
                                        uint8_t*, int, int, int, unsigned long long, unsigned long long, T*,      \
                                        double*, long long*, int*, int*, cudaStream_t);                           \
  template cudaError_t kattr_sample<T>(const Geo&, size_t, int*, size_t);
#endif

#ifdef PEPS_PART_BOUND
template <typename T>
cudaError_t launch_bound(const Geo& g, const Plan& p, int grid, size_t smem, const T* Tpad, const uint8_t* S, int Ns,
                         int cut, const T* envs, const double* logs, const TermTab& tt, double* bout, double* logabs,
                         double* phase, int* status, cudaStream_t s) {
  return with_geo_for<T>(g, [&](auto gg) {
    k_bound<T, decltype(gg)><<<grid, cta_threads(sizeof(typename Scal<T>::R), g.n, 1), smem, s>>>(gg, p, Tpad, S, Ns, cut, envs, logs, tt, bout, logabs, phase,
                                                          status);
    return cudaGetLastError();
  });
}
PEPS_KATTR(kattr_bound, k_bound, cta_threads(sizeof(typename Scal<T>::R), g.n, 1))
#define PEPS_INST_BOUND(T)                                                                                        \
  template cudaError_t launch_bound<T>(const Geo&, const Plan&, int, size_t, const T*, const uint8_t*, int, int,  \
                                       const T*, const double*, const TermTab&, double*, double*, double*, int*,  \
                                       cudaStream_t);                                                             \
  template cudaError_t kattr_bound<T>(const Geo&, size_t, int*, size_t);
#endif

#ifdef PEPS_DEFINE_COMMON
cudaError_t launch_rotate(int N, int d, const long long* site_off, const RotM& M, const double* in, int in_cplx,
                          double* out, cudaStream_t s) {
  k_rotate_theta<<<N < 1024 ? N : 1024, 256, 0, s>>>(N, d, site_off, M, in, in_cplx, out);
  return cudaGetLastError();
}
cudaError_t launch_bound_combine(const Geo& g, int Ns, int nt, const uint8_t* S, const double* bout, const DiagTab& dg,
                                 double* eloc, cudaStream_t s) {
  const int blocks = (Ns * 32 + 255) / 256;
  k_bound_combine<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(g, Ns, nt, S, bout, dg, eloc);
  return cudaGetLastError();
}
cudaError_t launch_combine(const Geo& g, int Ns, const uint8_t* S, const double* rowout, const double* pairout,
                           int use_rows_all, int use_pairs, const DiagTab& dg, double* logabs, double* phase,
                           double* eloc, cudaStream_t s) {
  const int blocks = (Ns * 32 + 255) / 256;
  k_combine<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(g, Ns, S, rowout, pairout, use_rows_all, use_pairs, dg, logabs, phase, eloc);
  return cudaGetLastError();
}
#endif

}  // namespace peps
