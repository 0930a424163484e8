// Channel form of the sweep: torn lines plus lagged couplings (cut entries
// that are not branches, e.g. controlled sources), and block Jacobi.
//
// Per sub-circuit P, sweep k (Sec. VI, Eq. 11 with the lagged couplings of
// the cut moved to the right-hand side with one sweep of delay, reading R2):
//   K_P x_P = b_P + sum_ports beta_s w_in(s) e_l(s) - sum_lag rho_q z_q e_i(q)
// with z_q = x_j(q) of the previous sweep (read from tile Q).  Condensed:
//   [w_out; y] = E_P [w_in; z] + [c; y0],   y = the node voltages of P that
// other tiles' lagged entries read ("probes").  E_P is built column by column
// from banded solves: input a with right-hand side sigma_a e_loc(a)
// (sigma = beta for a port, -rho for a lagged entry) gives, for outputs o,
//   E(o, a) = scale_o y(loc(o)) + [a, o are the same port] (W - 2g)/(W + 2g),
//   scale = 2 W beta for a port output, 1 for a probe.
// Block Jacobi is the case without lines: every cut entry is lagged and
// K_P = A_PP, x_P^k = A_PP^-1 (b_P - sum_Q A_PQ x_Q^(k-1)) (Sec. X).
//
// Residual of sweep k at row i: torn branch s (twin t):
//   ((W - 2g) u_s + (W + 2g) u_t - w_in(s) - w_in(t)) / 2  (waves carried as w / d),
// lagged entry q: rho_q (z_q - x_j^k)   (z_q = x_j^(k-1) was used).
#include <algorithm>
#include <cmath>

#include "band.cuh"
#include "gridctl.cuh"
#include "ptx.h"
#include "vtm_internal.h"

namespace vtm {

// one warp per input channel: column `a` of E_P (stored as row a of E_P^T)
__global__ void build_general_kernel(const int32_t* __restrict__ node_off,
                                     const int32_t* __restrict__ bwv,
                                     const int64_t* __restrict__ band_off,
                                     const double* __restrict__ Lc, const double* __restrict__ Uc,
                                     const int32_t* __restrict__ in_tile,
                                     const int32_t* __restrict__ in_off,
                                     const int32_t* __restrict__ out_off,
                                     const int32_t* __restrict__ in_loc,
                                     const int32_t* __restrict__ in_own_out,
                                     const double* __restrict__ sigma,
                                     const int32_t* __restrict__ out_loc,
                                     const double* __restrict__ scale,
                                     const double* __restrict__ diag,
                                     const int64_t* __restrict__ E_off,
                                     const int32_t* __restrict__ E_ld, double* __restrict__ E) {
  extern __shared__ double y[];
  const int a = blockIdx.x;
  const int t = in_tile[a];
  const int n = node_off[t + 1] - node_off[t];
  const int lane = threadIdx.x;
  for (int i = lane; i < n; i += 32) y[i] = 0.0;
  __syncwarp();
  const int la = in_loc[a];
  if (lane == 0) y[la] = sigma[a];
  __syncwarp();
  warp_band_solve_any(y, n, bwv[t], Lc + band_off[t], Uc + band_off[t], la);
  const int o0 = out_off[t], no = out_off[t + 1] - o0;
  double* row = E + E_off[t] + (size_t)(a - in_off[t]) * E_ld[t];
  const int own = in_own_out[a];
  for (int q = lane; q < no; q += 32) {
    const int o = o0 + q;
    double v = scale[o] * y[out_loc[o]];
    if (o == own) v += diag[o];
    row[q] = v;
  }
}

// c_o = scale_o x0(loc(o)) for every output (one block per tile)
__global__ void general_const_kernel(const int32_t* __restrict__ node_off,
                                     const int32_t* __restrict__ out_off,
                                     const int32_t* __restrict__ out_loc,
                                     const double* __restrict__ scale,
                                     const double* __restrict__ x0, double* __restrict__ c) {
  const int t = blockIdx.x;
  const int base = node_off[t];
  for (int o = out_off[t] + threadIdx.x; o < out_off[t + 1]; o += blockDim.x)
    c[o] = scale[o] * x0[base + out_loc[o]];
}

// v(row node) += sum of sigma_a * input_a over the inputs of that row (fixed order)
__global__ void general_inject_kernel(const int32_t* __restrict__ node_off,
                                      const int32_t* __restrict__ in_off,
                                      const int32_t* __restrict__ in_loc,
                                      const int32_t* __restrict__ res_perm,
                                      const uint8_t* __restrict__ res_run,
                                      const double* __restrict__ sigma,
                                      const double* __restrict__ in_state, double* __restrict__ v) {
  const int t = blockIdx.x;
  const int a0 = in_off[t], ni = in_off[t + 1] - a0;
  for (int k = threadIdx.x; k < ni; k += blockDim.x) {
    const int nr = res_run[a0 + k];
    if (!nr) continue;
    double acc = 0.0;
    for (int q = 0; q < nr; ++q) {
      const int a = a0 + res_perm[a0 + k + q];
      acc += sigma[a] * in_state[a];
    }
    v[node_off[t] + in_loc[a0 + res_perm[a0 + k]]] += acc;
  }
}

__device__ double gblock_sum(double v) {
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double tot = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += red[i];
  __syncthreads();
  return tot;
}

__device__ double gblock_sum_array(const double* __restrict__ a, int count) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += a[i];
  return gblock_sum(acc);
}

// One CTA per tile; the products run in KS groups of blockDim / KS threads:
// group g takes the inputs a = g, g + KS, ... of each output, the KS partial
// sums meet in shared memory and are added in group order (more loads in
// flight per output than one thread walking every input: a tile's E_P streams
// with only a few CTAs per SM).
template <int KS>
__global__ void __launch_bounds__(1024) general_sweep_kernel(
    const double* __restrict__ E, const int64_t* __restrict__ E_off, const int32_t* __restrict__ E_ld,
    const int32_t* __restrict__ in_off, const int32_t* __restrict__ out_off,
    const int32_t* __restrict__ in_src, const uint8_t* __restrict__ in_kind,
    const int32_t* __restrict__ in_twin, const int32_t* __restrict__ in_own_out,
    const double* __restrict__ coef, const double* __restrict__ dsc, const int32_t* __restrict__ res_perm,
    const uint8_t* __restrict__ res_run, const double* __restrict__ c, double* __restrict__ gin,
    double* __restrict__ gout, int64_t n_in, int64_t n_out, SweepCtrl* __restrict__ ctrl,
    double* __restrict__ partials, double* __restrict__ hist, int hist_len, int nparts) {
  extern __shared__ double sm[];
  __shared__ int s_k, s_flag;
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    s_k = *((volatile int*)&ctrl->k);
    s_flag = *((volatile int*)&ctrl->flag);
  }
  __syncthreads();
  if (s_flag) return;
  const int k = s_k;
  const int t = blockIdx.x;
  const int a0 = in_off[t], ni = in_off[t + 1] - a0;
  const int o0 = out_off[t], no = out_off[t + 1] - o0;
  double* vin = sm;       // [max_in]
  double* rc = sm + ni;   // [max_in]
  double* part = rc + ni;  // [KS][blockDim / KS]
  const double* pin = gin + (size_t)((k - 1) & 1) * n_in;
  const double* pout = gout + (size_t)((k - 1) & 1) * n_out;
  double* cin = gin + (size_t)(k & 1) * n_in;
  double* cout_ = gout + (size_t)(k & 1) * n_out;
  for (int q = threadIdx.x; q < ni; q += blockDim.x) {
    const int a = a0 + q;
    double vi = 0.0, r = 0.0;
    if (k > 1) {
      const double src = pout[in_src[a]];
      vi = src;
      if (in_kind[a] == 0) {
        const double wi_s = pin[a], wo_s = pout[in_own_out[a]];
        const double wi_t = pin[in_twin[a]], wo_t = src;
        // coef = g/W, dsc = d of the line (waves carried as w / d)
        const double Ss = wi_s + wo_s, St = wi_t + wo_t;
        r = 0.5 * dsc[a] * (0.5 * (Ss + St) - coef[a] * (Ss - St) - wi_s - wi_t);
      } else {
        r = coef[a] * (pin[a] - src);
      }
    }
    vin[q] = vi;
    rc[q] = r;
  }
  __syncthreads();
  double sq = 0.0;
  if (k > 1) {
    for (int q = threadIdx.x; q < ni; q += blockDim.x) {
      const int nr = res_run[a0 + q];
      if (nr) {
        double r = 0.0;
        for (int e = 0; e < nr; ++e) r += rc[res_perm[a0 + q + e]];
        sq += r * r;
      }
    }
  }
  const double tile_sq = gblock_sum(sq);
  const double* Eb = E + E_off[t];
  const int ld = E_ld[t];
  const int to = (int)blockDim.x / KS, g = threadIdx.x / to, ql = threadIdx.x % to;
  for (int q0 = 0; q0 < no; q0 += to) {
    const int q = q0 + ql;
    double acc = 0.0;
    if (q < no) {
#pragma unroll 4
      for (int a = g; a < ni; a += KS) acc += __ldg(Eb + (size_t)a * ld + q) * vin[a];
    }
    part[g * to + ql] = acc;
    __syncthreads();
    if (g == 0 && q < no) {
      double tot = c[o0 + q];
      for (int gg = 0; gg < KS; ++gg) tot += part[gg * to + ql];
      cout_[o0 + q] = tot;
    }
    __syncthreads();
  }
  for (int q = threadIdx.x; q < ni; q += blockDim.x) cin[a0 + q] = vin[q];
  if (threadIdx.x == 0) {
    partials[t] = tile_sq;
    __threadfence();
    s_last = atomicAdd(&ctrl->counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const double tot = gblock_sum_array(partials, nparts);
  if (threadIdx.x == 0) {
    int flag = 0;
    if (k > 1) {
      const int ks = k - 1;
      if (hist && ks <= hist_len) hist[ks - 1] = sqrt(tot / ctrl->bnorm2);
      if (ks == 1) ctrl->first_res2 = tot;
      ctrl->last_res2 = tot;
      if (!isfinite(tot) || (ks > 1 && tot > 1e12 * ctrl->first_res2 && ctrl->first_res2 > 0)) {
        flag = 3;
      } else if (tot <= ctrl->tol2) {
        flag = 1;
        ctrl->conv_sweep = ks;
      }
    }
    if (!flag && k >= ctrl->k_max) flag = 2;
    ctrl->counter = 0u;
    ctrl->k = k + 1;
    __threadfence();
    ctrl->flag = flag;
  }
}

// 16-byte asynchronous copies into shared memory, completing in groups
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The same sweeps in one cooperative launch, one bounded grid barrier per sweep (the
// control warp of gridctl.cuh).  A CTA owns a contiguous range of output pairs -- of
// one tile or several -- of equal cost (pairs times inputs): thread (pair, group) takes
// the inputs group, group + G, ... of its pair, so that every SM's FP64 pipe has the
// same work, which no split into whole tiles or slabs gives (460 slabs of 64 outputs on
// 152 SMs: 4 on some, 3 on most).  As many of a thread's elements of E_P as fit stay in
// shared memory for the whole solve; the rest stream from L2 through a ring of
// asynchronous copies that never stops: E_P does not change, so the first elements of
// sweep k + 1 are on their way while barrier k is awaited.  The residual of sweep k - 1
// is formed in that wait; what its rows need of w_in(k - 1) are the w_out(k - 2) the
// waves came from, so no incident value is stored before the last sweep.
// Slots of w_out: 8 (sweeps k - 2 to k + 1 may be in use at once, and the iterate that
// is kept is up to five sweeps old when every CTA has stopped).
// Bound by the FP64 pipe and the chain barrier - gather - products - sums around it.
// Measured, VCCS grid 640 x 640 in 100 tiles (46 MB of E_P, 9.8 us of FP64 pipe): one CTA
// per tile and launch 39 us per sweep, slabs of 64 outputs 24 us, here 16.5 us; solves of
// 100 sweeps on 1024 x 1024 in 256 tiles 17.9 -> 6.5 ms, 24 x 24 in 9 tiles 1.39 -> 0.98.
// Plans with more output pairs per SM than threads (over 230k outputs: 1024 x 1024 in
// tiles of 16 x 16) keep one CTA per tile: slabs of outputs were slower there (100
// sweeps in tiles of 16 x 16 14.8 ms against 24.2, of 8 x 8 21.6 against 44.3).
constexpr int kGenThreads = 768;  // and a control warp: 80 registers per thread
constexpr int kGenRing = 4, kGenMinSlots = 8;
// elements (pairs of outputs times an input) per thread below which fewer CTAs share the work
template <bool PORTS>
constexpr int kGenMinElems = PORTS ? 2 : 8;
struct GenCta {
  int32_t pair0, np;   // first output pair, pairs
  int32_t in0, nin;    // inputs of the tiles it touches
  int32_t q0, q1;      // residual entries (whole runs)
  int32_t i0, i1;      // inputs it stores after the last sweep
};
struct GenRes {
  const double* E;
  const int64_t* E_off;
  const int32_t *E_ld, *in_off, *out_off, *pair_off;
  const GenCta* ctas;
  const int32_t *in_src, *in_own_out, *res_in;
  const uint8_t *in_kind, *res_run;
  const double *coef, *dsc, *c;
  const double2* kd;  // port form: (g/W, d)
  double *gin, *gout;
  int64_t n_in, n_out;
  SweepCtrl* ctrl;
  unsigned long long* bar;
  double *part, *hist;
  int hist_len, nparts, nslots, vmax;
  uint32_t max_polls;
};

// PORTS: the sweeps of a plan without lagged couplings, FP64 throughout -- E_P = T_P, the
// inputs and outputs of a tile its ports in their order, the source of an input its twin.
// The last sweep leaves (w_in, w_out) pairs in gin.  For symmetric plans of up to 256 ports
// per tile, like kernel 13.  Measured per sweep, kernel 1 -> here: 64 tiles of 256 ports
// (27 MB of T_P, 7.7 us of busy FP64 pipe) 19 -> 11.1 us; 169 tiles of 128 ports 18.4 -> 9.3 us;
// 9 tiles of 128 ports 16.4 -> 7.0 us.  CTAs with as little as two elements per thread:
// 81 tiles of 124 ports 7.1 us, with at least eight 8.6 us (the channel form keeps eight:
// its inputs gather from more tiles).
template <bool PORTS>
__global__ void __launch_bounds__(kGenThreads + 32, 1) general_resident_kernel(const GenRes A) {
  constexpr int NT = kGenThreads, NW = NT / 32, S = kGenRing;
  extern __shared__ __align__(16) unsigned char gsm[];
  __shared__ int s_flag;
  __shared__ double s_part[2][NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_flag = 0;
  if (tid < NW) s_part[0][tid] = s_part[1][tid] = 0.0;
  __syncthreads();
  if (warp == NW) {
    res_control(A.ctrl, A.bar, A.part, A.hist, A.hist_len, A.max_polls, &s_flag, s_part[0], NW, NW, lane);
    return;
  }
  // shared memory: [nslots][NT] elements | [NT] sums | [vmax] incident values | [vmax] their sources |
  // [2 NT] output ids
  double2* slots = reinterpret_cast<double2*>(gsm) + tid;
  double2* red = reinterpret_cast<double2*>(gsm) + (size_t)A.nslots * NT;
  double* vin = reinterpret_cast<double*>(red + NT);
  int32_t* src = reinterpret_cast<int32_t*>(vin + A.vmax);
  int32_t* oid = src + A.vmax;
  const GenCta C = A.ctas[blockIdx.x];
  const int np = C.np, G = np > 0 ? NT / np : 0;
  const int l = np > 0 ? tid % np : 0, g = np > 0 ? tid / np : 0;
  int cnt = 0, vofs = 0, ld = 0;
  const double* Ep = A.E;
  if (g < G) {
    int lo = 0, hi = A.nparts;  // the tile of the pair
    const int pg = C.pair0 + l;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (A.pair_off[mid] <= pg) lo = mid;
      else hi = mid;
    }
    const int m = 2 * (pg - A.pair_off[lo]), ni = A.in_off[lo + 1] - A.in_off[lo];
    ld = A.E_ld[lo];
    cnt = ni > g ? (ni - g + G - 1) / G : 0;
    Ep = A.E + A.E_off[lo] + m + (size_t)g * ld;
    vofs = A.in_off[lo] - C.in0 + g;
    if (g == 0) {
      const int no = A.out_off[lo + 1] - A.out_off[lo], o = A.out_off[lo] + m;
      oid[2 * l] = o;
      oid[2 * l + 1] = m + 1 < no ? o + 1 : -1;
    }
  }
  for (int q = tid; q < C.nin; q += NT) src[q] = A.in_src[C.in0 + q];
  const size_t step = (size_t)G * ld;
  // elements 0 .. nres - 1 stay; the others pass through slots nslots - S ..
  const int nres = cnt <= A.nslots ? cnt : A.nslots - S, nstr = cnt - nres;
  double2* ring = slots + (size_t)(A.nslots - S) * NT;
  for (int i = 0; i < nres; ++i) cp_async16(slots + i * NT, Ep + i * step);
  cp_async_commit_group();
  cp_async_wait_group<0>();
  int an = 0, sn = 0;
  auto issue = [&]() {  // the next streamed element, round and round
    cp_async16(ring + sn * NT, Ep + (size_t)(nres + an) * step);
    cp_async_commit_group();
    an = an + 1 == nstr ? 0 : an + 1;
    sn = (sn + 1) & (S - 1);
  };
  if (nstr > 0)
#pragma unroll
    for (int b = 0; b < S - 1; ++b) issue();
  int sl = 0, k = 1;
  for (;; ++k) {
    __syncthreads();  // the waves of sweep k - 1 are out and the flag is read
    if (*((volatile int*)&s_flag)) break;
    const double* prev = A.gout + (size_t)((k - 1) & (kGenSlots - 1)) * A.n_out;
    for (int q = tid; q < C.nin; q += NT) vin[q] = __ldcg(prev + src[q]);
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
    double x = 0.0, y = 0.0;
    const double* v = vin + vofs;
#pragma unroll 4
    for (int i = 0; i < nres; ++i) {
      const double2 e = slots[i * NT];
      const double w = *v;
      x += e.x * w;
      y += e.y * w;
      v += G;
    }
    for (int i = 0; i < nstr; ++i) {
      issue();
      cp_async_wait_group<S - 1>();  // this thread's oldest element has landed
      const double2 e = ring[sl * NT];
      const double w = *v;
      x += e.x * w;
      y += e.y * w;
      v += G;
      sl = (sl + 1) & (S - 1);
    }
    red[tid] = make_double2(x, y);
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
    double* cur = A.gout + (size_t)(k & (kGenSlots - 1)) * A.n_out;
    const double* rs = reinterpret_cast<const double*>(red);
    for (int q = tid; q < 2 * np; q += NT) {
      const int o = oid[q];
      if (o < 0) continue;
      double tot = __ldg(A.c + o);
#pragma unroll 8
      for (int b = 0; b < G; ++b) tot += rs[(size_t)b * 2 * np + q];
      cur[o] = tot;
    }
    __syncthreads();  // every wave of sweep k is written
    if (k > 1) {  // the residual of sweep k - 1, while the grid barrier is awaited
      const double* pp = A.gout + (size_t)((k - 2) & (kGenSlots - 1)) * A.n_out;
      double sq = 0.0;
      for (int q = C.q0 + tid; q < C.q1; q += NT) {
        const int nr = A.res_run[q];
        if (!nr) continue;
        double r = 0.0;
        for (int e = 0; e < nr; ++e) {
          const int a = PORTS ? q + e : A.res_in[q + e], s = A.in_src[a];
          const double wo_t = __ldcg(prev + s), wi_s = __ldcg(pp + s);
          if (!PORTS && A.in_kind[a] != 0) {
            r += A.coef[a] * (wi_s - wo_t);
          } else {
            const int own = PORTS ? a : A.in_own_out[a];
            const double wo_s = __ldcg(prev + own), wi_t = __ldcg(pp + own);
            const double Ss = wi_s + wo_s, St = wi_t + wo_t;
            const double2 kd = PORTS ? __ldg(A.kd + a) : make_double2(A.coef[a], A.dsc[a]);
            r += 0.5 * kd.y * (0.5 * (Ss + St) - kd.x * (Ss - St) - wi_s - wi_t);
          }
        }
        sq += r * r;
      }
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, o);
      if (lane == 0) s_part[k & 1][warp] = sq;
    }
  }
  cp_async_wait_group<0>();  // no copy into shared memory outlives the CTA
  const int flag = *((volatile int*)&s_flag);
  if (flag == 5) return;
  // the decision of sweep k - 1 closed sweep k - 3: its iterate, or the one before
  const int it = flag == 1 ? k - 4 : k - 3;
  const double* from = A.gout + (size_t)((it - 1) & (kGenSlots - 1)) * A.n_out;
  for (int a = C.i0 + tid; a < C.i1; a += NT) {
    const double w = __ldcg(from + A.in_src[a]);
    if constexpr (PORTS)
      reinterpret_cast<double2*>(A.gin)[a] =
          make_double2(w, __ldcg(A.gout + (size_t)(it & (kGenSlots - 1)) * A.n_out + a));
    else A.gin[(size_t)(it & 1) * A.n_in + a] = w;
  }
}

// the CTAs of the resident form; gen_ctas is -1 where it does not apply
template <bool PORTS>
static vtm_status plan_resident(vtm_plan_s* P) {
  P->gen_ctas = -1;
  const std::vector<int32_t>&in_off = PORTS ? P->port_off : P->in_off, &out_off = PORTS ? P->port_off : P->out_off;
  const std::vector<uint8_t>& run = PORTS ? P->port_run : P->res_run;
  const int64_t n_in = PORTS ? (int64_t)P->port_node.size() : P->n_in, n_out = PORTS ? n_in : P->n_out;
  int coop = 0, sms = 152;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, P->device);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, P->device);
  if (!coop || n_in == 0 || n_out == 0) return VTM_OK;
  std::vector<int32_t> pair_off(P->nparts + 1, 0), res_in(PORTS ? 0 : n_in);
  int64_t cost = 0;  // elements of E_P in pairs, and the sums
  auto pairs = [&](int32_t t) { return (out_off[t + 1] - out_off[t] + 1) / 2; };
  auto pair_cost = [&](int32_t t) { return (int64_t)(in_off[t + 1] - in_off[t]) + 4; };
  for (int32_t t = 0; t < P->nparts; ++t) {
    pair_off[t + 1] = pair_off[t] + pairs(t);
    cost += pairs(t) * pair_cost(t);
    if (!PORTS)
      for (int32_t a = in_off[t]; a < in_off[t + 1]; ++a) res_in[a] = in_off[t] + P->res_perm[a];
  }
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, cost / (kGenMinElems<PORTS> * kGenThreads)));
  std::vector<GenCta> ctas(grid);
  auto run_start = [&](int64_t q) {
    while (q < n_in && !run[q]) ++q;
    return (int32_t)q;
  };
  int32_t t = 0, pr = 0;  // next pair: pair `pr` of tile t
  int64_t done = 0;
  int32_t vmax = 1;
  for (int b = 0; b < grid; ++b) {
    GenCta& c = ctas[b];
    const int64_t upto = cost * (b + 1) / grid;
    while (t < P->nparts && pr >= pairs(t)) {
      ++t;
      pr = 0;
    }
    c.pair0 = t < P->nparts ? pair_off[t] + pr : pair_off[P->nparts];
    c.np = 0;
    c.in0 = t < P->nparts ? in_off[t] : 0;
    int32_t last = t;
    while (t < P->nparts && done < upto) {
      if (pr >= pairs(t)) {
        ++t;
        pr = 0;
        continue;
      }
      const int64_t pc = pair_cost(t);
      const int32_t take = (int32_t)std::min<int64_t>(pairs(t) - pr, (upto - done + pc - 1) / pc);
      c.np += take;
      pr += take;
      done += take * pc;
      last = t;
    }
    c.nin = c.np > 0 ? in_off[last + 1] - c.in0 : 0;
    vmax = std::max(vmax, c.nin);
    if (c.np > kGenThreads) return VTM_OK;
    c.i0 = (int32_t)(n_in * b / grid);
    c.i1 = (int32_t)(n_in * (b + 1) / grid);
    c.q0 = run_start(c.i0);
    c.q1 = run_start(c.i1);
  }
  vmax = (vmax + 1) / 2 * 2;
  const int64_t fixed = (int64_t)kGenThreads * 16 + 12 * (int64_t)vmax + 8 * kGenThreads;
  auto* kern = general_resident_kernel<PORTS>;
  int optin = 0, fits = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, P->device);
  cudaFuncAttributes fa{};
  VTM_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
  const int nslots = (int)((optin - (int64_t)fa.sharedSizeBytes - fixed) / (kGenThreads * 16));
  if (nslots < kGenMinSlots) return VTM_OK;
  P->gen_smem = fixed + (int64_t)nslots * kGenThreads * 16;
  VTM_CUDA_TRY(allow_smem(kern, (size_t)P->gen_smem));
  VTM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fits, kern, kGenThreads + 32, (size_t)P->gen_smem));
  if (fits < 1) return VTM_OK;
  cudaStream_t s = P->stream;
  VTM_TRY(upload(P->d_gen_ctas, ctas, s));
  VTM_TRY(upload(P->d_gen_pair, pair_off, s));
  if (PORTS) VTM_TRY(dev_alloc(P->d_gout, kGenSlots * n_out * sizeof(double)));
  else VTM_TRY(upload(P->d_gen_res, res_in, s));
  VTM_TRY(dev_alloc(P->d_gen_part, 64 + 2 * (size_t)grid * sizeof(double)));
  VTM_CUDA_TRY(cudaStreamSynchronize(s));  // the host lists are about to go
  P->gen_nslots = nslots;
  P->gen_vmax = vmax;
  P->gen_ctas = grid;
  return VTM_OK;
}

// (without the memory for it the plan keeps one launch per sweep)
template <bool PORTS>
static vtm_status plan_resident_if_room(vtm_plan_s* P) {
  const vtm_status st = plan_resident<PORTS>(P);
  if (st != VTM_ENOMEM) return st;
  P->gen_ctas = -1;
  return VTM_OK;
}

template <bool PORTS>
static cudaError_t launch_resident(vtm_plan_s* P, double* hist, int hist_len) {
  cudaStream_t s = P->stream;
  GenRes a{};
  a.ctas = P->d_gen_ctas.as<GenCta>();
  a.pair_off = P->d_gen_pair.as<int32_t>();
  a.gout = P->d_gout.as<double>();
  if constexpr (PORTS) {
    a.E = P->d_T64.as<double>();
    a.E_off = P->tabs.T_off.as<int64_t>();
    a.E_ld = P->tabs.T_ld.as<int32_t>();
    a.in_off = a.out_off = P->tabs.port_off.as<int32_t>();
    a.in_src = P->d_twin.as<int32_t>();
    a.res_run = P->d_run.as<uint8_t>();
    a.kd = P->d_kd.as<double2>();
    a.c = P->d_c64.as<double>();
    a.gin = P->d_state64.as<double>();
    a.n_in = a.n_out = (int64_t)P->port_node.size();
  } else {
    a.E = P->d_E.as<double>();
    a.E_off = P->d_E_off.as<int64_t>();
    a.E_ld = P->d_E_ld.as<int32_t>();
    a.in_off = P->d_in_off.as<int32_t>();
    a.out_off = P->d_out_off.as<int32_t>();
    a.in_src = P->d_in_src.as<int32_t>();
    a.in_own_out = P->d_in_own_out.as<int32_t>();
    a.res_in = P->d_gen_res.as<int32_t>();
    a.in_kind = P->d_in_kind.as<uint8_t>();
    a.res_run = P->d_res_run.as<uint8_t>();
    a.coef = P->d_in_coef.as<double>();
    a.dsc = P->d_in_d.as<double>();
    a.c = P->d_cg.as<double>();
    a.gin = P->d_gin.as<double>();
    a.n_in = P->n_in;
    a.n_out = P->n_out;
  }
  a.ctrl = P->d_ctrl.as<SweepCtrl>();
  a.bar = reinterpret_cast<unsigned long long*>(P->d_gen_part.p);
  a.part = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(P->d_gen_part.p) + 64);
  a.hist = hist;
  a.hist_len = hist_len;
  a.nparts = P->nparts;
  a.nslots = P->gen_nslots;
  a.vmax = P->gen_vmax;
  a.max_polls = (uint32_t)P->opts.wait_polls;
  cudaError_t e = cudaMemsetAsync(P->d_gen_part.p, 0, 64, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.gout, 0, a.n_out * sizeof(double), s);  // slot 0: the first sweep's waves
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)general_resident_kernel<PORTS>, dim3(P->gen_ctas),
                                     dim3(kGenThreads + 32), args, (size_t)P->gen_smem, s);
}

// The port form for run_sweeps: true where it serves this many sweeps.
vtm_status port_resident_prepare(vtm_plan_s* P, int budget, bool* ok) {
  if (P->gen_ctas == 0) VTM_TRY(plan_resident_if_room<true>(P));
  *ok = P->gen_ctas > 0 && res_counts(budget, P->gen_ctas);
  return VTM_OK;
}
cudaError_t launch_port_resident(vtm_plan_s* P, double* hist, int hist_len) {
  return launch_resident<true>(P, hist, hist_len);
}

static vtm_status general_sweeps_resident(vtm_plan_s* P, int budget, double* hist, int hist_len, int* sweep_out,
                                          int* flag_out) {
  cudaStream_t s = P->stream;
  VTM_CUDA_TRY(cudaEventRecord(P->evs0, s));
  VTM_CUDA_TRY(launch_resident<false>(P, hist, hist_len));
  VTM_CUDA_TRY(cudaEventRecord(P->evs1, s));
  VTM_CUDA_TRY(cudaMemcpyAsync(P->h_ctrl, P->d_ctrl.p, sizeof(SweepCtrl), cudaMemcpyDeviceToHost, s));
  VTM_CUDA_TRY(cudaStreamSynchronize(s));
  float ms = 0.f;
  VTM_CUDA_TRY(cudaEventElapsedTime(&ms, P->evs0, P->evs1));
  P->sweep_ms += ms;
  const SweepCtrl& r = *P->h_ctrl;
  P->sweep_launch_count += std::max(r.k - 1, 1);  // sweeps run by the one launch
  P->launch_count += 1;
  if (r.flag == 5) {
    set_detail("vtm_solve: a bounded wait of the resident sweeps ran out");
    return VTM_ETIMEOUT;
  }
  *flag_out = r.flag;
  *sweep_out = r.flag == 1 ? r.conv_sweep : std::min(r.k - 1, budget);
  return VTM_OK;
}

vtm_status build_general_operators(vtm_plan_s* P) {
  cudaStream_t s = P->stream;
  const size_t bytes = std::max<int64_t>(P->E_elems, 8) * sizeof(double);
  VTM_TRY(dev_alloc(P->d_E, bytes));
  VTM_CUDA_TRY(cudaMemsetAsync(P->d_E.p, 0, bytes, s));
  if (P->n_in > 0) {
    const size_t smem = (size_t)P->max_nodes * sizeof(double);
    if (smem > 200 * 1024) {
      set_detail("vtm_factor: a sub-circuit with more than 25600 nodes has cut couplings");
      return VTM_EINVAL;
    }
    VTM_CUDA_TRY(cudaFuncSetAttribute(build_general_kernel,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    build_general_kernel<<<(unsigned)P->n_in, 32, smem, s>>>(
        P->tabs.node_off.as<int32_t>(), P->tabs.bw.as<int32_t>(), P->tabs.band_off.as<int64_t>(),
        P->d_Lc.as<double>(), P->d_Uc.as<double>(), P->d_in_tile.as<int32_t>(),
        P->d_in_off.as<int32_t>(), P->d_out_off.as<int32_t>(), P->d_in_loc.as<int32_t>(),
        P->d_in_own_out.as<int32_t>(), P->d_in_sigma.as<double>(), P->d_out_loc.as<int32_t>(),
        P->d_out_scale.as<double>(), P->d_out_diag.as<double>(), P->d_E_off.as<int64_t>(),
        P->d_E_ld.as<int32_t>(), P->d_E.as<double>());
    VTM_CUDA_TRY(cudaGetLastError());
  }
  VTM_CUDA_TRY(cudaStreamSynchronize(s));
  return VTM_OK;
}

vtm_status general_const(vtm_plan_s* P, const double* x0) {
  general_const_kernel<<<P->nparts, 128, 0, P->stream>>>(
      P->tabs.node_off.as<int32_t>(), P->d_out_off.as<int32_t>(), P->d_out_loc.as<int32_t>(),
      P->d_out_scale.as<double>(), x0, P->d_cg.as<double>());
  P->launch_count++;
  VTM_CUDA_TRY(cudaGetLastError());
  return VTM_OK;
}

vtm_status general_sweeps(vtm_plan_s* P, double bnorm2, double target2, int budget, double* hist,
                          int hist_len, int* sweep_out, int* flag_out) {
  cudaStream_t s = P->stream;
  SweepCtrl h{};
  h.k = 1;
  h.k_max = budget;
  h.tol2 = target2;
  h.bnorm2 = bnorm2 > 0 ? bnorm2 : 1.0;
  *P->h_ctrl = h;
  VTM_CUDA_TRY(cudaMemcpyAsync(P->d_ctrl.p, P->h_ctrl, sizeof(SweepCtrl), cudaMemcpyHostToDevice, s));
  if (P->gen_ctas == 0) VTM_TRY(plan_resident_if_room<false>(P));
  // (the barrier word holds as many arrivals and sweeps as res_counts allows; above that one
  // launch per sweep)
  if (P->gen_ctas > 0 && res_counts(budget, P->gen_ctas))
    return general_sweeps_resident(P, budget, hist, hist_len, sweep_out, flag_out);
  VTM_CUDA_TRY(cudaMemsetAsync(P->d_gin.p, 0, 2 * std::max<int64_t>(P->n_in, 1) * sizeof(double), s));
  VTM_CUDA_TRY(cudaMemsetAsync(P->d_gout.p, 0, 2 * std::max<int64_t>(P->n_out, 1) * sizeof(double), s));
  // four groups of up to 256 threads per tile (one output each; eight groups
  // of 128 measured slower on the 1024^2 VCCS grid)
  constexpr int KS = 4;
  const int to = P->max_out <= 64 ? 64 : (P->max_out <= 128 ? 128 : 256);
  const int threads = KS * to;
  const size_t smem = (2 * (size_t)std::max(P->max_in, 1) + threads) * sizeof(double);
  if (smem > 48 * 1024)
    VTM_CUDA_TRY(cudaFuncSetAttribute(general_sweep_kernel<KS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
  int launched = 0;
  while (true) {
    const int m = (int)std::min<int64_t>(P->opts.check_every, (int64_t)budget + 1 - launched);
    VTM_CUDA_TRY(cudaEventRecord(P->evs0, s));
    for (int i = 0; i < m; ++i)
      general_sweep_kernel<KS><<<P->nparts, threads, smem, s>>>(
          P->d_E.as<double>(), P->d_E_off.as<int64_t>(), P->d_E_ld.as<int32_t>(),
          P->d_in_off.as<int32_t>(), P->d_out_off.as<int32_t>(), P->d_in_src.as<int32_t>(),
          P->d_in_kind.as<uint8_t>(), P->d_in_twin.as<int32_t>(), P->d_in_own_out.as<int32_t>(),
          P->d_in_coef.as<double>(), P->d_in_d.as<double>(), P->d_res_perm.as<int32_t>(),
          P->d_res_run.as<uint8_t>(),
          P->d_cg.as<double>(), P->d_gin.as<double>(), P->d_gout.as<double>(), P->n_in, P->n_out,
          P->d_ctrl.as<SweepCtrl>(), P->d_partials.as<double>(), hist, hist_len, P->nparts);
    VTM_CUDA_TRY(cudaGetLastError());
    launched += m;
    VTM_CUDA_TRY(cudaEventRecord(P->evs1, s));
    VTM_CUDA_TRY(cudaMemcpyAsync(P->h_ctrl, P->d_ctrl.p, sizeof(SweepCtrl), cudaMemcpyDeviceToHost, s));
    VTM_CUDA_TRY(cudaStreamSynchronize(s));
    float bms = 0.f;
    VTM_CUDA_TRY(cudaEventElapsedTime(&bms, P->evs0, P->evs1));
    P->sweep_ms += bms;
    P->sweep_launch_count += m;
    P->launch_count += m;
    if (P->h_ctrl->flag || launched > budget) break;
  }
  const SweepCtrl& r = *P->h_ctrl;
  *flag_out = r.flag;
  *sweep_out = r.flag == 1 ? r.conv_sweep : std::min(r.k - 1, budget);
  return VTM_OK;
}

vtm_status general_inject(vtm_plan_s* P, int sweep, double* v) {
  general_inject_kernel<<<P->nparts, 128, 0, P->stream>>>(
      P->tabs.node_off.as<int32_t>(), P->d_in_off.as<int32_t>(), P->d_in_loc.as<int32_t>(),
      P->d_res_perm.as<int32_t>(), P->d_res_run.as<uint8_t>(), P->d_in_sigma.as<double>(),
      P->d_gin.as<double>() + (size_t)(sweep & 1) * P->n_in, v);
  P->launch_count++;
  VTM_CUDA_TRY(cudaGetLastError());
  return VTM_OK;
}

}  // namespace vtm
