// Single-column band solves of half bandwidths above 32: a CTA per tile and
// column, rows in blocks of 32, the unit-triangular diagonal blocks applied by
// their inverses.
//
// With the multipliers divided by the pivots (see band.cuh) the forward pass
// is u = M^-1 v with M unit lower, y(j) = u(j) Lc[j][0], and the backward pass
// the same in reversed row order over Uc.  In pass coordinates (row j forward,
// n - 1 - j backward) both read column j's multipliers at offsets 1..bw, so one
// code serves both.  Per block of 32 rows: t = v + (the updates of the earlier
// blocks), u = M_JJ^-1 t (32 x 32, inverted once per factorisation), then the
// block's 32 columns update the next K = (31 + bw) / 32 blocks.  Warp w takes
// a quarter of the columns of both products; its update of a later block stays in its own
// registers (lane = row) and is added across the warps only when that block's
// turn comes.  The chain per 32 rows is two CTA barriers, against 32 dependent
// warp steps (a shared-memory round trip each) in band_solve_tiles_kernel.
//
// What bounds it: FP64 the FP64 pipe (2 FMA per clock and SM: n (bw + 32) FMA
// per pass), FP32 the chain of barriers; a block's columns (contiguous in the
// band storage) and its inverse arrive by bulk copies into a ring of stages,
// so no load latency is on the chain.  Measured per solve against the
// row-by-row kernel (one warp per tile):
//   FP64  256 tiles of 4096 rows, bw 64: 2720 -> 734 us (the pipe needs 506 us
//         at two tiles on the fullest SM); 100 tiles, bw 99, LU: 4057 -> 622 us;
//         150 boxes of up to 1782 rows, bw <= 112: 1770 -> 287 us
//   FP32  the same three shapes: 936 -> 179 us (bw 64), 1058 -> 92 us (bw <= 112)
// With several columns a CTA takes four (each multiplier read once for them): FP64,
// 110 boxes of up to 2028 rows, bw <= 126, 18 columns: 5.2 ms with the batched
// row-by-row kernel, 1.62 ms here.
// Two warps per tile (fewer cross-warp sums, 112 instead of 128 FP64
// instructions per block) measured 745, 916 and 423 us: too few in flight.
#include <algorithm>

#include "ptx.h"
#include "vtm_internal.h"

namespace vtm {

constexpr int kBbN = 32;                 // rows per block
constexpr uint32_t kBbPolls = 1u << 24;  // mbarrier polls before giving up

// Skeel condition of the diagonal blocks M (largest row sum of |M^-1| |M|) up to which
// their inverses serve.  A product with the inverse is off by u |M^-1| |t| <= u |M^-1| |M| |u|,
// so by this many u of the largest element, the bound that substitution has too.  Where no
// column of K_P outweighs its diagonal |M^-1| <= 1; thermal grids measure 3, resistor and
// power grids 20 to 26, VCCS grids 22 to 28.  Beyond the limit -- LU of a matrix with
// large multipliers, say -- the solves substitute row by row, whose residual stays at a few u all
// the same: 64 rows, half bandwidth 40 and multipliers of -1.8 below the diagonal left
// 2e-9 by inverses, 3e-16 by substitution.
constexpr float kBbMaxCond = 256.f;

// Inverses of the unit-triangular diagonal blocks, one warp per (block, pass):
// lane q keeps column q of the inverse and substitutes through the block.
// inv[(first block of the tile + k) 1024 + q 32 + r]; rows past n are identity.
__global__ void __launch_bounds__(128) band_inverse_kernel(
    const int32_t* __restrict__ node_off, const int32_t* __restrict__ bwv, const int64_t* __restrict__ band_off,
    const int32_t* __restrict__ blk_off, int nparts, const double* __restrict__ Lc,
    const double* __restrict__ Uc, double* __restrict__ Li, double* __restrict__ Ui, int* __restrict__ cond) {
  __shared__ double sm[4][kBbN * (kBbN + 1)];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = blockIdx.x * 4 + warp;
  if (g >= blk_off[nparts]) return;
  int lo = 0, hi = nparts - 1;  // the tile of block g
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (blk_off[mid] <= g) lo = mid;
    else hi = mid - 1;
  }
  const int t = lo, s = (g - blk_off[t]) * kBbN;
  const int n = node_off[t + 1] - node_off[t], bw = bwv[t], B = bw + 1;
  const bool fwd = blockIdx.y == 0;
  const double* f = (fwd ? Lc : Uc) + band_off[t];
  double* M = sm[warp];  // M[r][p], r > p
  for (int q = 0; q < kBbN; ++q) {
    const int a = lane - q, j = s + q;
    double v = 0.0;
    if (a >= 1 && a <= bw && s + lane < n) v = f[(int64_t)(fwd ? j : n - 1 - j) * B + a];
    M[lane * (kBbN + 1) + q] = v;
  }
  __syncwarp();
  double x[kBbN];
  float rs = 1.f;  // row sum of |M|
#pragma unroll
  for (int r = 0; r < kBbN; ++r) {
    double acc = r == lane ? 1.0 : 0.0;
#pragma unroll
    for (int p = 0; p < r; ++p) acc -= M[r * (kBbN + 1) + p] * x[p];
    x[r] = acc;
    rs += fabsf((float)M[lane * (kBbN + 1) + r]);
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < kBbN; ++r) M[lane * (kBbN + 1) + r] = x[r];
  __syncwarp();
  float c = 0.f;  // row `lane` of |M^-1| |M|, summed
#pragma unroll
  for (int q = 0; q < kBbN; ++q) c += fabsf((float)M[q * (kBbN + 1) + lane]) * __shfl_sync(0xffffffffu, rs, q);
  for (int o = 16; o > 0; o >>= 1) c = fmaxf(c, __shfl_xor_sync(0xffffffffu, c, o));
  // (bits of positive floats order like the floats; a NaN counts as too large)
  if (lane == 0) atomicMax(cond, __float_as_int(c <= kBbMaxCond ? c : INFINITY));
  double* out = (fwd ? Li : Ui) + (int64_t)g * kBbN * kBbN;
#pragma unroll 4
  for (int q = 0; q < kBbN; ++q) out[q * kBbN + lane] = M[q * (kBbN + 1) + lane];
}

// elements of one stage: 32 columns from the 16-byte boundary below the
// first, then the 32 x 32 inverse
template <class FT>
__host__ __device__ constexpr int bb_stage_elems(int B) {
  constexpr int kVec = 16 / sizeof(FT);
  return (kBbN * B + 2 * kVec - 1) / kVec * kVec + kBbN * kBbN;
}

// the warps' partial sums of one row, added as a tree; `step` between the warps
template <int NW, class FT>
__device__ __forceinline__ FT sum_warps(const FT* r, int step) {
  static_assert(NW == 4, "");
  return (r[0] + r[step]) + (r[2 * step] + r[3 * step]);
}

// NC columns at once (each multiplier is read once for all of them)
template <class FT, int K, int NW, int NC, bool FWD>
__device__ __forceinline__ bool bb_pass(const FT* __restrict__ cols, const FT* __restrict__ inv, int n, int bw,
                                        FT* v, int64_t stride, int nc, FT* ring, int stage_elems, int S,
                                        uint64_t* bars, uint32_t& par, FT* red, int* s_fail) {
  constexpr int C = kBbN / NW;  // band columns per warp
  constexpr int RW = NC * kBbN;  // one warp's row of `red`
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int B = bw + 1;
  const int nblk = (n + kBbN - 1) / kBbN;
  auto first_col = [&](int b) { return FWD ? b * kBbN : n - min(n, (b + 1) * kBbN); };
  auto issue = [&](int b) {  // thread 0: block b into its stage
    const int c0 = first_col(b), c1 = FWD ? min(n, (b + 1) * kBbN) : n - b * kBbN;
    const uintptr_t a = reinterpret_cast<uintptr_t>(cols + (int64_t)c0 * B);
    const uintptr_t a0 = a & ~(uintptr_t)15;
    const uint32_t bytes = (uint32_t)(((a - a0) + (size_t)(c1 - c0) * B * sizeof(FT) + 15) & ~(size_t)15);
    FT* dst = ring + (size_t)(b % S) * stage_elems;
    uint64_t* bar = &bars[b % S];
    mbar_arrive_expect_tx(bar, bytes + (uint32_t)(kBbN * kBbN * sizeof(FT)));
    bulk_copy_g2s(dst, reinterpret_cast<const void*>(a0), bytes, bar);
    bulk_copy_g2s(dst + stage_elems - kBbN * kBbN, inv + (int64_t)b * kBbN * kBbN, kBbN * kBbN * sizeof(FT), bar);
  };
  auto src = [&](int j, int x) -> FT { return j < n && x < nc ? v[x * stride + (FWD ? j : n - 1 - j)] : FT(0); };
  if (threadIdx.x == 0) {
    fence_proxy_async_smem();  // the stages' earlier reads come before the copies
    for (int b = 0; b < S && b < nblk; ++b) issue(b);
  }
  FT acc[K][NC];  // this warp's updates of the next K blocks, lane = row
  FT vt[NC];
#pragma unroll
  for (int x = 0; x < NC; ++x) {
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k][x] = FT(0);
    vt[x] = src(lane, x);
  }
  FT* mine = red + (2 * NW + warp) * RW;  // this warp's copy of t, then of -u
  for (int b = 0; b < nblk; ++b) {
    const int s = b * kBbN, sl = b % S;
    FT vn[NC];
#pragma unroll
    for (int x = 0; x < NC; ++x) {
      vn[x] = src(s + kBbN + lane, x);
      red[warp * RW + x * kBbN + lane] = acc[0][x];
    }
    if (!mbar_wait_bounded(&bars[sl], (par >> sl) & 1u, kBbPolls)) *(volatile int*)s_fail = 1;
    par ^= 1u << sl;
    __syncthreads();
    if (*(volatile int*)s_fail) {
      // a copy did not land: wait (bounded) for the stages still in flight
      for (int i = 1; i < S && b + i < nblk; ++i) {
        const int sj = (b + i) % S;
        mbar_wait_bounded(&bars[sj], (par >> sj) & 1u, kBbPolls);
      }
      return false;
    }
    if (threadIdx.x == 0 && b > 0 && b + S - 1 < nblk) {  // block b - 1 is read: refill its stage
      fence_proxy_async_smem();
      issue(b + S - 1);
    }
    const FT* st = ring + (size_t)sl * stage_elems;
    const FT* iv = st + stage_elems - kBbN * kBbN + warp * C * kBbN + lane;
#pragma unroll
    for (int x = 0; x < NC; ++x) mine[x * kBbN + lane] = vt[x] + sum_warps<NW>(red + x * kBbN + lane, RW);
    __syncwarp();
    {
      constexpr int P = NC == 1 ? 4 : 1;  // chains per column
      FT part[NC][P];
#pragma unroll
      for (int x = 0; x < NC; ++x)
#pragma unroll
        for (int y = 0; y < P; ++y) part[x][y] = FT(0);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const FT m = iv[c * kBbN];
#pragma unroll
        for (int x = 0; x < NC; ++x) part[x][c % P] += m * mine[x * kBbN + warp * C + c];
      }
#pragma unroll
      for (int x = 0; x < NC; ++x) {
        if constexpr (P == 4) part[x][0] = (part[x][0] + part[x][1]) + (part[x][2] + part[x][3]);
        red[(NW + warp) * RW + x * kBbN + lane] = part[x][0];
      }
    }
    __syncthreads();
    FT u[NC];
#pragma unroll
    for (int x = 0; x < NC; ++x) u[x] = sum_warps<NW>(red + NW * RW + x * kBbN + lane, RW);
    __syncwarp();
#pragma unroll
    for (int x = 0; x < NC; ++x) mine[x * kBbN + lane] = -u[x];
    __syncwarp();
    const int c0 = first_col(b);
    constexpr int kMask = 16 / sizeof(FT) - 1;
    const int dl = (int)((reinterpret_cast<uintptr_t>(cols + (int64_t)c0 * B) / sizeof(FT)) & kMask);
    const int last = (FWD ? min(n, s + kBbN) : n - s) - c0 - 1;  // columns in the stage, less one
    // column q of the block: element 32 k - q + lane is row 32 k + lane's multiplier
    const FT* col = st + dl + (FWD ? warp * C : last - warp * C) * B + lane - warp * C;
    const int step = (FWD ? B : -B) - 1;
    const int amax = min(bw, n - 1 - s);  // no row past n: 32 k + lane <= n - 1 - s as well
#pragma unroll
    for (int k = 1; k <= K; ++k) {
      constexpr int P = NC == 1 ? 2 : 1;
      FT y[NC][P];
#pragma unroll
      for (int x = 0; x < NC; ++x) {
        y[x][0] = k < K ? acc[k < K ? k : 0][x] : FT(0);
        if constexpr (P == 2) y[x][1] = FT(0);
      }
      const bool row = kBbN * k + lane <= n - 1 - s;
#pragma unroll
      for (int c4 = 0; c4 < C; c4 += 4) {
        const int q0 = warp * C + c4;
        if (kBbN * k - q0 - 3 <= amax) {  // (the whole warp) any of the four columns reaches these rows
#pragma unroll
          for (int c = c4; c < c4 + 4; ++c) {
            const int a = kBbN * k - (warp * C + c) + lane;
            const FT m = (row && a <= bw) ? col[kBbN * k + c * step] : FT(0);
#pragma unroll
            for (int x = 0; x < NC; ++x) y[x][c % P] += m * mine[x * kBbN + warp * C + c];
          }
        }
      }
#pragma unroll
      for (int x = 0; x < NC; ++x) {
        if constexpr (P == 2) acc[k - 1][x] = y[x][0] + y[x][1];
        else acc[k - 1][x] = y[x][0];
      }
    }
    if (s + lane < n) {
      const FT dg = st[dl + (FWD ? lane : last - lane) * B];
#pragma unroll
      for (int x = 0; x < NC; ++x)  // a column per warp in turn
        if (warp == (x & (NW - 1)) && x < nc) v[x * stride + (FWD ? s + lane : n - 1 - s - lane)] = u[x] * dg;
    }
#pragma unroll
    for (int x = 0; x < NC; ++x) vt[x] = vn[x];
  }
  return true;
}

template <class FT, int K, int NW, int NC>
__global__ void __launch_bounds__(32 * NW) band_solve_blk_kernel(
    const int32_t* __restrict__ node_off, const int32_t* __restrict__ bwv, const int64_t* __restrict__ band_off,
    const int32_t* __restrict__ blk_off, const int32_t* __restrict__ order, const FT* __restrict__ Lc,
    const FT* __restrict__ Uc, const FT* __restrict__ Li, const FT* __restrict__ Ui, FT* __restrict__ v,
    int64_t stride, int nparts, int ncols, int stage_elems, int S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[8];
  __shared__ int s_fail;
  __shared__ __align__(16) FT red[3 * NW * NC * kBbN];
  FT* ring = reinterpret_cast<FT*>(smem_raw);
  const int groups = (ncols + NC - 1) / NC;  // of one tile side by side: largest tiles first
  const int t = order[blockIdx.x / groups];
  const int col = blockIdx.x % groups * NC, nc = min(NC, ncols - col);
  const int off = node_off[t], n = node_off[t + 1] - off, bw = bwv[t];
  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) mbar_init(&bars[i], 1);
    fence_mbar_init();
    s_fail = 0;
  }
  __syncthreads();
  FT* vg = v + (int64_t)col * stride + off;
  const int64_t io = (int64_t)blk_off[t] * kBbN * kBbN;
  uint32_t par = 0;
  bool ok = bb_pass<FT, K, NW, NC, true>(Lc + band_off[t], Li + io, n, bw, vg, stride, nc, ring, stage_elems, S, bars,
                                         par, red, &s_fail);
  __syncthreads();  // y of the whole tile before the backward pass reads it
  if (ok)
    ok = bb_pass<FT, K, NW, NC, false>(Uc + band_off[t], Ui + io, n, bw, vg, stride, nc, ring, stage_elems, S, bars, par,
                                       red, &s_fail);
  if (!ok)  // the refinement reports the NaN as a divergence
    for (int i = threadIdx.x; i < n; i += 32 * NW)
      for (int x = 0; x < nc; ++x) vg[x * stride + i] = FT(NAN);
}

// Half bandwidths this form serves: above 32 (up to 32 the warp-per-tile
// kernels already keep the SMs full) and up to 256.
bool band_blk_eligible(const vtm_plan_s* P) { return P->max_bw > 32 && P->max_bw <= 256; }

// The inverted diagonal blocks of the current factors (vtm_factor).
vtm_status band_blk_prepare(vtm_plan_s* P) {
  P->bb_ok = false;
  if (!band_blk_eligible(P)) return VTM_OK;
  cudaStream_t s = P->stream;
  if (P->bb_blocks == 0) {
    std::vector<int32_t> off(P->nparts + 1, 0), order(P->nparts);
    for (int32_t t = 0; t < P->nparts; ++t) {
      off[t + 1] = off[t] + (P->node_off[t + 1] - P->node_off[t] + kBbN - 1) / kBbN;
      order[t] = t;
    }
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {  // largest tiles first
      return P->node_off[a + 1] - P->node_off[a] > P->node_off[b + 1] - P->node_off[b];
    });
    VTM_TRY(upload(P->d_bb_off, off, s));
    VTM_TRY(upload(P->d_bb_order, order, s));
    VTM_CUDA_TRY(cudaStreamSynchronize(s));  // the host tables are about to go
    P->bb_blocks = off[P->nparts];
  }
  // Where the memory for the inverses runs out (512 bytes per unknown, 768 with FP32
  // sweeps) the solves stay with the row-by-row kernels
  const int64_t ne = (int64_t)P->bb_blocks * kBbN * kBbN;
  const bool f32 = P->opts.precision != VTM_PREC_FP64;
  const size_t sz[4] = {sizeof(double), sizeof(double), sizeof(float), sizeof(float)};
  DevBuf* const inv[4] = {&P->d_bb_Li, &P->d_bb_Ui, &P->d_bb_Li32, &P->d_bb_Ui32};
  for (int i = 0; i < (f32 ? 4 : 2); ++i) {
    const vtm_status st = dev_alloc(*inv[i], ne * sz[i]);
    if (st == VTM_ENOMEM) {
      for (DevBuf* b : inv) dev_free(*b);
      return VTM_OK;
    }
    VTM_TRY(st);
  }
  int* d_cond = P->d_err.as<int>() + 1;
  VTM_CUDA_TRY(cudaMemsetAsync(d_cond, 0, sizeof(int), s));
  band_inverse_kernel<<<dim3((P->bb_blocks + 3) / 4, 2), 128, 0, s>>>(
      P->tabs.node_off.as<int32_t>(), P->tabs.bw.as<int32_t>(), P->tabs.band_off.as<int64_t>(),
      P->d_bb_off.as<int32_t>(), P->nparts, P->d_Lc.as<double>(), P->d_Uc.as<double>(), P->d_bb_Li.as<double>(),
      P->d_bb_Ui.as<double>(), d_cond);
  VTM_CUDA_TRY(cudaGetLastError());
  if (f32) {
    convert_f32(P->d_bb_Li.as<double>(), P->d_bb_Li32.as<float>(), ne, s);
    convert_f32(P->d_bb_Ui.as<double>(), P->d_bb_Ui32.as<float>(), ne, s);
  }
  float cond = 0.f;
  VTM_CUDA_TRY(cudaMemcpyAsync(&cond, d_cond, sizeof(float), cudaMemcpyDeviceToHost, s));
  VTM_CUDA_TRY(cudaStreamSynchronize(s));
  P->bb_ok = cond <= kBbMaxCond;
  return VTM_OK;
}

template <class FT>
static void launch_blk_t(vtm_plan_s* P, FT* v, const FT* Lc, const FT* Uc, const FT* Li, const FT* Ui, int ncols,
                         int64_t stride, cudaStream_t s) {
  constexpr int NW = 4;
  const int stage = bb_stage_elems<FT>(P->max_bw + 1);
  // as many stages as leave room for the tiles an SM holds at once
  const size_t bytes = (size_t)stage * sizeof(FT);
  const int S = (int)std::max<size_t>(2, std::min<size_t>(sizeof(FT) == 8 ? 3 : 6, 110 * 1024 / bytes));
  // few tiles: ask for so much shared memory that the scheduler cannot put more
  // than ceil(tiles / SMs) of them on one SM while others stay empty
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, P->device);
  const bool multi = ncols >= 3;  // four columns per CTA
  const int per_sm = (P->nparts * (multi ? (ncols + 3) / 4 : ncols) + sms - 1) / sms;
  const size_t smem = std::max(S * bytes, per_sm <= 3 ? (size_t)(224 / (per_sm + 1) + 1) * 1024 : 0);
  auto go = [&](auto* kern, int nc) {
    allow_smem(kern, smem);
    kern<<<P->nparts * ((ncols + nc - 1) / nc), 32 * NW, smem, s>>>(
        P->tabs.node_off.as<int32_t>(), P->tabs.bw.as<int32_t>(), P->tabs.band_off.as<int64_t>(),
        P->d_bb_off.as<int32_t>(), P->d_bb_order.as<int32_t>(), Lc, Uc, Li, Ui, v, stride, P->nparts, ncols, stage, S);
  };
  const int K = (31 + P->max_bw) / 32;
  if (K <= 2) multi ? go(band_solve_blk_kernel<FT, 2, NW, 4>, 4) : go(band_solve_blk_kernel<FT, 2, NW, 1>, 1);
  else if (K <= 4) multi ? go(band_solve_blk_kernel<FT, 4, NW, 4>, 4) : go(band_solve_blk_kernel<FT, 4, NW, 1>, 1);
  else multi ? go(band_solve_blk_kernel<FT, 8, NW, 4>, 4) : go(band_solve_blk_kernel<FT, 8, NW, 1>, 1);
}

bool launch_band_solve_blk(vtm_plan_s* P, double* v, int ncols, int64_t stride, cudaStream_t s) {
  if (!P->bb_ok) return false;
  launch_blk_t<double>(P, v, P->d_Lc.as<double>(), P->d_Uc.as<double>(), P->d_bb_Li.as<double>(),
                       P->d_bb_Ui.as<double>(), ncols, stride, s);
  return true;
}

bool launch_band_solve_blk(vtm_plan_s* P, float* v, int ncols, int64_t stride, cudaStream_t s) {
  if (!P->bb_ok || !P->d_bb_Li32.p) return false;
  launch_blk_t<float>(P, v, P->d_Lc32.as<float>(), P->d_Uc32.as<float>(), P->d_bb_Li32.as<float>(),
                      P->d_bb_Ui32.as<float>(), ncols, stride, s);
  return true;
}

}  // namespace vtm
