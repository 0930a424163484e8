// Reflection matrices of symmetric plans by blocked solves of 32 ports at a time.
//
// T_P needs G = K_P^-1 between port nodes only, and G is symmetric: with the
// ports sorted by their row, the solve for port q starts its forward pass at its
// own row (everything above is zero) and ends its backward pass there (G(s, q)
// for rows above comes from the solve of s).  That is half of the arithmetic of
// a full solve per port, and with 32 ports per work item each band column is
// used 32 times from shared memory.
//
// One CTA per work item (tile, 32 ports of neighbouring rows), taken from a
// queue, longest first.  The item's 32 right-hand sides live in a ring of rows
// in shared memory.  Per block of 32 rows: U = M_JJ^-1 V (the inverted unit
// diagonal blocks of bandblk.cu's set-up, zero triangle skipped), then the
// block's 32 columns update the rows below within the band; columns and inverse
// of the next block arrive by cp.async meanwhile.  The forward results wait in a
// global scratch array (one slab per resident CTA) for the backward pass.
// Every product is a 2 x 2 register tile per thread: GB300's FP64 pipe (2 FMA
// per clock and SM) is the bound, not shared memory.
// Measured: 256 tiles of 4096 rows, bw 64, 240 ports: 72.3 ms with a warp per port
// and a full solve each, 35.2 ms here (27 ms of FP64 pipe).  Half bandwidths up
// to 32 keep the warp per port: its solves stream through registers there and
// need no inverted blocks (256 tiles of 32 x 32: 3.03 ms against 2.84 + 0.43 ms
// for the inverses).
#include <algorithm>

#include "ptx.h"
#include "vtm_internal.h"

namespace vtm {

constexpr int kRfN = 32;         // rows per block
constexpr int kRfC = 32;         // ports (right-hand sides) per work item
constexpr int kRfThreads = 256;

struct __align__(16) ReflItem {
  int32_t tile, first, count, row0;  // first port in the tile's row order, ports, its row
};

// rows of the ring: a block, the rows its columns reach, one row of padding (a
// multiple of 32)
__host__ __device__ constexpr int rf_ring(int bw) { return (bw + 34 + 31) / 32 * 32; }
__host__ __device__ constexpr size_t rf_smem(int bw) {
  return sizeof(double) * ((size_t)rf_ring(bw) * kRfC + kRfN * kRfC + 2 * ((size_t)kRfN * (bw + 1) + kRfN * kRfN));
}

__device__ __forceinline__ void rf_copy8(double* smem, const double* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void rf_copy16(double* smem, const double* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}

struct RfTile {
  int n, bw, B, R;
  const double *cols, *inv;  // band columns and inverted blocks of the pass
};

// One pass over the 32-row blocks from pass row `start` (a multiple of 32) to
// `stop`.  A row enters the ring with its right-hand side: the unit vectors of
// the ports at `loc` (forward) or its row of `y` (backward).  out(s, stage, last)
// takes the block's result from U.
template <bool FWD, class Out>
__device__ __forceinline__ void rf_pass(const RfTile& T, int start, int stop, const int* loc, const double* y,
                                        double* ring, double* U, double* stage, Out&& out) {
  const int tid = threadIdx.x, cp = 2 * (tid & 15), rp = 2 * (tid >> 4);
  const int n = T.n, bw = T.bw, B = T.B, R = T.R;
  const int nst = kRfN * B + kRfN * kRfN;
  auto row = [&](int j) { return ring + (j % R) * kRfC; };
  auto init_rows = [&](int j0) {  // 32 pass rows from j0 into the ring
    if (FWD) {
      for (int e = tid; e < kRfN * kRfC; e += kRfThreads) {
        const int j = j0 + (e >> 5), c = e & 31;
        row(j)[c] = loc[c] == j ? 1.0 : 0.0;
      }
    } else {
      for (int e = tid; e < kRfN * kRfC / 2; e += kRfThreads) {
        const int j = j0 + (e >> 4), c = 2 * (e & 15);
        if (j < stop) rf_copy16(row(j) + c, y + (int64_t)(n - 1 - j) * kRfC + c);
        else *reinterpret_cast<double2*>(row(j) + c) = make_double2(0.0, 0.0);
      }
    }
  };
  auto load_stage = [&](int s) {
    double* st = stage + ((s / kRfN) & 1) * nst;
    const int c0 = FWD ? s : n - min(n, s + kRfN), c1 = FWD ? min(n, s + kRfN) : n - s;
    const double* src = T.cols + (int64_t)c0 * B;
    for (int e = tid; e < (c1 - c0) * B; e += kRfThreads) rf_copy8(st + e, src + e);
    const double* iv = T.inv + (int64_t)(s / kRfN) * kRfN * kRfN;
    double* di = st + kRfN * B;
    for (int e = tid; e < kRfN * kRfN; e += kRfThreads) rf_copy8(di + e, iv + e);
  };
  for (int j = start; j < start + R; j += kRfN) init_rows(j);
  load_stage(start);
  for (int s = start; s < stop; s += kRfN) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (s + kRfN < stop) load_stage(s + kRfN);
    const double* st = stage + ((s / kRfN) & 1) * nst;
    const double* iv = st + kRfN * B;
    const double* V = row(s);  // the block's rows are adjacent: R and s are multiples of 32
    double a00 = 0.0, a01 = 0.0, a10 = 0.0, a11 = 0.0;
#pragma unroll 4
    for (int k = 0; k < rp + 2; ++k) {
      const double2 m = *reinterpret_cast<const double2*>(iv + k * kRfN + rp);
      const double2 v = *reinterpret_cast<const double2*>(V + k * kRfC + cp);
      a00 += m.x * v.x;
      a01 += m.x * v.y;
      a10 += m.y * v.x;
      a11 += m.y * v.y;
    }
    *reinterpret_cast<double2*>(U + rp * kRfC + cp) = make_double2(a00, a01);
    *reinterpret_cast<double2*>(U + (rp + 1) * kRfC + cp) = make_double2(a10, a11);
    __syncthreads();
    const int last = (FWD ? min(n, s + kRfN) : n - s) - (FWD ? s : n - min(n, s + kRfN)) - 1;
    out(s, st, last);
    init_rows(s + R);  // the block's slots take the rows that enter next
    const int rmax = min(kRfN - 1 + bw, stop - 1 - s);  // last row the block's columns reach
    for (int r = kRfN + rp; r <= rmax; r += kRfN) {
      double* v = row(s + r) + cp;
      double b00 = 0.0, b01 = 0.0, b10 = 0.0, b11 = 0.0;
      const int q0 = max(0, r - bw);  // the first column that reaches row r
      const int a1 = s + r + 1 < stop ? bw : -1;  // row r + 1 may lie past the pass
#pragma unroll 4
      for (int q = q0; q < kRfN; ++q) {
        const double* col = st + (FWD ? q : last - q) * B + r - q;
        const double m0 = col[0], m1 = r + 1 - q <= a1 ? col[1] : 0.0;
        const double2 u = *reinterpret_cast<const double2*>(U + q * kRfC + cp);
        b00 += m0 * u.x;
        b01 += m0 * u.y;
        b10 += m1 * u.x;
        b11 += m1 * u.y;
      }
      double2 x = *reinterpret_cast<double2*>(v);
      x.x -= b00;
      x.y -= b01;
      *reinterpret_cast<double2*>(v) = x;
      x = *reinterpret_cast<double2*>(v + kRfC);
      x.x -= b10;
      x.y -= b11;
      *reinterpret_cast<double2*>(v + kRfC) = x;
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kRfThreads, 2) build_reflection_blk_kernel(
    const ReflItem* __restrict__ items, int nitems, int* __restrict__ queue, const int32_t* __restrict__ node_off,
    const int32_t* __restrict__ bwv, const int64_t* __restrict__ band_off, const int32_t* __restrict__ blk_off,
    const double* __restrict__ Lc, const double* __restrict__ Uc, const double* __restrict__ Li,
    const double* __restrict__ Ui, const int32_t* __restrict__ port_off, const int32_t* __restrict__ port_loc,
    const int32_t* __restrict__ by_row, const double* __restrict__ bin, const double* __restrict__ bout,
    const double* __restrict__ rho, const int64_t* __restrict__ T_off, const int32_t* __restrict__ T_ld,
    double* __restrict__ scratch, int64_t slab, double* __restrict__ Tm) {
  extern __shared__ __align__(16) double rsm[];
  __shared__ int s_item;
  __shared__ int loc[kRfC], prt[kRfC];  // the item's ports: row and local index
  const int tid = threadIdx.x;
  double* y = scratch + blockIdx.x * slab;  // forward results, [row][32]
  while (true) {
    if (tid == 0) s_item = atomicAdd(queue, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= nitems) return;
    const ReflItem d = items[it];
    const int t = d.tile, p0 = port_off[t], p = port_off[t + 1] - p0;
    RfTile T;
    T.n = node_off[t + 1] - node_off[t];
    T.bw = bwv[t];
    T.B = T.bw + 1;
    T.R = rf_ring(T.bw);
    double* ring = rsm;
    double* U = ring + T.R * kRfC;
    double* stage = U + kRfN * kRfC;
    const int32_t* order = by_row + p0;
    if (tid < kRfC) {
      const int q = tid < d.count ? order[d.first + tid] : -1;
      prt[tid] = q;
      loc[tid] = q >= 0 ? port_loc[p0 + q] : -1;
    }
    __syncthreads();
    const int n = T.n, B = T.B;
    const int64_t io = (int64_t)blk_off[t] * kRfN * kRfN;
    T.cols = Lc + band_off[t];
    T.inv = Li + io;
    const int start = d.row0 / kRfN * kRfN;
    rf_pass<true>(T, start, n, loc, nullptr, ring, U, stage, [&](int s, const double* st, int) {
      for (int e = tid; e < kRfN * kRfC; e += kRfThreads) {
        const int r = e >> 5, c = e & 31;
        if (s + r < n) y[(int64_t)(s + r) * kRfC + c] = U[e] * st[r * B];
      }
    });
    __threadfence();  // y of every thread before the backward pass reads it
    __syncthreads();
    T.cols = Uc + band_off[t];
    T.inv = Ui + io;
    double* Tb = Tm + T_off[t];
    const int ld = T_ld[t];
    int hi = p;  // ports of the rows not yet passed are order[0 .. hi)
    rf_pass<false>(T, 0, n - d.row0, loc, y, ring, U, stage, [&](int s, const double* st, int last) {
      // rows n - 1 - s down to n - 32 - s: their ports against the item's
      const int top = n - 1 - s;
      int lo = hi;
      {  // first port at or above row top - 31 (every thread the same search)
        int a = 0, b = hi;
        while (a < b) {
          const int m = (a + b) >> 1;
          if (port_loc[p0 + order[m]] < top - (kRfN - 1)) a = m + 1;
          else b = m;
        }
        lo = a;
      }
      for (int e = tid; e < (hi - lo) * kRfC; e += kRfThreads) {
        const int c = e & 31, sp = order[lo + (e >> 5)], q = prt[c];
        const int ls = port_loc[p0 + sp];
        if (q >= 0 && ls >= loc[c]) {
          const int r = top - ls;  // pass row within the block
          const double g = U[r * kRfC + c] * st[(last - r) * B];
          double v = bout[p0 + sp] * g * bin[p0 + q];
          if (sp == q) v += rho[p0 + q];
          Tb[(int64_t)q * ld + sp] = v;
          if (ls > loc[c]) Tb[(int64_t)sp * ld + q] = bout[p0 + q] * g * bin[p0 + sp];
        }
      }
      hi = lo;
    });
  }
}

// Symmetric plans of half bandwidth 33 up to what ring and stages leave room for
// (about 220); vtm_factor has made the inverted diagonal blocks.
static bool reflect_blk_eligible(const vtm_plan_s* P) {
  return P->symmetric && !P->general && !P->port_node.empty() && P->bb_ok && rf_smem(P->max_bw) <= 222 * 1024;
}

// *done = false where it does not serve
vtm_status build_reflections_blk(vtm_plan_s* P, bool* done) {
  cudaStream_t s = P->stream;
  *done = false;
  if (!reflect_blk_eligible(P)) return VTM_OK;
  if (P->refl_items == 0) {
    const size_t npt = P->port_node.size();
    std::vector<int32_t> by_row(npt);
    std::vector<ReflItem> items;
    for (int32_t t = 0; t < P->nparts; ++t) {
      const int32_t p0 = P->port_off[t], p = P->port_off[t + 1] - p0;
      for (int32_t q = 0; q < p; ++q) by_row[p0 + q] = q;
      std::stable_sort(by_row.begin() + p0, by_row.begin() + p0 + p,
                       [&](int32_t a, int32_t b) { return P->port_loc[p0 + a] < P->port_loc[p0 + b]; });
      for (int32_t f = 0; f < p; f += kRfC)
        items.push_back(ReflItem{t, f, std::min(kRfC, p - f), P->port_loc[p0 + by_row[p0 + f]]});
    }
    auto cost = [&](const ReflItem& d) {
      return (int64_t)(P->node_off[d.tile + 1] - P->node_off[d.tile] - d.row0) * (P->bw[d.tile] + 16);
    };
    std::stable_sort(items.begin(), items.end(), [&](const ReflItem& a, const ReflItem& b) { return cost(a) > cost(b); });
    VTM_TRY(upload(P->d_refl_items, items, s));
    VTM_TRY(upload(P->d_refl_order, by_row, s));
    VTM_CUDA_TRY(cudaStreamSynchronize(s));  // the host lists are about to go
    P->refl_items = (int)items.size();
  }
  const size_t smem = rf_smem(P->max_bw);
  VTM_CUDA_TRY(allow_smem(build_reflection_blk_kernel, smem));
  int sms = 152, per_sm = 1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, P->device);
  VTM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_reflection_blk_kernel, kRfThreads, smem));
  const int grid = std::min(P->refl_items, std::max(1, per_sm) * sms);
  const int64_t slab = (int64_t)P->max_nodes * kRfC;
  const vtm_status st = dev_alloc(P->d_refl_scratch, (size_t)grid * slab * sizeof(double));
  if (st == VTM_ENOMEM) return VTM_OK;  // a warp per port needs none
  VTM_TRY(st);
  *done = true;
  int* queue = P->d_err.as<int>() + 4;
  cudaMemsetAsync(queue, 0, sizeof(int), s);
  build_reflection_blk_kernel<<<grid, kRfThreads, smem, s>>>(
      P->d_refl_items.as<ReflItem>(), P->refl_items, queue, P->tabs.node_off.as<int32_t>(),
      P->tabs.bw.as<int32_t>(), P->tabs.band_off.as<int64_t>(), P->d_bb_off.as<int32_t>(), P->d_Lc.as<double>(),
      P->d_Uc.as<double>(), P->d_bb_Li.as<double>(), P->d_bb_Ui.as<double>(), P->tabs.port_off.as<int32_t>(),
      P->d_port_loc.as<int32_t>(), P->d_refl_order.as<int32_t>(), P->d_beta.as<double>(), P->d_bout.as<double>(),
      P->d_rho.as<double>(), P->tabs.T_off.as<int64_t>(), P->tabs.T_ld.as<int32_t>(), P->d_refl_scratch.as<double>(), slab,
      P->d_T64.as<double>());
  VTM_CUDA_TRY(cudaGetLastError());
  return VTM_OK;
}

}  // namespace vtm
