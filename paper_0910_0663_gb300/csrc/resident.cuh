// Kernel 13: every sweep of an inner solve in one cooperative launch, one grid
// barrier per sweep, the reflection blocks held in shared memory.
//
// For plans of few sub-circuits the arithmetic of a sweep takes a microsecond or
// two and the launch-per-sweep kernels spend the rest on kernel boundaries:
// launch, sweep-number ticket, reading blocks and port tables back from L2.
// Here CTA b keeps tiles b, b + grid, ... for the whole solve: TPC tiles of WPT
// warps each and a control warp.
//   * The warps of a tile split its packed 16x16 blocks (column-major order,
//     equal contiguous ranges, two blocks of a column at a time); each adds row
//     and column parts into sums of its own, added over the warps in order at the
//     end.  The last blocks of each range, as many as fit, stay in shared memory;
//     the others stream from L2 through two register slots, loaded while the grid
//     barrier is awaited.
//   * Arithmetic as in kernel 9 (FP32, BF16, FP16 storage; tiles of up to 256 ports) and
//     kernel 12 (FP64 plans: hi + lo FP32 pairs, double-float; up to 128 ports, and only
//     where kernel 12 is the fastest of the launch-per-sweep kernels: elsewhere FP64 plans
//     sweep in FP64, in one launch by general_resident_kernel<true> of general.cu).
//   * The residual terms of sweep k - 1 (from what the gather of sweep k read) are
//     formed while the grid barrier is awaited, so nothing but the waves is on the
//     critical path.  The control warp publishes the CTA's partial one sweep later,
//     arrives at the barrier and polls it (bounded); CTA 0's takes the decisions.
//     Partials of sweep k are out with barrier k + 1, closed in sweep k + 2 (which
//     judges iterate k - 1), and the decision rides in the barrier word and ends
//     every CTA before sweep k + 3: four wave slots.
// Plans that one SM holds take sweep_small_kernel (below) instead.
// What bounds it: the chain barrier (about 1.5 us) - gather - blocks - sums; for
// double-float the FP32 pipe and the latency of its chains in the block loop (30k
// instructions per sweep of a 256-port tile).  Measured per sweep, best
// launch-per-sweep kernel -> this one:
//   FP64  1504 tiles of 128 ports 36 -> 31 us; 121 tiles of 80 ports 13.3 -> 4.0 us (the FP64
//         resident form 6.7 us)
//   FP32  256 tiles of 256 ports 13.6 -> 6.7 us; 1232 tiles of 116 ports 13.3 -> 11 us
//   FP16  256 tiles of 128 ports 6 -> 3.2 us
// With more than 11 (FP64) or 15 tiles per SM (2048^2 in 4096 tiles) the
// one-warp-per-tile kernels stay: shared memory then holds few of the blocks.
#pragma once

#include "gridctl.cuh"

namespace vtm {

// tile warps per CTA: with the control warp 128 registers per thread, and 168 for
// double-float
constexpr int res_warps(bool df) { return df ? 11 : 15; }
constexpr int kResSlots = 4;

template <class TT>
struct ResMode {  // FP32 and 16-bit storage
  using WV = float;      // a wave
  using AC = float;      // a sum
  using PAIR = float2;   // (w_in, w_out)
  using KD = float2;
  using CV = float;
  static constexpr int kBlkBytes = kSymB * kSymB * (int)sizeof(TT);
};
template <>
struct ResMode<double> {  // double-float
  using WV = df;
  using AC = dacc;
  using PAIR = float4;
  using KD = float4;
  using CV = float2;
  static constexpr int kBlkBytes = kSymB * kSymB * 8;
};

struct ResArgs {
  const void* Tp;
  const TileDesc* tdesc;
  const int32_t* twin;
  const void* kd;
  const uint8_t* run;
  const void* c;
  void* state3;
  int64_t nports;
  SweepCtrl* ctrl;
  unsigned long long* bar;  // the barrier word (gridctl.cuh)
  double* part;             // [2][grid]
  double* hist;
  int hist_len, nparts, pp, tpc, wpt, nres;
  uint32_t max_polls;
};

// The incident waves of a tile in shared memory.  Double-float keeps them in the
// pairs its instructions take -- (w, w) for the columns of a block, (w(r), w(r + 8))
// for its rows, each with the negated high parts -- so that no operand has to be
// assembled from single registers.
template <class TT>
struct ResWaves {
  static constexpr int kBytes = 4;  // per port
  float* w;
  __device__ ResWaves(unsigned char* base, int pp) : w(reinterpret_cast<float*>(base)) {}
  __device__ float get(int s) const { return w[s]; }
  __device__ void set(int s, float v) { w[s] = v; }
};
template <>
struct ResWaves<double> {
  static constexpr int kBytes = 36;
  float4 *col4, *row4;  // {h, h, l, l} per port; {h(r), h(r+8), l(r), l(r+8)} per row pair
  float2 *coln, *rown;  // the negated high parts
  __device__ ResWaves(unsigned char* base, int pp) {
    col4 = reinterpret_cast<float4*>(base);
    row4 = col4 + pp;
    coln = reinterpret_cast<float2*>(row4 + pp / 2);
    rown = coln + pp;
  }
  __device__ df get(int s) const {
    const float4 v = col4[s];
    return {v.x, v.z};
  }
  __device__ void set(int s, df v) {
    col4[s] = make_float4(v.h, v.h, v.l, v.l);
    coln[s] = make_float2(-v.h, -v.h);
    const int i = (s / kSymB) * 8 + (s & 7), o = (s >> 3) & 1;
    float* r = reinterpret_cast<float*>(row4 + i);
    r[o] = v.h;
    r[2 + o] = v.l;
    reinterpret_cast<float*>(rown + i)[o] = -v.h;
  }
};

// bytes of shared memory apart from the resident blocks: per tile the incident
// waves, outgoing waves, what the residual needs, twins; per warp the sums
template <class TT>
__host__ __device__ constexpr size_t res_base_bytes(int pp, int tpc, int warps) {
  using M = ResMode<TT>;
  return (size_t)tpc * pp * (ResWaves<TT>::kBytes + 4 * sizeof(typename M::WV) + 4) +
         (size_t)warps * pp * sizeof(typename M::AC);
}

// One lane's share of a packed block: rows r1 and r1 + 8 (r1 = lane / 4),
// columns 4 (lane % 4) .. + 3.
template <class TT>
struct ResBlock {
  typename SymLoad<TT>::raw r;
  __device__ void load(const void* tile, int idx, int lane) {
    r = SymLoad<TT>::load(reinterpret_cast<const TT*>(tile) + (size_t)idx * kSymB * kSymB, lane);
  }
  __device__ void pair() {}
  __device__ void put(unsigned char* slot, int lane) const {
    if constexpr (std::is_same<TT, float>::value) {
      reinterpret_cast<float4*>(slot)[lane] = r.a;
      reinterpret_cast<float4*>(slot)[lane + 32] = r.b;
    } else {
      reinterpret_cast<uint4*>(slot)[lane] = r;
    }
  }
  __device__ void get(const unsigned char* slot, int lane) {
    r = SymLoad<TT>::load_shared(reinterpret_cast<const TT*>(slot), lane);
  }
  __device__ void values(float4& a, float4& b) const {
    if constexpr (std::is_same<TT, float>::value) {
      a = r.a;
      b = r.b;
    } else {
      const float2 e0 = Pair16<TT>::f2(r.x), e1 = Pair16<TT>::f2(r.y);
      const float2 e2 = Pair16<TT>::f2(r.z), e3 = Pair16<TT>::f2(r.w);
      a = make_float4(e0.x, e0.y, e1.x, e1.y);
      b = make_float4(e2.x, e2.y, e3.x, e3.y);
    }
  }
};
template <>
struct ResBlock<double> {
  float4 h01, h23, l01, l23;  // columns (0, 1) and (2, 3): {row r1, r1 + 8, row r1, r1 + 8}
  // from the stored form (hi block, lo block, row-major): straight into pairs
  __device__ void load(const void* tile, int idx, int lane) {
    const float4* p = reinterpret_cast<const float4*>(tile) + (size_t)idx * 128 + lane;
    h01 = __ldg(p);
    h23 = __ldg(p + 32);
    l01 = __ldg(p + 64);
    l23 = __ldg(p + 96);
  }
  __device__ void pair() {  // (row r1 columns 0..3, row r1 + 8 columns 0..3) -> pairs of rows
    const float4 a = h01, b = h23, c = l01, d = l23;
    h01 = make_float4(a.x, b.x, a.y, b.y);
    h23 = make_float4(a.z, b.z, a.w, b.w);
    l01 = make_float4(c.x, d.x, c.y, d.y);
    l23 = make_float4(c.z, d.z, c.w, d.w);
  }
  __device__ void put(unsigned char* slot, int lane) const {
    float4* p = reinterpret_cast<float4*>(slot) + lane;
    p[0] = h01;
    p[32] = h23;
    p[64] = l01;
    p[96] = l23;
  }
  __device__ void get(const unsigned char* slot, int lane) {
    const float4* p = reinterpret_cast<const float4*>(slot) + lane;
    h01 = p[0];
    h23 = p[32];
    l01 = p[64];
    l23 = p[96];
  }
};

// A warp's sums over its block range: row() gives the row part of a block (valid in
// lanes with bit 1 clear, for row `row_of`) and keeps its column part in registers
// until the column (or the range) ends.
__device__ __forceinline__ int res_row_of(int lane) { return (lane >> 2) + ((lane & 1) ? 8 : 0); }

template <class TT>
struct ResApply {
  float2 ca01, ca23;
  __device__ void clear() { ca01 = ca23 = make_float2(0.f, 0.f); }
  static __device__ float add(float a, float b) { return a + b; }
  __device__ float row(const ResBlock<TT>& blk, int bi, int bj, int lane, const ResWaves<TT>& wv) {
    const float* w_in = wv.w;
    constexpr unsigned FULL = 0xffffffffu;
    const int r1 = lane >> 2, cg = lane & 3;
    const bool b0 = lane & 1;
    float4 va, vb;
    blk.values(va, vb);
    const float2 a01 = make_float2(va.x, va.y), a23 = make_float2(va.z, va.w);
    const float2 b01 = make_float2(vb.x, vb.y), b23 = make_float2(vb.z, vb.w);
    const float4 wc = *reinterpret_cast<const float4*>(w_in + bj * kSymB + cg * 4);
    const float2 wc01 = make_float2(wc.x, wc.y), wc23 = make_float2(wc.z, wc.w);
    const float2 pa = __ffma2_rn(a23, wc23, __fmul2_rn(a01, wc01));
    const float2 pb = __ffma2_rn(b23, wc23, __fmul2_rn(b01, wc01));
    const float x1 = pa.x + pa.y, x2 = pb.x + pb.y;
    float t = (b0 ? x2 : x1) + __shfl_xor_sync(FULL, b0 ? x1 : x2, 1);
    t += __shfl_xor_sync(FULL, t, 2);
    if (bi != bj) {
      const float wr1 = w_in[bi * kSymB + r1], wr2 = w_in[bi * kSymB + r1 + 8];
      const float2 w1 = make_float2(wr1, wr1), w2 = make_float2(wr2, wr2);
      ca01 = __ffma2_rn(b01, w2, __ffma2_rn(a01, w1, ca01));
      ca23 = __ffma2_rn(b23, w2, __ffma2_rn(a23, w1, ca23));
    }
    return t;
  }
  __device__ void flush(int bj, int lane, float* acc) {
    constexpr unsigned FULL = 0xffffffffu;
    const int cg = lane & 3;
    const bool b4 = lane & 16, b3 = lane & 8;
    float k0 = b4 ? ca23.x : ca01.x, k1 = b4 ? ca23.y : ca01.y;
    k0 += __shfl_xor_sync(FULL, b4 ? ca01.x : ca23.x, 16);
    k1 += __shfl_xor_sync(FULL, b4 ? ca01.y : ca23.y, 16);
    float t1 = (b3 ? k1 : k0) + __shfl_xor_sync(FULL, b3 ? k0 : k1, 8);
    t1 += __shfl_xor_sync(FULL, t1, 4);
    if (!(lane & 4)) acc[bj * kSymB + cg * 4 + (b4 ? 2 : 0) + (b3 ? 1 : 0)] += t1;
  }
};
template <>
struct ResApply<double> {
  dacc2 ca[4];  // per column, the two rows as halves
  __device__ void clear() {
#pragma unroll
    for (int j = 0; j < 4; ++j) ca[j] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  }
  static __device__ dacc add(dacc a, dacc b) { return dacc_add(a, b); }
  __device__ dacc row(const ResBlock<double>& v, int bi, int bj, int lane, const ResWaves<double>& wv) {
    constexpr unsigned FULL = 0xffffffffu;
    const int cg = lane & 3;
    const bool b0 = lane & 1;
    const float2 h[4] = {make_float2(v.h01.x, v.h01.y), make_float2(v.h01.z, v.h01.w),
                         make_float2(v.h23.x, v.h23.y), make_float2(v.h23.z, v.h23.w)};
    const float2 l[4] = {make_float2(v.l01.x, v.l01.y), make_float2(v.l01.z, v.l01.w),
                         make_float2(v.l23.x, v.l23.y), make_float2(v.l23.z, v.l23.w)};
    const float4* wc = wv.col4 + bj * kSymB + cg * 4;
    const float2* wn = wv.coln + bj * kSymB + cg * 4;
    dacc2 x;
    {
      const float4 w = wc[0];
      x = dacc2_first(h[0], l[0], make_float2(w.x, w.y), make_float2(w.z, w.w));
    }
#pragma unroll
    for (int j = 1; j < 4; ++j) {
      const float4 w = wc[j];
      dacc2_fma(x, h[j], l[j], make_float2(w.x, w.y), wn[j], make_float2(w.z, w.w));
    }
    if (bi != bj) {
      const float4 w = wv.row4[bi * 8 + (lane >> 2)];
      const float2 n = wv.rown[bi * 8 + (lane >> 2)];
#pragma unroll
      for (int j = 0; j < 4; ++j) dacc2_fma(ca[j], h[j], l[j], make_float2(w.x, w.y), n, make_float2(w.z, w.w));
    }
    const dacc x1 = dacc2_lo(x), x2 = dacc2_hi(x);
    dacc t = dacc_add(b0 ? x2 : x1, shfl_xor_dacc(b0 ? x1 : x2, 1));
    return dacc_add(t, shfl_xor_dacc(t, 2));
  }
  __device__ void flush(int bj, int lane, dacc* acc) {
    const int cg = lane & 3;
    const bool b4 = lane & 16, b3 = lane & 8;
    dacc c[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) c[j] = dacc_add(dacc2_lo(ca[j]), dacc2_hi(ca[j]));
    dacc k0 = b4 ? c[2] : c[0], k1 = b4 ? c[3] : c[1];
    k0 = dacc_add(k0, shfl_xor_dacc(b4 ? c[0] : c[2], 16));
    k1 = dacc_add(k1, shfl_xor_dacc(b4 ? c[1] : c[3], 16));
    dacc t1 = dacc_add(b3 ? k1 : k0, shfl_xor_dacc(b3 ? k0 : k1, 8));
    t1 = dacc_add(t1, shfl_xor_dacc(t1, 4));
    if (!(lane & 4)) {
      dacc& o = acc[bj * kSymB + cg * 4 + (b4 ? 2 : 0) + (b3 ? 1 : 0)];
      o = dacc_add(o, t1);
    }
  }
};

// Squared node residuals of sweep k - 1 over the ports s = first, first + step, ...
// of a tile (the lanes of a warp), scaled by a power of two (see pow2_exponent);
// the sum in lane 0.  sv: own (w_in, w_out) and the twin's w_in of sweep k - 1; wv:
// the twin's w_out of sweep k - 1, that is the incident wave of sweep k.
template <class TT, int PPL>
__device__ __forceinline__ double res_partial(const typename ResMode<TT>::WV* sv,
                                              const ResWaves<TT>& wv, const uint8_t* __restrict__ run,
                                              const typename ResMode<TT>::KD* __restrict__ kd, int pp, int p,
                                              int first, int step) {
  using WV = typename ResMode<TT>::WV;
  constexpr bool DF = std::is_same<TT, double>::value;
  constexpr unsigned FULL = 0xffffffffu;
  WV r[PPL];
  float rmax = 0.f;
#pragma unroll
  for (int m = 0; m < PPL; ++m) {
    const int s = first + step * m;
    r[m] = WV{};
    const int nr = s < p ? (int)__ldg(run + s) : 0;
    for (int q = s; q < s + nr; ++q) {
      if constexpr (DF) r[m] = df_add(r[m], port_residual_df(sv[q], sv[pp + q], sv[2 * pp + q], wv.get(q), __ldg(kd + q)));
      else r[m] += port_residual<float>(sv[q], sv[pp + q], sv[2 * pp + q], wv.get(q), __ldg(kd + q));
    }
    if constexpr (DF) rmax = fmaxf(rmax, fabsf(r[m].h));
    else rmax = fmaxf(rmax, fabsf(r[m]));
  }
  const int e = pow2_exponent(warp_max(rmax));
  const float sc = pow2f(-e);
  WV sq = WV{};
#pragma unroll
  for (int m = 0; m < PPL; ++m) {
    if constexpr (DF) {
      const df v = {r[m].h * sc, r[m].l * sc};
      sq = df_add(sq, df_mul(v, v));
    } else {
      sq += (r[m] * sc) * (r[m] * sc);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    if constexpr (DF) sq = df_add(sq, df{__shfl_down_sync(FULL, sq.h, o), __shfl_down_sync(FULL, sq.l, o)});
    else sq += __shfl_down_sync(FULL, sq, o);
  }
  double v;
  if constexpr (DF) v = (double)sq.h + (double)sq.l;
  else v = (double)sq;
  return v * pow2d(2 * e);
}

template <class TT, int PPL>
__global__ void __launch_bounds__(32 * (res_warps(std::is_same<TT, double>::value) + 1), 1)
    sweep_resident_kernel(const ResArgs A) {
  using M = ResMode<TT>;
  using WV = typename M::WV;
  using AC = typename M::AC;
  using PAIR = typename M::PAIR;
  using KD = typename M::KD;
  constexpr bool DF = std::is_same<TT, double>::value;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int B = kSymB;  // PPL: ports per lane, ceil(pp / (32 WPT))
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flag;
  __shared__ double s_part[2][16];  // residual partials of a sweep
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nthreads = blockDim.x, nw = (nthreads >> 5) - 1;
  const int pp = A.pp, tpc = A.tpc, wpt = A.wpt;
  // shared memory: resident blocks | [tpc][pp] w_in, w_out | [tpc][3][pp] the
  // residual's own (w_in, w_out) and the twin's w_in | [nw][pp] sums | [tpc][pp] twins
  unsigned char* sm = smem_raw + (size_t)nw * A.nres * M::kBlkBytes;
  WV* wo_all = reinterpret_cast<WV*>(sm + (size_t)tpc * pp * ResWaves<TT>::kBytes);
  WV* sv_all = wo_all + (size_t)tpc * pp;
  AC* acc_all = reinterpret_cast<AC*>(sv_all + 3 * (size_t)tpc * pp);
  int* tw_all = reinterpret_cast<int*>(acc_all + (size_t)nw * pp);
  if (tid == 0) s_flag = 0;
  if (tid < 32) s_part[0][tid] = 0.0;
  __syncthreads();
  if (warp == nw) {
    // ---- control warp ----
    res_control(A.ctrl, A.bar, A.part, A.hist, A.hist_len, A.max_polls, &s_flag, s_part[0], 16, nw, lane);
  } else {
    // ---- tile warps ----
    const int slot = warp / wpt, part = warp % wpt;
    const int g = slot * gridDim.x + blockIdx.x;
    TileDesc dsc{};
    if (g < A.nparts) dsc = A.tdesc[g];
    const int p0 = dsc.p0, p = dsc.p;
    const int nb = (p + B - 1) / B, nblk = nb * (nb + 1) / 2;
    const int q0 = (int)((long long)nblk * part / wpt), q1 = (int)((long long)nblk * (part + 1) / wpt);
    const int nstream = max(0, q1 - q0 - A.nres);  // blocks q0 .. q0 + nstream - 1 come from L2
    unsigned char* res = smem_raw + (size_t)warp * A.nres * M::kBlkBytes;
    const void* Tl = DF ? (const void*)(reinterpret_cast<const float*>(A.Tp) + 2 * dsc.Tp_off)
                        : (const void*)(reinterpret_cast<const TT*>(A.Tp) + dsc.Tp_off);
    ResWaves<TT> wv(sm + (size_t)slot * pp * ResWaves<TT>::kBytes, pp);
    WV* wo = wo_all + (size_t)slot * pp;
    WV* sv = sv_all + 3 * (size_t)slot * pp;
    int* tws = tw_all + (size_t)slot * pp;
    AC* acc = acc_all + (size_t)warp * pp;
    // block q of the column-major order: column bj, row bi
    int bj0 = (int)((sqrtf(8.f * q0 + 1.f) - 1.f) * 0.5f);
    while (bj0 * (bj0 + 1) / 2 > q0) --bj0;
    while ((bj0 + 1) * (bj0 + 2) / 2 <= q0) ++bj0;
    const int bi0 = q0 - bj0 * (bj0 + 1) / 2;
    auto packed = [&](int bi, int bj) { return bi * nb - bi * (bi - 1) / 2 + bj - bi; };
    {
      int bi = bi0, bj = bj0;
      for (int q = q0; q < q1; ++q) {
        if (q - q0 >= nstream) {
          ResBlock<TT> v;
          v.load(Tl, packed(bi, bj), lane);
          v.pair();
          v.put(res + (size_t)(q - q0 - nstream) * M::kBlkBytes, lane);
        }
        if (bi < bj) {
          ++bi;
        } else {
          ++bj;
          bi = 0;
        }
      }
    }
    for (int s = lane + 32 * part; s < nb * B; s += 32 * wpt) {
      wv.set(s, WV{});  // stays zero past p
      wo[s] = WV{};
      tws[s] = s < p ? A.twin[p0 + s] : 0;
    }
    auto group_sync = [&]() {
      if (wpt == 1) __syncwarp();
      else asm volatile("bar.sync %0, %1;" ::"r"(1 + slot), "r"(32 * wpt) : "memory");
    };
    // streamed blocks: two register slots, (sbi, sbj) the next one to load
    ResBlock<TT> pf[2];
    int sbi = bi0, sbj = bj0, sq = 0;
    auto stream_next = [&](ResBlock<TT>& d) {
      if (sq < nstream) {
        d.load(Tl, packed(sbi, sbj), lane);
        if (sbi < sbj) {
          ++sbi;
        } else {
          ++sbj;
          sbi = 0;
        }
      }
      ++sq;
    };
    const PAIR* gstate = reinterpret_cast<const PAIR*>(A.state3);
    const int rowp = res_row_of(lane);
    const bool row_owner = !(lane & 2);
    for (int k = 1;; ++k) {
      sbi = bi0;
      sbj = bj0;
      sq = 0;
      stream_next(pf[0]);
      stream_next(pf[1]);
      for (int s = lane; s < nb * B; s += 32) acc[s] = AC{};
      __syncthreads();  // the waves of sweep k - 1 are out and the flag is read
      if (*((volatile int*)&s_flag)) break;
      const size_t ps = (size_t)((k - 1) % kResSlots) * A.nports, cs = (size_t)(k % kResSlots) * A.nports;
      const PAIR* prev = gstate + ps;
      PAIR* cur = reinterpret_cast<PAIR*>(A.state3) + cs;
      // incident waves
      if (k > 1) {
        PAIR wt[PPL];
#pragma unroll
        for (int m = 0; m < PPL; ++m) {
          const int s = lane + 32 * (part + wpt * m);
          if (s < p) wt[m] = __ldcg(prev + tws[s]);
        }
#pragma unroll
        for (int m = 0; m < PPL; ++m) {
          const int s = lane + 32 * (part + wpt * m);
          if (s < p) {
            sv[s] = wv.get(s);
            sv[pp + s] = wo[s];
            if constexpr (DF) {
              sv[2 * pp + s] = {wt[m].x, wt[m].y};
              wv.set(s, {wt[m].z, wt[m].w});
            } else {
              sv[2 * pp + s] = wt[m].x;
              wv.set(s, wt[m].y);
            }
          }
        }
      }
      group_sync();
      // the warp's blocks, two of a column at a time
      ResApply<TT> ap;
      ap.clear();
      int bi = bi0, bj = bj0;
      auto end_column = [&]() {
        __syncwarp();  // the diagonal block's row part is in before the column's
        if (bj > 0) ap.flush(bj, lane, acc);
        __syncwarp();  // and the column part before later rows add to this block
        ap.clear();
        ++bj;
        bi = 0;
      };
      auto one = [&](const ResBlock<TT>& v) {
        const AC t = ap.row(v, bi, bj, lane, wv);
        if (row_owner) acc[bi * B + rowp] = ResApply<TT>::add(acc[bi * B + rowp], t);
        if (bi < bj) ++bi;
        else end_column();
      };
      auto two = [&](const ResBlock<TT>& v0, const ResBlock<TT>& v1) {  // rows bi, bi + 1 <= bj
        const AC a0 = acc[bi * B + rowp], a1 = acc[(bi + 1) * B + rowp];
        const AC t0 = ap.row(v0, bi, bj, lane, wv), t1 = ap.row(v1, bi + 1, bj, lane, wv);
        if (row_owner) {
          acc[bi * B + rowp] = ResApply<TT>::add(a0, t0);
          acc[(bi + 1) * B + rowp] = ResApply<TT>::add(a1, t1);
        }
        bi += 2;
        if (bi > bj) end_column();
      };
      int q = q0;
      for (; q - q0 < nstream; ++q) {
        ResBlock<TT> v = pf[0];
        pf[0] = pf[1];
        stream_next(pf[1]);
        v.pair();
        one(v);
      }
      const unsigned char* at = res;
      while (q < q1) {
        ResBlock<TT> v0, v1;
        v0.get(at, lane);
        if (bi < bj && q + 1 < q1) {
          v1.get(at + M::kBlkBytes, lane);
          two(v0, v1);
          q += 2;
          at += 2 * M::kBlkBytes;
        } else {
          one(v0);
          ++q;
          at += M::kBlkBytes;
        }
      }
      if (bi > 0) {  // the range ended inside a column
        __syncwarp();
        ap.flush(bj, lane, acc);
      }
      group_sync();
      // outputs: the tile's warps in order, then c (FP32: c first)
      for (int s = lane + 32 * part; s < p; s += 32 * wpt) {
        const AC* a = acc_all + (size_t)(slot * wpt) * pp + s;
        if constexpr (DF) {
          const float2 c0 = __ldg(reinterpret_cast<const float2*>(A.c) + p0 + s);
          dacc o = a[0];
#pragma unroll 4
          for (int w = 1; w < wpt; ++w) o = dacc_add(o, a[(size_t)w * pp]);
          o = dacc_add(dacc{c0.x, c0.y}, o);  // c last: its low part would round every sum before it
          const df v = dacc_value(o), wi = wv.get(s);
          wo[s] = v;
          cur[p0 + s] = make_float4(wi.h, wi.l, v.h, v.l);
        } else {
          float o = __ldg(reinterpret_cast<const float*>(A.c) + p0 + s);
#pragma unroll 4
          for (int w = 0; w < wpt; ++w) o += a[(size_t)w * pp];
          wo[s] = o;
          cur[p0 + s] = make_float2(wv.get(s), o);
        }
      }
      __syncthreads();  // every wave of sweep k is written
      if (k > 1) {  // the residual, while the grid barrier is awaited
        const double v = res_partial<TT, PPL>(sv, wv, A.run + p0, reinterpret_cast<const KD*>(A.kd) + p0, pp, p,
                                              lane + 32 * part, 32 * wpt);
        if (lane == 0) s_part[k & 1][warp] = v;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The same for a plan that one SM holds: one CTA, waves and full matrices in
// shared memory, one CTA barrier per sweep.  A lane is a row: tile t of pp rows
// takes pp / 32 warps, and row s adds T(s, q) w(q) over q, two columns per step
// (the halves of the paired instructions) -- no cross-lane sums, so a third of
// the packed form's instructions per tile of 32 ports.  Seven more warps form the
// residual of sweep k - 1 from its wave slot while sweep k runs, the last warp
// closes the sweep before.  Issue-bound.
// Measured: 16 tiles of up to 32 ports in double-float 5.4 us per launch of the best
// other kernel, 2.6 us here (5.3 us with the packed blocks of the form above).
// ---------------------------------------------------------------------------

constexpr int kSmallRows = 16, kSmallSide = 7;  // most row warps; residual warps
constexpr int kSmallPorts = 32 * kSmallSide * 4;  // four ports per lane of the residual warps

// residual term of a port from the (w_in, w_out) pairs of both ends
__device__ __forceinline__ df res_term(float4 o, float4 t, float4 kd) {
  return port_residual_df({o.x, o.y}, {o.z, o.w}, {t.x, t.y}, {t.z, t.w}, kd);
}
__device__ __forceinline__ float res_term(float2 o, float2 t, float2 kd) {
  return port_residual<float>(o.x, o.y, t.x, t.y, kd);
}

// matrices, incident waves, wave slots and port tables
template <class TT>
__host__ __device__ constexpr size_t small_bytes(int pr, int tiles, int64_t nports) {
  using M = ResMode<TT>;
  return (size_t)tiles * pr * pr * sizeof(typename M::WV) + (size_t)tiles * pr * sizeof(typename M::WV) +
         (size_t)nports * (kResSlots * sizeof(typename M::PAIR) + sizeof(typename M::KD) + 4 + 4);
}

template <class TT>
__global__ void __launch_bounds__(32 * (kSmallRows + kSmallSide + 1), 1) sweep_small_kernel(const ResArgs A) {
  using M = ResMode<TT>;
  using WV = typename M::WV;
  using PAIR = typename M::PAIR;
  using KD = typename M::KD;
  constexpr bool DF = std::is_same<TT, double>::value;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int B = kSymB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // the decision of sweep k in word (k + 1) & 1, read behind barrier k + 1: every warp leaves at
  // the same sweep (one word could be read late, with the decision that this sweep has just made)
  __shared__ int s_flag[2];
  __shared__ double s_part[2][kSmallSide];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthreads = blockDim.x;
  const int pr = A.pp;           // rows and columns of a tile: a multiple of 32
  const int rpt = pr / 32, nrow = A.nparts * rpt;
  const int np = (int)A.nports;
  // matrices: step q / 2 (DF) or q / 4 of row s as one float4 -- {h q, h q+1, l q, l q+1} or four columns
  float4* Ts = reinterpret_cast<float4*>(smem_raw);
  constexpr int CPS = DF ? 2 : 4;  // columns per step
  const int nstep = pr / CPS;
  float4* ws = Ts + (size_t)A.nparts * nstep * pr;  // incident waves in the same steps
  PAIR* st = reinterpret_cast<PAIR*>(ws + (size_t)A.nparts * nstep);
  KD* kds = reinterpret_cast<KD*>(st + (size_t)kResSlots * np);
  int* tws = reinterpret_cast<int*>(kds + np);
  int* runs = tws + np;
  for (int t = 0; t < A.nparts; ++t) {
    const TileDesc d = A.tdesc[t];
    const int nb = (d.p + B - 1) / B;
    float* Tf = reinterpret_cast<float*>(Ts + (size_t)t * nstep * pr);
    for (int e = tid; e < pr * pr; e += nthreads) {
      const int s = e % pr, q = e / pr;
      float h = 0.f, l = 0.f;
      if (s < d.p && q < d.p) {
        int r = s, c = q;  // the packed entry on or above the block diagonal
        if (r / B > c / B) {
          r = q;
          c = s;
        }
        const int bi = r / B, bj = c / B, w = (r % B) * B + c % B;
        const size_t blk = bi * nb - bi * (bi - 1) / 2 + bj - bi;
        if constexpr (DF) {
          const float* x = reinterpret_cast<const float*>(A.Tp) + 2 * d.Tp_off + blk * 2 * B * B;
          h = x[w];
          l = x[B * B + w];
        } else if constexpr (sizeof(TT) == 4) {
          h = reinterpret_cast<const float*>(A.Tp)[d.Tp_off + blk * B * B + w];
        } else {  // lane order of a 16-bit block: row l/4 (+ 8), columns 4 (l%4) ..
          const int rr = r % B, cc = c % B;
          const int ln = (rr & 7) * 4 + cc / 4;
          h = Pair16<TT>::f(reinterpret_cast<const TT*>(A.Tp)[d.Tp_off + blk * B * B + ln * 8 + (rr >> 3) * 4 + cc % 4]);
        }
      }
      float* o = Tf + ((size_t)(q / CPS) * pr + s) * 4 + q % CPS;
      o[0] = h;
      if (DF) o[2] = l;
    }
  }
  for (int s = tid; s < np; s += nthreads) {
    tws[s] = A.twin[s];
    runs[s] = A.run[s];
    kds[s] = reinterpret_cast<const KD*>(A.kd)[s];
  }
  for (int i = tid; i < A.nparts * nstep; i += nthreads) ws[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid < 2) s_flag[tid] = 0;
  if (tid < 2 * kSmallSide) s_part[0][tid] = 0.0;
  // row warps: tile, row, port
  const int tile = warp / rpt, row = 32 * (warp % rpt) + lane;
  int port = -1, tw = 0, nst = 0;
  float2 c0 = make_float2(0.f, 0.f);
  if (warp < nrow) {
    const TileDesc d = A.tdesc[tile];
    nst = (d.p + 2 * CPS - 1) / (2 * CPS) * 2;  // whole pairs of steps: columns past p are zero
    if (row < d.p) {
      port = d.p0 + row;
      tw = A.twin[port];
      if constexpr (DF) c0 = reinterpret_cast<const float2*>(A.c)[port];
      else c0.x = reinterpret_cast<const float*>(A.c)[port];
    }
  }
  ResDecision dec;
  dec.load(A.ctrl);
  for (int k = 1;; ++k) {
    __syncthreads();  // the waves of sweep k - 1 and the flag
    if (*((volatile int*)&s_flag[k & 1])) break;
    const PAIR* prev = st + (size_t)((k - 1) % kResSlots) * np;
    if (warp < nrow) {
      float4* wt = ws + (size_t)tile * nstep;
      WV wi = WV{};
      if (port >= 0 && k > 1) {
        const PAIR v = prev[tw];
        float* o = reinterpret_cast<float*>(wt + row / CPS) + row % CPS;
        if constexpr (DF) {
          wi = {v.z, v.w};
          o[0] = v.z;
          o[2] = v.w;
        } else {
          wi = v.y;
          o[0] = v.y;
        }
      }
      if (rpt == 1) __syncwarp();
      else asm volatile("bar.sync %0, %1;" ::"r"(1 + tile), "r"(32 * rpt) : "memory");
      const float4* Tr = Ts + (size_t)tile * nstep * pr + row;
      if constexpr (DF) {
        dacc2 a = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, b = a;
#pragma unroll 2
        for (int i = 0; i < nst; i += 2) {
          const float4 t0 = Tr[(size_t)i * pr], w0 = wt[i];
          const float2 h0 = make_float2(w0.x, w0.y);
          dacc2_fma(a, make_float2(t0.x, t0.y), make_float2(t0.z, t0.w), h0, f2neg(h0), make_float2(w0.z, w0.w));
          const float4 t1 = Tr[(size_t)(i + 1) * pr], w1 = wt[i + 1];
          const float2 h1 = make_float2(w1.x, w1.y);
          dacc2_fma(b, make_float2(t1.x, t1.y), make_float2(t1.z, t1.w), h1, f2neg(h1), make_float2(w1.z, w1.w));
        }
        // c last: in a chain's E its low part would cost a rounding at 2^-48 |c| per step
        const dacc t = dacc_add(dacc_add(dacc2_lo(a), dacc2_hi(a)), dacc_add(dacc2_lo(b), dacc2_hi(b)));
        const df o = dacc_value(dacc_add(dacc{c0.x, c0.y}, t));
        if (port >= 0) st[(size_t)(k % kResSlots) * np + port] = make_float4(wi.h, wi.l, o.h, o.l);
      } else {
        float2 a = make_float2(c0.x, 0.f), b = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int i = 0; i < nst; ++i) {
          const float4 t = Tr[(size_t)i * pr], w = wt[i];
          a = __ffma2_rn(make_float2(t.x, t.y), make_float2(w.x, w.y), a);
          b = __ffma2_rn(make_float2(t.z, t.w), make_float2(w.z, w.w), b);
        }
        if (port >= 0) st[(size_t)(k % kResSlots) * np + port] = make_float2(wi, (a.x + b.x) + (a.y + b.y));
      }
    } else if (warp < nrow + kSmallSide) {
      // residual of sweep k - 1 at the nodes whose ports start at s
      const int sv = warp - nrow;
      if (k > 1) {
        WV r[4];
        int nr[4];
        float rmax = 0.f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int s = lane + 32 * (sv + kSmallSide * m);
          nr[m] = s < np ? runs[s] : 0;
          r[m] = WV{};
          if (nr[m]) r[m] = res_term(prev[s], prev[tws[s]], kds[s]);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int s = lane + 32 * (sv + kSmallSide * m);
          for (int q = s + 1; q < s + nr[m]; ++q) {  // further branches of the node
            const WV t = res_term(prev[q], prev[tws[q]], kds[q]);
            if constexpr (DF) r[m] = df_add(r[m], t);
            else r[m] += t;
          }
          if constexpr (DF) rmax = fmaxf(rmax, fabsf(r[m].h));
          else rmax = fmaxf(rmax, fabsf(r[m]));
        }
        const int e = pow2_exponent(warp_max(rmax));
        const float sc = pow2f(-e);
        WV sq = WV{};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          if (32 * kSmallSide * m >= np) break;
          if constexpr (DF) {
            const df v = {r[m].h * sc, r[m].l * sc};
            sq = df_add(sq, df_mul(v, v));
          } else {
            sq += (r[m] * sc) * (r[m] * sc);
          }
        }
        for (int o = 16; o > 0; o >>= 1) {
          if constexpr (DF) sq = df_add(sq, df{__shfl_down_sync(FULL, sq.h, o), __shfl_down_sync(FULL, sq.l, o)});
          else sq += __shfl_down_sync(FULL, sq, o);
        }
        if (lane == 0) {
          double v;
          if constexpr (DF) v = (double)sq.h + (double)sq.l;
          else v = (double)sq;
          s_part[k & 1][sv] = v * pow2d(2 * e);
        }
      }
    } else if (lane == 0 && k > 1) {
      // close sweep k - 1 (the residual of sweep k - 2)
      const double* v = s_part[(k - 1) & 1];
      const double t = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + v[6]);
      const int f = dec.close(k - 1, t, A.hist, A.hist_len);
      if (f) {
        dec.store(A.ctrl, k - 1, f);
        *((volatile int*)&s_flag[(k + 1) & 1]) = f;
      }
    }
  }
  // the slot the host recovers from
  volatile SweepCtrl* ct = A.ctrl;
  const int flag = ct->flag;
  const int ks = (flag == 1 || flag == 4) ? ct->conv_sweep : min(ct->k - 1, ct->k_max);
  const PAIR* src = st + (size_t)(ks % kResSlots) * np;
  PAIR* dst = reinterpret_cast<PAIR*>(A.state3) + (size_t)(ks % kResSlots) * np;
  for (int i = tid; i < np; i += nthreads) dst[i] = src[i];
}

}  // namespace vtm
