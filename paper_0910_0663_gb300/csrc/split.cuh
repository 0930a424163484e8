// Batched FP64 sweep on the tensor cores (FP64 plans).
//
// GB300's FP64 pipe (2 FMA per clock and SM) bounds every FP64 product of the
// batched sweep; its 16-bit tensor pipe is three orders of magnitude wider.  Both
// operands are therefore cut into nine signed base-128 digits (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numerical Algorithms 59, 2012): with 2^E above a row's (T_P) or a
// column's (W, per 256 inputs) largest entry, x = 2^(E - 62) sum_i d_i 2^(7 (8 - i)),
// |d_i| <= 64, exact to 2^(E - 63).  Digits are BF16 numbers, products of digits
// integers of at most 2^12, and the sums of the groups g = i + j over 256 inputs
// stay below 9 2^20 < 2^24: the FP32 accumulators hold them exactly.  Groups g > 8
// are left out: less than 2^-58 of the largest |T w| of the row and column each
// (FP64 products round at 2^-53 of their own size, their sum at 2^-53 of itself).
// The nine group sums join as 64-bit integers, one FP64 rounding per 256 inputs.
//
// Fixed point serves where the waves of a tile are of one size.  Where they are not (a
// column with one hot node decays by 2^-40 across a box), the large ones would leave an
// error of 2^-58 of themselves in outputs that are small, with a small entry of T_P at
// their place.  So a column's chunk whose largest wave is more than 2^6 above the largest
// of some eight neighbouring inputs of the tile is multiplied in FP64 instead, by the
// warps that join (dg_graded).  Measured, one hot node per column, 30 boxes, converged to
// 1e-10: entries 1e-30 of the peak were off by 0.3 of themselves, now by 1e-7 like the FP64
// kernel's; 110 boxes, every column hot, 2 / 18 / 64 columns: 0.89 / 3.0 / 8.5 ms per sweep
// (CUDA cores 6.9 ms at any count).  Columns of random currents are not graded; the blocks'
// maxima cost them 1 to 5% (18 columns 0.258 -> 0.260 ms).
//
// Per sweep two launches.  batch_digits_kernel: the incident waves (twins' outgoing
// ones) and their digits in the B operand's core matrices (a CTA per 256 ports), the
// residual of sweep k - 1 in FP64 (a CTA per 64 ports); its last CTA closes the sweep
// before, so a converged sweep never reads T_P.  batch_sweep_digits_kernel (persistent,
// one CTA per SM; an item is 128 outputs and up to 24 columns): tcgen05.mma with the
// nine groups of sums side by side in TMEM (below), T_P's digits (built once per
// factorisation, 18 bytes per entry) and W's by bulk copies through a ring of five
// steps, two sets of accumulators so that a chunk is joined while the next one runs.
// Bound: HBM (18 bytes of digits per entry of T_P).  Measured per sweep, thermal grid
// of 147,456 nodes in 110 boxes, 18 columns: FP64 CUDA cores 6.54 ms; digits with
// mma.sync 0.08 + 0.43 ms (its rate, about 4 cycles per m16n8k16 and SM); here
// 0.06 + 0.20 ms, the same bits (1.03 GB per sweep: 0.15 ms at the copy rate).
// Errors of the iterates against quad precision are those of the FP64 kernel to two
// digits (1 to 20 sweeps; 3e-16 thermal, 8e-15 grids), and those of converged solutions
// against a refined one, entry by entry, too (random columns 2.5e-11, hot ones 2e-11 at a
// tolerance of 1e-14).  Against the CUDA cores, per sweep: 2 tiles of 10 ports 19 us / 28,
// 16 of 32 ports 23 / 48, 64 of 256 ports 46 / 526, 110 boxes 260 / 6800 (18 columns).

constexpr int kDg = 9;          // digits
constexpr int kDgChunk = 16;    // 16-input blocks between two joins of the group sums
constexpr int kDgStages = 5;
constexpr int kDgSpan = 6;      // binary orders between the waves of a tile that the digits may serve
constexpr int kDgMaxNt = 3;     // 8-column groups per work item (nine groups of 24 columns: 216 of 256 TMEM columns)

// biased exponent of |v| (0x7ff: not finite)
__device__ __forceinline__ int exp_bits(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff); }

// the nine digits of v 2^(62 - E), most significant first; |v| <= 2^E.  From the
// bits alone: the FP64 pipe has the residual to do.
__device__ __forceinline__ void digits_of(double v, int E, int (&d)[kDg]) {
  const long long u = __double_as_longlong(v);
  const int e = (int)((u >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)u & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = max(e, 1) - 1075 + 62 - E;  // v 2^(62 - E) = +- m 2^sh, sh <= 9
  if (sh >= 0) m <<= min(sh, 10);            // (min: a non-finite v)
  else if (sh > -64) m = (m + (1ull << (-sh - 1))) >> -sh;
  else m = 0;
  long long x = u < 0 ? -(long long)m : (long long)m;
#pragma unroll
  for (int i = kDg - 1; i > 0; --i) {
    const int r = (int)((x + 64) & 127) - 64;
    d[i] = r;
    x = (x - r) >> 7;
  }
  d[0] = (int)x;
}

__device__ __forceinline__ uint32_t bf16_pair(int lo, int hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn((float)lo, (float)hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// E of every output row of T_P (port): 32 rows per CTA step, the columns over its warps
__global__ void __launch_bounds__(256) row_exponents_kernel(const double* __restrict__ T,
                                                            const int64_t* __restrict__ T_off,
                                                            const int32_t* __restrict__ T_ld,
                                                            const int32_t* __restrict__ port_off,
                                                            int* __restrict__ E) {
  __shared__ int mx[8][32];
  const int t = blockIdx.x, p0 = port_off[t], p = port_off[t + 1] - p0, ld = T_ld[t];
  const double* Tb = T + T_off[t];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int s0 = 32 * blockIdx.y; s0 < p; s0 += 32 * gridDim.y) {
    int m = 0;
    if (s0 + lane < p)
      for (int q = warp; q < p; q += 8) m = max(m, exp_bits(Tb[(size_t)q * ld + s0 + lane]));
    mx[warp][lane] = m;
    __syncthreads();
    if (warp == 0 && s0 + lane < p) {
      for (int w = 1; w < 8; ++w) m = max(m, mx[w][lane]);
      E[p0 + s0 + lane] = m - 1022;
    }
    __syncthreads();
  }
}

// T_P's digits in the canonical K-major layout of tcgen05.mma without swizzle (8 x 8
// core matrices of 128 bytes, the two of a row group's 16 inputs adjacent): per tile,
// blocks of 128 outputs, per block every step of 16 inputs, per step the nine digits
// of the block's row groups.  A block's last row group may be ragged, its steps
// shorter; what a short step leaves of its stage only reaches rows past the tile.
__host__ __device__ __forceinline__ int dg_groups(int p, int m) { return min(16, (p - 128 * m + 7) / 8); }

__global__ void __launch_bounds__(256) pack_digits_kernel(const double* __restrict__ T,
                                                          const int64_t* __restrict__ T_off,
                                                          const int32_t* __restrict__ T_ld,
                                                          const int32_t* __restrict__ port_off,
                                                          const int64_t* __restrict__ dg_off,
                                                          const int* __restrict__ E, uint2* __restrict__ out) {
  const int t = blockIdx.x, p0 = port_off[t], p = port_off[t + 1] - p0, ld = T_ld[t];
  const int nb = (p + 15) / 16, ng = (p + 7) / 8;
  const double* Tb = T + T_off[t];
  // a warp takes 16 inputs of a row group: lane = (quad of inputs, row)
  const int lane = threadIdx.x & 31, row = lane & 7, kq = lane >> 3;
  for (int b = blockIdx.y * 8 + (threadIdx.x >> 5); b < nb * ng; b += gridDim.y * 8) {
    const int gr = b / nb, kb = b - gr * nb, m = gr / 16, rg = dg_groups(p, m);
    const int s = 8 * gr + row, q = 16 * kb + 4 * kq;
    int d[4][kDg];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const double v = s < p && q + e < p ? Tb[(size_t)(q + e) * ld + s] : 0.0;
      digits_of(v, s < p ? E[p0 + s] : 0, d[e]);
    }
    uint2* o = out + dg_off[t] * 2 + ((int64_t)m * nb * 16 + (int64_t)kb * rg) * kDg * 32 + (gr & 15) * 32 +
               (kq >> 1) * 16 + row * 2 + (kq & 1);
#pragma unroll
    for (int i = 0; i < kDg; ++i)
      o[(int64_t)i * rg * 32] = make_uint2(bf16_pair(d[0][i], d[1][i]), bf16_pair(d[2][i], d[3][i]));
  }
}

// A chunk's waves of a column, [smallest block << 16 | largest exponent] (biased): graded
// where the largest is more than kDgSpan above the smallest block of the tile.
constexpr int kDgNoBlock = 0x7ff;
__device__ __forceinline__ bool dg_graded(int wx, int tile_min) { return (wx & 0xffff) - tile_min > kDgSpan; }

// Work item of the digits kernel: 256 ports of a tile (digits), or kDgRes (residual).
constexpr int kDgRes = 64;  // (128: 60 us a launch instead of 58)
struct __align__(16) DgChunk {
  int32_t tile, m0, kb, pad;  // first port in the tile, first 16-input block of W's digits
};

__global__ void __launch_bounds__(256) batch_digits_kernel(
    const DgChunk* __restrict__ chunks, int nchunks, const int32_t* __restrict__ port_off,
    const int32_t* __restrict__ twin, const double2* __restrict__ kd, const uint8_t* __restrict__ run,
    double* __restrict__ state, int64_t nports,
    int R, int NT, int ny, uint32_t* __restrict__ wd, int* __restrict__ wexp, BatchCtrl* __restrict__ ctrl,
    double* __restrict__ partials, const double* __restrict__ tol2, double* __restrict__ hist, int hist_len) {
  __shared__ double rsq[256];
  __shared__ int stw[16 * kDgChunk];
  __shared__ int cmax[64], bmin[64];  // per column: largest exponent, smallest largest of eight inputs
  __shared__ int s_k, s_flag;
  __shared__ bool s_last;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_k = *((volatile int*)&ctrl->k);
    s_flag = *((volatile int*)&ctrl->flag);
  }
  if (tid < 64) {
    cmax[tid] = 0;
    bmin[tid] = kDgNoBlock;
  }
  __syncthreads();
  if (s_flag) return;
  const int k = s_k;
  const DgChunk ch = chunks[blockIdx.x];
  const int p0 = port_off[ch.tile], p = port_off[ch.tile + 1] - p0;
  const double* prev = state + (size_t)((k - 1) & 1) * nports * 2 * R;
  // thread = (row slot, column): rows tid / R, + G, ...
  const int G = 256 / R, g = tid / R, r = tid - g * R;
  const size_t R2 = 2 * (size_t)R;
  if ((int)blockIdx.x >= nchunks) {
    // residual of sweep k - 1 at the nodes whose ports start in these kDgRes; with
    // a = w_out(s) - w_in(t), b = w_out(t) - w_in(s) the term of batch_residual is
    // d/2 ((a + b)/2 - (g/W) (a - b)): seven FP64 operations (their rate bounds it)
    const int ticket = blockIdx.x - nchunks, nres = gridDim.x - nchunks;
    double sq = 0.0;
    if (k > 1 && g < G) {
      const int s1 = p0 + min(p, ch.m0 + kDgRes);
#pragma unroll 4
      for (int s = p0 + ch.m0 + g; s < s1; s += G) {
        const int nr = run[s];
        double sum = 0.0;
        for (int q = s; q < s + nr; ++q) {
          const double* a = prev + (size_t)q * R2 + r;
          const double* b = prev + (size_t)twin[q] * R2 + r;
          const double wi_s = a[0], wo_s = a[R], wi_t = b[0], wo_t = b[R];
          const double2 k2 = kd[q];
          const double da = wo_s - wi_t, db = wo_t - wi_s;
          sum = fma(k2.y, fma(0.5, da + db, -(k2.x * (da - db))), sum);
        }
        sq = fma(sum, sum, sq);
      }
    }
    rsq[tid] = sq;
    __syncthreads();
    if (tid < R) {
      double a = 0.0;
      for (int i = 0; i < G; ++i) a += rsq[i * R + tid];
      partials[(size_t)ticket * R + tid] = 0.25 * a;  // the halves of d/2
    }
    __syncthreads();
    batch_item_done(ctrl, ticket, nres, R, partials, rsq);
  } else {
    const int m1 = min(p, ch.m0 + 16 * kDgChunk);
    double* cur = state + (size_t)(k & 1) * nports * 2 * R;
    // this sweep's incident waves and the largest exponent of each column
    const int nrow = m1 - ch.m0;
    for (int i = tid; i < nrow; i += 256) stw[i] = twin[p0 + ch.m0 + i];
    __syncthreads();
    if (g < G) {
      int mx = 0;
#pragma unroll 4
      for (int i = g; i < nrow; i += G) {
        const double w = k > 1 ? prev[(size_t)stw[i] * R2 + R + r] : 0.0;
        cur[(size_t)(p0 + ch.m0 + i) * R2 + r] = w;
        mx = max(mx, w != 0.0 ? exp_bits(w) : 0);
      }
      if (mx) atomicMax(&cmax[r], mx);
    }
    __syncthreads();
    // digits, a pair of rows per item, in the K-major core matrices of the B operand:
    // [16 inputs][column group of the items][digit][8 columns][input half][column][input]
    const int kbn = k > 1 ? (m1 - ch.m0 + 15) / 16 : 0, nt = NT * ny;
    const int w = tid & 63;
#pragma unroll 2
    for (int u = tid >> 6; u < kbn * nt; u += 4) {  // (a warp together)
      const int n = u % nt, kb = u / nt;
      const int c = 8 * n + ((w >> 2) & 7), i = 16 * kb + 8 * (w >> 5) + 2 * (w & 3);
      int d0[kDg], d1[kDg];
      const bool col = c < R;
      const double v0 = col && i < nrow ? prev[(size_t)stw[i] * R2 + R + c] : 0.0;
      const double v1 = col && i + 1 < nrow ? prev[(size_t)stw[i + 1] * R2 + R + c] : 0.0;
      const int E = col ? cmax[c] - 1022 : 0;
      digits_of(v0, E, d0);
      digits_of(v1, E, d1);
      uint32_t* o = wd + (((size_t)(ch.kb + kb) * ny + n / NT) * kDg * NT + n % NT) * 64 + w;
#pragma unroll
      for (int j = 0; j < kDg; ++j) o[(size_t)j * NT * 64] = bf16_pair(d0[j], d1[j]);
      // the largest of eight inputs (four lanes), unless fewer than four are left of the tile
      int e8 = max(exp_bits(v0), exp_bits(v1));
      e8 = max(e8, __shfl_xor_sync(0xffffffffu, e8, 1));
      e8 = max(e8, __shfl_xor_sync(0xffffffffu, e8, 2));
      if ((w & 3) == 0 && col && nrow - (16 * kb + 8 * (w >> 5)) >= 4) atomicMin(&bmin[c], e8);
    }
    __syncthreads();
    if (tid < 64) wexp[blockIdx.x * 64 + tid] = bmin[tid] << 16 | cmax[tid];
  }
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(&ctrl->counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  batch_finish(ctrl, partials, gridDim.x - nchunks, R, tol2, hist, hist_len, k, rsq);
}

// Work item of the sweep: 128 outputs of a tile.
struct __align__(16) DgItem {
  int32_t tile, m, kb, chunk;  // block of 128 outputs; W's first 16-input step and first chunk of the tile
  int64_t off;                 // the tile's digits (16-byte units)
  int64_t pad;
};

// Per step of 16 inputs nine tcgen05.mma (M = 128): digit i of T_P against the digits
// 0 .. 8 - i of W side by side (N = (9 - i) nc columns), accumulated at TMEM column
// i nc -- so the product of digits i and j lands in group i + j, and the first MMA of a
// chunk clears all groups.  N is a multiple of 16: with an odd number of column groups
// the last eight columns of an MMA go to a tenth group that nothing reads.
constexpr int kDgThreads = 320;    // warp 0: copies; warp 1: MMAs; eight warps join
constexpr uint32_t kDgABytes = kDg * 128 * 16 * 2;
constexpr uint32_t kDgTmem = 256;  // TMEM columns per accumulator set (two sets)
constexpr uint32_t dg_b_bytes(int NT) { return kDg * NT * 256; }
constexpr uint32_t dg_stage(int NT) { return kDgABytes + dg_b_bytes(NT) + 256; }  // (+ the rounded-up N)
constexpr size_t dg_smem(int NT) { return kDgStages * (size_t)dg_stage(NT) + 1024; }

// canonical K-major, no swizzle: 128 bytes between the two core matrices of 16 inputs,
// 256 between row groups
__device__ __forceinline__ uint64_t dg_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | (uint64_t)(128 >> 4) << 16 | (uint64_t)(256 >> 4) << 32 | (uint64_t)1 << 46;
}
__device__ __forceinline__ void dg_mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t n, uint32_t acc) {
  // F32 accumulate, BF16 A and B, both K-major, M = 128
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}
// four columns of the nine groups, this warp's 32 rows
__device__ __forceinline__ void dg_ld(uint32_t addr, uint32_t nc, uint32_t (&v)[kDg][4]) {
#define DG_R(g) "=r"(v[g][0]), "=r"(v[g][1]), "=r"(v[g][2]), "=r"(v[g][3])
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%36];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%37];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%38];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%39];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%40];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%41];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%42];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28,%29,%30,%31}, [%43];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%32,%33,%34,%35}, [%44];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : DG_R(0), DG_R(1), DG_R(2), DG_R(3), DG_R(4), DG_R(5), DG_R(6), DG_R(7), DG_R(8)
      : "r"(addr), "r"(addr + nc), "r"(addr + 2 * nc), "r"(addr + 3 * nc), "r"(addr + 4 * nc), "r"(addr + 5 * nc),
        "r"(addr + 6 * nc), "r"(addr + 7 * nc), "r"(addr + 8 * nc)
      : "memory");
#undef DG_R
}

// The group sums joined: S = sum_g v_g 2^(7 (8 - g)), |v_g| <= (g + 1) 2^20.  In pairs
// (below 2^31), then two exact halves hi 2^35 + lo (|hi| < 2^45, |lo| < 2^51) that
// become doubles by adding them to the bits of 1.5 2^52: four FP64 operations with the
// scaling in place of a dozen (64-bit conversions and ldexp made the joins, 13.8 k
// cycles of the FP64 pipe per 256 inputs, longer than the products of short tiles).
__device__ __forceinline__ double dg_join(const uint32_t (&v)[kDg]) {
  int x[kDg];
#pragma unroll
  for (int g = 0; g < kDg; ++g) x[g] = __float2int_rn(__uint_as_float(v[g]));
  const long long hi = (long long)(x[0] * 128 + x[1]) * 16384 + (x[2] * 128 + x[3]);
  const long long lo = ((long long)(x[4] * 128 + x[5]) * 16384 + (x[6] * 128 + x[7])) * 128 + x[8];
  constexpr double M = 6755399441055744.0;  // 1.5 2^52
  constexpr long long MB = 0x4338000000000000ll;
  return fma(__longlong_as_double(hi + MB) - M, 34359738368.0, __longlong_as_double(lo + MB) - M);
}

__global__ void __launch_bounds__(kDgThreads, 1) batch_sweep_digits_kernel(
    const DgItem* __restrict__ items, int nitems, int NT, int ny, const int32_t* __restrict__ port_off,
    const unsigned char* __restrict__ Td, const int* __restrict__ texp, const unsigned char* __restrict__ wd,
    const int* __restrict__ wexp, const double* __restrict__ T64, const int64_t* __restrict__ T_off,
    const int32_t* __restrict__ T_ld, const double* __restrict__ c, double* __restrict__ state, int64_t nports, int R,
    BatchCtrl* __restrict__ ctrl) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  __shared__ uint64_t full[kDgStages], empty[kDgStages], tfull[2], tempty[2], ufull[2], uempty[2], drain;
  __shared__ volatile int s_unit[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_k, s_flag;
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_flag = *((volatile int*)&ctrl->flag);
    s_k = *((volatile int*)&ctrl->k) - 1;  // the digits kernel has closed the sweep before
    s_abort = 0;
    for (int i = 0; i < kDgStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 8);
      mbar_init(&ufull[i], 1);
      mbar_init(&uempty[i], 9);
    }
    mbar_init(&drain, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (s_flag) return;
  const int k = s_k, total = nitems * ny;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(2 * kDgTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem, nc = 8 * NT;
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dsm + 1023) & ~(uintptr_t)1023);
  const uint32_t stage = dg_stage(NT), bbytes = dg_b_bytes(NT);
  // Every wait is bounded; one that runs out sets flag 5 (VTM_ETIMEOUT), and each role
  // goes on to its end without waiting, copying or issuing.
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (s_abort) return false;
    if (mbar_wait_bounded(bar, parity, kTcPolls)) return true;
    atomicCAS(&ctrl->flag, 0, 5);
    s_abort = 1;
    return false;
  };
  uint32_t issued = 0;
  if (warp == 0) {
    // units (an item and a column group, the largest first) from a counter: the SMs' shares
    // of the bandwidth differ, equal shares of the bytes leave the slowest 1.3 times the mean
    if (lane == 0) {
      uint32_t g = 0;
      int next = (int)atomicAdd(&ctrl->work, 1u);
      for (uint32_t u = 0;; ++u) {
        const int idx = next < total ? next : -1;
        if (u >= 2 && !wait(&uempty[u & 1], ((u >> 1) - 1) & 1)) break;
        s_unit[u & 1] = idx;
        mbar_arrive(&ufull[u & 1]);
        if (idx < 0) break;
        next = (int)atomicAdd(&ctrl->work, 1u);
        if (k == 1) continue;
        const DgItem it = items[idx / ny];
        const int y = idx % ny, p = port_off[it.tile + 1] - port_off[it.tile], nb = (p + 15) / 16;
        const uint32_t dig = dg_groups(p, it.m) * 256;  // bytes of a digit's rows
        const unsigned char* a = Td + it.off * 16 + (int64_t)it.m * nb * kDgABytes;
        const unsigned char* b = wd + ((int64_t)it.kb * ny + y) * bbytes;
        for (int kb = 0; kb < nb; ++kb, ++g) {
          const uint32_t st = g % kDgStages;
          if (g >= kDgStages && !wait(&empty[st], (g / kDgStages - 1) & 1)) break;
          if (s_abort) break;
          unsigned char* dst = base + st * stage;
          mbar_arrive_expect_tx(&full[st], kDg * dig + bbytes);
          issued = g + 1;
          if (dig == 4096) {
            bulk_copy_g2s(dst, a, kDgABytes, &full[st]);
          } else {
            for (int i = 0; i < kDg; ++i) bulk_copy_g2s(dst + i * 4096, a + i * dig, dig, &full[st]);
          }
          bulk_copy_g2s(dst + kDgABytes, b, bbytes, &full[st]);
          a += kDg * dig;
          b += (int64_t)ny * bbytes;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      uint32_t g = 0, ch = 0;
      for (uint32_t u = 0;; ++u) {
        if (!wait(&ufull[u & 1], (u >> 1) & 1)) break;
        const int idx = s_unit[u & 1];
        mbar_arrive(&uempty[u & 1]);
        if (idx < 0) break;
        if (k == 1) continue;
        const int tile = items[idx / ny].tile, nb = (port_off[tile + 1] - port_off[tile] + 15) / 16;
        for (int kb = 0; kb < nb; ++kb, ++g) {
          const uint32_t st = g % kDgStages, buf = ch & 1;
          const bool first = kb % kDgChunk == 0;
          if (first && ch >= 2 && !wait(&tempty[buf], ((ch >> 1) - 1) & 1)) break;
          if (!wait(&full[st], (g / kDgStages) & 1)) break;
          tc_fence_after();
          const uint32_t a0 = smem_u32(base + st * stage), b0 = a0 + kDgABytes, d0 = tmem + buf * kDgTmem;
          const uint64_t bd = dg_desc(b0);
#pragma unroll
          for (int i = 0; i < kDg; ++i)
            dg_mma(d0 + i * nc, dg_desc(a0 + i * 4096), bd, ((kDg - i) * nc + 15) & ~15u, (first && i == 0) ? 0u : 1u);
          tc_commit(&empty[st]);
          if (kb % kDgChunk == kDgChunk - 1 || kb == nb - 1) {
            tc_commit(&tfull[buf]);
            ++ch;
          }
        }
      }
    }
  } else {
    // eight warps: TMEM lanes 32 (warp % 4).., quads of columns h, h + 2, ...
    const int quarter = warp & 3, h = (warp - 2) >> 2, nq = 2 * NT;
    uint32_t ch = 0;
    double* cur = state + (size_t)(k & 1) * nports * 2 * R;
    for (uint32_t unit = 0;; ++unit) {
      if (!__all_sync(0xffffffffu, wait(&ufull[unit & 1], (unit >> 1) & 1))) break;  // (the warp together)
      const int idx = s_unit[unit & 1];
      __syncwarp();
      if (lane == 0) mbar_arrive(&uempty[unit & 1]);
      if (idx < 0) break;
      const DgItem it = items[idx / ny];
      const int c0 = (idx % ny) * (int)nc, p0 = port_off[it.tile], p = port_off[it.tile + 1] - p0, nb = (p + 15) / 16;
      const int s = 128 * it.m + 32 * quarter + lane;
      double out[kDgMaxNt][4];
#pragma unroll
      for (int u = 0; u < kDgMaxNt; ++u)
#pragma unroll
        for (int e = 0; e < 4; ++e) out[u][e] = 0.0;
      if (k > 1) {
        const int nch = (nb + kDgChunk - 1) / kDgChunk;
        const bool mine = lane < (int)nc && c0 + lane < R;
        int tmin = kDgNoBlock;  // the tile's smallest block in column c0 + lane
        for (int j = 0; j < nch; ++j) tmin = min(tmin, mine ? wexp[(it.chunk + j) * 64 + c0 + lane] >> 16 : kDgNoBlock);
        for (int j = 0; j < nch; ++j, ++ch) {
          const uint32_t buf = ch & 1;
          const int wp = mine ? wexp[(it.chunk + j) * 64 + c0 + lane] : 0;
          const int wx = (wp & 0xffff) - 1022;
          const uint32_t graded = __ballot_sync(0xffffffffu, mine && dg_graded(wp, tmin));  // by column
          if (!__all_sync(0xffffffffu, wait(&tfull[buf], (ch >> 1) & 1))) break;  // (the warp together)
          tc_fence_after();
#pragma unroll
          for (int u = 0; u < kDgMaxNt; ++u) {
            const int q = h + 2 * u;
            if (q >= nq) break;
            uint32_t v[kDg][4];
            dg_ld(tmem + ((uint32_t)(32 * quarter) << 16) + buf * kDgTmem + 4 * q, nc, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (c0 + 4 * q + e >= R) break;
              if (graded >> (4 * q + e) & 1) continue;
              const int we = __shfl_sync(0xffffffffu, wx, 4 * q + e);
              uint32_t x[kDg];
#pragma unroll
              for (int g = 0; g < kDg; ++g) x[g] = v[g][e];
              const double S = dg_join(x);
              if (we > -960 && we < 960) out[u][e] = fma(S, __longlong_as_double((long long)(we + 1023) << 52), out[u][e]);
              else out[u][e] += ldexp(S, we);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&tempty[buf]);
          if (graded) {  // these columns' 256 inputs in FP64, in the digits' scale
            const int ld = T_ld[it.tile], t0 = 16 * kDgChunk * j, nt = min(p - t0, 16 * kDgChunk), sr = min(s, p - 1);
            const double* Tr = T64 + T_off[it.tile] + (size_t)t0 * ld + sr;
            const int te = texp[p0 + sr] - 68;
#pragma unroll
            for (int u = 0; u < kDgMaxNt; ++u) {
              const int q = h + 2 * u;
              const uint32_t four = q < nq ? graded >> (4 * q) & 15u : 0u;
              if (!four) continue;
              double a[4] = {0.0, 0.0, 0.0, 0.0};
              const double* wr = cur + (size_t)(p0 + t0) * 2 * R + c0 + 4 * q;
              for (int t = 0; t < nt; t += 8) {
                double T[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) T[i] = t + i < nt ? __ldg(Tr + (size_t)(t + i) * ld) : 0.0;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (four >> e & 1) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                      if (t + i < nt) a[e] = fma(T[i], wr[(size_t)(t + i) * 2 * R + e], a[e]);
                  }
              }
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (four >> e & 1) out[u][e] += ldexp(a[e], -te);
            }
          }
        }
      }
      if (s < p && !s_abort) {
        const size_t ps = (size_t)(p0 + s);
        const int te = texp[ps] - 68;
#pragma unroll
        for (int u = 0; u < kDgMaxNt; ++u) {
          const int q = h + 2 * u;
          if (q >= nq) break;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int col = c0 + 4 * q + e;
            if (col < R) cur[ps * 2 * R + R + col] = c[ps * R + col] + ldexp(out[u][e], te);
          }
        }
      }
    }
  }
  __syncwarp();
  // after an abort: copies in flight land before the CTA's shared memory goes, and the
  // MMAs issued complete before its TMEM (both bounded)
  if (warp == 0 && lane == 0 && s_abort)
    for (uint32_t g = issued > kDgStages ? issued - kDgStages : 0; g < issued; ++g)
      mbar_wait_bounded(&full[g % kDgStages], (g / kDgStages) & 1, kTcPolls);
  if (warp == 1 && lane == 0 && s_abort) {
    tc_commit(&drain);
    mbar_wait_bounded(&drain, 0, kTcPolls);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kDgTmem) : "memory");
}
