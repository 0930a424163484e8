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
// Per sweep two launches.  batch_digits_kernel: the incident waves (twins' outgoing
// ones) and their digits in the B fragment order of mma.m16n8k16 (a CTA per 256
// ports), the residual of sweep k - 1 in FP64 (a CTA per 32 ports); its last CTA
// closes the sweep before, so a converged sweep never reads T_P.  batch_sweep_digits_kernel (a CTA
// per 128 outputs and up to 24 columns, 8 warps of 16 outputs): 45 MMAs per 16
// inputs and 8 columns, T_P's digits (fragment order, built once per
// factorisation, 18 bytes per entry) and W's through a three-stage cp.async ring.
// Bound: the rate of mma.sync (about 4 cycles per m16n8k16 and SM); its floor in HBM
// traffic (18 bytes of digits per entry) is a third of that at 24 columns.  Measured
// per sweep, thermal grid of 147,456 nodes in 110 boxes, 18 columns: FP64 CUDA
// cores 6.54 ms, here 0.08 + 0.43 ms (the same with 15 warps of 8 columns: 0.45).
// Errors of the iterates against quad precision are those of the FP64 kernel to two
// digits (1 to 20 sweeps; 3e-16 thermal, 8e-15 grids).

constexpr int kDg = 9;          // digits
constexpr int kDgChunk = 16;    // 16-input blocks between two joins of the group sums
constexpr int kDgStages = 3;
constexpr int kDgMaxNt = 3;     // 8-column groups per work item
constexpr int kDgBlocks = 8;    // 16-output blocks (warps) per work item

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

// T_P's digits: block (mb, kb) of a tile at (off + mb nb + kb) 9 32 uint4s, digit i
// at [i][lane] = the lane's A fragment (rows g, g + 8, columns 2t, 2t + 1, 2t + 8, 2t + 9)
__global__ void __launch_bounds__(256) pack_digits_kernel(const double* __restrict__ T,
                                                          const int64_t* __restrict__ T_off,
                                                          const int32_t* __restrict__ T_ld,
                                                          const int32_t* __restrict__ port_off,
                                                          const int64_t* __restrict__ dg_off,
                                                          const int* __restrict__ E, uint4* __restrict__ out) {
  const int t = blockIdx.x, p0 = port_off[t], p = port_off[t + 1] - p0, ld = T_ld[t];
  const int nb = (p + 15) / 16;
  const double* Tb = T + T_off[t];
  const int lane = threadIdx.x & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int b = blockIdx.y * 8 + (threadIdx.x >> 5); b < nb * nb; b += gridDim.y * 8) {
    const int mb = b / nb, kb = b - mb * nb;
    int d[8][kDg];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int s = 16 * mb + g + 8 * ((e >> 1) & 1), q = 16 * kb + t2 + (e & 1) + 8 * (e >> 2);
      const double v = s < p && q < p ? Tb[(size_t)q * ld + s] : 0.0;
      digits_of(v, s < p ? E[p0 + s] : 0, d[e]);
    }
    uint4* o = out + (dg_off[t] + b) * kDg * 32 + lane;
#pragma unroll
    for (int i = 0; i < kDg; ++i)
      o[i * 32] = make_uint4(bf16_pair(d[0][i], d[1][i]), bf16_pair(d[2][i], d[3][i]), bf16_pair(d[4][i], d[5][i]),
                             bf16_pair(d[6][i], d[7][i]));
  }
}

// Work item of the digits kernel: 256 ports of a tile (digits), or 32 (residual).
struct __align__(16) DgChunk {
  int32_t tile, m0, kb, pad;  // first port in the tile, first 16-input block of W's digits
};

__global__ void __launch_bounds__(256) batch_digits_kernel(
    const DgChunk* __restrict__ chunks, int nchunks, const int32_t* __restrict__ port_off,
    const int32_t* __restrict__ twin, const double2* __restrict__ kd, const uint8_t* __restrict__ run,
    double* __restrict__ state, int64_t nports,
    int R, int nt, uint2* __restrict__ wd, int* __restrict__ wexp, BatchCtrl* __restrict__ ctrl,
    double* __restrict__ partials, const double* __restrict__ tol2, double* __restrict__ hist, int hist_len) {
  __shared__ double rsq[32][64];
  __shared__ double red[64];
  __shared__ int cmax[64];
  __shared__ int s_k, s_flag;
  __shared__ bool s_last;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_k = *((volatile int*)&ctrl->k);
    s_flag = *((volatile int*)&ctrl->flag);
  }
  if (tid < 64) {
    red[tid] = 0.0;
    cmax[tid] = 0;
  }
  __syncthreads();
  if (s_flag) return;
  const int k = s_k;
  const DgChunk ch = chunks[blockIdx.x];
  const int p0 = port_off[ch.tile], p = port_off[ch.tile + 1] - p0;
  const double* prev = state + (size_t)((k - 1) & 1) * nports * 2 * R;
  if ((int)blockIdx.x >= nchunks) {
    // residual of sweep k - 1 at the nodes whose ports start in these 32
    const int ticket = blockIdx.x - nchunks, nres = gridDim.x - nchunks;
    if (k > 1) batch_residual<double, double>(twin, kd, run, prev, p0, ch.m0, min(p, ch.m0 + 32), R, rsq, red);
    for (int r = tid; r < R; r += 256) partials[(size_t)ticket * R + r] = k > 1 ? red[r] : 0.0;
    __syncthreads();
    batch_item_done(ctrl, ticket, nres, R, partials, &rsq[0][0]);
  } else {
    const int m1 = min(p, ch.m0 + 16 * kDgChunk);
    double* cur = state + (size_t)(k & 1) * nports * 2 * R;
    // this sweep's incident waves and the largest exponent of each column
    for (int i = tid; i < (m1 - ch.m0) * R; i += 256) {
      const int s = p0 + ch.m0 + i / R, r = i % R;
      const double w = k > 1 ? prev[(size_t)twin[s] * 2 * R + R + r] : 0.0;
      cur[(size_t)s * 2 * R + r] = w;
      if (w != 0.0) atomicMax(&cmax[r], exp_bits(w));
    }
    __syncthreads();
    if (tid < 64) wexp[blockIdx.x * 64 + tid] = cmax[tid] - 1022;
    // digits, a pair of rows per item: (16-input block, column group, lane, half)
    const int kbn = k > 1 ? (m1 - ch.m0 + 15) / 16 : 0;
    uint32_t* out = reinterpret_cast<uint32_t*>(wd);
    for (int i = tid; i < kbn * nt * 64; i += 256) {
      const int h = i & 1, lane = (i >> 1) & 31, u = i >> 6, n = u % nt, kb = u / nt;
      const int c = 8 * n + (lane >> 2), q = ch.m0 + 16 * kb + 2 * (lane & 3) + 8 * h;
      int d0[kDg], d1[kDg];
      const bool col = c < R;
      const double v0 = col && q < p ? prev[(size_t)twin[p0 + q] * 2 * R + R + c] : 0.0;
      const double v1 = col && q + 1 < p ? prev[(size_t)twin[p0 + q + 1] * 2 * R + R + c] : 0.0;
      const int E = col ? cmax[c] - 1022 : 0;
      digits_of(v0, E, d0);
      digits_of(v1, E, d1);
      uint32_t* o = out + ((size_t)(ch.kb + kb) * nt + n) * kDg * 64 + lane * 2 + h;
#pragma unroll
      for (int j = 0; j < kDg; ++j) o[j * 64] = bf16_pair(d0[j], d1[j]);
    }
  }
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(&ctrl->counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  batch_finish(ctrl, partials, gridDim.x - nchunks, R, tol2, hist, hist_len, k, &rsq[0][0]);
}

// Work item of the sweep: up to kDgBlocks 16-output blocks of a tile.
struct __align__(16) DgItem {
  int32_t tile, mb0, kb, chunk;  // first 16-output block; W's first block and first chunk of the tile
  int64_t off;                   // block (0, 0) of the tile's digits
  int64_t pad;
};

template <int NT>
__global__ void __launch_bounds__(32 * kDgBlocks, 1) batch_sweep_digits_kernel(
    const DgItem* __restrict__ items, const int32_t* __restrict__ port_off, const uint4* __restrict__ Td,
    const int* __restrict__ texp, const uint2* __restrict__ wd, const int* __restrict__ wexp, int nt_all, int ny,
    const double* __restrict__ c, double* __restrict__ state, int64_t nports, int R,
    const BatchCtrl* __restrict__ ctrl) {
  extern __shared__ __align__(16) unsigned char dsm[];
  const int flag = *((volatile const int*)&ctrl->flag);
  if (flag) return;
  const int k = *((volatile const int*)&ctrl->k) - 1;  // the digits kernel has closed the sweep before
  // the column groups of an item run side by side (its T_P digits from HBM once)
  const DgItem it = items[blockIdx.x / ny];
  const int n0 = (blockIdx.x % ny) * NT;  // first 8-column group
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int p0 = port_off[it.tile], p = port_off[it.tile + 1] - p0, nb = (p + 15) / 16;
  const int mb = it.mb0 + warp;
  const bool active = mb < nb;
  constexpr int kA = kDg * 32;       // uint4s of one warp's T_P digits per stage
  constexpr int kB = NT * kDg * 32;  // uint2s of the W digits per stage
  constexpr size_t kStage = kDgBlocks * kA * sizeof(uint4) + kB * sizeof(uint2);
  const int nn = min(NT, nt_all - n0);  // column groups this item has
  auto issue = [&](int kb) {
    if (kb < nb) {
      unsigned char* st = dsm + (kb % kDgStages) * kStage;
      if (active) {
        const uint4* src = Td + (it.off + (int64_t)mb * nb + kb) * kA + lane;
        uint4* dst = reinterpret_cast<uint4*>(st) + warp * kA + lane;
#pragma unroll
        for (int i = 0; i < kDg; ++i) cp_async16_cg(dst + i * 32, src + i * 32);
      }
      const uint4* bsrc = reinterpret_cast<const uint4*>(wd + ((int64_t)(it.kb + kb) * nt_all + n0) * kDg * 32);
      uint4* bdst = reinterpret_cast<uint4*>(st) + kDgBlocks * kA;
      for (int e = tid; e < nn * kDg * 16; e += 32 * kDgBlocks) cp_async16_cg(bdst + e, bsrc + e);
    }
    cp_async_commit();
  };
  float acc[NT][kDg][4];
  double out[NT][4];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      out[n][e] = 0.0;
#pragma unroll
      for (int g = 0; g < kDg; ++g) acc[n][g][e] = 0.f;
    }
  const int g8 = lane >> 2, t2 = 2 * (lane & 3);
  // the group sums of a chunk joined: S = sum_g acc_g 2^(7 (8 - g)), exact in two
  // 64-bit halves, scaled by the chunk's column exponents
  auto join = [&](int chunk) {
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      if (n >= nn) break;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        long long hi = 0, lo = 0;
#pragma unroll
        for (int g = 0; g < 4; ++g) hi = hi * 128 + __float2int_rn(acc[n][g][e]);
#pragma unroll
        for (int g = 4; g < kDg; ++g) lo = lo * 128 + __float2int_rn(acc[n][g][e]);
        const double S = fma((double)hi, 34359738368.0, (double)lo);  // hi 2^35 + lo
        out[n][e] += ldexp(S, wexp[chunk * 64 + 8 * (n0 + n) + t2 + (e & 1)]);
#pragma unroll
        for (int g = 0; g < kDg; ++g) acc[n][g][e] = 0.f;
      }
    }
  };
  if (k > 1) {
#pragma unroll
    for (int b = 0; b < kDgStages - 1; ++b) issue(b);
    for (int kb = 0; kb < nb; ++kb) {
      cp_async_wait<kDgStages - 2>();
      __syncthreads();  // the stage has landed; the one refilled below is read
      issue(kb + kDgStages - 1);
      if (active) {
        const unsigned char* st = dsm + (kb % kDgStages) * kStage;
        const uint4* As = reinterpret_cast<const uint4*>(st) + warp * kA + lane;
        const uint2* Bs = reinterpret_cast<const uint2*>(st + kDgBlocks * kA * sizeof(uint4)) + lane;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if (n < nn) {
            uint2 b[kDg];
#pragma unroll
            for (int j = 0; j < kDg; ++j) b[j] = Bs[(n * kDg + j) * 32];
#pragma unroll
            for (int i = 0; i < kDg; ++i) {
              const uint4 a = As[i * 32];
#pragma unroll
              for (int j = 0; i + j < kDg; ++j) mma_bf16(acc[n][i + j], a.x, a.y, a.z, a.w, b[j].x, b[j].y);
            }
          }
        }
        if (kb % kDgChunk == kDgChunk - 1 || kb == nb - 1) join(it.chunk + kb / kDgChunk);
      }
    }
    cp_async_wait<0>();
  }
  if (!active) return;
  double* cur = state + (size_t)(k & 1) * nports * 2 * R;
#pragma unroll
  for (int n = 0; n < NT; ++n) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int s = 16 * mb + g8 + 8 * (e >> 1), r = 8 * (n0 + n) + t2 + (e & 1);
      if (s < p && r < R) {
        const size_t ps = (size_t)(p0 + s);
        cur[ps * 2 * R + R + r] = c[ps * R + r] + ldexp(out[n][e], texp[ps] - 68);
      }
    }
  }
}
