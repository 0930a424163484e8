// Values on the device: checks of a new set of values, line coefficients, the
// band of K_P.
//
// Everything here follows from A's values by elementwise work over the
// nonzeros, the cut pairs or the ports, so vtm_set_values and vtm_factor run it
// where the values are: the host assembled the band twice per refactorisation
// and sent it over the link (1024^2 grid in 256 tiles: set_values + factor spent
// about 100 of 200 ms there; 512^2: 17 of 28 ms).  The host keeps a copy of the
// values and of the port coefficients only for what asks for them
// (ensure_host_vals, ensure_host_ports).  Bound by HBM: the values and columns
// once (12 bytes per nonzero) and the band written once.
#include <algorithm>
#include <cmath>

#include "vtm_internal.h"

namespace vtm {

static int grid_of(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16)); }

// bad |= 1: a value is not finite; |= 2: A(i, j) != A(j, i)
__global__ void __launch_bounds__(256) check_values_kernel(const int64_t* __restrict__ rowptr,
                                                           const int32_t* __restrict__ col,
                                                           const double* __restrict__ vals, int64_t n,
                                                           int symmetric, int* __restrict__ bad) {
  int b = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    for (int64_t q = rowptr[i]; q < rowptr[i + 1]; ++q) {
      const double v = vals[q];
      if (!isfinite(v)) b |= 1;
      const int32_t j = col[q];
      if (symmetric && j > i) {
        int64_t lo = rowptr[j], hi = rowptr[j + 1];  // columns ascend within a row
        while (lo < hi) {
          const int64_t mid = (lo + hi) >> 1;
          if (col[mid] < i) lo = mid + 1;
          else hi = mid;
        }
        if (lo >= rowptr[j + 1] || col[lo] != i || vals[lo] != v) b |= 2;
      }
    }
  if (b) atomicOr(bad, b);
}

// bad |= 4: a cut pair gained or lost its line, or a lagged coupling appeared
// (flags: 1 the pair carries a line, 2 / 4 its first / second entry is lagged)
__global__ void check_cuts_kernel(const int64_t* __restrict__ p1, const int64_t* __restrict__ p2,
                                  const uint8_t* __restrict__ flags, int64_t ncut,
                                  const double* __restrict__ vals, int lines, int* __restrict__ bad) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ncut; e += (int64_t)gridDim.x * blockDim.x) {
    const double a1 = p1[e] >= 0 ? vals[p1[e]] : 0.0, a2 = p2[e] >= 0 ? vals[p2[e]] : 0.0;
    const double g = -(a1 + a2) / 2.0;
    const bool wire = lines && g > 0;
    const double r1 = wire ? a1 + g : a1, r2 = wire ? a2 + g : a2;
    const int f = flags[e];
    if (wire != (bool)(f & 1) || (r1 != 0.0 && !(f & 2)) || (r2 != 0.0 && !(f & 4))) atomicOr(bad, 4);
  }
}

// Per port: conductance, line admittance (kind 0: one W; 1, 2: alpha 2 g; 3:
// given) and the coefficients the kernels use (see vtm_internal.h).  Waves are
// carried as w / d with d = 1 for one W on every line, else sqrt(W_s) (power
// waves), which keeps the condensed operator symmetric for a symmetric A.
// bad[0] |= 8: a conductance is not positive; bad[1]: first port with a bad W.
__global__ void port_coefs_kernel(const int64_t* __restrict__ pij, const int64_t* __restrict__ pji,
                                  const double* __restrict__ vals, int64_t npt, int kind, double alpha,
                                  double* __restrict__ pg, double* __restrict__ pW, double* __restrict__ pd,
                                  double* __restrict__ bin, double* __restrict__ bout, float* __restrict__ bin32,
                                  float* __restrict__ bout32, double* __restrict__ rho, double2* __restrict__ kd,
                                  float2* __restrict__ kd32, float4* __restrict__ kddf, int* __restrict__ bad) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < npt; s += (int64_t)gridDim.x * blockDim.x) {
    const double a1 = pij[s] >= 0 ? vals[pij[s]] : 0.0, a2 = pji[s] >= 0 ? vals[pji[s]] : 0.0;
    const double g = -(a1 + a2) / 2.0;
    if (!(g > 0)) atomicOr(bad, 8);
    const double W = kind == 3 ? pW[s] : (kind == 0 ? alpha : alpha * 2.0 * g);
    if (!(W > 0) || !isfinite(W)) atomicMin(bad + 1, (int)s);
    const double d = kind == 0 ? 1.0 : sqrt(W);
    const double beta = 2 * g / (2 * g + W);
    pg[s] = g;
    pW[s] = W;
    pd[s] = d;
    const double bi = beta * d, bo = 2.0 * W * beta / d;
    bin[s] = bi;
    bout[s] = bo;
    bin32[s] = (float)bi;
    bout32[s] = (float)bo;
    rho[s] = (W - 2.0 * g) / (W + 2.0 * g);
    const double x = g / W;
    kd[s] = make_double2(x, d);
    const float xh = (float)x, dh = (float)d;
    kd32[s] = make_float2(xh, dh);
    kddf[s] = make_float4(xh, (float)(x - (double)xh), dh, (float)(d - (double)dh));
  }
}

// channel form: the remainder of each lagged entry after the branch part
__global__ void lag_rho_kernel(const int64_t* __restrict__ pos, const int64_t* __restrict__ back,
                               const double* __restrict__ vals, int64_t nl, int lines, double* __restrict__ rho) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nl; q += (int64_t)gridDim.x * blockDim.x) {
    const double a = pos[q] >= 0 ? vals[pos[q]] : 0.0, b = back[q] >= 0 ? vals[back[q]] : 0.0;
    const double g = -(a + b) / 2.0;
    rho[q] = lines && g > 0 ? a + g : a;
  }
}

// channel form, per input: residual coefficients (g/W and d of a port, rho of a
// lagged entry) and right-hand-side weight (beta d or -rho); per output: scale
// (2 W beta / d or 1) and the diagonal reflection term of a port
__global__ void channel_coefs_kernel(const int32_t* __restrict__ in_item, const uint8_t* __restrict__ in_kind,
                                     int64_t n_in, const int32_t* __restrict__ out_item, int64_t n_out,
                                     const double2* __restrict__ kd, const double* __restrict__ bin,
                                     const double* __restrict__ bout, const double* __restrict__ rho,
                                     const double* __restrict__ lag, double* __restrict__ coef,
                                     double* __restrict__ dsc, double* __restrict__ sigma,
                                     double* __restrict__ scale, double* __restrict__ diag) {
  const int64_t step = (int64_t)gridDim.x * blockDim.x, id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (int64_t a = id; a < n_in; a += step) {
    const int32_t it = in_item[a];
    if (in_kind[a] == 0) {
      coef[a] = kd[it].x;
      dsc[a] = kd[it].y;
      sigma[a] = bin[it];
    } else {
      coef[a] = lag[it];
      dsc[a] = 0.0;
      sigma[a] = -lag[it];
    }
  }
  for (int64_t o = id; o < n_out; o += step) {
    const int32_t it = out_item[o];
    scale[o] = it >= 0 ? bout[it] : 1.0;
    diag[o] = it >= 0 ? rho[it] : 0.0;
  }
}

// The band of K_P, a CTA per tile: A_PP (lower part into Lc, the upper into Uc
// for LU), then g - 4 g^2/(2 g + W) of every torn branch onto its node's
// diagonal, the ports of a node in order.
__global__ void __launch_bounds__(256) assemble_band_kernel(
    const int32_t* __restrict__ node_off, const int32_t* __restrict__ bwv, const int64_t* __restrict__ band_off,
    const int32_t* __restrict__ perm, const int32_t* __restrict__ iperm, const int64_t* __restrict__ rowptr,
    const int32_t* __restrict__ col, const double* __restrict__ vals, const int32_t* __restrict__ port_off,
    const int32_t* __restrict__ port_loc, const uint8_t* __restrict__ run, const double* __restrict__ pg,
    const double* __restrict__ pW, double* __restrict__ Lc, double* __restrict__ Uc) {
  const int t = blockIdx.x;
  const int off = node_off[t], cnt = node_off[t + 1] - off, B = bwv[t] + 1;
  double* lc = Lc + band_off[t];
  double* uc = Uc ? Uc + band_off[t] : nullptr;
  for (int l = threadIdx.x; l < cnt; l += blockDim.x) {
    const int32_t i = perm[off + l];
    for (int64_t q = rowptr[i]; q < rowptr[i + 1]; ++q) {
      const int m = iperm[col[q]] - off;
      if (m < 0 || m >= cnt) continue;  // another tile's node
      if (m <= l) lc[(int64_t)m * B + (l - m)] = vals[q];
      else if (uc) uc[(int64_t)m * B + (m - l)] = vals[q];
    }
  }
  __syncthreads();
  for (int s = port_off[t] + threadIdx.x; s < port_off[t + 1]; s += blockDim.x) {
    const int nr = run[s];
    if (!nr) continue;
    double* d = lc + (int64_t)port_loc[s] * B;
    double v = *d;
    for (int q = s; q < s + nr; ++q) {
      const double g = pg[q], W = pW[q];
      v += g - 4 * g * g / (2 * g + W);
    }
    *d = v;
  }
}

// New values against the plan: what vtm_set_values refuses.
vtm_status check_values(vtm_plan_s* P, const double* d_vals) {
  cudaStream_t s = P->stream;
  int* bad = P->d_err.as<int>();
  VTM_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), s));
  check_values_kernel<<<grid_of(P->n), 256, 0, s>>>(P->d_rowptr.as<int64_t>(), P->d_colidx.as<int32_t>(), d_vals,
                                                    P->n, P->symmetric ? 1 : 0, bad);
  const int64_t ncut = (int64_t)P->cut_p1.size();
  if (ncut > 0) {
    if (!P->d_cut_flags.p) {
      VTM_TRY(upload(P->d_cut_p1, P->cut_p1, s));
      VTM_TRY(upload(P->d_cut_p2, P->cut_p2, s));
      VTM_TRY(upload(P->d_cut_flags, P->cut_flags, s));
    }
    check_cuts_kernel<<<grid_of(ncut), 256, 0, s>>>(P->d_cut_p1.as<int64_t>(), P->d_cut_p2.as<int64_t>(),
                                                    P->d_cut_flags.as<uint8_t>(), ncut, d_vals,
                                                    P->method == VTM_METHOD_VTM ? 1 : 0, bad);
  }
  VTM_CUDA_TRY(cudaGetLastError());
  int h = 0;
  VTM_CUDA_TRY(cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  VTM_CUDA_TRY(cudaStreamSynchronize(s));
  if (h & 1) set_detail("vtm_set_values: non-finite value");
  else if (h & 2) set_detail("vtm_set_values: the plan was made for a symmetric matrix");
  else if (h & 4) set_detail("vtm_set_values: the set of torn lines or lagged couplings changed");
  return h ? VTM_EINVAL : VTM_OK;
}

// Port (and channel) coefficients of the plan's values and admittance choice.
vtm_status assemble_ports(vtm_plan_s* P) {
  cudaStream_t s = P->stream;
  const int64_t npt = (int64_t)P->port_node.size();
  const size_t np1 = (size_t)std::max<int64_t>(npt, 1);
  P->host_ports = false;
  if (!P->d_ppij.p) {
    VTM_TRY(upload(P->d_ppij, P->port_pos_ij, s));
    VTM_TRY(upload(P->d_ppji, P->port_pos_ji, s));
    for (vtm::DevBuf* b : {&P->d_port_g, &P->d_port_W, &P->d_port_d, &P->d_beta, &P->d_bout, &P->d_rho})
      VTM_TRY(dev_alloc(*b, np1 * sizeof(double)));
    VTM_TRY(dev_alloc(P->d_kd, np1 * sizeof(double2)));
    VTM_TRY(dev_alloc(P->d_kddf, np1 * sizeof(float4)));
    VTM_TRY(dev_alloc(P->d_kd32, np1 * sizeof(float2)));
    VTM_TRY(dev_alloc(P->d_beta32, np1 * sizeof(float)));
    VTM_TRY(dev_alloc(P->d_bout32, np1 * sizeof(float)));
  }
  int kind = 3;
  double alpha = 1.0;
  if (P->w_kind == VTM_W_ALPHA) {
    kind = 0;
    alpha = P->W;
  } else if (P->w_kind == VTM_W_DIAG) {
    kind = 1;
  } else if (P->w_kind == VTM_W_WOB) {
    kind = 2;
    alpha = P->w_alpha;
  } else {  // partial Schur complements or the caller's own: from the host
    std::vector<double> W;
    VTM_TRY(host_admittance(P, W));
    VTM_TRY(upload(P->d_port_W, W, s));
    VTM_CUDA_TRY(cudaStreamSynchronize(s));
  }
  int* bad = P->d_err.as<int>();
  const int init[2] = {0, INT32_MAX};
  VTM_CUDA_TRY(cudaMemcpyAsync(bad, init, sizeof(init), cudaMemcpyHostToDevice, s));
  if (npt > 0)
    port_coefs_kernel<<<grid_of(npt), 256, 0, s>>>(
        P->d_ppij.as<int64_t>(), P->d_ppji.as<int64_t>(), P->d_vals.as<double>(), npt, kind, alpha,
        P->d_port_g.as<double>(), P->d_port_W.as<double>(), P->d_port_d.as<double>(), P->d_beta.as<double>(),
        P->d_bout.as<double>(), P->d_beta32.as<float>(), P->d_bout32.as<float>(), P->d_rho.as<double>(),
        P->d_kd.as<double2>(), P->d_kd32.as<float2>(), P->d_kddf.as<float4>(), bad);
  if (P->general) {
    const int64_t nl = (int64_t)P->lag_i.size();
    if (!P->d_in_item.p) {
      VTM_TRY(upload(P->d_lag_pos, P->lag_pos, s));
      VTM_TRY(upload(P->d_lag_back, P->lag_back, s));
      VTM_TRY(dev_alloc(P->d_lag_rho, std::max<int64_t>(nl, 1) * sizeof(double)));
      VTM_TRY(upload(P->d_in_item, P->in_item, s));
      VTM_TRY(upload(P->d_out_item, P->out_item, s));
      const size_t ni = std::max<int64_t>(P->n_in, 1) * sizeof(double), no = std::max<int64_t>(P->n_out, 1) * sizeof(double);
      VTM_TRY(dev_alloc(P->d_in_coef, ni));
      VTM_TRY(dev_alloc(P->d_in_d, ni));
      VTM_TRY(dev_alloc(P->d_in_sigma, ni));
      VTM_TRY(dev_alloc(P->d_out_scale, no));
      VTM_TRY(dev_alloc(P->d_out_diag, no));
    }
    if (nl > 0)
      lag_rho_kernel<<<grid_of(nl), 256, 0, s>>>(P->d_lag_pos.as<int64_t>(), P->d_lag_back.as<int64_t>(),
                                                 P->d_vals.as<double>(), nl, P->method == VTM_METHOD_VTM ? 1 : 0,
                                                 P->d_lag_rho.as<double>());
    channel_coefs_kernel<<<grid_of(P->n_in + P->n_out), 256, 0, s>>>(
        P->d_in_item.as<int32_t>(), P->d_in_kind.as<uint8_t>(), P->n_in, P->d_out_item.as<int32_t>(), P->n_out,
        P->d_kd.as<double2>(), P->d_beta.as<double>(), P->d_bout.as<double>(), P->d_rho.as<double>(),
        P->d_lag_rho.as<double>(), P->d_in_coef.as<double>(), P->d_in_d.as<double>(), P->d_in_sigma.as<double>(),
        P->d_out_scale.as<double>(), P->d_out_diag.as<double>());
  }
  VTM_CUDA_TRY(cudaGetLastError());
  int h[2];
  VTM_CUDA_TRY(cudaMemcpyAsync(h, bad, sizeof(h), cudaMemcpyDeviceToHost, s));
  VTM_CUDA_TRY(cudaStreamSynchronize(s));
  if (h[0]) {
    set_detail("vtm_set_values: a torn branch lost its positive conductance");
    return VTM_EINVAL;
  }
  if (h[1] != INT32_MAX) {
    set_detail("line admittance not positive at port " + std::to_string(h[1]));
    return VTM_EINVAL;
  }
  return VTM_OK;
}

vtm_status assemble_band(vtm_plan_s* P) {
  cudaStream_t s = P->stream;
  const size_t bytes = P->band_elems * sizeof(double);
  VTM_CUDA_TRY(cudaMemsetAsync(P->d_Lc.p, 0, bytes, s));
  if (!P->symmetric) VTM_CUDA_TRY(cudaMemsetAsync(P->d_Uc.p, 0, bytes, s));
  if (!P->d_iperm.p) VTM_TRY(upload(P->d_iperm, P->iperm, s));
  assemble_band_kernel<<<P->nparts, 256, 0, s>>>(
      P->tabs.node_off.as<int32_t>(), P->tabs.bw.as<int32_t>(), P->tabs.band_off.as<int64_t>(),
      P->d_perm.as<int32_t>(), P->d_iperm.as<int32_t>(), P->d_rowptr.as<int64_t>(), P->d_colidx.as<int32_t>(),
      P->d_vals.as<double>(), P->tabs.port_off.as<int32_t>(), P->d_port_loc.as<int32_t>(), P->d_run.as<uint8_t>(),
      P->d_port_g.as<double>(), P->d_port_W.as<double>(), P->d_Lc.as<double>(),
      P->symmetric ? nullptr : P->d_Uc.as<double>());
  VTM_CUDA_TRY(cudaGetLastError());
  return VTM_OK;
}

template <class T>
static vtm_status download(std::vector<T>& h, const DevBuf& b, size_t count, cudaStream_t s) {
  h.resize(count);
  if (count) VTM_CUDA_TRY(cudaMemcpyAsync(h.data(), b.p, count * sizeof(T), cudaMemcpyDeviceToHost, s));
  return VTM_OK;
}

// h_vals follows the device's values
vtm_status ensure_host_vals(vtm_plan_s* P) {
  if (P->host_vals) return VTM_OK;
  VTM_TRY(download(P->h_vals, P->d_vals, (size_t)P->nnz, P->stream));
  VTM_CUDA_TRY(cudaStreamSynchronize(P->stream));
  P->host_vals = true;
  return VTM_OK;
}

// port_g, port_W and port_d follow the device's
vtm_status ensure_host_ports(vtm_plan_s* P) {
  if (P->host_ports) return VTM_OK;
  const size_t npt = P->port_node.size();
  VTM_TRY(download(P->port_g, P->d_port_g, npt, P->stream));
  VTM_TRY(download(P->port_W, P->d_port_W, npt, P->stream));
  VTM_TRY(download(P->port_d, P->d_port_d, npt, P->stream));
  VTM_CUDA_TRY(cudaStreamSynchronize(P->stream));
  P->host_ports = true;
  return VTM_OK;
}

}  // namespace vtm
