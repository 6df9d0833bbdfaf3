// Device assembly of the stiffness matrices A_k of every input PCE term
// (Sec. 2.1, Eqs. inputlogn and Galerkin_L_exp) on the shared 5-point
// pattern, stored slot-major (ELL) for the operator apply.
//
// c_bar_k(e) = c_0(e) prod_i g_i(e)^{alpha_ki} / sqrt(alpha_ki!),
// c_0(e) = exp(g0 + 1/2 sum_i g_i(e)^2)       (lognormal input PCE)
// A_k[r][c] = sum_{triangles e containing edge rc} c_bar_k(e) K_e[r][c]
// with the unit P1 element matrices of the two right triangles of a cell.
#include <algorithm>
#include <cmath>

#include "sg_internal.h"
#include "sg_stencil.h"

namespace sg {

sg_status DevBuf::alloc(size_t nbytes) {
  free_();
  if (nbytes == 0) nbytes = 16;
  cudaError_t e = cudaMalloc(&ptr, nbytes);
  if (e != cudaSuccess) {
    ptr = nullptr;
    set_error(std::string("cudaMalloc: ") + cudaGetErrorString(e));
    return SG_ERR_NOMEM;
  }
  bytes = nbytes;
  cudaMemset(ptr, 0, nbytes);
  return SG_OK;
}

void DevBuf::free_() {
  if (ptr) cudaFree(ptr);
  ptr = nullptr;
  bytes = 0;
}

namespace {

// c_bar for input terms [k0, k0 + kn) on every triangle: out[(k - k0) * E + e]
__global__ void k_cbar(const double* __restrict__ gfield, const int* __restrict__ mi_in,
                       const double* __restrict__ inv_sqrt_fact, int L, int64_t E, double g0,
                       int k0, int kn, double* __restrict__ out) {
  int64_t total = int64_t(kn) * E;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < total;
       t += int64_t(gridDim.x) * blockDim.x) {
    int kl = int(t / E);
    int64_t e = t - int64_t(kl) * E;
    int k = k0 + kl;
    double s2 = 0.0, prod = 1.0;
    for (int i = 0; i < L; ++i) {
      double gi = gfield[int64_t(i) * E + e];
      s2 += gi * gi;
      int d = mi_in[k * L + i];
      for (int j = 0; j < d; ++j) prod *= gi;
    }
    out[t] = exp(g0 + 0.5 * s2) * prod * inv_sqrt_fact[k];
  }
}

// Five-slot ELL values for input terms [k0, k0 + kn).  Slot order (ascending
// column): south, west, centre, east, north.  Thread per (row, term).
__global__ void k_fine_ell(const double* __restrict__ cb, int N, int64_t n, int64_t ldr, int k0,
                           int kn, double* __restrict__ v64) {
  const int m = N - 1;
  const int64_t E = 2LL * N * N;
  int64_t total = int64_t(kn) * n;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < total;
       t += int64_t(gridDim.x) * blockDim.x) {
    int kl = int(t / n);
    int64_t r = t - int64_t(kl) * n;
    int i = int(r % m) + 1, j = int(r / m) + 1;
    const double* c = cb + int64_t(kl) * E;
    double v[5];
    p1_stencil<double>(c, N, i, j, v);
    int k = k0 + kl;
    for (int s = 0; s < 5; ++s) {
      int64_t idx = (int64_t(k) * 5 + s) * ldr + r;
      v64[idx] = v[s];
    }
  }
}

// conductance of edge e of a mesh of N x N cells with the coefficient field
// c over its triangles: the horizontal edge (i,j)-(i+1,j) (i = 0..N-1, j =
// 1..N-1) at (j-1) N + i, half the sum of the lower triangle of cell (i,j)
// and the upper one of cell (i,j-1); the vertical edge (i,j)-(i,j+1) (i =
// 1..N-1, j = 0..N-1) at N (N-1) + j (N-1) + i - 1, half the sum of the
// upper triangle of cell (i,j) and the lower one of cell (i-1,j).  A row of
// A(c) is then the sum over its four edges of w (x_r - x_neighbour) (the
// rows of the P1 element matrices sum to zero).
template <typename T>
__device__ __forceinline__ T edge_conductance(const T* c, int N, int64_t e) {
  const int m = N - 1;
  auto lo = [&](int ci, int cj) { return c[2LL * (int64_t(cj) * N + ci)]; };
  auto up = [&](int ci, int cj) { return c[2LL * (int64_t(cj) * N + ci) + 1]; };
  if (e < int64_t(N) * m) {
    const int i = int(e % N), j = int(e / N) + 1;
    return T(0.5) * (lo(i, j) + up(i, j - 1));
  }
  const int64_t e2 = e - int64_t(N) * m;
  const int i = int(e2 % m) + 1, j = int(e2 / m);
  return T(0.5) * (up(i, j) + lo(i - 1, j));
}

// FP64 conductances of input terms [k0, k0 + kn), w[k * vkst + e]; thread
// per (term, edge)
__global__ void k_flux_values64(const double* __restrict__ cb, int N, int64_t vkst, int k0, int kn,
                                double* __restrict__ w) {
  const int64_t E = 2LL * N * N, ne = 2LL * N * (N - 1), total = int64_t(kn) * ne;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < total;
       t += int64_t(gridDim.x) * blockDim.x) {
    const int kl = int(t / ne);
    const int64_t e = t - int64_t(kl) * ne;
    w[int64_t(k0 + kl) * vkst + e] = edge_conductance(cb + int64_t(kl) * E, N, e);
  }
}

// conductances of input terms [k0, k0 + kn) into the edge form's blocks
// (EdgeVals), every position of the term; lanes without an edge get zero
template <typename Tc>
__global__ void k_edge_values(const Tc* __restrict__ cb, int N, int KT, const int* __restrict__ off,
                              const int* __restrict__ pos, const double* __restrict__ scale, int k0, int kn,
                              float* __restrict__ v32, double* __restrict__ v64) {
  const int m = N - 1, ntile = (N + 30) / 31;
  const int64_t E = 2LL * N * N, per = int64_t(N) * ntile * 64, total = int64_t(kn) * per;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < total;
       t += int64_t(gridDim.x) * blockDim.x) {
    const int kl = int(t / per);
    const int64_t q = t - int64_t(kl) * per;  // ((j ntile + tile) 2 + vertical) 32 + lane
    const int lane = int(q & 31), ver = int(q >> 5) & 1;
    const int64_t b = q >> 6;
    const int tile = int(b % ntile), j = int(b / ntile), e = 31 * tile + lane;
    int64_t edge = -1;
    if (ver) {
      if (lane < 31 && e + 1 <= m) edge = int64_t(N) * m + int64_t(j) * m + e;
    } else if (j >= 1 && e < N) {
      edge = int64_t(j - 1) * N + e;
    }
    const double w = edge >= 0 ? scale[k0 + kl] * double(edge_conductance(cb + int64_t(kl) * E, N, edge)) : 0.0;
    for (int u = off[k0 + kl]; u < off[k0 + kl + 1]; ++u) {
      const int64_t at = (((q >> 5) * (KT / 4) + pos[u] / 4) * 32 + lane) * 4 + pos[u] % 4;
      if (v32) v32[at] = float(w);
      if (v64) v64[at] = w;
    }
  }
}

// All terms at once: CTA per (node row, tile, direction), warp per four
// consecutive positions, which a lane writes as one 16- or 32-byte piece (a
// thread per term writes single words 16 bytes apart: 80 us at 128^2, K = 210
// for 55 MB in and out)
// FP32 coefficients: scale = hi + lo in FP32 (the conversions and products of
// FP64 run at 1/64 of the FP32 rate: 65 us; now 21).
template <typename Tc>
__global__ void __launch_bounds__(256) k_edge_values_all(const Tc* __restrict__ cb, int N, int KT,
                                                         const int* __restrict__ term,
                                                         const double* __restrict__ scale,
                                                         const float2* __restrict__ scale2, float* __restrict__ v32,
                                                         double* __restrict__ v64) {
  const int m = N - 1, ntile = (N + 30) / 31, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t E = 2LL * N * N, q = blockIdx.x;
  const int ver = int(q & 1), tile = int((q >> 1) % ntile), j = int((q >> 1) / ntile), e = 31 * tile + lane;
  // the edge's two triangles (edge_conductance), or none
  int64_t t0 = -1, t1 = -1;
  if (ver) {
    if (lane < 31 && e + 1 <= m) {
      t0 = 2 * (int64_t(j) * N + e + 1) + 1;
      t1 = 2 * (int64_t(j) * N + e);
    }
  } else if (j >= 1 && e < N) {
    t0 = 2 * (int64_t(j) * N + e);
    t1 = 2 * (int64_t(j - 1) * N + e) + 1;
  }
#pragma unroll 2
  for (int g = threadIdx.x >> 5; g < KT / 4; g += nw) {
    const int4 k4 = reinterpret_cast<const int4*>(term)[g];
    const int k[4] = {k4.x, k4.y, k4.z, k4.w};
    Tc w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      w[u] = k[u] >= 0 && t0 >= 0 ? Tc(0.5) * (cb[k[u] * E + t0] + cb[k[u] * E + t1]) : Tc(0);
    const int64_t at = (q * (KT / 4) + g) * 32 + lane;
    if constexpr (sizeof(Tc) == 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2 s = scale2[k[u] >= 0 ? k[u] : 0];
        w[u] = fmaf(w[u], s.x, w[u] * s.y);
      }
      if (v32) reinterpret_cast<float4*>(v32)[at] = make_float4(w[0], w[1], w[2], w[3]);
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] *= scale[k[u] >= 0 ? k[u] : 0];
      if (v32) reinterpret_cast<float4*>(v32)[at] = make_float4(float(w[0]), float(w[1]), float(w[2]), float(w[3]));
    }
    if (v64) {
      reinterpret_cast<double2*>(v64)[2 * at] = make_double2(w[0], w[1]);
      reinterpret_cast<double2*>(v64)[2 * at + 1] = make_double2(w[2], w[3]);
    }
  }
}

__global__ void k_round_values(const double* __restrict__ v64, float* __restrict__ v32, int64_t len) {
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < len; t += int64_t(gridDim.x) * blockDim.x)
    v32[t] = float(v64[t]);
}

// Coefficients of the triangles of the nested 2h mesh: the mean over the
// four fine triangles inside (the gradients of the coarse basis are constant
// on a coarse triangle, so R_0 A(c) R_0^T is the P1 stiffness of that mean).
// Coarse cell (I, J), fine cell (i, j) = (2I, 2J): its lower triangle holds
// lo(i, j), lo(i+1, j), up(i+1, j), lo(i+1, j+1), its upper triangle
// up(i, j), up(i, j+1), lo(i, j+1), up(i+1, j+1).
__global__ void k_coarse_coef(const double* __restrict__ cb, int N, int kn, double* __restrict__ out) {
  const int Nc = N / 2;
  const int64_t E = 2LL * N * N, Ec = 2LL * Nc * Nc, total = int64_t(kn) * Nc * Nc;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < total; t += int64_t(gridDim.x) * blockDim.x) {
    const int kl = int(t / (int64_t(Nc) * Nc));
    const int64_t cell = t - int64_t(kl) * Nc * Nc;
    const int i = 2 * int(cell % Nc), j = 2 * int(cell / Nc);
    const double* c = cb + int64_t(kl) * E;
    auto lo = [&](int ci, int cj) { return c[2LL * (int64_t(cj) * N + ci)]; };
    auto up = [&](int ci, int cj) { return c[2LL * (int64_t(cj) * N + ci) + 1]; };
    double* o = out + int64_t(kl) * Ec + 2 * cell;
    o[0] = 0.25 * (lo(i, j) + lo(i + 1, j) + up(i + 1, j) + lo(i + 1, j + 1));
    o[1] = 0.25 * (up(i, j) + up(i, j + 1) + lo(i, j + 1) + up(i + 1, j + 1));
  }
}

}  // namespace

sg_status ell_f32(const Ell& A, int K, cudaStream_t st) {
  if (A.v32.ptr) return SG_OK;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (st) SG_CUDA(cudaStreamIsCapturing(st, &cs));
  if (cs != cudaStreamCaptureStatusNone) {
    set_error("the FP32 slot values must exist before a capture");
    return SG_ERR_ARG;
  }
  const int64_t len = int64_t(K) * A.S * A.ldr;
  DevBuf v;
  SG_TRY(v.alloc(size_t(len) * 4));
  k_round_values<<<4 * 152, 256, 0, st>>>(A.v64.as<double>(), v.as<float>(), len);
  note_launch();
  SG_CUDA(cudaGetLastError());
  SG_CUDA(cudaStreamSynchronize(st));
  A.v32 = std::move(v);
  return SG_OK;
}

sg_status edge_alloc(const sg_problem* pr, int N, bool f32, bool f64, EdgeVals& out) {
  out.N = N;
  const size_t len = size_t(N) * ((N + 30) / 31) * 64 * pr->edge_terms.KT;
  if (f32 && !out.v32.ptr) SG_TRY(out.v32.alloc(len * sizeof(float)));
  if (f64 && !out.v64.ptr) SG_TRY(out.v64.alloc(len * sizeof(double)));
  return SG_OK;
}

template <typename Tc>
sg_status edge_values(const sg_problem* pr, const Tc* coef, int k0, int kn, EdgeVals& out, cudaStream_t st) {
  const EdgeTerms& T = pr->edge_terms;
  k_edge_values<Tc><<<8 * 152, 256, 0, st>>>(coef, out.N, T.KT, T.off.as<int>(), T.pos.as<int>(), T.scale.as<double>(),
                                             k0, kn, out.v32.as<float>(), out.v64.as<double>());
  note_launch();
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}
template sg_status edge_values<float>(const sg_problem*, const float*, int, int, EdgeVals&, cudaStream_t);
template sg_status edge_values<double>(const sg_problem*, const double*, int, int, EdgeVals&, cudaStream_t);

template <typename Tc>
sg_status edge_values_all(const sg_problem* pr, const Tc* coef, EdgeVals& out, cudaStream_t st) {
  const EdgeTerms& T = pr->edge_terms;
  const int64_t blocks = 2 * int64_t(out.N) * ((out.N + 30) / 31);
  k_edge_values_all<Tc><<<unsigned(blocks), 256, 0, st>>>(coef, out.N, T.KT, T.term.as<int>(), T.scale.as<double>(),
                                                          T.scale2.as<float2>(), out.v32.as<float>(), out.v64.as<double>());
  note_launch();
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}
template sg_status edge_values_all<float>(const sg_problem*, const float*, EdgeVals&, cudaStream_t);
template sg_status edge_values_all<double>(const sg_problem*, const double*, EdgeVals&, cudaStream_t);

static sg_status edge_terms_build(sg_problem* pr) {
  const std::vector<int> term = jit_edge_terms(pr);
  std::vector<int> off(pr->K + 1, 0), pos(term.size());
  for (int k : term)
    if (k >= 0) ++off[k + 1];
  for (int k = 0; k < pr->K; ++k) off[k + 1] += off[k];
  std::vector<int> at(off.begin(), off.end() - 1);
  for (size_t q = 0; q < term.size(); ++q)
    if (term[q] >= 0) pos[at[term[q]]++] = int(q);
  EdgeTerms& T = pr->edge_terms;
  T.KT = int(term.size());
  T.R = jit_edge_rotations(pr);
  SG_TRY(T.off.alloc(off.size() * 4));
  SG_TRY(T.pos.alloc(pos.size() * 4));
  SG_CUDA(cudaMemcpy(T.off.ptr, off.data(), off.size() * 4, cudaMemcpyHostToDevice));
  SG_TRY(T.term.alloc(term.size() * 4));
  SG_CUDA(cudaMemcpy(T.term.ptr, term.data(), term.size() * 4, cudaMemcpyHostToDevice));
  const std::vector<double> scale = jit_edge_scale(pr);
  SG_TRY(T.scale.alloc(scale.size() * 8));
  SG_CUDA(cudaMemcpy(T.scale.ptr, scale.data(), scale.size() * 8, cudaMemcpyHostToDevice));
  std::vector<float2> scale2(scale.size());
  for (size_t k = 0; k < scale.size(); ++k) {
    const float hi = float(scale[k]);
    scale2[k] = make_float2(hi, float(scale[k] - double(hi)));
  }
  SG_TRY(T.scale2.alloc(scale2.size() * 8));
  SG_CUDA(cudaMemcpy(T.scale2.ptr, scale2.data(), scale2.size() * 8, cudaMemcpyHostToDevice));
  SG_CUDA(cudaMemcpy(T.pos.ptr, pos.data(), pos.size() * 4, cudaMemcpyHostToDevice));
  return SG_OK;
}

sg_status coarse_edge_build(sg_problem* pr, EdgeVals& out) {
  const int K = pr->K, N = pr->N, Nc = N / 2, KC = 32;
  SG_TRY(edge_alloc(pr, Nc, true, false, out));
  DevBuf dcb, dcc;
  SG_TRY(dcb.alloc(size_t(KC) * pr->E * sizeof(double)));
  SG_TRY(dcc.alloc(size_t(KC) * 2 * Nc * Nc * sizeof(double)));
  for (int k0 = 0; k0 < K; k0 += KC) {
    const int kn = std::min(KC, K - k0);
    SG_TRY(element_coefficients(pr, k0, kn, dcb.as<double>(), nullptr));
    k_coarse_coef<<<4 * 152, 256>>>(dcb.as<double>(), N, kn, dcc.as<double>());
    note_launch();
    SG_TRY(edge_values<double>(pr, dcc.as<double>(), k0, kn, out, nullptr));
  }
  SG_CUDA(cudaDeviceSynchronize());
  return SG_OK;
}

sg_status flux_values64(sg_problem* pr, double* w, int64_t vkst) {
  const int K = pr->K, N = pr->N, KC = 32;
  DevBuf dcb;
  SG_TRY(dcb.alloc(size_t(KC) * pr->E * sizeof(double)));
  for (int k0 = 0; k0 < K; k0 += KC) {
    const int kn = std::min(KC, K - k0);
    SG_TRY(element_coefficients(pr, k0, kn, dcb.as<double>(), nullptr));
    k_flux_values64<<<4 * 152, 256>>>(dcb.as<double>(), N, vkst, k0, kn, w);
    note_launch();
    SG_CUDA(cudaGetLastError());
  }
  SG_CUDA(cudaDeviceSynchronize());
  return SG_OK;
}

sg_status assemble_fine(sg_problem* pr) {
  const int S = 5, K = pr->K, L = pr->L, N = pr->N;
  const int64_t n = pr->n, E = pr->E, ldr = round_up(n, 64);
  Ell& A = pr->fine;
  A.S = S;
  A.n = n;
  A.ldr = ldr;
  // column indices: neighbour or the row itself for padding slots
  std::vector<int32_t> col(size_t(S) * ldr, 0);
  const int m = N - 1;
  for (int64_t r = 0; r < ldr; ++r) {
    if (r >= n) {
      for (int s = 0; s < S; ++s) col[s * ldr + r] = 0;
      continue;
    }
    int i = int(r % m) + 1, j = int(r / m) + 1;
    col[0 * ldr + r] = int32_t(j > 1 ? r - m : r);
    col[1 * ldr + r] = int32_t(i > 1 ? r - 1 : r);
    col[2 * ldr + r] = int32_t(r);
    col[3 * ldr + r] = int32_t(i < m ? r + 1 : r);
    col[4 * ldr + r] = int32_t(j < m ? r + m : r);
  }
  SG_TRY(A.col.alloc(col.size() * sizeof(int32_t)));
  SG_CUDA(cudaMemcpy(A.col.ptr, col.data(), col.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
  SG_TRY(A.v64.alloc(size_t(K) * S * ldr * sizeof(double)));
  // the conductances of the edge form from the same coefficients
  const bool edges = jit_eligible(pr) && n > 0;
  if (edges) {
    SG_TRY(edge_terms_build(pr));
    SG_TRY(edge_alloc(pr, N, true, false, pr->edge));
  }

  const int KC = 32;
  DevBuf dcb;
  SG_TRY(dcb.alloc(size_t(KC) * E * sizeof(double)));
  for (int k0 = 0; k0 < K; k0 += KC) {
    int kn = std::min(KC, K - k0);
    SG_TRY(element_coefficients(pr, k0, kn, dcb.as<double>(), nullptr));
    k_fine_ell<<<4 * 152, 256>>>(dcb.as<double>(), N, n, ldr, k0, kn, A.v64.as<double>());
    note_launch();
    if (edges) SG_TRY(edge_values<double>(pr, dcb.as<double>(), k0, kn, pr->edge, nullptr));
    SG_CUDA(cudaGetLastError());
  }
  SG_CUDA(cudaDeviceSynchronize());
  return SG_OK;
}

sg_status gfield_upload(sg_problem* pr) {
  DevBuf& g = pr->gfield_dev;
  if (g.ptr) return SG_OK;
  SG_TRY(g.alloc(std::max<size_t>(1, pr->gfield.size()) * 8));
  if (!pr->gfield.empty()) SG_CUDA(cudaMemcpy(g.ptr, pr->gfield.data(), pr->gfield.size() * 8, cudaMemcpyHostToDevice));
  return SG_OK;
}

sg_status element_coefficients(sg_problem* pr, int k0, int kn, double* out, cudaStream_t st) {
  const int K = pr->K, L = pr->L;
  if (!pr->mi_in_dev.ptr) {
    std::vector<double> isf(K, 1.0);
    std::vector<int32_t> mi = pr->mi_in;
    if (L == 0) mi.assign(1, 0);
    for (int k = 0; k < K; ++k) {
      double f = 1.0;
      for (int i = 0; i < L; ++i)
        for (int v = 2; v <= mi[size_t(k) * L + i]; ++v) f *= v;
      isf[k] = 1.0 / std::sqrt(f);
    }
    SG_TRY(gfield_upload(pr));
    SG_TRY(pr->isf_dev.alloc(isf.size() * sizeof(double)));
    SG_CUDA(cudaMemcpy(pr->isf_dev.ptr, isf.data(), isf.size() * sizeof(double), cudaMemcpyHostToDevice));
    SG_TRY(pr->mi_in_dev.alloc(mi.size() * sizeof(int32_t)));
    SG_CUDA(cudaMemcpy(pr->mi_in_dev.ptr, mi.data(), mi.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
  }
  k_cbar<<<4 * 152, 256, 0, st>>>(pr->gfield_dev.as<double>(), pr->mi_in_dev.as<int>(), pr->isf_dev.as<double>(), L,
                                  pr->E, pr->g0, k0, kn, out);
  note_launch();
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

// Triples re-ordered by (a, k, b) and split into input-term chunks of kc for
// the shared-memory apply; off[a * (nchunk + 1) + c] is the first triple of
// output a with k >= c * kc.
sg_status build_triple_tables(sg_problem* pr, TripleTables& t, int S) {
  const int P = pr->P, K = pr->K;
  const int64_t T = pr->T;
  // chunk of input terms: the FP64 tile of 32 rows must fit in shared memory
  const size_t budget = 200 * 1024;
  const size_t fixed = size_t(S * P + P) * 32 * sizeof(double);
  int kc = 1;
  if (fixed < budget) kc = int((budget - fixed) / (size_t(S) * 32 * sizeof(double)));
  kc = std::max(1, std::min(kc, K));
  if (kc >= 8) kc = kc / 8 * 8;
  t.kc = kc;
  t.nchunk = (K + kc - 1) / kc;
  std::vector<int64_t> order(T);
  for (int64_t i = 0; i < T; ++i) order[i] = i;
  std::sort(order.begin(), order.end(), [&](int64_t x, int64_t y) {
    const int32_t* a = &pr->kab[3 * x];
    const int32_t* b = &pr->kab[3 * y];
    if (a[1] != b[1]) return a[1] < b[1];
    if (a[0] != b[0]) return a[0] < b[0];
    return a[2] < b[2];
  });
  std::vector<int32_t> tk(T), tb(T), off(size_t(P) * (t.nchunk + 1));
  std::vector<double> g64(T);
  std::vector<float> g32(T);
  for (int64_t i = 0; i < T; ++i) {
    tk[i] = pr->kab[3 * order[i] + 0];
    tb[i] = pr->kab[3 * order[i] + 2];
    g64[i] = pr->g[order[i]];
    g32[i] = float(g64[i]);
  }
  int64_t pos = 0;
  for (int a = 0; a < P; ++a) {
    for (int c = 0; c <= t.nchunk; ++c) {
      int kstart = std::min(c * kc, K);
      while (pos < T && pr->kab[3 * order[pos] + 1] == a && tk[pos] < kstart) ++pos;
      off[size_t(a) * (t.nchunk + 1) + c] = int32_t(pos);
    }
    while (pos < T && pr->kab[3 * order[pos] + 1] == a) ++pos;
  }
  SG_TRY(t.tk.alloc(T * sizeof(int32_t)));
  SG_TRY(t.tb.alloc(T * sizeof(int32_t)));
  SG_TRY(t.g64.alloc(T * sizeof(double)));
  SG_TRY(t.g32.alloc(T * sizeof(float)));
  SG_TRY(t.off.alloc(off.size() * sizeof(int32_t)));
  SG_CUDA(cudaMemcpy(t.tk.ptr, tk.data(), T * sizeof(int32_t), cudaMemcpyHostToDevice));
  SG_CUDA(cudaMemcpy(t.tb.ptr, tb.data(), T * sizeof(int32_t), cudaMemcpyHostToDevice));
  SG_CUDA(cudaMemcpy(t.g64.ptr, g64.data(), T * sizeof(double), cudaMemcpyHostToDevice));
  SG_CUDA(cudaMemcpy(t.g32.ptr, g32.data(), T * sizeof(float), cudaMemcpyHostToDevice));
  SG_CUDA(cudaMemcpy(t.off.ptr, off.data(), off.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
  return SG_OK;
}

}  // namespace sg
