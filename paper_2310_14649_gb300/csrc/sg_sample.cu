// Batched deterministic solves for Monte Carlo verification of the SG
// solution (Sec. 4.1, Fig. mcs_verify_poisson: the paper compares the SG
// mean, standard deviation and pdf with 40,000 Monte Carlo samples).
//
// Sample s draws xi_s in R^L and solves the deterministic problem
//     -div( c_s grad u_s ) = 1,  u_s = 0 on the boundary,
//     c_s(e) = exp( g0 + sum_i g_i(e) xi_{s,i} )      (the exact lognormal
// field of Eq. KLE at the element centroids, not its chaos expansion) with
// the same P1 discretisation as the SG system.  One CTA solves one sample
// entirely in shared memory by Jacobi-preconditioned conjugate gradients
// in FP32: the search direction, the edge conductances and the inverse
// diagonal live in shared memory, the iterate, the residual and the thread's
// own search direction in registers.
#include <algorithm>
#include <cmath>

#include "sg_df.h"
#include "sg_exp_df.h"
#include "sg_internal.h"

namespace sg {
namespace {

constexpr int kSampThreads = 512;      // most threads of a CTA
constexpr int kSampMaxNodes = 10240;   // meshes up to N = 102
constexpr int kSampMaxRun = 21;        // most nodes of a thread (m = 101: 5 runs of a column)

// The sums over a block and the scalars of the CG recurrence are carried in
// double-FP32: GB300 runs FP64 at 1/64 of its FP32 rate, and the FP64 sums
// this replaces (every thread adding 64 partial sums per reduction) were 90 %
// of an iteration.
// float(a / b): the quotient of the high words corrected by its remainder
__device__ __forceinline__ float df_div(Df a, Df b) {
  const float q = __fdiv_rn(a.h, b.h);
  const float r = __fmaf_rn(-q, b.h, a.h);
  return __fadd_rn(q, __fdiv_rn(__fadd_rn(r, __fmaf_rn(-q, b.l, a.l)), b.h));
}
__device__ __forceinline__ Df df_of(double v) {
  const float h = float(v);
  return {h, float(v - double(h))};
}

// Block-wide sums of NV (1 or 2) values (every thread receives them):
// butterflies in the warps, then every warp sums the warps' results.  The
// slots alternate between two halves of red, so one barrier per call is
// enough.  512 threads: the butterflies cost the same instructions in every
// warp, and with 1,024 threads they were a third of an iteration (7.2 us
// against 4.0 us at N = 100).
template <int NV>
__device__ __forceinline__ void block_sum(const float (&v)[NV], float2* red, int& turn, int nwarps, Df (&s)[NV]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2* slot = red + 32 * turn;
  turn ^= 1;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    Df x{v[q], 0.f};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      x = df_add(x, Df{__shfl_xor_sync(0xffffffffu, x.h, o), __shfl_xor_sync(0xffffffffu, x.l, o)});
    if (lane == 0) slot[16 * q + warp] = make_float2(x.h, x.l);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int l = lane & 15;
    const float2 t = l < nwarps ? slot[16 * q + l] : make_float2(0.f, 0.f);
    Df x{t.x, t.y};
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
      x = df_add(x, Df{__shfl_xor_sync(0xffffffffu, x.h, o), __shfl_xor_sync(0xffffffffu, x.l, o)});
    s[q] = two_sum(x.h, x.l);
  }
}

// Edge conductances of the P1 stencil (Sec. 2.1): the horizontal edge
// (i,j)-(i+1,j) couples the lower triangle of cell (i,j) and the upper one
// of cell (i,j-1), wx = (c_lo(i,j) + c_up(i,j-1)) / 2; the vertical edge
// (i,j)-(i,j+1) couples the upper triangle of cell (i,j) and the lower one
// of cell (i-1,j), wy = (c_up(i,j) + c_lo(i-1,j)) / 2.  Row (i,j) of A(c):
// diagonal = the four conductances around the node, off-diagonals = minus
// the conductance of the edge (edges to boundary nodes are dropped: the
// search direction is stored with a border of zeros).
//
// A thread owns a run of HN vertically adjacent nodes of one column, lanes
// adjacent columns: the vertical neighbours inside a run are its registers
// and every shared-memory access of a warp is to consecutive words.  Per
// iteration a node costs seven shared words and three barriers a CTA.  304
// samples at N = 100 (two waves of one CTA per SM): 21.4 ms with FP64 block
// sums and interleaved nodes, now 2.0 ms (4.0 us per iteration); what
// bounds it now is the shared-memory words (1.2 us) and the latency of the
// three barriers and two butterflies of an iteration.
// Shared memory: p [(N+1)^2] with its border, the inverse diagonal [n]
// (both first hold the 2 N^2 triangle coefficients), wx [m N], wy [N m],
// the reduction slots.
template <typename To, int HN>
__global__ void __launch_bounds__(kSampThreads, 1)
    k_sample_pcg(int N, int L, int runs, const double* __restrict__ gfield, double g0, const double* __restrict__ xi,
                 double h2, double rtol, int max_it, To* __restrict__ U, int64_t ldu, int* __restrict__ its_max) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = N - 1, S = N + 1;
  const int64_t E = 2LL * N * N;
  float2* red = reinterpret_cast<float2*>(smem_raw);   // [2][2][16]
  float* p = reinterpret_cast<float*>(red + 64);       // [S][S], node (i, j) at j S + i
  float* dinv = p + S * S;                             // [m][m]
  float* wx = dinv + m * m;                            // [m][N]: (i = 0..N-1, j = 1..m)
  float* wy = wx + m * N;                              // [N][m]: (i = 1..m, j = 0..m)
  float* cb = p;                                       // [2 N^2] while wx and wy are formed
  __shared__ double sxi[16];
  const int64_t s = blockIdx.x;
  const int nthr = blockDim.x, nwarps = nthr >> 5;
  if (threadIdx.x < L) sxi[threadIdx.x] = xi[s * L + threadIdx.x];
  __syncthreads();
  for (int e = threadIdx.x; e < 2 * N * N; e += nthr) {
    double a = g0;
    for (int i = 0; i < L; ++i) a += gfield[int64_t(i) * E + e] * sxi[i];
    const Df d = df_of(a);
    cb[e] = exp_df(d.h, d.l);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < m * N; t += nthr) {
    const int i = t % N, j = t / N + 1;  // edge (i,j)-(i+1,j)
    wx[t] = 0.5f * (cb[2 * (j * N + i)] + cb[2 * ((j - 1) * N + i) + 1]);
  }
  for (int t = threadIdx.x; t < N * m; t += nthr) {
    const int i = t % m + 1, j = t / m;  // edge (i,j)-(i,j+1)
    wy[t] = 0.5f * (cb[2 * (j * N + i) + 1] + cb[2 * (j * N + i - 1)]);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < S * S; t += nthr) p[t] = 0.0f;
  __syncthreads();
  // column i, rows j0 .. j0 + cnt - 1
  const int run = threadIdx.x / m, i = threadIdx.x - run * m + 1;
  const int j0 = run * HN + 1, cnt = run < runs ? min(HN, m - j0 + 1) : 0;
  float* pc = p + j0 * S + i;
  const float* we = wx + (j0 - 1) * N + i;
  const float* wv = wy + (j0 - 1) * m + i - 1;  // south edge of the run's first node
  float* di = dinv + (j0 - 1) * m + i - 1;
  float x[HN], r[HN], pr[HN];
  float rz_loc = 0.0f, bb_loc = 0.0f;
#pragma unroll
  for (int k = 0; k < HN; ++k) {
    x[k] = 0.0f;
    r[k] = 0.0f;
    pr[k] = 0.0f;
    if (k < cnt) {
      const float d = we[k * N] + we[k * N - 1] + wv[(k + 1) * m] + wv[k * m];
      const float dv = 1.0f / d;
      di[k * m] = dv;
      r[k] = float(h2);
      pr[k] = r[k] * dv;
      pc[k * S] = pr[k];
      rz_loc += r[k] * r[k] * dv;
      bb_loc += r[k] * r[k];
    }
  }
  int turn = 0;
  Df sums[2];
  block_sum<2>({rz_loc, bb_loc}, red, turn, nwarps, sums);
  Df rz = sums[0];
  const Df tol2 = df_of(rtol * rtol * (double(sums[1].h) + double(sums[1].l)));
  int it = 0;
  for (; it < max_it; ++it) {
    __syncthreads();  // p complete
    float q[HN];
    float pq_loc = 0.0f;
    if (cnt > 0) {
      float ws = wv[0], pS = pc[-S];
      const float pTop = pc[cnt * S];
#pragma unroll
      for (int k = 0; k < HN; ++k) {
        q[k] = 0.0f;
        if (k < cnt) {
          const float e = we[k * N], w = we[k * N - 1], wn = wv[(k + 1) * m];
          const float pN = (k + 1 < cnt && k + 1 < HN) ? pr[(k + 1) % HN] : pTop;
          float v = (e + w + wn + ws) * pr[k];
          v -= w * pc[k * S - 1];
          v -= e * pc[k * S + 1];
          v -= ws * pS;
          v -= wn * pN;
          q[k] = v;
          pq_loc += pr[k] * v;
          ws = wn;
          pS = pr[k];
        }
      }
    }
    Df pq[1];
    block_sum<1>({pq_loc}, red, turn, nwarps, pq);
    if (!(pq[0].h > 0.0f)) break;
    const float alpha = df_div(rz, pq[0]);
    float rr_loc = 0.0f, rzn_loc = 0.0f;
#pragma unroll
    for (int k = 0; k < HN; ++k) {
      if (k < cnt) {
        x[k] += alpha * pr[k];
        r[k] -= alpha * q[k];
        rr_loc += r[k] * r[k];
        rzn_loc += r[k] * r[k] * di[k * m];
      }
    }
    block_sum<2>({rr_loc, rzn_loc}, red, turn, nwarps, sums);
    const Df rr = sums[0], rzn = sums[1];
    if ((rr.h - tol2.h) + (rr.l - tol2.l) <= 0.0f) {
      ++it;
      break;
    }
    const float beta = df_div(rzn, rz);
    rz = rzn;
    // every thread read its neighbours' p before the first sum's barrier
#pragma unroll
    for (int k = 0; k < HN; ++k)
      if (k < cnt) {
        pr[k] = r[k] * di[k * m] + beta * pr[k];
        pc[k * S] = pr[k];
      }
  }
#pragma unroll
  for (int k = 0; k < HN; ++k)
    if (k < cnt) U[s * ldu + int64_t(j0 - 1 + k) * m + i - 1] = To(x[k]);
  if (threadIdx.x == 0) atomicMax(its_max, it);
}

size_t sample_smem(int N) {
  const int64_t m = N - 1, S = N + 1;
  return 64 * sizeof(float2) + size_t(S * S + m * m + 2 * m * N) * 4;
}

// the shortest run of nodes per thread (of the instantiated lengths) whose
// m x ceil(m / run) threads fit a CTA: short runs keep more warps in flight
int sample_run(int m) {
  for (int h : {1, 2, 4, 8, 12, 16, 20, kSampMaxRun})
    if (int64_t(m) * ((m + h - 1) / h) <= kSampThreads) return h;
  return 0;
}

template <typename To, int HN>
sg_status sample_launch(const sg_problem* pr, int64_t S, const double* gfield, const double* xi, double rtol,
                        int max_it, To* U, int64_t ldu, int* its, cudaStream_t st) {
  const int m = pr->N - 1, runs = (m + HN - 1) / HN;
  const double h = 1.0 / pr->N;
  const size_t smem = sample_smem(pr->N);
  SG_CUDA(cudaFuncSetAttribute(k_sample_pcg<To, HN>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
  k_sample_pcg<To, HN><<<unsigned(S), unsigned(round_up(int64_t(m) * runs, 32)), smem, st>>>(
      pr->N, pr->L, runs, gfield, pr->g0, xi, h * h, rtol, max_it, U, ldu, its);
  note_launch();
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

template <typename To>
sg_status sample_dispatch(const sg_problem* pr, int64_t S, const double* gfield, const double* xi, double rtol,
                          int max_it, To* U, int64_t ldu, int* its, cudaStream_t st) {
  switch (sample_run(pr->N - 1)) {
    case 1: return sample_launch<To, 1>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    case 2: return sample_launch<To, 2>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    case 4: return sample_launch<To, 4>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    case 8: return sample_launch<To, 8>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    case 12: return sample_launch<To, 12>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    case 16: return sample_launch<To, 16>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    case 20: return sample_launch<To, 20>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
    default: return sample_launch<To, kSampMaxRun>(pr, S, gfield, xi, rtol, max_it, U, ldu, its, st);
  }
}

}  // namespace
}  // namespace sg

using namespace sg;

extern "C" sg_status sg_sample_solve(sg_problem* pr, const double* xi, int64_t S, sg_dtype dtype, void* U,
                                     int64_t ldu, double rtol, int max_it, int* its_max, void* stream) {
  SG_ARG(pr && xi && U, "sg_sample_solve: NULL argument");
  SG_ARG(dtype == SG_F64 || dtype == SG_F32, "sg_sample_solve: bad dtype");
  SG_ARG(S >= 0 && S <= 0x7fffffff, "sg_sample_solve: sample count out of range");
  SG_ARG(ldu >= pr->n, "sg_sample_solve: leading dimension < n");
  SG_ARG(rtol > 0 && max_it > 0, "sg_sample_solve: rtol and max_it must be > 0");
  SG_ARG(pr->L >= 1 && pr->L <= 16, "sg_sample_solve: needs 1 <= L <= 16 KL modes");
  SG_ARG(pr->n <= kSampMaxNodes && sample_run(pr->N - 1) > 0 && sample_smem(pr->N) <= 227 * 1024,
         "sg_sample_solve: the mesh is too large for one CTA per sample (N <= 102)");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the KL modes at the element centroids, once per problem
  SG_TRY(gfield_upload(pr));
  const DevBuf& g = pr->gfield_dev;
  DevBuf itsd;
  SG_TRY(itsd.alloc(sizeof(int)));
  SG_CUDA(cudaMemsetAsync(itsd.ptr, 0, sizeof(int), st));
  if (S > 0) {
    if (dtype == SG_F32)
      SG_TRY(sample_dispatch<float>(pr, S, dp<double>(g), xi, rtol, max_it, static_cast<float*>(U), ldu,
                                    dp<int>(itsd), st));
    else
      SG_TRY(sample_dispatch<double>(pr, S, dp<double>(g), xi, rtol, max_it, static_cast<double*>(U), ldu,
                                     dp<int>(itsd), st));
  }
  int its = 0;
  SG_CUDA(cudaMemcpyAsync(&its, itsd.ptr, sizeof(int), cudaMemcpyDeviceToHost, st));
  SG_CUDA(cudaStreamSynchronize(st));
  if (its_max) *its_max = its;
  if (S > 0 && its >= max_it) {
    set_error("sg_sample_solve: a sample reached max_it before rtol");
    return SG_NOT_CONVERGED;
  }
  return SG_OK;
}
