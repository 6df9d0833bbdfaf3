// Galerkin operator apply (Sec. 2.1, Eq. Galerkin_L_exp, Kronecker form):
//     Y = sum_k A_k X G_k^T,
//     y_r[a] = sum_{s} sum_{(k,a,b) in T} v_k^{r,s} g_kab x_{col(r,s)}[b],
// over an ELL family of K matrices with S slots per row.
//
// Shared-memory tile kernel: one CTA owns 32 consecutive rows (lane = row)
// and all P output modes; its warps split the output modes.  The 32-row
// tile of X gathered through the slot columns (S x P values per row) and a
// chunk of kc input terms of the matrix values (S x kc per row) are staged
// in shared memory, laid out [.][lane] so every access is bank-conflict
// free; the triple list of each output mode is walked warp-uniformly.
#include <algorithm>

#include "sg_solver.h"

namespace sg {

namespace {

template <typename T>
struct ApplyArgs {
  const int* col;
  const T* V;
  int64_t ldr, n;
  int S, K, P;
  const T* X;
  int64_t ldx;
  const T* F;  // optional: Y = F - A(X)
  int64_t ldf;
  T* Y;
  int64_t ldy;
  const int* tk;
  const int* tb;
  const T* tg;
  const int* off;
  int kc, nchunk;
};

template <typename T>
__global__ void __launch_bounds__(256) k_apply_tile(ApplyArgs<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* xs = reinterpret_cast<T*>(smem_raw);  // [S][P][32]
  T* vs = xs + size_t(p.S) * p.P * 32;     // [S][kc][32]
  T* ys = vs + size_t(p.S) * p.kc * 32;    // [P][32]
  const int lane = threadIdx.x, w = threadIdx.y, W = blockDim.y;
  const int64_t r = int64_t(blockIdx.x) * 32 + lane;
  const bool valid = r < p.n;
  const int S = p.S, P = p.P, kc = p.kc;

  for (int sb = w; sb < S * P; sb += W) {
    int s = sb / P, b = sb - s * P;
    T v = T(0);
    if (valid) v = p.X[int64_t(b) * p.ldx + p.col[int64_t(s) * p.ldr + r]];
    xs[sb * 32 + lane] = v;
  }
  for (int a = w; a < P; a += W) ys[a * 32 + lane] = T(0);

  for (int c = 0; c < p.nchunk; ++c) {
    const int k0 = c * kc;
    __syncthreads();
    for (int sk = w; sk < S * kc; sk += W) {
      int s = sk / kc, kk = sk - s * kc, k = k0 + kk;
      T v = T(0);
      if (valid && k < p.K) v = p.V[(int64_t(k) * S + s) * p.ldr + r];
      vs[sk * 32 + lane] = v;
    }
    __syncthreads();
    for (int a = w; a < P; a += W) {
      T acc = ys[a * 32 + lane];
      const int t0 = p.off[a * (p.nchunk + 1) + c], t1 = p.off[a * (p.nchunk + 1) + c + 1];
      for (int t = t0; t < t1; ++t) {
        const int kk = p.tk[t] - k0, b = p.tb[t];
        T sum = T(0);
        for (int s = 0; s < S; ++s) sum += vs[(s * kc + kk) * 32 + lane] * xs[(s * P + b) * 32 + lane];
        acc += p.tg[t] * sum;
      }
      ys[a * 32 + lane] = acc;
    }
  }
  __syncthreads();
  if (valid) {
    for (int a = w; a < P; a += W) {
      T y = ys[a * 32 + lane];
      if (p.F) y = p.F[int64_t(a) * p.ldf + r] - y;
      p.Y[int64_t(a) * p.ldy + r] = y;
    }
  }
}

// ---------------------------------------------------------------------------
// Assembled FP64 apply.  GB300's FP64 units (2 FMAs per clock and SM) bound
// FP64 applies: the generated kernel spends two FP64 operations per triple
// and slot (2,395 triples at P = 35), one P x P block per edge P^2 FMAs, and
// each edge's flux B^e (x_hi - x_lo) is formed once for both of its nodes, as
// in the generated FP32 edge form: about 2.1 P^2 FMAs per row against 5 P^2
// for a block per stencil slot.  An apply with cold caches, before and now:
// 881 and 397 us at 256^2, P = 35 (the operations alone 255 us), 4.96 and 1.89
// ms at 256^2, P = 84, 16.4 and 10.2 us at 32^2, P = 6.  Lane: a column of the tile (AsmBlocks): its
// node's west edge from the lane itself, its east edge's flux from the next
// lane; the CTA marches up its strip of rows and keeps the flux through a
// row's upper edges for the next row; warps and CTA groups share the outputs,
// a warp's outputs in registers.  The differences of up to 64 modes stand in
// shared memory.  B_ab and B_ba are one stored value, read by two warps of
// the CTA (the second from L1 or L2).
// ---------------------------------------------------------------------------

// Blocks from the slot values: thread per edge (in the order of AsmBlocks) and
// pairs p = blockIdx.y, blockIdx.y + gridDim.y, ...  The conductance of an
// edge between two unknowns is minus their slot value.  A row's slot values
// add up to the conductances of its edges to the Dirichlet boundary; those
// edges act on the same difference, so the first of them (west, east, south,
// north) takes the sum and the others zero.
__global__ void k_edge_blocks64(int N, int strip, int64_t len, int S, int64_t ldr, const int* __restrict__ col,
                                int npair, const int* __restrict__ pptr, const int* __restrict__ pk,
                                const double* __restrict__ pg, const double* __restrict__ V, double* __restrict__ C) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= len) return;
  const int m = N - 1, lane = int(q & 31), visits = 2 * strip + 1;
  const int64_t t = (q >> 5) / visits, column = 31 * t + lane;
  const int visit = int((q >> 5) % visits), ver = visit % 2 == 0;
  // the edge's nodes (i, j), (i2, j2); r: the row of one that is an unknown
  const int64_t sn = column / N;
  const int e = int(column - sn * N), j = int(std::min<int64_t>(N, sn * strip + (visit + 1) / 2));
  const int i = e + ver, i2 = e + 1, j2 = j + ver;
  const bool in = i >= 1 && i <= m && j >= 1 && j <= m, in2 = i2 >= 1 && i2 <= m && j2 >= 1 && j2 <= m;
  const int64_t r = int64_t((in ? j : j2) - 1) * m + (in ? i : i2) - 1;
  int s0 = 0, s1 = 0;  // the conductance is sign x the sum over slots s0 .. s1 - 1
  double sign = 1.0;
  if (in && in2) {
    const int64_t r2 = int64_t(j2 - 1) * m + i2 - 1;
    for (int s = 0; s < S; ++s)
      if (col[s * ldr + r] == r2) {
        s0 = s;
        s1 = s + 1;
      }
    sign = -1.0;
  } else if (in || in2) {
    const int iu = in ? i : i2, ju = in ? j : j2;  // the unknown
    const bool first = ver ? iu > 1 && iu < m && (j == 0 || ju > 1) : i == 0 || iu > 1;
    if (first) s1 = S;
  }
  for (int p = blockIdx.y; p < npair; p += gridDim.y) {
    double c = 0.0;
    if (s1 > s0)
      for (int u = pptr[p]; u < pptr[p + 1]; ++u) {
        const double* v = V + int64_t(pk[u]) * S * ldr + r;
        double x = v[s0 * ldr];
        for (int s = s0 + 1; s < s1; ++s) x += v[s * ldr];
        c = fma(pg[u], sign * x, c);
      }
    C[((q >> 5) * npair + p) * 32 + lane] = c;
  }
}

constexpr int kAsmModes = 64;  // modes whose differences are in shared memory at a time
constexpr int kAsmWarps = 16;

struct AsmArgs {
  int N, P, npair, strip, W, G;
  const double* C;
  const double* X;
  int64_t ldx;
  const double* F;
  int64_t ldf;
  double* Y;
  int64_t ldy;
};

// packed index of (a, b): the pair's row starts at lo P - lo (lo + 1) / 2
__device__ __forceinline__ int pair_index(int P, int a, int b) {
  const int lo = min(a, b), hi = max(a, b);
  return lo * P - lo * (lo + 1) / 2 + hi;
}

// f += sum_b B_ab d_b over modes b0 .. b0 + nb - 1 (d: [64][32], lane's column)
__device__ __forceinline__ double asm_dot(const double* __restrict__ C, int P, int a, int b0, int nb, const double* d,
                                          double f) {
  int b = 0;
  for (; b + 8 <= nb; b += 8) {
    double c[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = C[int64_t(pair_index(P, a, b0 + b + u)) * 32];
#pragma unroll
    for (int u = 0; u < 8; ++u) f = fma(c[u], d[(b + u) * 32], f);
  }
  for (; b < nb; ++b) f = fma(C[int64_t(pair_index(P, a, b0 + b)) * 32], d[b * 32], f);
  return f;
}

// the same over two edges: f += sum_b C_ab d_b, f2 += sum_b C2_ab d2_b
__device__ __forceinline__ void asm_dot2(const double* __restrict__ C, const double* __restrict__ C2, int P, int a,
                                         int b0, int nb, const double* d, const double* d2, double& f, double& f2) {
  constexpr int U = 4;
  int b = 0;
  for (; b + U <= nb; b += U) {
    double c[U], c2[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t o = int64_t(pair_index(P, a, b0 + b + u)) * 32;
      c[u] = C[o];
      c2[u] = C2[o];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      f = fma(c[u], d[(b + u) * 32], f);
      f2 = fma(c2[u], d2[(b + u) * 32], f2);
    }
  }
  for (; b < nb; ++b) {
    const int64_t o = int64_t(pair_index(P, a, b0 + b)) * 32;
    f = fma(C[o], d[b * 32], f);
    f2 = fma(C2[o], d2[b * 32], f2);
  }
}

template <int MO>
__global__ void __launch_bounds__(32 * kAsmWarps, 2) k_apply_edge64(const __grid_constant__ AsmArgs p) {
  extern __shared__ double ds[];  // [3][min(P, 64)][32]: west, upper, lower edge
  const int P = p.P, N = p.N, m = N - 1, lane = threadIdx.x, w = threadIdx.y;
  const int g = blockIdx.x % p.G;
  const int bc = min(P, kAsmModes);
  double* dh = ds + lane;
  double* dv = dh + bc * 32;
  double* dl = dv + bc * 32;
  const int64_t t = blockIdx.x / p.G, column = 31 * t + lane, sn = column / N;
  const int i = int(column - sn * N);  // node column to the west; the lane's own node is i + 1
  const int j0 = 1 + int(sn) * p.strip;
  const double* C = p.C + t * (2 * p.strip + 1) * p.npair * 32 + lane;
  double lower[MO];
#pragma unroll
  for (int o = 0; o < MO; ++o) lower[o] = 0.0;
  for (int k = 0; k < p.strip; ++k) {
    const int j = j0 + k;
    const bool in0 = i >= 1 && j <= m, in1 = i + 1 <= m && j <= m;
    const double* Ch = C + int64_t(2 * k + 1) * p.npair * 32;
    const double* Cv = Ch + int64_t(p.npair) * 32;
    const int64_t r = int64_t(j - 1) * m + i;  // the lane's own node
    double fh[MO], fv[MO];
#pragma unroll
    for (int o = 0; o < MO; ++o) fh[o] = fv[o] = 0.0;
    for (int b0 = 0; b0 < P; b0 += kAsmModes) {
      const int nb = min(kAsmModes, P - b0);
      __syncthreads();
#pragma unroll 4
      for (int b = w; b < nb; b += p.W) {
        const double* x = p.X + int64_t(b0 + b) * p.ldx + r;
        const double x1 = in1 ? x[0] : 0.0;
        const double x0 = in0 ? x[-1] : 0.0;
        const double x2 = in1 && j < m ? x[m] : 0.0;
        dh[b * 32] = x1 - x0;
        dv[b * 32] = x2 - x1;
        if (k == 0) dl[b * 32] = x1 - (in1 && j > 1 ? x[-m] : 0.0);
      }
      __syncthreads();
#pragma unroll
      for (int o = 0; o < MO; ++o) {
        const int a = g + p.G * (w + p.W * o);
        if (a < P) {
          if (k == 0) lower[o] = asm_dot(C, P, a, b0, nb, dl, lower[o]);
          asm_dot2(Ch, Cv, P, a, b0, nb, dh, dv, fh[o], fv[o]);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < MO; ++o) {
      const int a = g + p.G * (w + p.W * o);
      const double east = __shfl_down_sync(0xffffffffu, fh[o], 1);
      const double y = (fh[o] - east) + (lower[o] - fv[o]);
      lower[o] = fv[o];
      if (a < P && lane < 31 && in1)
        p.Y[int64_t(a) * p.ldy + r] = p.F ? p.F[int64_t(a) * p.ldf + r] - y : y;
    }
  }
}

template <typename T> const T* vals_of(const Ell& A);
template <> const double* vals_of<double>(const Ell& A) { return A.v64.as<double>(); }
template <> const float* vals_of<float>(const Ell& A) { return A.v32.as<float>(); }
template <typename T> const T* g_of(const TripleTables& t);
template <> const double* g_of<double>(const TripleTables& t) { return t.g64.as<double>(); }
template <> const float* g_of<float>(const TripleTables& t) { return t.g32.as<float>(); }

}  // namespace

template <typename T>
sg_status apply_ell(const Ell& A, const TripleTables& tri, int P, int K, const T* X, int64_t ldx,
                    const T* F, int64_t ldf, T* Y, int64_t ldy, cudaStream_t st) {
  ApplyArgs<T> a;
  a.col = A.col.as<int>();
  a.V = vals_of<T>(A);
  a.ldr = A.ldr;
  a.n = A.n;
  a.S = A.S;
  a.K = K;
  a.P = P;
  a.X = X;
  a.ldx = ldx;
  a.F = F;
  a.ldf = ldf;
  a.Y = Y;
  a.ldy = ldy;
  a.tk = tri.tk.as<int>();
  a.tb = tri.tb.as<int>();
  a.tg = g_of<T>(tri);
  a.off = tri.off.as<int>();
  a.kc = tri.kc;
  a.nchunk = tri.nchunk;
  const size_t smem = (size_t(A.S) * P + size_t(A.S) * tri.kc + P) * 32 * sizeof(T);
  static bool attr_set[2] = {false, false};
  bool& set = attr_set[sizeof(T) == 8 ? 1 : 0];
  if (!set) {
    SG_CUDA(cudaFuncSetAttribute(k_apply_tile<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 227 * 1024));
    set = true;
  }
  const int W = std::min(8, P);
  dim3 block(32, W);
  dim3 grid(unsigned((A.n + 31) / 32));
  if (A.n == 0) return SG_OK;
  k_apply_tile<T><<<grid, block, smem, st>>>(a); note_launch();
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

sg_status apply_attrs_init() {
  SG_CUDA(cudaFuncSetAttribute(k_apply_tile<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  SG_CUDA(cudaFuncSetAttribute(k_apply_tile<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  return SG_OK;
}

Profiler::~Profiler() {
  for (auto& r : pool) {
    if (r.a) cudaEventDestroy(r.a);
    if (r.b) cudaEventDestroy(r.b);
  }
}

sg_status Profiler::begin(int kind, cudaStream_t st, size_t& slot) {
  if (used == pool.size()) {
    Rec r;
    SG_CUDA(cudaEventCreate(&r.a));
    SG_CUDA(cudaEventCreate(&r.b));
    pool.push_back(r);
  }
  slot = used++;
  pool[slot].kind = kind;
  SG_CUDA(cudaEventRecord(pool[slot].a, st));
  return SG_OK;
}

sg_status Profiler::end(size_t slot, cudaStream_t st) {
  SG_CUDA(cudaEventRecord(pool[slot].b, st));
  return SG_OK;
}

sg_status Profiler::read(int kind, int64_t* launches, double* ms) {
  int64_t cnt = 0;
  double tot = 0.0;
  for (size_t i = 0; i < used; ++i) {
    if (pool[i].kind != kind) continue;
    SG_CUDA(cudaEventSynchronize(pool[i].b));
    float t = 0.0f;
    SG_CUDA(cudaEventElapsedTime(&t, pool[i].a, pool[i].b));
    tot += t;
    ++cnt;
  }
  if (launches) *launches = cnt;
  if (ms) *ms = tot;
  return SG_OK;
}

void pair_lists(const sg_problem* pr, std::vector<int>& pptr, std::vector<int>& pk, std::vector<double>& pg) {
  const int P = pr->P;
  const int npair = P * (P + 1) / 2;
  // (k, g) list of every packed pair a <= b
  std::vector<std::vector<std::pair<int, double>>> lst(npair);
  for (int64_t t = 0; t < pr->T; ++t) {
    const int k = pr->kab[3 * t], a = pr->kab[3 * t + 1], b = pr->kab[3 * t + 2];
    if (a > b) continue;
    lst[size_t(a) * P - size_t(a) * (a - 1) / 2 + (b - a)].push_back({k, pr->g[t]});
  }
  pptr.assign(npair + 1, 0);
  pk.clear();
  pg.clear();
  for (int q = 0; q < npair; ++q) {
    for (const auto& e : lst[q]) {
      pk.push_back(e.first);
      pg.push_back(e.second);
    }
    pptr[q + 1] = int(pk.size());
  }
}

sg_status asm_prepare(sg_problem* pr, bool coarse, cudaStream_t st) {
  AsmBlocks& B = coarse ? coarse_asm(pr) : pr->asm_fine;
  if (B.tried || pr->asm_mode == 1) return SG_OK;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  SG_CUDA(cudaStreamIsCapturing(st, &cs));
  if (cs != cudaStreamCaptureStatusNone) return SG_OK;
  B.tried = true;
  const int P = pr->P, N = coarse ? pr->N / 2 : pr->N, m = N - 1;
  const int npair = P * (P + 1) / 2;
  if (m <= 0) return SG_OK;
  // An SM's CTAs share its FP64 units: the strip and the split of the outputs
  // over groups of CTAs with the fewest CTAs per SM x visits x work of a
  // visit (its outputs, and the differences, worth about two); one CTA alone
  // on an SM leaves a quarter of its time to latencies.  Measured at 256^2, P =
  // 35, us by strip and groups: (4, 1) 416, (8, 1) 400, (16, 1) 494, (4, 4)
  // 399, (16, 4) 510; 200^2, P = 56: (3, 1) 582, (8, 1) 909, (3, 4) 594, (16,
  // 1) 961.
  auto tiles_of = [&](int strip) { return (int64_t((m + strip - 1) / strip) * N + 30) / 31; };
  int strip = 1, groups = 1;
  int64_t best = 0;
  for (int s = 1; s <= 16; ++s)
    for (int outs = std::min(P, kAsmModes); outs >= std::min(P, 4); --outs) {
      const int g = (P + outs - 1) / outs;
      const int64_t per_sm = (tiles_of(s) * g + 151) / 152;
      const int64_t cost = (per_sm == 1 ? 5 : 4 * per_sm) * (2 * s + 1) * (outs + 2);
      if (best == 0 || cost < best) {
        best = cost;
        strip = s;
        groups = g;
      }
    }
  const int64_t tiles = tiles_of(strip);
  const size_t bytes = size_t(tiles) * (2 * strip + 1) * 32 * npair * sizeof(double);
  if (pr->asm_mode == 0) {
    // automatic: only while the blocks take at most a quarter of free memory
    size_t fr = 0, tot = 0;
    SG_CUDA(cudaMemGetInfo(&fr, &tot));
    if (bytes > fr / 4) return SG_OK;
  }
  std::vector<int> pptr, pk;
  std::vector<double> pg;
  pair_lists(pr, pptr, pk, pg);
  const Ell& A = coarse ? coarse_ell(pr) : pr->fine;
  DevBuf dptr, dk, dg, c;
  SG_TRY(c.alloc(bytes));
  SG_TRY(dptr.alloc(pptr.size() * 4));
  SG_TRY(dk.alloc(std::max<size_t>(1, pk.size()) * 4));
  SG_TRY(dg.alloc(std::max<size_t>(1, pg.size()) * 8));
  SG_CUDA(cudaMemcpy(dptr.ptr, pptr.data(), pptr.size() * 4, cudaMemcpyHostToDevice));
  if (!pk.empty()) {
    SG_CUDA(cudaMemcpy(dk.ptr, pk.data(), pk.size() * 4, cudaMemcpyHostToDevice));
    SG_CUDA(cudaMemcpy(dg.ptr, pg.data(), pg.size() * 8, cudaMemcpyHostToDevice));
  }
  const int64_t len = int64_t(bytes / sizeof(double)) / npair;
  const int64_t nb = (len + 127) / 128;
  k_edge_blocks64<<<dim3(unsigned(nb), unsigned(std::min<int64_t>({npair, 65535, std::max<int64_t>(1, 152 * 64 / nb)}))),
                    128, 0, st>>>(N, strip, len, A.S, A.ldr, A.col.as<int>(), npair, dptr.as<int>(), dk.as<int>(),
                                  dg.as<double>(), A.v64.as<double>(), c.as<double>());
  note_launch();
  SG_CUDA(cudaGetLastError());
  SG_CUDA(cudaStreamSynchronize(st));
  B.N = N;
  B.strip = strip;
  B.groups = groups;
  B.npair = npair;
  B.c = std::move(c);
  return SG_OK;
}

template <int MO>
static sg_status asm_launch(const AsmArgs& a, dim3 grid, size_t smem, cudaStream_t st) {
  k_apply_edge64<MO><<<grid, dim3(32, a.W), smem, st>>>(a);
  note_launch();
  SG_CUDA(cudaGetLastError());
  return SG_OK;
}

sg_status apply_asm64(const sg_problem* pr, const AsmBlocks& B, const double* X, int64_t ldx, const double* F,
                      int64_t ldf, double* Y, int64_t ldy, cudaStream_t st) {
  const int N = B.N, m = N - 1, P = pr->P;
  AsmArgs a;
  a.N = N;
  a.P = P;
  a.npair = B.npair;
  a.strip = B.strip;
  a.G = B.groups;
  a.W = std::min(kAsmWarps, (P + a.G - 1) / a.G);
  a.C = B.c.as<double>();
  a.X = X;
  a.ldx = ldx;
  a.F = F;
  a.ldf = ldf;
  a.Y = Y;
  a.ldy = ldy;
  const int64_t tiles = (int64_t((m + a.strip - 1) / a.strip) * N + 30) / 31;
  const dim3 grid(unsigned(tiles * a.G));
  const size_t smem = size_t(3) * std::min(P, kAsmModes) * 32 * sizeof(double);
  const int mo = (P + a.G * a.W - 1) / (a.G * a.W);
  switch (mo) {
    case 1: return asm_launch<1>(a, grid, smem, st);
    case 2: return asm_launch<2>(a, grid, smem, st);
    case 3: return asm_launch<3>(a, grid, smem, st);
    default: return asm_launch<4>(a, grid, smem, st);
  }
}

bool solver_edge(const sg_problem* pr) {
  return jit_eligible(pr) && (pr->jit_cfg_user[0] ? pr->jit_cfg[0].flux != 0 : pr->flux_allowed && pr->P <= 48);
}

bool coarse_edge_form(const sg_problem* pr) {
  return solver_edge(pr) && (pr->jit_cfg_user[0] || pr->N * pr->p <= 800);
}

// generated family of an FP32 apply: a solve on the slot form while the fine
// family's own (untuned) form is the edge form has a family for it
static int fp32_family(const sg_problem* pr, bool coarse, bool solver) {
  if (coarse) return 1;
  return solver && jit_config(pr, 0).flux && !solver_edge(pr) ? 6 : 0;
}

template <typename T>
sg_status apply_any(sg_problem* pr, bool coarse, const T* X, int64_t ldx, const T* F, int64_t ldf, T* Y,
                    int64_t ldy, cudaStream_t st, bool solver) {
  const Ell& A = coarse ? coarse_ell(pr) : pr->fine;
  if (sizeof(T) == 8) {
    const AsmBlocks& B = coarse ? coarse_asm(pr) : pr->asm_fine;
    if (B.c.ptr)
      return apply_asm64(pr, B, reinterpret_cast<const double*>(X), ldx, reinterpret_cast<const double*>(F),
                         ldf, reinterpret_cast<double*>(Y), ldy, st);
  }
  if (pr->apply_mode != 1 && jit_eligible(pr)) {
    const int which = sizeof(T) == 8 ? 2 + coarse : fp32_family(pr, coarse, solver);
    if (sizeof(T) == 4 && jit_config(pr, which).flux)
      return jit_edge_launch<T>(pr, which, coarse ? coarse_edge(pr) : pr->edge, X, ldx, F, ldf, Y, ldy, st);
    if (sizeof(T) == 4) SG_TRY(ell_f32(A, pr->K, st));
    return jit_apply_launch(pr, which, A, X, ldx, F, ldf, Y, ldy, st);
  }
  if (sizeof(T) == 4) SG_TRY(ell_f32(A, pr->K, st));
  return apply_ell<T>(A, coarse ? coarse_tri(pr) : pr->tri, pr->P, pr->K, X, ldx, F, ldf, Y, ldy, st);
}

sg_status fp32_values(sg_problem* pr) {
  const bool generated = pr->apply_mode != 1 && jit_eligible(pr);
  if (!generated || !jit_config(pr, 0).flux || (pr->solver && !solver_edge(pr)))
    SG_TRY(ell_f32(pr->fine, pr->K, nullptr));
  if (!pr->solver) return SG_OK;
  const bool edge = jit_eligible(pr) && jit_config(pr, 1).flux;
  if (edge) SG_TRY(coarse_edge_prepare(pr));
  return edge && generated ? SG_OK : ell_f32(coarse_ell(pr), pr->K, nullptr);
}

sg_status apply_prepare32(sg_problem* pr, bool coarse, cudaStream_t st) {
  if (pr->apply_mode != 1 && jit_eligible(pr)) {
    const int which = fp32_family(pr, coarse, true);
    SG_TRY(jit_apply_build(pr, which));
    if (jit_config(pr, which).flux) return SG_OK;
  }
  return ell_f32(coarse ? coarse_ell(pr) : pr->fine, pr->K, st);
}

template sg_status apply_any<double>(sg_problem*, bool, const double*, int64_t, const double*, int64_t, double*,
                                     int64_t, cudaStream_t, bool);
template sg_status apply_any<float>(sg_problem*, bool, const float*, int64_t, const float*, int64_t, float*,
                                    int64_t, cudaStream_t, bool);

template <typename T>
sg_status apply_op(sg_problem* pr, bool coarse, const T* X, int64_t ldx, const T* F, int64_t ldf, T* Y,
                   int64_t ldy, cudaStream_t st, bool solver) {
  if (sizeof(T) == 8) SG_TRY(asm_prepare(pr, coarse, st));
  size_t slot = 0;
  const bool on = pr->prof.on;
  if (on) SG_TRY(pr->prof.begin((coarse ? 2 : 0) + (sizeof(T) == 8 ? 1 : 0), st, slot));
  SG_TRY(apply_any<T>(pr, coarse, X, ldx, F, ldf, Y, ldy, st, solver));
  if (on) SG_TRY(pr->prof.end(slot, st));
  return SG_OK;
}

template sg_status apply_op<double>(sg_problem*, bool, const double*, int64_t, const double*, int64_t, double*,
                                    int64_t, cudaStream_t, bool);
template sg_status apply_op<float>(sg_problem*, bool, const float*, int64_t, const float*, int64_t, float*,
                                   int64_t, cudaStream_t, bool);

template sg_status apply_ell<double>(const Ell&, const TripleTables&, int, int, const double*, int64_t,
                                     const double*, int64_t, double*, int64_t, cudaStream_t);
template sg_status apply_ell<float>(const Ell&, const TripleTables&, int, int, const float*, int64_t,
                                    const float*, int64_t, float*, int64_t, cudaStream_t);

}  // namespace sg
