// Internal declarations of libsg (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "sg.h"

namespace sg {

void set_error(const std::string& msg);
// process-wide count of kernel launches made by the library
void note_launch();
// adds n (possibly negative) to the launch count: kernels executed inside
// graphs, minus kernel nodes counted while a graph was being recorded
void note_launches(int64_t n);
int64_t launch_count();
int64_t launch_count();

#define SG_CUDA(call)                                                                    \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess) {                                                             \
      ::sg::set_error(std::string(#call) + ": " + cudaGetErrorString(e_));               \
      return SG_ERR_CUDA;                                                                \
    }                                                                                    \
  } while (0)

#define SG_TRY(call)                    \
  do {                                  \
    sg_status s_ = (call);              \
    if (s_ != SG_OK) return s_;         \
  } while (0)

#define SG_ARG(cond, msg)               \
  do {                                  \
    if (!(cond)) {                      \
      ::sg::set_error(msg);             \
      return SG_ERR_ARG;                \
    }                                   \
  } while (0)

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Device buffer owned by a handle.
struct DevBuf {
  void* ptr = nullptr;
  size_t bytes = 0;
  DevBuf() = default;
  DevBuf(const DevBuf&) = delete;
  DevBuf& operator=(const DevBuf&) = delete;
  DevBuf(DevBuf&& o) noexcept : ptr(o.ptr), bytes(o.bytes) {
    o.ptr = nullptr;
    o.bytes = 0;
  }
  DevBuf& operator=(DevBuf&& o) noexcept {
    if (this != &o) {
      free_();
      ptr = o.ptr;
      bytes = o.bytes;
      o.ptr = nullptr;
      o.bytes = 0;
    }
    return *this;
  }
  ~DevBuf() { free_(); }
  sg_status alloc(size_t nbytes);
  void free_();
  template <typename T> T* as() const { return static_cast<T*>(ptr); }
};

template <typename T> inline T* dp(const DevBuf& b) { return static_cast<T*>(b.ptr); }

// ELL ("sliced by slot") storage of a family of K matrices sharing one
// pattern with at most S entries per row: col[s * ldr + r] and
// val[(k * S + s) * ldr + r].  Padding entries carry col = r, value 0.
struct Ell {
  int S = 0;
  int64_t n = 0, ldr = 0;
  DevBuf col;      // int32 S x ldr
  DevBuf v64;      // double K x S x ldr
  mutable DevBuf v32;  // float  K x S x ldr, rounded from v64 where the slot form runs (ell_f32)
};

// The same family in the edge form: one conductance per edge of a mesh of
// N x N cells, in the order the generated kernel reads them.  Tile t of a
// node row j holds the horizontal edges (e, j)-(e + 1, j), e = 31 t + lane,
// of its 32 lanes (the last one again in the next tile) and the vertical
// edges (e + 1, j)-(e + 1, j + 1) above them, every position kk of the
// kernel's order of input terms (EdgeTerms):
//     v[((((j ntile + t) 2 + vertical) KT / 4 + kk / 4) 32 + lane) 4 + kk % 4],  ntile = ceil(N / 31),
// KT a multiple of 4, the values scaled as the kernel wants them (EdgeTerms).
struct EdgeVals {
  int N = 0;
  DevBuf v32, v64;  // v64: nonlinear operators only
};
// Where the conductances of input term k go: positions pos[off[k]] ..
// pos[off[k + 1] - 1] of KT.
struct EdgeTerms {
  int KT = 0, R = 1;  // positions; turns of the kernel's loop over orbits (KT / R positions each)
  DevBuf off, pos;        // int32 K + 1, KT
  DevBuf term;            // int32 KT: the term at a position, -1 for padding
  DevBuf scale;           // double K: factor of the stored conductances
  DevBuf scale2;          // float2 K: the same as hi + lo
};

// The Galerkin operator of an N x N mesh with each edge's P x P block summed
// once (FP64), B_ab^e = sum_k g_kab w_k(e) (symmetric: a <= b stored, packed
// row by row), in the order the apply reads them: the node rows are cut into
// strips of `strip` rows, the strips' N edge columns laid side by side, and
// tile t holds columns 31 t + lane (the last one again in the next tile);
// visit 0 of a tile is the vertical edges below the strip's first row, visits
// 2 k + 1 and 2 k + 2 the horizontal edges of its row k and the vertical ones
// above,
//     c[((t (2 strip + 1) + visit) npair + pair) 32 + lane],
// one contiguous run per tile.  Column e of a strip: the horizontal edge
// (e, j)-(e + 1, j), the vertical edges of node column e + 1.  Built on demand
// for FP64 applies.
struct AsmBlocks {
  int N = 0, npair = 0, strip = 1, groups = 1;
  bool tried = false;  // the policy was applied (built or declined)
  DevBuf c;
};

// The fine operator in the edge-flux form with each edge's P x P block
// summed once, B_ab^e = sum_k g_kab w_k(e) (symmetric: a <= b stored,
// packed row by row), each entry split into two FP32 numbers hi + lo;
// layout [npair][lde].  A row of the operator is sum over its four edges of
// B^e (x_r - x_neighbour), the neighbour's term dropped on the Dirichlet
// boundary.  Built on demand for the refinement residuals.
struct FluxDf {
  int npair = 0;
  int64_t lde = 0;
  bool tried = false;  // the policy was applied (built or declined)
  DevBuf b;            // float2 [npair][lde]
  DevBuf xs;           // float2 [P][ldr]: the split iterate
};

struct SolverState;
void solver_free(sg_problem* pr);
struct NewtonWork;
void newton_free(sg_problem* pr);
struct Cnn;
void cnn_free(sg_problem* pr);

// Triple products re-ordered by output mode a, then k, then b, split into
// chunks of input terms [c*kc, (c+1)*kc) for the shared-memory apply.
struct TripleTables {
  int kc = 0, nchunk = 0;
  DevBuf tk, tb;   // int32 T
  DevBuf g64, g32; // T
  DevBuf off;      // int32 P x (nchunk + 1)
};

// Optional per-launch timing (bench mode): CUDA events bracket each launch
// or phase on its stream; read() sums the elapsed times per kind.  Kernel
// kinds: 0 fine apply FP32, 1 fine apply FP64, 2 coarse apply FP32, 3
// coarse apply FP64, 4 RAS local solve FP32, 5 RAS local solve FP64.
// Phase kinds of the host-driven solve (a phase holds the kernels it
// launches, so kinds 4 and 5 lie inside kind 6): 6 smoother, 7 coarse
// correction (restriction, coarse GMRES graph, interpolation), 8 Arnoldi
// step (Gram-Schmidt, Givens rotation, normalisation), 9 refinement step
// bookkeeping (FP64 residual norm, conversion to FP32, the update of x).
constexpr int kProfKinds = 10;
struct Profiler {
  bool on = false;
  struct Rec {
    cudaEvent_t a = nullptr, b = nullptr;
    int kind = 0;
  };
  std::vector<Rec> pool;
  size_t used = 0;
  sg_status begin(int kind, cudaStream_t st, size_t& slot);
  sg_status end(size_t slot, cudaStream_t st);
  sg_status read(int kind, int64_t* launches, double* ms);
  void reset() { used = 0; }
  ~Profiler();
};

// Brackets a phase with profiler events when the profiler is on (errors of
// the event calls are ignored: timing never fails a solve).
struct ProfScope {
  Profiler* p;
  cudaStream_t st;
  size_t slot = 0;
  bool on;
  ProfScope(Profiler* p_, int kind, cudaStream_t st_) : p(p_), st(st_), on(p_ && p_->on) {
    if (on && p->begin(kind, st, slot) != SG_OK) on = false;
  }
  void stop() {
    if (on) p->end(slot, st);
    on = false;
  }
  ~ProfScope() { stop(); }
};

// Register-specialised apply compiled at setup time (sg_jit.cpp).  Four
// families: which = 0 fine FP32, 1 coarse FP32, 2 fine FP64, 3 coarse FP64,
// and of the library's own: 4 and 5, the nonlinear operators in FP32 and FP64
// (edge form), 6 the fine FP32 operator of solves in the slot form
// (solver_edge).
constexpr int kJitFamilies = 4;
constexpr int kJitAllFamilies = 7;
constexpr int kJitMaxP = 128;
constexpr int kJitGeneratorVersion = 12;  // bump when the generated code changes
constexpr int64_t kJitMaxT = 40000;
struct JitConfig {
  int rows = 1;        // rows per thread (2: paired FP32 FMA)
  int groups = 1;      // output groups (warp groups of 4 warps)
  int igroups = 1;     // input groups (partial sums meet in shared memory)
  int sgroups = 1;     // stencil-slot groups (partial sums meet in shared memory)
  int prefetch = 8;    // input terms loaded ahead
  int min_blocks = 1;  // CTAs per SM requested from the register allocator
  int stages = 0;      // 0: matrix values prefetched into registers; >= 2: staged through shared
                       // memory by cp.async in blocks of `prefetch` terms, stages - 1 blocks ahead
  int cgroups = 1;     // output groups as separate 128-thread CTAs (no register cap from wide CTAs)
  int warps = 4;       // warps per group (rows per group = 32 x warps x rows): narrow groups keep
                       // several slot or input groups within one register-rich CTA
  int flux = 0;        // 1: edge form (FP32 families): each edge's flux sum_k w_k G_k (x_hi - x_lo)
                       // formed once, conductances stored once per edge
  int strip = 4;       // edge form: node rows a lane marches over
};
struct JitApply {
  cudaLibrary_t lib = nullptr;
  cudaKernel_t kern = nullptr;
  bool from_cache = false;
  double compile_s = 0.0;
};

}  // namespace sg

struct sg_problem {
  int device = 0;
  int N = 0, L = 0, p = 0, q = 0, P = 0, K = 0;
  int64_t n = 0, nnzA = 0, T = 0, E = 0;
  double sigma2 = 0, bx = 0, by = 0, g0 = 0;
  std::vector<int32_t> mi_out, mi_in;  // P x L, K x L
  std::vector<int32_t> kab;            // T x 3, ordered k, a, b
  std::vector<int64_t> num;            // T
  std::vector<double> g;               // T
  std::vector<double> gfield;          // L x E
  std::vector<int32_t> rowptr, colidx; // shared CSR pattern
  std::vector<double> b;               // load vector (n)
  std::vector<double> a0;              // A_0 values on the CSR pattern (host)

  sg::Ell fine;                        // A_k on the device
  sg::TripleTables tri;
  int64_t ld = 0;                      // internal leading dimension of blocks
  sg::SolverState* solver = nullptr;   // preconditioner + solver workspaces
  sg::Cnn* cnn = nullptr;              // learned smoother network
  sg::NewtonWork* nl = nullptr;        // nonlinear problem: coefficients, operators, triple lists
  sg::DevBuf gfield_dev;               // KL modes at the element centroids
  sg::DevBuf mi_in_dev, isf_dev;       // input multi-indices, 1 / sqrt(k!) (element_coefficients)
  sg::Profiler prof;
  sg::JitApply* jit[sg::kJitAllFamilies] = {};     // specialised apply per family (fine/coarse x f32/f64)
  sg::JitConfig jit_cfg[sg::kJitAllFamilies];
  bool jit_cfg_set[sg::kJitAllFamilies] = {};
  bool jit_cfg_user[sg::kJitAllFamilies] = {};  // configured or tuned by the program
  sg::DevBuf mdot_partial, mdot_counter;  // scratch of sg_mdot
  int apply_mode = 0;                  // 0 auto, 1 shared-memory kernel, 2 specialised
  sg::AsmBlocks asm_fine;              // assembled FP64 blocks of the fine operator
  sg::EdgeVals edge;                   // edge form of the fine operator (FP32 conductances)
  sg::EdgeTerms edge_terms;            // order of the input terms in the edge form
  bool flux_allowed = true;            // fine FP32 applies may use the edge form
  int wait_limit = 1 << 22;            // mbarrier polls of a tcgen05 completion wait
  int asm_mode = 0;                    // FP64 applies: 0 auto, 1 never assembled, 2 always
  sg::FluxDf fdf;                      // double-FP32 edge blocks of the fine operator
  int res_mode = 0;                    // refinement residuals: 0 auto, 1 FP64 applies, 2 double-FP32 edge blocks
};

namespace sg {
// setup helpers (sg_setup.cpp)
std::vector<int32_t> multi_indices(int L, int p);
// <He_a He_b He_c> (integer, textbook linearisation formula)
int64_t he_triple_1d(int a, int b, int c);
sg_status build_host(sg_problem* pr, const sg_kl_desc* kl);
// device assembly (sg_assemble.cu)
sg_status assemble_fine(sg_problem* pr);
// lognormal input coefficients c_bar_k(e) of terms [k0, k0 + kn) at every
// element, written as out[(k - k0) E + e] (FP64 device array) on `st`; the
// field modes and index tables go to the device on the first call
sg_status gfield_upload(sg_problem* pr);
sg_status element_coefficients(sg_problem* pr, int k0, int kn, double* out, cudaStream_t st);
// the edge conductances of every input term in FP64, w[k * vkst + e] (the
// edge numbering of EdgeVals); synchronous
sg_status flux_values64(sg_problem* pr, double* w, int64_t vkst);
// FP32 conductances of the coarse operator R_0 A_k R_0^T on the nested 2h
// mesh (its triangles carry the mean of the four fine triangles inside);
// synchronous
sg_status coarse_edge_build(sg_problem* pr, EdgeVals& out);
// storage of the edge form on a mesh of N x N cells (either precision), and
// its values from coefficients [kn][2 N^2] over the triangles of that mesh,
// input terms [k0, k0 + kn); v32 and v64 where allocated
sg_status edge_alloc(const sg_problem* pr, int N, bool f32, bool f64, EdgeVals& out);
template <typename Tc>
sg_status edge_values(const sg_problem* pr, const Tc* coef, int k0, int kn, EdgeVals& out, cudaStream_t st);
// the same for all terms at once
template <typename Tc>
sg_status edge_values_all(const sg_problem* pr, const Tc* coef, EdgeVals& out, cudaStream_t st);
// the FP32 five- or seven-slot values of an ELL family (rounded from the
// FP64 ones when they are not there yet, see fp32_values; synchronous then,
// never while `st` is capturing)
sg_status ell_f32(const Ell& A, int K, cudaStream_t st);
sg_status build_triple_tables(sg_problem* pr, TripleTables& t, int S);
// apply (sg_apply.cu)
template <typename T>
sg_status apply_ell(const Ell& A, const TripleTables& tri, int P, int K, const T* X, int64_t ldx,
                    const T* F, int64_t ldf, T* Y, int64_t ldy, cudaStream_t st);
std::string jit_apply_source(const sg_problem* pr, const JitConfig& c, bool fp64 = false);
std::string jit_edge_source(const sg_problem* pr, const JitConfig& c, bool fp64);
JitConfig jit_default_config(const sg_problem* pr, int which);
JitConfig jit_slot_config(const sg_problem* pr, int which);  // the same in the five-slot form
// turns of the edge form's loop, and the input term at each position of its
// conductance blocks
int jit_edge_rotations(const sg_problem* pr);
std::vector<int> jit_edge_terms(const sg_problem* pr);  // -1: padding
std::vector<double> jit_edge_scale(const sg_problem* pr);
// the configuration in use (or to be used) by one family
JitConfig jit_config(const sg_problem* pr, int which);
size_t jit_smem_bytes(const sg_problem* pr, const JitConfig& c, bool fp64 = false);
sg_status jit_autotune(sg_problem* pr, int which, int force, double* best_ms);
sg_status jit_apply_build(sg_problem* pr, int which);
void jit_free(sg_problem* pr, int which);
sg_status jit_configure(sg_problem* pr, int which, const JitConfig& c);
// the form a family runs on untuned becomes the program's own choice (solver_edge)
sg_status jit_keep(sg_problem* pr, int which);
bool jit_eligible(const sg_problem* pr);
sg_status jit_apply_launch(sg_problem* pr, int which, const Ell& A, const double* X, int64_t ldx, const double* F,
                           int64_t ldf, double* Y, int64_t ldy, cudaStream_t st);
sg_status jit_apply_launch(sg_problem* pr, int which, const Ell& A, const float* X, int64_t ldx, const float* F,
                           int64_t ldf, float* Y, int64_t ldy, cudaStream_t st);
// the same over the edge form (the family's configuration has flux = 1)
template <typename T>
sg_status jit_edge_launch(sg_problem* pr, int which, const EdgeVals& A, const T* X, int64_t ldx, const T* F,
                          int64_t ldf, T* Y, int64_t ldy, cudaStream_t st);
// Whether FP32 solves run on the edge form: what the program configured or
// tuned for the fine family, else P <= 48.  A mixed solve that stops at a
// relative residual of 1e-8 carries the rounding error of its FP32 operator:
// 1.1e-9 of the solution at 384^2, P = 70 in the five-slot form, 2e-11 in the
// edge form (below 2e-11 in either up to P = 35).  Above the line untuned
// handles keep the five-slot form and with it the solutions they have
// returned all along, digit for digit; the edge form is nearer the exact
// solution and several times faster (345 us against 1.29 ms an apply at that
// size), and sg_apply_flux(prob, 1) selects it.
bool solver_edge(const sg_problem* pr);
// whether coarse solves use the coarse edge form and the folded V-cycle
// (sg_precond_setup decides it once, Precond::coarse_edge): in solves that use
// the edge form, and (untuned) while N p <= 800.  A coarse
// solve to the default tolerance (1e-5) in FP32 returns the rounding error of
// its operator amplified by the condition of the coarse matrix: the two
// forms' corrections differ by 1.2e-5 at 256^2, p = 3, 1.5e-5 at 320^2, p = 3
// and 1.6e-5 at 256^2, p = 4 (1.0e-5 at 200^2, p = 3, 5e-6 at 256^2, p = 2),
// and beyond the line by more than FP32 results may move.
bool coarse_edge_form(const sg_problem* pr);
// the FP32 slot values of the operators that run on the slot form (and the
// coarse conductances where that operator runs on the edge form), with the
// handle, its preconditioner or the choice of the form: a first apply may be
// captured and neither allocates nor waits.  Synchronous.
sg_status fp32_values(sg_problem* pr);
// FP32 values the applies of a solve need, built before any capture
sg_status apply_prepare32(sg_problem* pr, bool coarse, cudaStream_t st);
// assembled FP64 blocks (sg_apply.cu): build per the problem's policy (no-op
// once tried; never while `st` is capturing), and the apply over them
sg_status asm_prepare(sg_problem* pr, bool coarse, cudaStream_t st);
// (k, g_kab) list of every packed pair a <= b (pair index a P - a (a - 1) / 2
// + b - a): pair q owns entries [pptr[q], pptr[q + 1]) of pk, pg
void pair_lists(const sg_problem* pr, std::vector<int>& pptr, std::vector<int>& pk, std::vector<double>& pg);
// refinement residuals (sg_resid_df.cu): the double-FP32 edge blocks built
// per the problem's policy (no-op once tried; never while `st` is
// capturing), and R = F - A X (FP64 in and out) over them, or with the FP64
// apply when they are not built
sg_status resid_prepare(sg_problem* pr, cudaStream_t st);
sg_status resid_df(sg_problem* pr, const double* F, int64_t ldf, const double* X, int64_t ldx, double* R,
                   int64_t ldr, cudaStream_t st);
sg_status refine_residual(sg_problem* pr, const double* F, int64_t ldf, const double* X, int64_t ldx, double* R,
                          int64_t ldr, cudaStream_t st);
sg_status apply_asm64(const sg_problem* pr, const AsmBlocks& B, const double* X, int64_t ldx, const double* F,
                      int64_t ldf, double* Y, int64_t ldy, cudaStream_t st);
// (solver: the form FP32 solves use, solver_edge)
// the operator apply without timing: assembled blocks (FP64, when built),
// else the specialised kernel, else the shared-memory kernel
template <typename T>
sg_status apply_any(sg_problem* pr, bool coarse, const T* X, int64_t ldx, const T* F, int64_t ldf, T* Y,
                    int64_t ldy, cudaStream_t st, bool solver = false);
// apply_ell on the fine (coarse = false) or coarse family of a problem,
// timed when the problem's profiler is on
template <typename T>
sg_status apply_op(sg_problem* pr, bool coarse, const T* X, int64_t ldx, const T* F, int64_t ldf, T* Y,
                   int64_t ldy, cudaStream_t st, bool solver = false);
}  // namespace sg
