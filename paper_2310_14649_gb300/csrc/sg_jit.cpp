// Register-specialised Galerkin apply (Sec. 2.1, Eq. Galerkin_L_exp):
//     y_r[a] = sum_s sum_{(k,a,b)} v_k^{r,s} g_kab x_{col(r,s)}[b].
//
// The triple list depends only on (L, p, q), so at setup the library writes
// a CUDA kernel in which every nonzero g_kab is an immediate operand and
// every accumulator y[a] and gathered value x[b] lives in a named register.
// Per stencil slot a thread gathers the P values of its rows' neighbours,
// then streams the K matrix values of that slot (coalesced across the warp:
// lanes hold consecutive rows) and, for each input term k, updates the
// outputs coupled to it:  y_a += v_k * (sum_b g_kab x_b).
//
// Tile shape (chosen by the autotuner, cached per problem shape):
//   R  rows per thread: 1, or 2 adjacent rows packed in float2 registers
//      and updated with the paired FP32 FMA of sm_100+ (one instruction for
//      two rows; matrix values loaded as 8-byte pairs);
//   H  output groups: the P outputs are split into H contiguous ranges of
//      about T/H triples each, one range per group of 4 warps, so the
//      registers per thread stay bounded for large P;
//   HI input groups: the gathered x[b] are split into HI ranges as well;
//      each (output, input) group accumulates partial sums that meet in
//      shared memory, in a fixed order, before the single write of Y;
//   SG slot groups: the stencil slots are dealt round-robin to SG groups
//      (more threads for small row counts such as the coarse operator);
//   pf input terms whose values are loaded ahead of use;
//   mb CTAs per SM requested from the register allocator.
// Kernels are compiled for sm_103a with NVRTC and cached on disk by a hash
// of their source.  The same kernel serves the fine (5 slots) and the
// coarse (7 slots) family.
#include <nvrtc.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <sstream>
#include <sys/stat.h>
#include <unistd.h>

#include "sg_solver.h"

namespace sg {

namespace {

uint64_t fnv1a(const std::string& s) {
  uint64_t h = 1469598103934665603ull;
  for (unsigned char c : s) {
    h ^= c;
    h *= 1099511628211ull;
  }
  return h;
}

std::string cache_dir() {
  const char* env = std::getenv("SG_JIT_CACHE");
  if (env && *env) return env;
  const char* home = std::getenv("HOME");
  return std::string(home && *home ? home : "/tmp") + "/.cache/sg_gb300";
}

void mkdirs(const std::string& path) {
  std::string cur;
  std::stringstream ss(path);
  std::string part;
  if (!path.empty() && path[0] == '/') cur = "/";
  while (std::getline(ss, part, '/')) {
    if (part.empty()) continue;
    cur += part + "/";
    mkdir(cur.c_str(), 0755);
  }
}

std::string hexf(float g) {
  uint32_t u;
  std::memcpy(&u, &g, 4);
  char b[16];
  std::snprintf(b, sizeof b, "0x%08x", u);
  return b;
}

std::string hexd(double g) {
  uint64_t u;
  std::memcpy(&u, &g, 8);
  char b[24];
  std::snprintf(b, sizeof b, "0x%016llxull", (unsigned long long)u);
  return b;
}

// contiguous output ranges [lo_h, hi_h) with about T/H triples each
std::vector<int> output_split(const sg_problem* pr, int H) {
  std::vector<int64_t> per_a(pr->P, 0);
  for (int64_t t = 0; t < pr->T; ++t) per_a[pr->kab[3 * t + 1]]++;
  std::vector<int> cut(H + 1, pr->P);
  cut[0] = 0;
  int64_t acc = 0;
  int h = 1;
  for (int a = 0; a < pr->P && h < H; ++a) {
    acc += per_a[a];
    if (acc * H >= int64_t(h) * pr->T) cut[h++] = a + 1;
  }
  for (int i = 1; i <= H; ++i) cut[i] = std::max(cut[i], cut[i - 1]);
  return cut;
}

// H output groups of about T / H triples for the split into separate CTAs,
// outputs that share input terms together: a group reads only the values of
// its own input terms (the union over its outputs), so every output joins
// the group whose union it enlarges least
std::vector<int> output_groups(const sg_problem* pr, int H) {
  const int P = pr->P;
  std::vector<std::vector<int>> terms(P);
  std::vector<int64_t> weight(P, 0);
  for (int64_t t = 0; t < pr->T; ++t) {
    const int k = pr->kab[3 * t], a = pr->kab[3 * t + 1];
    if (terms[a].empty() || terms[a].back() != k) terms[a].push_back(k);
    ++weight[a];
  }
  std::vector<int> group(P, -1);
  int64_t acc = 0;
  int left = P;
  for (int h = 0; h < H && left > 0; ++h) {
    std::vector<char> have(pr->K, 0);
    for (bool first = true; left > 0 && (first || h == H - 1 || acc * H < int64_t(h + 1) * pr->T); first = false) {
      int best = -1;
      int64_t cost = 0;
      for (int a = 0; a < P; ++a) {
        if (group[a] >= 0) continue;
        int64_t c = 0;
        for (int k : terms[a]) c += !have[k];
        if (first) c = -weight[a];  // a group starts from the heaviest output left
        if (best < 0 || c < cost) {
          best = a;
          cost = c;
        }
      }
      group[best] = h;
      acc += weight[best];
      --left;
      for (int k : terms[best]) have[k] = 1;
    }
  }
  return group;
}

}  // namespace

std::string jit_apply_source(const sg_problem* pr, const JitConfig& c, bool fp64) {
  // output groups either as 4-warp groups of one CTA (partial sums meet in
  // shared memory, registers capped by the CTA width) or as separate
  // 128-thread CTAs, group by group over the grid: the CTAs on an SM run the
  // same group's code, which stays in the instruction cache
  const bool csplit = c.cgroups > 1;
  const int P = pr->P, K = pr->K, R = fp64 ? 1 : c.rows, HO = csplit ? c.cgroups : c.groups,
            HI = csplit ? 1 : c.igroups, SG = csplit ? 1 : c.sgroups, pf = c.prefetch;
  // FP64 family: the same code over double values, inputs and outputs, the
  // coefficients as exact double immediates
  const char* T = fp64 ? "double" : "float";
  const std::string Ts = T;
  const int mb = c.min_blocks, NG = HO * HI * SG, NPART = HI * SG, W = csplit ? 4 : c.warps;
  const std::vector<int> cut = output_split(pr, HO);
  const std::vector<int> cgrp = csplit ? output_groups(pr, HO) : std::vector<int>();
  std::vector<int> icut(HI + 1);
  for (int i = 0; i <= HI; ++i) icut[i] = int(int64_t(P) * i / HI);
  // triples grouped by k, then by a
  std::vector<std::map<int, std::vector<std::pair<int, double>>>> by_k(K);
  for (int64_t t = 0; t < pr->T; ++t) {
    int k = pr->kab[3 * t], a = pr->kab[3 * t + 1], b = pr->kab[3 * t + 2];
    by_k[k][a].push_back({b, fp64 ? pr->g[t] : double(float(pr->g[t]))});
  }
  // paired rows take their coefficients from the constant bank (the paired
  // FMA has no immediate operand)
  std::map<uint32_t, int> gslot;
  std::vector<float> gvals;
  auto gref = [&](double gd) -> std::string {
    if (fp64) return "GD(" + hexd(gd) + ")";
    const float g = float(gd);
    if (R == 1) return "G(" + hexf(g) + ")";
    uint32_t u;
    std::memcpy(&u, &g, 4);
    auto it = gslot.find(u);
    int id;
    if (it == gslot.end()) {
      id = int(gvals.size());
      gslot[u] = id;
      gvals.push_back(g);
    } else {
      id = it->second;
    }
    return "gq2[" + std::to_string(id) + "]";
  };
  const char* ty = R == 2 ? "float2" : T;
  std::ostringstream body;
  std::string staged_table;
  // slot groups alone run the same code from different first slots: one
  // body with the slot offset taken from the group index (separate unrolled
  // bodies per group multiply the instruction footprint)
  const bool slot_only = !csplit && HO == 1 && HI == 1 && SG > 1;
  for (int g = 0; g < (slot_only ? 1 : NG); ++g) {
    const int ho = g / (HI * SG), hi = (g / SG) % HI, sgi = g % SG;
    const int lo = cut[ho], up = cut[ho + 1], blo = icut[hi], bup = icut[hi + 1];
    auto in_out = [&](int a) { return csplit ? cgrp[a] == ho : a >= lo && a < up; };
    auto in_grp = [&](int a, int b) { return in_out(a) && b >= blo && b < bup; };
    std::vector<int> ks;
    std::vector<char> need_b(P, 0), has_a(P, 0);
    for (int k = 0; k < K; ++k) {
      bool any = false;
      for (const auto& ga : by_k[k])
        for (const auto& e : ga.second)
          if (in_grp(ga.first, e.first)) {
            any = true;
            need_b[e.first] = 1;
            has_a[ga.first] = 1;
          }
      if (any) ks.push_back(k);
    }
    if (slot_only)
      body << "  {\n";
    else
      body << "  " << (g ? "else " : "") << "if (grp == " << g << ") {\n";
    for (int a = 0; a < P; ++a)
      if (has_a[a]) body << "    " << ty << " y" << a << (R == 2 ? " = make_float2(0.f, 0.f);\n" : (fp64 ? " = 0.0;\n" : " = 0.f;\n"));
    body << "#pragma unroll 1\n"
            "    for (int s = " << (slot_only ? std::string("grp") : std::to_string(sgi)) << "; s < S; s += " << SG
         << ") {\n";
    body << "      const " << Ts << "* xp0 = X + col[(long long)s * ldr + rr];\n";
    if (R == 2) body << "      const float* xp1 = X + col[(long long)s * ldr + rr + 1];\n";
    for (int b = 0; b < P; ++b) {
      if (!need_b[b]) continue;
      if (R == 2)
        body << "      const float2 x" << b << " = make_float2(__ldg(xp0 + (long long)" << b
             << " * ldx), __ldg(xp1 + (long long)" << b << " * ldx));\n";
      else
        body << "      const " << Ts << " x" << b << " = __ldg(xp0 + (long long)" << b << " * ldx);\n";
    }
    const bool staged = c.stages >= 2;
    if (!staged) body << "      const " << Ts << "* vp = V + (long long)s * ldr + rr;\n";
    auto load = [&](int k) {
      if (R == 2)
        body << "      const float2 v" << k << " = __ldg(reinterpret_cast<const float2*>(vp + (long long)" << k
             << " * kst));\n";
      else
        body << "      const " << Ts << " v" << k << " = __ldg(vp + (long long)" << k << " * kst);\n";
    };
    const int nk = int(ks.size());
    // staged: blocks of KB input terms arrive in shared memory (cp.async,
    // stages - 1 blocks ahead, across slot boundaries); each thread reads
    // back only the values it copied, so no barrier is needed
    const int KB = std::max(1, pf);
    if (!staged)
      for (int i = 0; i < std::min(nk, pf); ++i) load(ks[i]);
    for (int i = 0; i < nk; ++i) {
      if (staged && i % KB == 0) {
        if (i) body << "      }\n";
        body << "      {\n        asm volatile(\"cp.async.wait_group " << (c.stages - 2) << ";\" ::: \"memory\");\n"
             << "        issue_blk(gb + " << (c.stages - 1) << ", S, V, ldr, kst, rr, vsm);\n"
             << "        const " << Ts << "* vb = vsm + (gb % " << c.stages << ") * " << KB * 128 << ";\n"
             << "        ++gb;\n";
        for (int q = i; q < std::min(nk, i + KB); ++q)
          body << "        const " << Ts << " v" << ks[q] << " = vb[" << (q - i) * 128 << "];\n";
      }
      if (!staged && i + pf < nk) load(ks[i + pf]);
      const int k = ks[i];
      for (const auto& ga : by_k[k]) {
        const int a = ga.first;
        std::vector<std::pair<int, double>> lst;
        for (const auto& e : ga.second)
          if (in_grp(a, e.first)) lst.push_back(e);
        if (lst.empty()) continue;
        const char* fma = R == 2 ? "__ffma2_rn" : (fp64 ? "fma" : "fmaf");
        if (lst.size() == 1 && lst[0].second == 1.0) {
          body << "      y" << a << " = " << fma << "(v" << k << ", x" << lst[0].first << ", y" << a << ");\n";
          continue;
        }
        if (R == 2)
          body << "      { float2 t = __fmul2_rn(x" << lst[0].first << ", " << gref(lst[0].second) << ");";
        else
          body << "      { " << Ts << " t = x" << lst[0].first << " * " << gref(lst[0].second) << ";";
        for (size_t e = 1; e < lst.size(); ++e)
          body << " t = " << fma << "(x" << lst[e].first << ", " << gref(lst[e].second) << ", t);";
        body << " y" << a << " = " << fma << "(v" << k << ", t, y" << a << "); }\n";
      }
    }
    if (staged && nk > 0) body << "      }\n";
    body << "    }\n";
    if (staged) {
      // the table of input terms per block, for the copy helper
      std::ostringstream tab;
      const int NB = (nk + KB - 1) / KB;
      tab << "#define STG_NB " << NB << "\n__constant__ int c_ktab[" << std::max(1, NB * KB) << "] = {";
      for (int e = 0; e < NB * KB; ++e) tab << (e ? ", " : "") << (e < nk ? ks[e] : -1);
      if (NB * KB == 0) tab << "-1";
      tab << "};\n";
      staged_table = tab.str();
    }
    if (csplit) {  // this CTA's outputs, written straight from registers
      for (int a = 0; a < P; ++a) {
        if (!in_out(a)) continue;
        const std::string val = has_a[a] ? "y" + std::to_string(a) : std::string(fp64 ? "0.0" : "0.f");
        body << "    if (r < n) Y[(long long)" << a << " * ldy + r] = F ? F[(long long)" << a << " * ldf + r] - " << val
             << " : " << val << ";\n";
      }
      body << "  }\n";
      continue;
    }
    // partial sums of the input and slot groups meet in shared memory, in
    // group order; outputs this group never touches contribute zero
    for (int a = lo; a < up; ++a) {
      if (!has_a[a]) {
        for (int q = 0; q < R; ++q) body << "    part[" << a << " * " << 32 * W * R << " + lrow + " << q << "] = 0;\n";
        continue;
      }
      for (int q = 0; q < R; ++q) {
        const std::string val = R == 2 ? ("y" + std::to_string(a) + (q ? ".y" : ".x")) : ("y" + std::to_string(a));
        body << "    part[" << a << " * " << 32 * W * R << " + lrow + " << q << "] = " << val << ";\n";
      }
    }
    body << "  }\n";
  }
  std::ostringstream os;
  os << "// generated: Galerkin apply, P=" << P << " K=" << K << " T=" << pr->T << " R=" << R << " groups=" << HO
     << "x" << HI << "x" << SG << " pf=" << pf << " mb=" << mb << (fp64 ? " fp64" : "") << "\n";
  os << (fp64 ? "#define GD(h) __longlong_as_double(h)\n" : "#define G(h) __int_as_float(h)\n");
  if (c.stages >= 2) {
    const int KB = std::max(1, pf);
    os << staged_table;
    os << "__device__ __forceinline__ void cpa(" << Ts << "* d, const " << Ts << "* s) {\n"
          "  const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(d));\n"
          "  asm volatile(\"cp.async.ca.shared.global [%0], [%1], " << (fp64 ? 8 : 4) << ";\" :: \"r\"(a), \"l\"(s) : \"memory\");\n"
          "}\n"
          "// copy block gb (slot gb / NB, terms c_ktab[(gb % NB) * KB ...]) of this thread's row\n"
          "__device__ __forceinline__ void issue_blk(int gb, int S, const " << Ts << "* V, long long ldr, long long kst,\n"
          "                                           int rr, " << Ts << "* vsm) {\n"
          "  if (gb < S * STG_NB) {\n"
          "    const int s = gb / STG_NB, b = gb - s * STG_NB;\n"
          "    const " << Ts << "* vp = V + (long long)s * ldr + rr;\n"
          "    " << Ts << "* d = vsm + (gb % " << c.stages << ") * " << KB * 128 << ";\n"
          "#pragma unroll\n"
          "    for (int i = 0; i < " << KB << "; ++i) {\n"
          "      const int k = c_ktab[b * " << KB << " + i];\n"
          "      if (k >= 0) cpa(d + i * 128, vp + (long long)k * kst);\n"
          "    }\n"
          "  }\n"
          "  asm volatile(\"cp.async.commit_group;\" ::: \"memory\");\n"
          "}\n";
  }
  if (R == 2 && !gvals.empty()) {
    // both halves of each pair carry the same coefficient bits
    os << "__constant__ unsigned long long gq_bits[" << gvals.size() << "] = {";
    for (size_t i = 0; i < gvals.size(); ++i) {
      const std::string h = hexf(gvals[i]).substr(2);
      os << (i ? ", " : "") << "0x" << h << h << "ull";
    }
    os << "};\n#define gq2 (reinterpret_cast<const float2*>(gq_bits))\n";
  }
  const int rows_cta = 32 * W * R;
  if (csplit) {
    os << "extern \"C\" __global__ void __launch_bounds__(128, " << mb << ") " << (fp64 ? "sg_k1_f64" : "sg_k1")
       << "(\n"
          "    const " << Ts << "* __restrict__ V, const int* __restrict__ col, long long ldr, int n, int S,\n"
          "    const " << Ts << "* __restrict__ X, long long ldx, const " << Ts << "* __restrict__ F, long long ldf,\n"
          "    " << Ts << "* __restrict__ Y, long long ldy) {\n"
          "  const int nt = (n + 127) / 128, grp = blockIdx.x / nt;\n"
          "  const int r = (blockIdx.x - grp * nt) * 128 + threadIdx.x;\n"
          "  const int rr = r < n ? r : n - 1;\n"
          "  const long long kst = (long long)S * ldr;\n";
    os << body.str();
    os << "}\n";
    return os.str();
  }
  os << "extern \"C\" __global__ void __launch_bounds__(" << 32 * W * NG << ", " << mb << ") "
     << (fp64 ? "sg_k1_f64" : "sg_k1") << "(\n"
        "    const " << Ts << "* __restrict__ V, const int* __restrict__ col, long long ldr, int n, int S,\n"
        "    const " << Ts << "* __restrict__ X, long long ldx, const " << Ts << "* __restrict__ F, long long ldf,\n"
        "    " << Ts << "* __restrict__ Y, long long ldy) {\n"
        "  extern __shared__ " << Ts << " smem[];\n"
        "  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;\n"
        "  const int grp = warp / " << W << ";\n"
        "  const int lrow = (warp % " << W << ") * "
     << 32 * R << " + lane * " << R << ";\n"
     << "  const int r = blockIdx.x * " << rows_cta << " + lrow;\n"
     << "  const int rr = r < n ? r : (n - 1) & ~" << (R - 1) << ";\n"
     << "  const long long kst = (long long)S * ldr;\n";
  if (NG == 1) {
    os << "  " << Ts << "* part = smem;\n  (void)part;\n";
    if (c.stages >= 2)
      os << "  " << Ts << "* vsm = smem + lrow;\n"
         << "  for (int g0 = 0; g0 < " << (c.stages - 1) << "; ++g0) issue_blk(g0, S, V, ldr, kst, rr, vsm);\n"
         << "  int gb = 0;\n";
    // single group: write straight from registers
    std::string b = body.str();
    // drop the shared-memory hand-off of the single group
    std::ostringstream direct;
    std::istringstream in(b);
    std::string line;
    while (std::getline(in, line)) {
      if (line.find("part[") != std::string::npos) continue;
      direct << line << "\n";
      if (line == "    }") {  // end of the slot loop: write the outputs
        for (int a = 0; a < P; ++a)
          for (int q = 0; q < R; ++q) {
            const std::string val = R == 2 ? ("y" + std::to_string(a) + (q ? ".y" : ".x")) : ("y" + std::to_string(a));
            direct << "    if (r + " << q << " < n) Y[(long long)" << a << " * ldy + r + " << q << "] = F ? F[(long long)"
                   << a << " * ldf + r + " << q << "] - " << val << " : " << val << ";\n";
          }
      }
    }
    os << direct.str();
  } else {
    os << "  " << Ts << "* part = smem + (size_t)(grp % " << NPART << ") * " << P * rows_cta << ";\n";
    os << body.str();
    os << "  __syncthreads();\n";
    os << "  for (int e = threadIdx.x; e < " << P * rows_cta << "; e += " << 32 * W * NG << ") {\n"
          "    const int a = e / "
       << rows_cta << ", lr = e - a * " << rows_cta << ";\n"
       << "    const int row = blockIdx.x * " << rows_cta << " + lr;\n"
       << "    if (row >= n) continue;\n"
          "    " << Ts << " acc = smem[e];\n";
    for (int q = 1; q < NPART; ++q) os << "    acc += smem[" << q * P * rows_cta << " + e];\n";
    os << "    Y[(long long)a * ldy + row] = F ? F[(long long)a * ldf + row] - acc : acc;\n  }\n";
  }
  os << "}\n";
  return os.str();
}

// The cyclic shift of the random variables by L / R places maps the multi-
// index sets onto themselves and keeps every triple product, so the triples
// fall into orbits of R (a few shorter).  EdgeOrder holds the shift as index
// maps, the input terms' orbits and one representative per triple orbit, its
// input term being the first of its orbit.
struct EdgeOrder {
  int R = 1, Kr = 0;                   // Kr: orbits, rounded up to a multiple of 4 (one 16-byte load a lane);
                                       // the conductance of sigma^s of orbit i's first lies at position s Kr + i
  std::vector<int> sig_out;            // sigma on output indices
  std::vector<double> fac;             // alpha! of the output indices
  struct Tri {
    int i, a, b;                       // orbit of the input term, output, input
    double g;                          // integer coefficient; a short orbit is visited several times, g split over them
  };
  std::vector<Tri> tri;                // ordered by i
};

static std::vector<double> index_factorials(const std::vector<int32_t>& mi, int L, int n) {
  std::vector<double> f(n, 1.0);
  for (int r = 0; r < n; ++r)
    for (int d = 0; d < L; ++d)
      for (int v = 2; v <= mi[int64_t(r) * L + d]; ++v) f[r] *= v;
  return f;
}

std::vector<double> jit_edge_scale(const sg_problem* pr) {
  std::vector<double> f = index_factorials(pr->mi_in, pr->L, pr->K);
  for (double& v : f) v = std::sqrt(v);
  return f;
}

static std::vector<int> shift_map(const std::vector<int32_t>& mi, int L, int by) {
  const int n = L > 0 ? int(mi.size()) / L : 1;
  std::vector<int> out(n, 0);
  if (L == 0) return out;
  std::map<std::vector<int32_t>, int> at;
  for (int r = 0; r < n; ++r) at[std::vector<int32_t>(mi.begin() + int64_t(r) * L, mi.begin() + int64_t(r + 1) * L)] = r;
  for (int r = 0; r < n; ++r) {
    std::vector<int32_t> v(L);
    for (int d = 0; d < L; ++d) v[d] = mi[int64_t(r) * L + (d + by) % L];
    out[r] = at.at(v);
  }
  return out;
}

// R: the smallest divisor of L that leaves at most kBody triples in the loop
// body.  Straight-line code beyond the SM's instruction cache (64 KB) stalls
// on instruction fetch: at P = 84 (14,600 instructions an edge) 11 of 12
// cycles (ncu, no_instruction), 2.4 ms an apply at 512^2 against 0.56 ms with
// R = 6.  Below that the shorter body still helps a little (P = 35 at 256^2:
// R = 1 39.7 us, 2 37.4 us, 4 36.6 us).
int jit_edge_rotations(const sg_problem* pr) {
  constexpr int64_t kBody = 1000;
  for (int R = 1; R <= pr->L; ++R)
    if (pr->L % R == 0 && pr->T / R <= kBody) return R;
  return std::max(1, pr->L);
}

// the orbits of the input terms: orbit of each, first of each, the shift
struct TermOrbits {
  std::vector<int> sig, orbit, first;
};
static TermOrbits term_orbits(const sg_problem* pr) {
  TermOrbits t;
  const int L = pr->L, R = jit_edge_rotations(pr);
  t.sig = shift_map(pr->mi_in, L, R > 1 ? L / R : 0);
  t.orbit.assign(pr->K, -1);
  for (int k = 0; k < pr->K; ++k) {
    if (t.orbit[k] >= 0) continue;
    for (int q = k; t.orbit[q] < 0; q = t.sig[q]) t.orbit[q] = int(t.first.size());
    t.first.push_back(k);
  }
  return t;
}

std::vector<int> jit_edge_terms(const sg_problem* pr) {
  const TermOrbits t = term_orbits(pr);
  const int R = jit_edge_rotations(pr), Kr = int(round_up(int64_t(t.first.size()), 4));
  std::vector<int> term(size_t(R) * Kr, -1);
  for (int i = 0; i < int(t.first.size()); ++i)
    for (int s = 0, k = t.first[i]; s < R; ++s, k = t.sig[k]) term[size_t(s) * Kr + i] = k;
  return term;
}

static EdgeOrder edge_order(const sg_problem* pr) {
  EdgeOrder o;
  const int L = pr->L, R = jit_edge_rotations(pr);
  o.R = R;
  const TermOrbits terms = term_orbits(pr);
  const std::vector<int>&si = terms.sig, &orbit = terms.orbit, &first = terms.first;
  const std::vector<double> fin = index_factorials(pr->mi_in, L, pr->K);
  o.fac = index_factorials(pr->mi_out, L, pr->P);
  o.sig_out = shift_map(pr->mi_out, L, R > 1 ? L / R : 0);
  o.Kr = int(round_up(int64_t(first.size()), 4));
  // one representative per triple orbit: the smallest (a, b) among the
  // members whose input term is the orbit's first
  std::map<std::array<int, 3>, EdgeOrder::Tri> reps;
  for (int64_t t = 0; t < pr->T; ++t) {
    int k = pr->kab[3 * t], a = pr->kab[3 * t + 1], b = pr->kab[3 * t + 2];
    const int i = orbit[k], k0 = first[i];
    std::array<int, 3> best{i, pr->P, pr->P};
    for (int s = 0; s < R; ++s) {
      if (k == k0) best = std::min(best, std::array<int, 3>{i, a, b});
      k = si[k];
      a = o.sig_out[a];
      b = o.sig_out[b];
    }
    // a! b! <He_k He_a He_b> / (a! b! k!) = the integer prod C(a, c) C(b, c) c!, c = (a + b - k) / 2
    const double g = double(pr->num[t]) / fin[pr->kab[3 * t]];
    auto it = reps.find(best);
    if (it == reps.end())
      reps[best] = {i, best[1], best[2], g};
    else
      it->second.g += g;  // equal over the orbit: its length times g
  }
  for (auto& e : reps) {
    e.second.g = R == 1 ? e.second.g : e.second.g / R;
    o.tri.push_back(e.second);
  }
  return o;
}

// terms per staged chunk (a multiple of 4): at most `prefetch`, and a turn has at least
// stages - 1 chunks (the copies run that far ahead, into the next turn at most); Kr > 0, so
// at least two stages
static int edge_stages(const JitConfig& c, int Kr) { return std::max(2, std::min(c.stages, Kr / 4 + 1)); }
static int edge_chunk(const JitConfig& c, int Kr) {
  return 4 * std::max(1, std::min(c.prefetch / 4, Kr / 4 / (edge_stages(c, Kr) - 1)));
}

// Edge form (structured mesh of N x N cells, conductances w_k(e) stored once
// per edge): a warp's 32 lanes hold 32 consecutive horizontal edges of one
// node row, lane e the node right of its edge, and march up a strip of
// `strip` node rows.  Per row a lane forms the flux f = sum_k w_k G_k
// (x_hi - x_lo) of its horizontal edge and of the vertical edge north of its
// node, each once:
//     y = f_west - f_east + f_south - f_north,
// f_east from the next lane by a shuffle, f_south kept from the row below
// (y waits in shared memory, a word per output and thread).  So a strip
// computes 2 strip + 1 edges for `strip` rows where the gathering form
// computed four per row (and the five-slot form five products); the last
// lane of a tile repeats the first edge of the next (31 nodes a tile).
//
// In the unnormalised chaos the coefficients are small integers, 1 for most
// triples: with x'_b = x_b / sqrt(b!), w'_k = sqrt(k!) w_k and f_a = f'_a /
// sqrt(a!), f'_a = sum n_kab w'_k x'_b.  Every distinct integer of an input
// term is multiplied onto its conductance once and each triple is then one
// FMA on registers: 2,600 instructions an edge at P = 35 against 3,751 for
// products formed per (term, output).  Where that exceeds
// the instruction cache the code of one representative per triple orbit (see
// EdgeOrder) runs R times, the registers of x and f moved along the shift
// after each turn.
//
// Conductances lie in the order a warp reads them, [row][tile][horizontal,
// vertical][turn][orbit / 4][32 lanes][4] (EdgeVals), and stream through a ring of
// `stages` chunks of `prefetch` terms in shared memory by 16-byte cp.async:
// eight copies replace 32 loads, no register waits on HBM, and a thread
// needs 2 P registers for x and f, so 8 to 16 warps a SM are resident.
std::string jit_edge_source(const sg_problem* pr, const JitConfig& c, bool fp64) {
  const int P = pr->P, HO = c.cgroups, W = c.warps, TY = c.strip, es = fp64 ? 8 : 4;
  const std::string Ts = fp64 ? "double" : "float", Z = fp64 ? "0.0" : "0.f", fma = fp64 ? "fma" : "fmaf";
  const EdgeOrder o = edge_order(pr);
  const int R = o.R, Kr = o.Kr, S = edge_stages(c, Kr), CB = edge_chunk(c, Kr), nch = (Kr + CB - 1) / CB;
  // output groups: whole orbits, about T / HO triples each
  std::vector<int64_t> per_a(P, 0);
  for (int64_t t = 0; t < pr->T; ++t) per_a[pr->kab[3 * t + 1]]++;
  std::vector<int> group(P, -1);
  {
    int64_t acc = 0;
    int h = 0;
    for (int a = 0; a < P; ++a) {
      if (group[a] >= 0) continue;
      while (h < HO - 1 && acc * HO >= int64_t(h + 1) * pr->T) ++h;
      for (int q = a; group[q] < 0; q = o.sig_out[q]) {
        group[q] = h;
        acc += per_a[q];
      }
    }
  }
  // 1 / sqrt(a!) as a factor in the source, nothing for 1
  auto scale = [&](int a) -> std::string {
    if (o.fac[a] == 1.0) return "";
    const double r = 1.0 / std::sqrt(o.fac[a]);
    return "G(" + (fp64 ? hexd(r) : hexf(float(r))) + ") * ";
  };
  std::ostringstream os;
  os << "// generated: Galerkin apply, edge form, P=" << P << " K=" << pr->K << " T=" << pr->T << " R=" << R
     << " groups=" << HO << " warps=" << W << " strip=" << TY << " chunk=" << CB << "x" << S << " mb=" << c.min_blocks
     << (fp64 ? " fp64" : "") << "\n"
     << "#define G(h) " << (fp64 ? "__longlong_as_double(h)" : "__int_as_float(h)") << "\n"
     << "typedef " << Ts << " T;\n"
     << "// `rows` terms (of 32 lanes) from global to shared memory, 16 bytes a lane and copy\n"
     << "template <int rows> __device__ __forceinline__ void chunk(unsigned dst, const T* src, int lane) {\n"
     << "  constexpr int pieces = rows * " << 2 * es << ";\n"
     << "#pragma unroll\n"
     << "  for (int u = 0; u < (pieces + 31) / 32; ++u)\n"
     << "    if (u * 32 + 32 <= pieces || u * 32 + lane < pieces)\n"
     << "      asm volatile(\"cp.async.cg.shared.global [%0], [%1], 16;\" :: \"r\"(dst + (u * 32 + lane) * 16),\n"
     << "                   \"l\"(reinterpret_cast<const char*>(src) + (u * 32 + lane) * 16) : \"memory\");\n"
     << "}\n"
     << "__device__ __forceinline__ void ld4(T (&v)[4], const T* p) {\n"
     << (fp64 ? "  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];\n"
                "  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;\n"
              : "  const float4 a = *reinterpret_cast<const float4*>(p);\n"
                "  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;\n")
     << "}\n"
     << "__device__ __forceinline__ void commit() { asm volatile(\"cp.async.commit_group;\" ::: \"memory\"); }\n"
     << "__device__ __forceinline__ void arrived() { asm volatile(\"cp.async.wait_group " << S - 2
     << ";\" ::: \"memory\"); __syncwarp(); }\n"
     << "extern \"C\" __global__ void __launch_bounds__(" << 32 * W << ", " << c.min_blocks << ") "
     << (fp64 ? "sg_k1_f64" : "sg_k1") << "(\n"
     << "    const T* __restrict__ V, int N, const T* __restrict__ X, long long ldx, const T* F, long long ldf,\n"
     << "    T* Y, long long ldy) {\n"
     << "  const int m = N - 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;\n"
     << "  const int grp = blockIdx.x % " << HO << ", ntile = (N + 30) / 31;\n"
     << "  const int q = (blockIdx.x / " << HO << ") * " << W << " + warp, st = q / ntile, tile = q - st * ntile;\n"
     << "  const int j0 = st * " << TY << " + 1;\n"
     << "  if (j0 > m) return;  // whole warps\n"
     << "  const int j1 = min(m, j0 + " << TY - 1 << "), e = 31 * tile + lane, c = e + 1;\n"
     << "  const bool own = lane < 31 && c <= m;\n"
     << "  extern __shared__ __align__(16) T sm[];\n"
     << "  T* y = sm + warp * " << 32 * (P + S * CB) << " + lane;  // [output of the group][32]\n"
     << "  T* ring = y - lane + " << 32 * P << " + 4 * lane;        // [stage][term / 4][32][4]\n"
     << "  const unsigned rs = static_cast<unsigned>(__cvta_generic_to_shared(ring - 4 * lane));\n"
     << "  int stg = 0;  // stage of the next chunk\n";
  for (int g = 0; g < HO; ++g) {
    std::vector<char> need_b(P, 0);
    std::vector<int> outs;  // outputs of the group
    for (int a = 0; a < P; ++a)
      if (group[a] == g) outs.push_back(a);
    std::vector<std::vector<EdgeOrder::Tri>> by_i(Kr);
    for (const auto& t : o.tri)
      if (group[t.a] == g) {
        by_i[t.i].push_back(t);
        // the register of b holds every member of its orbit in turn
        for (int q = t.b; !need_b[q]; q = o.sig_out[q]) need_b[q] = 1;
      }
    os << "  " << (g ? "else " : "") << "if (grp == " << g << ") {\n"
       << "    // even strips march up, odd ones down, so the edges two strips share are read at the same\n"
       << "    // time.  Marching up, visit v = 0 is the vertical edges below the strip, then per row come its\n"
       << "    // horizontal edges (v odd) and the vertical edges above its nodes (v even); marching down,\n"
       << "    // above and below change places.  row(v): node row of a horizontal visit, the row below the\n"
       << "    // edges of a vertical one.\n"
       << "    const bool up = !(st & 1);\n"
       << "    const T sg = up ? (T)1 : (T)-1;\n"
       << "    auto row = [&](int v) { return up ? j0 - 1 + ((v + 1) >> 1) : j1 - (v >> 1); };\n"
       << "    auto block = [&](int v) -> const T* {\n"
       << "      return V + (((long long)row(v) * ntile + tile) * 2 + (v & 1 ? 0 : 1)) * " << 32ll * R * Kr << ";\n"
       << "    };\n"
       << "    const int nv = 2 * (j1 - j0 + 1) + 1;\n"
       << "    const T* vp = block(0);\n";
    for (int u = 0; u < S - 1; ++u)
      os << "    chunk<" << std::min(CB, Kr - u * CB) << ">(rs + " << u * CB * 32 * es << ", vp + " << 32 * u * CB
         << ", lane); commit();\n";
    os << "#pragma unroll 1\n"
          "    for (int v = 0; v < nv; ++v) {\n"
          "      const int j = row(v);\n"
          "      const bool hor = v & 1, in = e < N && (hor || c <= m);\n"
          "      // the edge's end nodes: hi right of or above lo (rows of X), absent on the boundary\n"
          "      const int rhi = hor ? (j - 1) * m + c - 1 : j * m + c - 1;\n"
          "      const int rlo = hor ? rhi - 1 : rhi - m;\n"
          "      const bool bhi = in && (hor ? c <= m : j < m), blo = in && (hor ? e > 0 : j > 0);\n"
          "      const T* xh = X + (bhi ? rhi : 0);\n"
          "      const T* xl = X + (blo ? rlo : 0);\n";
    for (int b = 0; b < P; ++b)
      if (need_b[b])
        os << "      T x" << b << " = " << scale(b) << "((bhi ? __ldg(xh + " << b << "ll * ldx) : " << Z
           << ") - (blo ? __ldg(xl + " << b << "ll * ldx) : " << Z << "));\n";
    for (int a : outs) os << "      T f" << a << " = " << Z << ";\n";
    if (R > 1)
      os << "#pragma unroll 1\n      for (int s = 0; s < " << R << "; ++s) {\n"
         << "      const T* np = s + 1 < " << R << " ? vp + " << 32 * Kr << " : v + 1 < nv ? block(v + 1) : nullptr;\n";
    else
      os << "      const T* np = v + 1 < nv ? block(v + 1) : nullptr;\n";
    for (int ch = 0; ch < nch; ++ch) {
      // chunk ch has arrived; the stage consumed before it takes the chunk S - 1 ahead
      const int nx = ch + S - 1;
      os << "      { arrived();\n"
            "        int ns = stg + " << S - 1 << "; if (ns >= " << S << ") ns -= " << S << ";\n";
      if (nx < nch)
        os << "        chunk<" << std::min(CB, Kr - nx * CB) << ">(rs + ns * " << CB * 32 * es << ", vp + "
           << 32 * nx * CB << ", lane);\n";
      else
        os << "        if (np) chunk<" << std::min(CB, Kr - (nx - nch) * CB) << ">(rs + ns * " << CB * 32 * es
           << ", np + " << 32 * (nx - nch) * CB << ", lane);\n";
      os << "        commit();\n"
            "        const T* w = ring + stg * " << CB * 32 << ";\n"
            "        if (++stg == " << S << ") stg = 0;\n";
      for (int i4 = ch * CB; i4 < std::min(Kr, (ch + 1) * CB); i4 += 4) {
        os << "        { T v[4]; ld4(v, w + " << 32 * (i4 - ch * CB) << ");\n";
        for (int i = i4; i < i4 + 4; ++i) {
          std::map<double, std::vector<EdgeOrder::Tri>> by_g;
          for (const auto& t : by_i[i]) by_g[fp64 ? t.g : double(float(t.g))].push_back(t);
          const std::string vi = "v[" + std::to_string(i - i4) + "]";
          for (const auto& e : by_g) {
            const bool unit = e.first == 1.0;
            os << "         ";
            if (!unit)
              os << " { const T t = " << vi << " * G(" << (fp64 ? hexd(e.first) : hexf(float(e.first))) << ");";
            for (const auto& t : e.second)
              os << " f" << t.a << " = " << fma << "(" << (unit ? vi : "t") << ", x" << t.b << ", f" << t.a << ");";
            os << (unit ? "\n" : " }\n");
          }
        }
        os << "        }\n";
      }
      os << "      }\n";
    }
    if (R > 1) {
      // x_b <- x_sigma(b), f_a <- f_sigma(a), cycle by cycle
      auto rotate = [&](const char* name, const std::vector<char>& in) {
        std::vector<char> done(P, 0);
        for (int a = 0; a < P; ++a) {
          if (!in[a] || done[a] || o.sig_out[a] == a) continue;
          os << "      { const T t = " << name << a << ";";
          int q = a;
          for (; o.sig_out[q] != a; q = o.sig_out[q]) {
            done[q] = 1;
            os << " " << name << q << " = " << name << o.sig_out[q] << ";";
          }
          done[q] = 1;
          os << " " << name << q << " = t; }\n";
        }
      };
      std::vector<char> mine(P, 0);
      for (int a : outs) mine[a] = 1;
      rotate("x", need_b);
      rotate("f", mine);
      os << "      vp = np;\n      }\n";
    } else {
      os << "      vp = np;\n";
    }
    for (int a : outs)
      if (o.fac[a] != 1.0) os << "      f" << a << " = " << scale(a) << "f" << a << ";\n";
    os << "      if (hor) {\n";
    for (size_t u = 0; u < outs.size(); ++u)
      os << "        y[" << 32 * u << "] += f" << outs[u] << " - __shfl_down_sync(0xffffffffu, f" << outs[u] << ", 1);\n";
    os << "      } else {\n"
          "        if (v && own) {\n"
          "          const long long r = (long long)((up ? j : j + 1) - 1) * m + c - 1;\n";
    // eight outputs at a time, their loads of F together (F may be Y: a load
    // behind a store waits for nothing but is not moved before it; 62 us an
    // apply with F at 256^2, P = 35 one by one, now 44; 37 without F)
    for (size_t u0 = 0; u0 < outs.size(); u0 += 8) {
      const size_t u1 = std::min(outs.size(), u0 + 8);
      os << "          {";
      for (size_t u = u0; u < u1; ++u)
        os << " const T g" << u << " = F ? F[" << outs[u] << "ll * ldf + r] : T(0);";
      os << "\n";
      for (size_t u = u0; u < u1; ++u)
        os << "            { const T o = " << fma << "(-sg, f" << outs[u] << ", y[" << 32 * u << "]); Y[" << outs[u]
           << "ll * ldy + r] = F ? g" << u << " - o : o; }\n";
      os << "          }\n";
    }
    os << "        }\n";
    for (size_t u = 0; u < outs.size(); ++u) os << "        y[" << 32 * u << "] = sg * f" << outs[u] << ";\n";
    os << "      }\n"
          "    }\n"
          "  }\n";
  }
  os << "}\n";
  return os.str();
}

size_t jit_smem_bytes(const sg_problem* pr, const JitConfig& c, bool fp64) {
  // edge form: the running output of every thread (any output group holds at most P)
  // and its warp's ring of conductance chunks
  if (c.flux) {
    const int Kr = pr->edge_terms.KT / std::max(1, pr->edge_terms.R);
    return (size_t(pr->P) + size_t(edge_stages(c, Kr)) * edge_chunk(c, Kr)) * 32 * c.warps * (fp64 ? sizeof(double) : sizeof(float));
  }
  if (c.cgroups > 1) return 0;
  if (c.stages >= 2) return size_t(c.stages) * std::max(1, c.prefetch) * 128 * (fp64 ? sizeof(double) : sizeof(float));
  if (c.groups * c.igroups * c.sgroups == 1) return 0;
  return size_t(c.igroups) * c.sgroups * pr->P * 32 * c.warps * c.rows * (fp64 ? sizeof(double) : sizeof(float));
}

// Compile (or load from the cache) one configuration.
static sg_status jit_compile(const std::string& src, cudaLibrary_t* lib, cudaKernel_t* kern, bool* cached,
                             double* seconds, int dev, bool fp64) {
  auto t0 = std::chrono::steady_clock::now();
  char key[32];
  std::snprintf(key, sizeof key, "%016llx", (unsigned long long)fnv1a(src + "|sm_103a|v" + std::to_string(kJitGeneratorVersion)));
  const std::string dir = cache_dir();
  const std::string path = dir + "/k1_" + key + ".cubin";
  std::vector<char> cubin;
  {
    std::ifstream in(path, std::ios::binary);
    if (in) cubin.assign(std::istreambuf_iterator<char>(in), std::istreambuf_iterator<char>());
  }
  if (cached) *cached = !cubin.empty();
  if (cubin.empty()) {
    nvrtcProgram prog;
    if (nvrtcCreateProgram(&prog, src.c_str(), "sg_k1.cu", 0, nullptr, nullptr) != NVRTC_SUCCESS) {
      set_error("NVRTC: cannot create the specialised apply program");
      return SG_ERR_CUDA;
    }
    const char* opts[] = {"--gpu-architecture=sm_103a", "-std=c++17", "--fmad=true", "-lineinfo"};
    nvrtcResult rc = nvrtcCompileProgram(prog, 4, opts);
    if (rc != NVRTC_SUCCESS) {
      size_t ls = 0;
      nvrtcGetProgramLogSize(prog, &ls);
      std::string log(ls, '\0');
      nvrtcGetProgramLog(prog, &log[0]);
      nvrtcDestroyProgram(&prog);
      set_error("NVRTC compile of the specialised apply failed: " + log.substr(0, 2000));
      return SG_ERR_CUDA;
    }
    size_t sz = 0;
    nvrtcGetCUBINSize(prog, &sz);
    cubin.resize(sz);
    nvrtcGetCUBIN(prog, cubin.data());
    nvrtcDestroyProgram(&prog);
    mkdirs(dir);
    const std::string tmp = path + ".tmp" + std::to_string(::getpid());
    std::ofstream out(tmp, std::ios::binary);
    if (out) {
      out.write(cubin.data(), std::streamsize(cubin.size()));
      out.close();
      std::rename(tmp.c_str(), path.c_str());
    }
  }
  SG_CUDA(cudaLibraryLoadData(lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0));
  SG_CUDA(cudaLibraryGetKernel(kern, *lib, fp64 ? "sg_k1_f64" : "sg_k1"));
  SG_CUDA(cudaKernelSetAttributeForDevice(*kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024, dev));
  if (seconds) *seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  return SG_OK;
}

// Edge form without tuning, for a mesh of N x N cells.  Registers: 2 P for x
// and f (output groups only where they do not fit), the resident CTAs they
// leave.  Strip: an SM works off two CTAs of four warps at a time whatever
// else is resident, and a warp's time is its 2 strip + 1 edge visits, so the
// strip with the fewest rounds x visits (measured: 23.7 to 24.6 us per round
// and visit at 384^2, P = 70 for strips of 1 to 4, 6.8 to 7.3 us at 256^2, P
// = 35).  Long strips lose: 27 us at 6 rows.  FP64 takes the same
// rule (single-warp CTAs, one an SM to a round: 0.67 instead of 0.58 ms at
// 128^2, P = 35 with the nonlinear problem's full chaos).
static JitConfig edge_default(const sg_problem* pr, int N, bool fp64) {
  JitConfig c;
  c.flux = 1;
  const int words = fp64 ? 2 : 1;
  c.cgroups = std::min(16, std::max(1, (2 * pr->P * words + 219) / 220));
  c.prefetch = 32;
  c.stages = 3;
  c.warps = 4;
  while (c.warps > 1 && jit_smem_bytes(pr, c, fp64) > 200 * 1024) c.warps /= 2;
  c.min_blocks = words * pr->P <= 42 ? 4 : words * pr->P <= 60 ? 3 : 2;
  const int64_t tiles = (N + 30) / 31;
  int64_t best = 0;
  for (int strip = 1; strip <= 4; ++strip) {
    const int64_t ctas = ((N - 1 + strip - 1) / strip * tiles + c.warps - 1) / c.warps * c.cgroups;
    const int64_t cost = (ctas + 2 * 152 - 1) / (2 * 152) * (2 * strip + 1);
    if (strip == 1 || cost < best) {
      best = cost;
      c.strip = strip;
    }
  }
  return c;
}

JitConfig jit_default_config(const sg_problem* pr, int which) {
  // a handle beyond the specialised kernel's limits has no edge form (its
  // applies run on the shared-memory kernel): it reports the slot shape
  if (jit_eligible(pr)) {
    if ((which == 0 && pr->flux_allowed) || which == 4) return edge_default(pr, pr->N, false);
    if (which == 1 && coarse_edge_default(pr)) return edge_default(pr, pr->N / 2, false);
    if (which == 5) return edge_default(pr, pr->N, true);
  }
  return jit_slot_config(pr, which);
}

JitConfig jit_slot_config(const sg_problem* pr, int which) {
  const bool fp64 = which == 2 || which == 3;
  JitConfig c;
  c.rows = 1;
  c.min_blocks = 1;
  if (pr->P > 48) {
    // large P: output groups as separate CTAs keep every register of a
    // 128-thread CTA for one group's outputs.  FP32 slot form at 384^2, P =
    // 70: 3 groups 1.29 ms, 5 1.27, 8 1.59 (3 contiguous ranges interleaved
    // over the grid: 2.13 ms); 300^2, P = 84: 3 groups 1.43, 5 1.61, 8 1.77
    c.prefetch = 8;
    c.cgroups = std::min(16, fp64 ? (pr->P + 15) / 16 : std::max(3, (pr->P + 27) / 28));
    return c;
  }
  c.prefetch = fp64 ? 16 : 32;
  // the coarse operator has a quarter of the rows: deal the slots to two
  // groups so that the grid still fills the GPU
  c.sgroups = which % 2 == 1 ? 2 : 1;
  return c;
}

JitConfig jit_config(const sg_problem* pr, int which) {
  return pr->jit_cfg_set[which] ? pr->jit_cfg[which] : jit_default_config(pr, which);
}

static bool jit_fp64(int which) { return which == 2 || which == 3 || which == 5; }

static std::string family_source(const sg_problem* pr, const JitConfig& c, bool fp64) {
  return c.flux ? jit_edge_source(pr, c, fp64) : jit_apply_source(pr, c, fp64);
}

sg_status jit_apply_build(sg_problem* pr, int which) {
  if (pr->jit[which] && pr->jit[which]->kern) return SG_OK;
  if (!pr->jit[which]) pr->jit[which] = new JitApply();
  JitApply& J = *pr->jit[which];
  if (!pr->jit_cfg_set[which]) {
    pr->jit_cfg[which] = jit_default_config(pr, which);
    pr->jit_cfg_set[which] = true;
  }
  const bool fp64 = jit_fp64(which);
  return jit_compile(family_source(pr, pr->jit_cfg[which], fp64), &J.lib, &J.kern, &J.from_cache, &J.compile_s,
                     pr->device, fp64);
}

sg_status jit_configure(sg_problem* pr, int which, const JitConfig& c) {
  const bool edge_ok = (which == 0 || which == 1) && c.rows == 1 && c.groups * c.igroups * c.sgroups == 1 &&
                       c.stages >= 2 && c.stages <= 8 && c.cgroups >= 1 && c.cgroups <= 16 && c.prefetch >= 1 &&
                       c.prefetch <= 64 &&
                       c.min_blocks >= 1 && c.min_blocks <= 8 && (c.warps == 1 || c.warps == 2 || c.warps == 4) &&
                       c.strip >= 1 && c.strip <= 64;
  const bool slot_ok =
      c.rows >= 1 && c.rows <= 2 && c.groups >= 1 && c.groups <= 4 && c.igroups >= 1 && c.igroups <= 4 &&
      c.sgroups >= 1 && c.sgroups <= 8 && c.groups * c.igroups * c.sgroups <= 8 && c.prefetch >= 0 &&
      c.prefetch <= 64 && c.min_blocks >= 1 && c.min_blocks <= 8 && (which < 2 || c.rows == 1) && c.stages >= 0 &&
      c.stages != 1 && c.stages <= 8 &&
      (c.stages < 2 || (c.rows == 1 && c.groups * c.igroups * c.sgroups == 1 && c.prefetch >= 1)) && c.cgroups >= 1 &&
      c.cgroups <= 16 &&
      (c.cgroups == 1 || (c.rows == 1 && c.groups * c.igroups * c.sgroups == 1 && c.stages == 0)) &&
      (c.warps == 1 || c.warps == 2 || c.warps == 4) && (c.warps == 4 || (c.stages == 0 && c.cgroups == 1));
  if (c.flux ? !edge_ok : !slot_ok) {
    set_error("sg_apply_config: rows in {1,2}; groups, igroups in [1,4]; sgroups in [1,8]; "
              "groups*igroups*sgroups <= 8; prefetch in [0,64]; min_blocks in [1,8]; FP64 families: rows 1; "
              "stages 0 or 2..8, staged only with one row and one group and prefetch >= 1; "
              "cgroups 1..16, split only with one row, one group and no staging; warps per group 1, 2 or 4, "
              "fewer than 4 only without staging or separate CTAs");
    return SG_ERR_ARG;
  }
  if (jit_smem_bytes(pr, c, which >= 2) > 200 * 1024) {
    set_error("sg_apply_config: the input-group hand-off does not fit in shared memory");
    return SG_ERR_ARG;
  }
  // recorded coarse-solve graphs reference the kernel about to be unloaded
  if (pr->jit[which] || (which == 0 && pr->jit[6]) || jit_config(pr, which).flux != c.flux) drop_recorded(pr);
  jit_free(pr, which);
  pr->jit_cfg[which] = c;
  pr->jit_cfg_set[which] = true;
  pr->jit_cfg_user[which] = true;
  if (which < 2) SG_TRY(fp32_values(pr));
  if (!jit_eligible(pr)) return SG_OK;
  return jit_apply_build(pr, which);
}

sg_status jit_keep(sg_problem* pr, int which) {
  const bool edge = solver_edge(pr);
  pr->jit_cfg[which] = jit_config(pr, which);
  pr->jit_cfg_set[which] = true;
  pr->jit_cfg_user[which] = true;
  // recorded coarse-solve graphs run the form solves used until now
  if (solver_edge(pr) != edge) drop_recorded(pr);
  return jit_eligible(pr) ? jit_apply_build(pr, which) : SG_OK;
}

void jit_free(sg_problem* pr, int which) {
  if (!pr->jit[which]) return;
  if (pr->jit[which]->lib) cudaLibraryUnload(pr->jit[which]->lib);
  delete pr->jit[which];
  pr->jit[which] = nullptr;
}

bool jit_eligible(const sg_problem* pr) { return pr->P <= kJitMaxP && pr->T <= kJitMaxT; }

template <typename T>
static sg_status launch_kernel(cudaKernel_t kern, const JitConfig& c, size_t smem, const Ell& A, const T* X,
                               int64_t ldx, const T* F, int64_t ldf, T* Y, int64_t ldy, cudaStream_t st) {
  if (A.n == 0) return SG_OK;
  const T* V = sizeof(T) == 8 ? reinterpret_cast<const T*>(A.v64.ptr) : reinterpret_cast<const T*>(A.v32.ptr);
  const int* col = dp<int>(A.col);
  long long ldr = A.ldr, lx = ldx, lf = ldf, ly = ldy;
  int n = int(A.n), S = A.S;
  void* args[] = {(void*)&V, (void*)&col, &ldr, &n, &S, (void*)&X, &lx, (void*)&F, &lf, (void*)&Y, &ly};
  const bool cs = c.cgroups > 1;
  const int64_t rows_per_cta = 32LL * (cs ? 4 : c.warps) * c.rows;
  dim3 grid(unsigned((A.n + rows_per_cta - 1) / rows_per_cta * (cs ? c.cgroups : 1))),
      block(unsigned(cs ? 128 : 32 * c.warps * c.groups * c.igroups * c.sgroups));
  SG_CUDA(cudaLaunchKernel((const void*)kern, grid, block, args, smem, st));
  note_launch();
  return SG_OK;
}

template <typename T>
static sg_status launch_edge(cudaKernel_t kern, const JitConfig& c, size_t smem, const EdgeVals& A, const T* X,
                             int64_t ldx, const T* F, int64_t ldf, T* Y, int64_t ldy, cudaStream_t st) {
  const T* V = sizeof(T) == 8 ? reinterpret_cast<const T*>(A.v64.ptr) : reinterpret_cast<const T*>(A.v32.ptr);
  if (!V) {
    set_error("the edge form's conductances are not on the device");
    return SG_ERR_ARG;
  }
  long long lx = ldx, lf = ldf, ly = ldy;
  int N = A.N;
  void* args[] = {(void*)&V, &N, (void*)&X, &lx, (void*)&F, &lf, (void*)&Y, &ly};
  const int64_t warps = int64_t((N - 1 + c.strip - 1) / c.strip) * ((N + 30) / 31);  // 31 nodes a tile
  const dim3 grid(unsigned((warps + c.warps - 1) / c.warps * c.cgroups)), block(unsigned(32 * c.warps));
  SG_CUDA(cudaLaunchKernel((const void*)kern, grid, block, args, smem, st));
  note_launch();
  return SG_OK;
}

template <typename T>
sg_status jit_edge_launch(sg_problem* pr, int which, const EdgeVals& A, const T* X, int64_t ldx, const T* F,
                          int64_t ldf, T* Y, int64_t ldy, cudaStream_t st) {
  SG_TRY(jit_apply_build(pr, which));
  const JitConfig& c = pr->jit_cfg[which];
  return launch_edge<T>(pr->jit[which]->kern, c, jit_smem_bytes(pr, c, sizeof(T) == 8), A, X, ldx, F, ldf, Y, ldy, st);
}
template sg_status jit_edge_launch<float>(sg_problem*, int, const EdgeVals&, const float*, int64_t, const float*,
                                          int64_t, float*, int64_t, cudaStream_t);
template sg_status jit_edge_launch<double>(sg_problem*, int, const EdgeVals&, const double*, int64_t, const double*,
                                           int64_t, double*, int64_t, cudaStream_t);

sg_status jit_apply_launch(sg_problem* pr, int which, const Ell& A, const float* X, int64_t ldx, const float* F,
                           int64_t ldf, float* Y, int64_t ldy, cudaStream_t st) {
  SG_TRY(jit_apply_build(pr, which));
  const JitConfig& c = pr->jit_cfg[which];
  return launch_kernel<float>(pr->jit[which]->kern, c, jit_smem_bytes(pr, c, false), A, X, ldx, F, ldf, Y, ldy, st);
}

sg_status jit_apply_launch(sg_problem* pr, int which, const Ell& A, const double* X, int64_t ldx, const double* F,
                           int64_t ldf, double* Y, int64_t ldy, cudaStream_t st) {
  SG_TRY(jit_apply_build(pr, which));
  const JitConfig& c = pr->jit_cfg[which];
  return launch_kernel<double>(pr->jit[which]->kern, c, jit_smem_bytes(pr, c, true), A, X, ldx, F, ldf, Y, ldy, st);
}

// --------------------------------------------------------------------------
// Autotuner: compile the candidate tile shapes, time each on this problem's
// fine operator (median of a few launches after a warm-up, CUDA events),
// keep the fastest and remember the choice in the cache directory, keyed by
// the triple structure, n and the device name.
// --------------------------------------------------------------------------
// A short list of tile shapes per family, from sweeps on GB300: small P
// keeps the whole row in one thread (more prefetch helps); large P splits
// outputs and inputs over warp groups; the coarse family (a quarter of the
// rows) adds stencil-slot groups to fill the GPU.  Values staged through
// shared memory by 4-byte cp.async measured half the bandwidth of the
// register prefetch at 256^2 / P = 35 (0.144 ms against 0.071 ms), so the
// staged shapes are available through sg_apply_config but not tuned.  Groups
// of one warp (every slot its own group) measured slower everywhere except
// the fine FP64 family, where two output by two slot groups of one warp
// each beat the 4-warp shapes by 10 % at 256^2 / P = 35.  Slot groups alone
// share one generated body (0.0526 -> 0.0487 ms for the coarse family's two
// slot groups at 127^2 coarse rows, P = 35).
static std::vector<JitConfig> candidates(const sg_problem* pr, int which) {
  if (which == 1 || (which == 0 && pr->flux_allowed)) {
    // edge form: strips against parallelism
    std::vector<JitConfig> out;
    const JitConfig d = edge_default(pr, which == 1 ? pr->N / 2 : pr->N, false);
    out.push_back(d);
    for (int strip : {1, 2, 3, 8})
      if (strip != d.strip) {
        out.push_back(d);
        out.back().strip = strip;
      }
    return out;
  }
  struct S7 {
    int r, g, i, s, pf, st, mb = 1, cg = 1, w = 4;
  };
  std::vector<S7> list;
  const bool fp64 = which >= 2;
  if (fp64) {
    // twice the register bytes per value: more output/input splitting, or
    // values staged through shared memory
    if (pr->P <= 48) {
      if (which == 2)
        list = {{1, 1, 1, 1, 16, 0}, {1, 1, 1, 1, 8, 0}, {1, 2, 1, 1, 16, 0}, {1, 1, 2, 1, 16, 0},
                {1, 2, 2, 1, 8, 0}, {1, 2, 1, 2, 8, 0, 1, 1, 1}};
      else
        list = {{1, 1, 1, 2, 16, 0}, {1, 1, 1, 4, 8, 0}, {1, 2, 1, 2, 8, 0}, {1, 1, 2, 2, 8, 0}};
    } else {
      list = {{1, 1, 1, 1, 8, 0, 1, 4}, {1, 1, 1, 1, 8, 0, 1, 6}, {1, 1, 1, 1, 8, 0, 1, 8},
              {1, 1, 1, 1, 4, 0, 1, 6}};
    }
  } else if (pr->P <= 48) {
    list = {{1, 1, 1, 1, 32, 0}, {1, 1, 1, 1, 16, 0}, {1, 1, 2, 1, 16, 0}, {1, 2, 1, 1, 16, 0}};
  } else {
    list = {{1, 1, 1, 1, 8, 0, 1, 3}, {1, 1, 1, 1, 8, 0, 1, 4}, {1, 1, 1, 1, 16, 0, 1, 4},
            {1, 1, 1, 1, 8, 0, 1, 6}, {1, 1, 1, 1, 4, 0, 1, 8}};
  }
  std::vector<JitConfig> out;
  for (const S7& e : list) {
    JitConfig c;
    c.rows = e.r;
    c.groups = e.g;
    c.igroups = e.i;
    c.sgroups = e.s;
    c.prefetch = e.pf;
    c.stages = e.st;
    c.min_blocks = e.mb;
    c.cgroups = e.cg;
    c.warps = e.w;
    if (jit_smem_bytes(pr, c, fp64) > 200 * 1024) continue;
    out.push_back(c);
  }
  if (out.empty()) out.push_back(jit_default_config(pr, which));
  return out;
}

static std::string tune_key(const sg_problem* pr, const Ell& A, bool fp64) {
  cudaDeviceProp prop{};
  cudaGetDeviceProperties(&prop, pr->device);
  std::ostringstream os;
  os << prop.name << "|v" << kJitGeneratorVersion << "|" << pr->P << "|" << pr->K << "|" << pr->T << "|" << A.n << "|"
     << A.S << (fp64 ? "|f64" : "");
  for (int64_t t = 0; t < pr->T; ++t) os << "," << pr->kab[3 * t] << ":" << pr->kab[3 * t + 1] << ":" << pr->kab[3 * t + 2];
  char key[32];
  std::snprintf(key, sizeof key, "%016llx", (unsigned long long)fnv1a(os.str()));
  return key;
}

sg_status jit_autotune(sg_problem* pr, int which, int force, double* best_ms) {
  if (!jit_eligible(pr)) {
    set_error("sg_apply_autotune: the specialised kernel is not available for this size");
    return SG_ERR_UNSUPPORTED;
  }
  const bool coarse = which % 2 == 1, fp64 = which >= 2;
  if (coarse && !pr->solver) {
    set_error("sg_apply_autotune: the coarse operator exists after sg_precond_setup");
    return SG_ERR_ARG;
  }
  const Ell& A = coarse ? coarse_ell(pr) : pr->fine;
  const std::string path = cache_dir() + "/tune_" + tune_key(pr, A, fp64) + (pr->flux_allowed ? "_fx" : "") + ".txt";
  if (!force) {
    std::ifstream in(path);
    JitConfig c;
    double ms = 0;
    if (in >> c.rows >> c.groups >> c.igroups >> c.sgroups >> c.prefetch >> c.min_blocks >> c.stages >> c.cgroups >>
        c.warps >> c.flux >> c.strip >> ms) {
      if (best_ms) *best_ms = ms;
      return jit_configure(pr, which, c);
    }
  }
  const int64_t len = int64_t(pr->P) * std::max<int64_t>(pr->ld, A.ldr);
  const size_t esz = fp64 ? 8 : 4;
  DevBuf X, Y;
  SG_TRY(X.alloc(len * esz));
  SG_TRY(Y.alloc(len * esz));
  cudaStream_t st;
  SG_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
  cudaEvent_t e0, e1;
  SG_CUDA(cudaEventCreate(&e0));
  SG_CUDA(cudaEventCreate(&e1));
  JitConfig best = jit_default_config(pr, which);
  double best_t = 1e30;
  sg_status status = SG_OK;
  for (const JitConfig& c : candidates(pr, which)) {
    cudaLibrary_t lib = nullptr;
    cudaKernel_t kern = nullptr;
    if (jit_compile(family_source(pr, c, fp64), &lib, &kern, nullptr, nullptr, pr->device, fp64) != SG_OK) continue;
    const size_t sm = jit_smem_bytes(pr, c, fp64);
    if (coarse && c.flux) status = coarse_edge_prepare(pr);
    else if (!fp64 && !c.flux) status = ell_f32(A, pr->K, nullptr);
    if (status != SG_OK) {
      cudaLibraryUnload(lib);
      break;
    }
    auto run = [&]() {
      if (c.flux)
        return launch_edge<float>(kern, c, sm, coarse ? coarse_edge(pr) : pr->edge, dp<float>(X), A.ldr, nullptr, 0, dp<float>(Y),
                           A.ldr, st);
      return fp64 ? launch_kernel<double>(kern, c, sm, A, dp<double>(X), A.ldr, nullptr, 0, dp<double>(Y), A.ldr, st)
                  : launch_kernel<float>(kern, c, sm, A, dp<float>(X), A.ldr, nullptr, 0, dp<float>(Y), A.ldr, st);
    };
    std::vector<float> ts;
    for (int rep = 0; rep < 7 && status == SG_OK; ++rep) {
      status = run();
      if (status != SG_OK) break;
      if (rep < 2) continue;
      cudaEventRecord(e0, st);
      run();
      cudaEventRecord(e1, st);
      cudaEventSynchronize(e1);
      float ms = 0;
      cudaEventElapsedTime(&ms, e0, e1);
      ts.push_back(ms);
    }
    cudaLibraryUnload(lib);
    if (status != SG_OK) break;
    std::sort(ts.begin(), ts.end());
    const double med = ts.empty() ? 1e30 : ts[ts.size() / 2];
    if (med < best_t) {
      best_t = med;
      best = c;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(st);
  SG_TRY(status);
  if (best_ms) *best_ms = best_t;
  mkdirs(cache_dir());
  std::ofstream out(path);
  if (out)
    out << best.rows << " " << best.groups << " " << best.igroups << " " << best.sgroups << " " << best.prefetch
        << " " << best.min_blocks << " " << best.stages << " " << best.cgroups << " " << best.warps << " " << best.flux
        << " " << best.strip << " " << best_t << "\n";
  return jit_configure(pr, which, best);
}

}  // namespace sg
