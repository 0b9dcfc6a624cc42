// The device arithmetic of the thread-per-cell kernels compiled for the CPU, one lane at a
// time, so that its numbers, and what they do on rare states, can be tested without a GPU:
//   host_kernels <command> <mechanism file> < doubles > doubles
// (9 species, except for the gather plan of the CTA-per-cell kernels).
// The CUDA keywords are defined away; the few intrinsics the sources use are given here.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <iterator>
#include <string>
#include <vector>

#define __CUDACC_RTC__
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))
#define __shared__
static inline long long __double_as_longlong(double x) {
  long long b;
  std::memcpy(&b, &x, 8);
  return b;
}
static inline double __longlong_as_double(long long b) {
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}
static inline double rcbrt(double x) { return 1.0 / std::cbrt(x); }
static inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static inline int min(int a, int b) { return a < b ? a : b; }
static inline long long min(long long a, long long b) { return a < b ? a : b; }
static inline int max(int a, int b) { return a > b ? a : b; }
static inline long long max(long long a, long long b) { return a > b ? a : b; }
using std::fma;
using std::fmax;
using std::fmin;
using std::isfinite;
using std::sqrt;
struct int4 { int x, y, z, w; };
// warp and block operations of the kernel bodies, which are not run here
static struct { int x; } threadIdx, blockIdx, blockDim, gridDim;
static inline void __syncthreads() {}
static inline int __syncthreads_or(int v) { return v; }
static inline int __any_sync(unsigned, bool v) { return v; }
static inline unsigned __ballot_sync(unsigned, bool v) { return v; }
template <class T>
static inline T __shfl_sync(unsigned, T v, int) { return v; }
static inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }
static inline int __popc(unsigned v) { return __builtin_popcount(v); }
template <class T>
static inline T atomicAdd(T* p, T v) { T o = *p; *p += v; return o; }
template <class T>
static inline T atomicMax(T* p, T v) { T o = *p; if (v > o) *p = v; return o; }
static inline long long clock64() { return 0; }

#include "chem_adjoint_body.cuh"
#include "large_plan.h"
#include "mech_host.h"

using namespace rde;

namespace {
constexpr int K = 9, N = K + 1;

FixThermo g_fix;

// the packed reaction records with the fixed-point thermo of a specialised kernel
struct FixReactions {
  static constexpr unsigned kInert = 0u;
  static constexpr bool kFix = true;
  static int kCpBits;
  static int dcp_bits(int k) { return g_fix.dcp_bits[k]; }
  static bool two_ranges(int) { return true; }
  static uint64_t th(int k, int r, int j) { return (uint64_t)g_fix.c[(size_t)(k * 2 + r) * 21 + j] + kFixBias; }
  template <class F>
  static void each(const MechView& m, F&& f) { GenericReactions::each(m, f); }
};
int FixReactions::kCpBits = 0;

std::vector<double> read_doubles() {
  std::vector<double> v;
  double x;
  while (std::fread(&x, 8, 1, stdin) == 1) v.push_back(x);
  return v;
}
void put(const double* p, size_t n) { std::fwrite(p, 8, n, stdout); }

// in: invp, y[N], u[4][N], w[4][N]; out: g[N], thA[R], thE[R] of hvp_sum and of jtw's
// dual-number evaluations summed over the stages
template <class RX>
void hvp(const MechView& m, const double* in) {
  const int R = m.hdr->R;
  std::vector<double> slots((size_t)(18 * K + 64) * kLaneThreads), g(N, 0.0), A(R, 0.0), E(R, 0.0);
  const Lane L{slots.data()};
  const double *y = in + 1, *U = in + 1 + N, *W = in + 1 + 5 * N;
  hvp_sum<K, 4, RX>(m, L, in[0], y, U, W, 0, 1, g.data(), A.data(), E.data(), 1);
  put(g.data(), N);
  put(A.data(), R);
  put(E.data(), R);
  std::vector<double> s(N, 0.0), part(N, 0.0);
  std::fill(A.begin(), A.end(), 0.0);
  std::fill(E.begin(), E.end(), 0.0);
  for (int st = 0; st < 4; ++st) {
    Dual yd[N];
    for (int i = 0; i < N; ++i) yd[i] = mk(y[i], U[st * N + i]);
    jtw<K, GenericReactions>(m, L, 0, in[0], yd, W + st * N, part.data(), A.data(), E.data(), 1);
    for (int i = 0; i < N; ++i) s[i] += part[i];
  }
  put(s.data(), N);
  put(A.data(), R);
  put(E.data(), R);
}

// in: (invp, y[N]) per state; out: f[N] per state, once without and once with the Jacobian
template <class RX>
void rhs(const MechView& m, const std::vector<double>& in) {
  std::vector<double> slots((size_t)Slots<K>::TOTAL * kLaneThreads);
  const Lane L{slots.data()};
  for (size_t at = 0; at < in.size(); at += 1 + N)
    for (int jac = 0; jac < 2; ++jac) {
      for (int i = 0; i < N; ++i) L[Slots<K>::ARG + i] = in[at + 1 + i];
      if (jac) RhsOf<RX>::template eval<K, true, Slots<K>>(m, L, in[at]);
      else RhsOf<RX>::template eval<K, false, Slots<K>>(m, L, in[at]);
      for (int i = 0; i < N; ++i) put(&L[Slots<K>::VEC + i], 1);
    }
}

// in: T per state; out, per state and species: Cp/R, the polynomial part of H/RT,
// d(Cp/R)/dT and G/RT in fixed point, then the same in FP64
void thermo(const MechView& m, const std::vector<double>& in) {
  for (double T : in) {
    RhsCtx cx{};
    cx.invT = recip(T);
    cx.lnT = log_tab(T, m.logtab);
    cx.zlnT = (uint64_t)to_fix(cx.lnT, 59);
    cx.zinvT = (uint64_t)to_fix(cx.invT, 70);
    for (int k = 0; k < K; ++k) {
      SpecPacked sp = m.sp[k];
      sp.h[0][5] = sp.h[1][5] = 0.0;
      double o[8], g;
      int64_t z;
      thermo_fix<true, FixReactions>(sp, k, T, (uint64_t)to_fix(T, 50), cx, o[0], o[1], z, o[2]);
      o[3] = fix_to_log(z, 0);
      thermo_fp64<true>(sp, T, cx.lnT, cx.invT, o[4], o[5], g, o[6]);
      o[7] = g;
      put(o, 8);
    }
  }
}

// the terms of the CTA-per-cell kernels' gather plan as the device reads them:
// (matrix row and column, or -1 - list and species; index into RS; coefficient)
void plan_terms(const unsigned char* image) {
  std::vector<unsigned char> plan;
  build_large_plan(image, &plan);
  const PlanView pl = plan_view(plan.data());
  const int KP = mech_view(image).hdr->K;
  auto term = [&](double row, double col, uint32_t u, const double* coef) {
    const double t[4] = {row, col, (double)(u & 0xffffu), coef[u >> 16]};
    put(t, 4);
  };
  for (int k = 0; k < KP; ++k) {
    for (int e = pl.spr_ptr[k]; e < pl.spr_ptr[k + 1]; ++e) term(-1, k, pl.spr[e], pl.coef);
    for (int e = pl.row_ptr[k]; e < pl.row_ptr[k + 1]; ++e) term(-2, k, pl.row[e], pl.coef);
  }
  for (int e = 0; e < KP * KP; ++e) {
    const PlanEntry en = pl.ent[e];
    for (int q = en.first; q < pl.ent[e + 1].first; ++q)
      term((en.kj >> 6) & 63, en.kj & 63, pl.con[q], pl.coef + (en.kj >> 12) * kPlanPage);
  }
}
}  // namespace

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  std::ifstream f(argv[2], std::ios::binary);
  const std::string text((std::istreambuf_iterator<char>(f)), std::istreambuf_iterator<char>());
  std::vector<unsigned char> image;
  std::string err;
  if (pack_mechanism(text.data(), text.size(), &image, &err) != 0) {
    std::fprintf(stderr, "%s\n", err.c_str());
    return 3;
  }
  const MechView m = mech_view(image.data());
  const std::string cmd = argv[1];
  if (cmd == "plan") {
    plan_terms(image.data());
    return 0;
  }
  if (m.hdr->K != K) return 4;
  const bool fixed = fix_thermo(m, &g_fix);
  FixReactions::kCpBits = g_fix.cp_bits;
  const std::vector<double> in = read_doubles();
  if (cmd == "hvp" || cmd == "hvp_fix") {
    if (in.size() != 1 + 9 * (size_t)N) return 5;
    if (cmd == "hvp") hvp<GenericReactions>(m, in.data());
    else if (fixed) hvp<FixReactions>(m, in.data());
    else return 6;
    return 0;
  }
  if (cmd == "rhs" || cmd == "rhs_fix") {
    if (in.size() % (1 + N)) return 5;
    if (cmd == "rhs") rhs<GenericReactions>(m, in);
    else if (fixed) rhs<FixReactions>(m, in);
    else return 6;
    return 0;
  }
  if (cmd == "thermo") {
    if (!fixed) return 6;
    thermo(m, in);
    return 0;
  }
  return 7;
}
