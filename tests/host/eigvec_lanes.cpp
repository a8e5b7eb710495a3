// The eigenvectors of T (tridiag_vec.cuh) compiled for the host: the 32 lanes of
// a warp as fibers that run one after the other from one meeting point
// (__syncwarp or a shuffle) to the next, in the order given.  Nothing promises
// lockstep between two meeting points, so every order has to give the same.
//
// stdin:  order (0 ascending, 1 descending, 2 random), n, then alpha (n),
//         beta (n) and theta (n, descending) in decimal or hexadecimal
// stdout: the n x n eigenvectors S, a row per line
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <random>
#include <vector>

#include <cuda_runtime.h>

using std::isfinite;

static struct { unsigned x; } threadIdx;

namespace lanes {
constexpr int N = 32;
ucontext_t ctx[N], home;
char stack_mem[N][1 << 18];
bool done[N];
float slot[2][N];
int phase[N];
void (*body)();

void meet() {
  const int lane = (int)threadIdx.x;
  swapcontext(&ctx[lane], &home);
}
void entry() {
  body();
  done[threadIdx.x] = true;
}
void run(void (*f)(), int order) {
  static std::mt19937 rng(1);
  body = f;
  for (int l = 0; l < N; ++l) {
    done[l] = false;
    phase[l] = 0;
    getcontext(&ctx[l]);
    ctx[l].uc_stack.ss_sp = stack_mem[l];
    ctx[l].uc_stack.ss_size = sizeof(stack_mem[l]);
    ctx[l].uc_link = &home;
    makecontext(&ctx[l], entry, 0);
  }
  std::vector<int> seq(N);
  std::iota(seq.begin(), seq.end(), 0);
  if (order == 1) std::reverse(seq.begin(), seq.end());
  for (;;) {
    if (order == 2) std::shuffle(seq.begin(), seq.end(), rng);
    int ran = 0;
    for (int l : seq) {
      if (done[l]) continue;
      threadIdx.x = (unsigned)l;
      swapcontext(&home, &ctx[l]);
      ++ran;
    }
    if (ran == 0) return;
    if (ran != N) std::abort();  // a lane left while others still meet
    if (std::all_of(done, done + N, [](bool d) { return d; })) return;
  }
}
}  // namespace lanes

static inline void __syncwarp() { lanes::meet(); }
static inline float __shfl_xor_sync(unsigned, float v, int m) {
  const int l = (int)threadIdx.x, b = lanes::phase[l];
  lanes::slot[b][l] = v;
  lanes::phase[l] ^= 1;
  lanes::meet();
  return lanes::slot[b][l ^ m];
}
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __fdividef(float a, float b) { return a / b; }
static inline float __double2float_rn(double x) { return (float)x; }

#include "../../paper_2607_19368_gb300/csrc/tridiag_vec.cuh"

namespace {
constexpr int MAXN = 128;
float2 d[MAXN], du[MAXN], du2[MAXN], dl[MAXN], y[MAXN], sa[MAXN], sb[MAXN];
unsigned char piv[MAXN];
std::vector<double> alpha, beta, theta, S;
int n, first, last;

void warp_body() {
  double tnorm;
  const double sc = sls::eig_scale(theta.data(), n, &tnorm);
  sls::eig_scaled_T(alpha.data(), beta.data(), n, sc, (int)threadIdx.x, 32, sa, sb);
  __syncwarp();
  sls::eigvec_cluster(n, theta.data(), S.data(), n, first, last, sc, tnorm, sa, sb, d, du, du2, dl,
                      y, piv);
}
}  // namespace

int main() {
  int order;
  if (std::scanf("%d %d", &order, &n) != 2 || n < 1 || n > MAXN) return 2;
  for (auto* v : {&alpha, &beta, &theta}) {
    v->resize(n);
    for (double& x : *v)
      if (std::scanf("%la", &x) != 1) return 2;
  }
  S.assign((size_t)n * n, 0.0);
  for (int m = 0; m < n; ++m) {
    sls::eig_cluster(theta.data(), n, m, first, last);
    if (first == m) lanes::run(warp_body, order);
  }
  for (int i = 0; i < n; ++i)
    for (int m = 0; m < n; ++m) std::printf("%a%c", S[(size_t)i * n + m], m + 1 < n ? ' ' : '\n');
  return 0;
}
