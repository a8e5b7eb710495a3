// Eigh(T) and Ritz vectors (Algorithm 1) after the implicit Lanczos of
// lanczos_kernel.cuh, plus the planning and launch of the Lanczos kernel.
//
// The r x r (r <= 128) tridiagonal T is solved on the device: Ritz values by
// Sturm-count multisection (a CTA of 256 shifts per eigenvalue when the
// launch has few, one warp of 32 shifts when it has many; double-float
// recurrence), eigenvectors by inverse iteration with
// partial-pivoting LU (double-float), with
// modified Gram-Schmidt inside clusters of nearly equal eigenvalues.  Finally
// U = Q S.
#include "lanczos_kernel.cuh"
#include "tridiag_vec.cuh"

namespace sls {

namespace {

// Lanczos steps kept for problem p, clamped to [0, r]: r_eff is set to -1
// before the Lanczos launch and keeps that value if a device-side wait of the
// kernel gave up, so the later kernels then treat the problem as empty.
SLS_DEV int reff_clamped(const LanczosBatch& bt, int p) {
  return min(bt.r, max(0, bt.r_eff[p]));
}

// ----------------------------------------------------------------------------
// Eigenvalues of T: multisection on Sturm counts.  The arithmetic of the
// recurrences is double-float on the FP32 pipes: float64 on this part has a
// 64-cycle dependent latency (and a divide of several hundred cycles), which
// a serial recurrence pays at every step.
// ----------------------------------------------------------------------------

// Ritz values of few problems: one CTA per eigenvalue, a shift per thread and
// round.  Bound by the double-float recurrence (about 70 instructions and a chain
// of 20 per row of T).  Three rounds in float32 come first and are widened by their
// error, and the first double-float round spans the widened interval ends
// included, so an eigenvalue outside it is found all the same.  r = 32: 33 -> 26 us,
// r = 64: 58 -> 46 (128 threads: the same).
constexpr int EIG_THREADS = 256;  // shifts per multisection round
constexpr float kInvShiftsF = 1.0f / (float)(EIG_THREADS + 1);
constexpr int EIG_F32_ROUNDS = 3;
constexpr float EIG_F32_MARGIN = 0x1p-18f;

__global__ void __launch_bounds__(EIG_THREADS)
tridiag_eigvals_cta_kernel(LanczosBatch bt) {
  __shared__ float2 sa[SLS_MAX_R], sb2[SLS_MAX_R];
  __shared__ int s_first[2][EIG_THREADS / 32];
  __shared__ double s_sc;
  __shared__ float2 s_lo, s_hi;  // the interval, double-float
  const int m = blockIdx.x, p = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  if (p >= nprob) return;
  const int r = bt.r;
  const int n = reff_clamped(bt, p);
  double* theta = bt.theta + (size_t)p * r;
  if (m >= n) {
    if (tid == 0) theta[m] = 0.0;
    return;
  }
  const double* a = bt.alpha + (size_t)p * r;
  const double* b = bt.beta + (size_t)p * r;
  if (warp == 0) {
    // Gershgorin interval, and a power-of-two scale that maps it into [-1, 1]
    double glo = DBL_MAX, ghi = -DBL_MAX;
    for (int i = lane; i < n; i += 32) {
      const double bl = (i > 0) ? fabs(b[i - 1]) : 0.0;
      const double br = (i < n - 1) ? fabs(b[i]) : 0.0;
      glo = fmin(glo, a[i] - bl - br);
      ghi = fmax(ghi, a[i] + bl + br);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
      ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
    }
    if (lane == 0) {
      const double big = fmax(fabs(glo), fabs(ghi));
      int ex = 0;
      frexp(big > 0.0 ? big : 1.0, &ex);
      const double sc = ldexp(1.0, -ex);  // exact scaling
      double lo = glo * sc, hi = ghi * sc;
      const double pad = 0x1p-40 * fmax(fabs(lo), fabs(hi)) + 0x1p-100;
      s_lo = f2(df_from_double(lo - pad));
      s_hi = f2(df_from_double(hi + pad));
      s_sc = sc;
    }
  }
  __syncthreads();
  const double sc = s_sc;
  for (int i = tid; i < n; i += EIG_THREADS) {
    sa[i] = f2(df_from_double(a[i] * sc));
    if (i < n - 1) {
      const double bs = b[i] * sc;
      sb2[i] = f2(df_from_double(bs * bs));
    }
  }
  __syncthreads();
  const int k = n - 1 - m;  // ascending index of the wanted eigenvalue
  int buf = 0;
  // first shift whose count exceeds k (EIG_THREADS: none), the same in every thread
  auto first_above = [&](int c) {
    const unsigned ball = __ballot_sync(0xffffffffu, c > k);
    if (lane == 0) s_first[buf][warp] = ball ? warp * 32 + __ffs(ball) - 1 : EIG_THREADS;
    __syncthreads();
    int f = EIG_THREADS;
#pragma unroll
    for (int w2 = 0; w2 < EIG_THREADS / 32; ++w2) f = min(f, s_first[buf][w2]);
    buf ^= 1;
    return f;
  };
  const dfloat lo0 = dfv(s_lo), hi0 = dfv(s_hi);
  dfloat lo = lo0, hi = hi0;
  {
    float fl = lo0.hi, fh = hi0.hi;
    for (int round = 0; round < EIG_F32_ROUNDS; ++round) {
      const float step = (fh - fl) * kInvShiftsF;
      const int f = first_above(sturm_count_f32(sa, sb2, n, fmaf(step, (float)(tid + 1), fl)));
      const float nl = fmaf(step, (float)f, fl);
      if (f < EIG_THREADS) fh = fmaf(step, (float)(f + 1), fl);
      fl = nl;
    }
    lo = df_make(fl - EIG_F32_MARGIN, 0.f);
    hi = df_make(fh + EIG_F32_MARGIN, 0.f);
    // shifts lo + t (hi - lo) / (EIG_THREADS - 1), both ends among them
    const dfloat step = df_mul_f(df_sub(hi, lo), 1.0f / (float)(EIG_THREADS - 1));
    const int f = first_above(sturm_count(sa, sb2, n, df_add(lo, df_mul_f(step, (float)tid))));
    const dfloat base = lo;
    lo = f > 0 ? df_add(base, df_mul_f(step, (float)(f - 1))) : lo0;
    hi = f < EIG_THREADS ? df_add(base, df_mul_f(step, (float)f)) : hi0;
  }
  for (int round = 0; round < 40; ++round) {
    const dfloat w = df_sub(hi, lo);
    // 2^-46 relative, or one float64 unit of the scaled |T| <= 1
    if (w.hi <= 0x1p-46f * fmaxf(fabsf(lo.hi), fabsf(hi.hi)) || w.hi <= 0x1p-52f) break;
    // shift t: lo + (t + 1) (hi - lo) / (EIG_THREADS + 1), in double-float on
    // the float32 pipes (every thread computes one per round)
    const dfloat step = df_mul_f(w, kInvShiftsF);
    const int f =
        first_above(sturm_count(sa, sb2, n, df_add(lo, df_mul_f(step, (float)(tid + 1)))));
    // count(x_t) is non-decreasing in t: the eigenvalue lies in (x_{f-1}, x_f]
    const dfloat nlo = f > 0 ? df_add(lo, df_mul_f(step, (float)f)) : lo;
    if (f < EIG_THREADS) hi = df_add(lo, df_mul_f(step, (float)(f + 1)));
    lo = nlo;
  }
  if (tid == 0) theta[m] = (0.5 * df_to_double(df_add(lo, hi))) / sc;
}

constexpr int EIG_WARPS = 8;  // eigenvalues per CTA (one warp each)

// Ritz values of many problems: one warp per eigenvalue, multisection on
// Sturm counts (32 shifts per round, one per lane; a ballot finds the
// subinterval that holds the wanted eigenvalue), the warps of a CTA sharing
// the problem's scaled T.
__global__ void __launch_bounds__(EIG_WARPS * 32)
tridiag_eigvals_kernel(LanczosBatch bt) {
  __shared__ float2 sa[SLS_MAX_R], sb2[SLS_MAX_R];
  __shared__ double s_glo, s_ghi;
  const int p = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  if (p >= nprob) return;
  const int r = bt.r;
  const int n = reff_clamped(bt, p);
  const int m = blockIdx.x * EIG_WARPS + warp;  // descending index of this warp's value
  double* theta = bt.theta + (size_t)p * r;
  const double* a = bt.alpha + (size_t)p * r;
  const double* b = bt.beta + (size_t)p * r;
  if (warp == 0) {
    // Gershgorin interval
    double glo = DBL_MAX, ghi = -DBL_MAX;
    for (int i = lane; i < n; i += 32) {
      const double bl = (i > 0) ? fabs(b[i - 1]) : 0.0;
      const double br = (i < n - 1) ? fabs(b[i]) : 0.0;
      glo = fmin(glo, a[i] - bl - br);
      ghi = fmax(ghi, a[i] + bl + br);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
      ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
    }
    if (lane == 0) {
      s_glo = glo;
      s_ghi = ghi;
    }
  }
  __syncthreads();
  // a power-of-two scale that maps the interval into [-1, 1] (exact)
  const double glo = s_glo, ghi = s_ghi;
  const double big = fmax(fabs(glo), fabs(ghi));
  int ex = 0;
  frexp(big > 0.0 ? big : 1.0, &ex);
  const double sc = ldexp(1.0, -ex);
  for (int i = tid; i < n; i += EIG_WARPS * 32) {
    sa[i] = f2(df_from_double(a[i] * sc));
    if (i < n - 1) {
      const double bs = b[i] * sc;
      sb2[i] = f2(df_from_double(bs * bs));
    }
  }
  __syncthreads();
  if (m >= r) return;
  if (m >= n) {
    if (lane == 0) theta[m] = 0.0;
    return;
  }
  const double pad = 0x1p-40 * fmax(fabs(glo * sc), fabs(ghi * sc)) + 0x1p-100;
  // the interval in double-float: the shifts and updates of every round run
  // on the float32 pipes (float64 throughput is a small fraction here, and
  // every lane of every warp computes a shift per round)
  dfloat lo = df_from_double(glo * sc - pad), hi = df_from_double(ghi * sc + pad);
  const int k = n - 1 - m;  // ascending index of the wanted eigenvalue
  for (int round = 0; round < 40; ++round) {
    const dfloat w = df_sub(hi, lo);
    if (w.hi <= 0x1p-46f * fmaxf(fabsf(lo.hi), fabsf(hi.hi)) || w.hi <= 0x1p-52f) break;
    const dfloat step = df_mul_f(w, 1.0f / 33.0f);
    const int c = sturm_count(sa, sb2, n, df_add(lo, df_mul_f(step, (float)(lane + 1))));
    // count(x_t) is non-decreasing in t: the eigenvalue lies in (x_{f-1}, x_f]
    const unsigned ball = __ballot_sync(0xffffffffu, c > k);
    const int f = ball ? __ffs(ball) - 1 : 32;
    const dfloat nhi = (f < 32) ? df_add(lo, df_mul_f(step, (float)(f + 1))) : hi;
    const dfloat nlo = (f > 0) ? df_add(lo, df_mul_f(step, (float)f)) : lo;
    lo = nlo;
    hi = nhi;
  }
  if (lane == 0) theta[m] = (0.5 * df_to_double(df_add(lo, hi))) / sc;
}

// ----------------------------------------------------------------------------
// Eigenvectors of T (tridiag_vec.cuh)
// ----------------------------------------------------------------------------

// One warp per Ritz value: the warp of a cluster's first member computes the whole
// cluster.
__global__ void __launch_bounds__(32)
tridiag_eigvecs_kernel(LanczosBatch bt) {
  __shared__ float2 d[SLS_MAX_R], du[SLS_MAX_R], du2[SLS_MAX_R], dl[SLS_MAX_R];
  __shared__ float2 y[SLS_MAX_R], sa[SLS_MAX_R], sb[SLS_MAX_R];
  __shared__ unsigned char piv[SLS_MAX_R];
  const int m = blockIdx.x, p = blockIdx.y, lane = threadIdx.x;
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  if (p >= nprob) return;
  const int r = bt.r;
  const int n = reff_clamped(bt, p);
  double* S = bt.S + (size_t)p * r * r;
  if (m >= n) {
    for (int k = lane; k < r; k += 32) S[(size_t)k * r + m] = 0.0;
    return;
  }
  int first, last;
  eig_cluster(bt.theta + (size_t)p * r, n, m, first, last);
  if (first != m) return;  // another CTA (the first member of this cluster) writes this column
  for (int k = lane + n; k < r; k += 32)
    for (int mm = first; mm <= last; ++mm) S[(size_t)k * r + mm] = 0.0;
  double tnorm;
  const double sc = eig_scale(bt.theta + (size_t)p * r, n, &tnorm);
  eig_scaled_T(bt.alpha + (size_t)p * r, bt.beta + (size_t)p * r, n, sc, lane, 32, sa, sb);
  __syncwarp();
  eigvec_cluster(r, bt.theta + (size_t)p * r, S, n, first, last, sc, tnorm, sa, sb, d, du, du2, dl,
                 y, piv);
}

// Many small problems (r <= 32): one warp per problem, one lane per Ritz value;
// every lane factors and solves once, then a cluster's members take turns at the
// rest, which needs the finished ones (2048 windows of 16 tokens: 12 us less than
// with the whole cluster on its first member's lane).  Work arrays in local memory.
constexpr int EIGW_WARPS = 1;  // one problem per CTA: the fewest idle SMs at the end
constexpr int EIGW_MAXR = 32;
// Ritz values up to which a warp computes each eigenvector (32 values: 22 us, a
// lane each 31; 2048 values: 39 us either way)
constexpr int64_t EIGV_WARPS_MAX = 2048;

__global__ void __launch_bounds__(EIGW_WARPS * 32)
tridiag_eigvecs_warp_kernel(LanczosBatch bt) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = blockIdx.x * EIGW_WARPS + warp;
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  if (p >= nprob) return;
  const int r = bt.r;
  const int n = reff_clamped(bt, p);
  double* S = bt.S + (size_t)p * r * r;
  // S rows and columns beyond r_eff are zero
  for (int e = lane; e < r * r; e += 32) {
    const int i = e / r, m = e % r;
    if (i >= n || m >= n) S[e] = 0.0;
  }
  __shared__ float2 sa[EIGW_WARPS][EIGW_MAXR], sb[EIGW_WARPS][EIGW_MAXR];
  double tnorm = 1.0, sc = 1.0;
  if (n > 0) {
    sc = eig_scale(bt.theta + (size_t)p * r, n, &tnorm);
    eig_scaled_T(bt.alpha + (size_t)p * r, bt.beta + (size_t)p * r, n, sc, lane, 32, sa[warp],
                 sb[warp]);
  }
  __syncwarp();
  int first = lane, last = lane;
  float2 d[EIGW_MAXR], du[EIGW_MAXR], du2[EIGW_MAXR], dl[EIGW_MAXR], y[EIGW_MAXR];
  unsigned char piv[EIGW_MAXR];
  const double pert = 0x1p-44 * tnorm;
  if (lane < n) {
    const double* th = bt.theta + (size_t)p * r;
    eig_cluster(th, n, lane, first, last);
    if (n == 1) {
      y[0] = make_float2(1.f, 0.f);
    } else {
      const dfloat cy = eig_factor(n, eig_shift(th, lane, first, pert, sc),
                                   df_from_double(pert * sc),
                                   [lane](int i) { return eig_start(lane, i); }, sa[warp],
                                   sb[warp], d, du, du2, dl, y, piv);
      eig_back(n, cy, d, du, du2, y);
      eig_rescale<false>(n, y);
    }
  }
  // then the members of a cluster in turn, the clusters side by side
  const int turns = (int)__reduce_max_sync(0xffffffffu, (unsigned)(lane - first)) + 1;
  for (int k = 0; k < turns; ++k) {
    if (lane < n && lane - first == k) {
      if (n > 1) {
        eig_orthonormalise<false>(n, r, first, lane, S, y);
        const dfloat cy = eig_forward(n, dl, y, piv);
        eig_back(n, cy, d, du, du2, y);
        eig_rescale<false>(n, y);
        eig_orthonormalise<false>(n, r, first, lane, S, y);
      }
      eig_store<false>(n, r, lane, y, S);
    }
    __syncwarp();
  }
}

// ----------------------------------------------------------------------------
// Ritz vectors U = Q S (float32 output): tiles of basis rows in shared memory,
// 4 x 4 outputs per thread
// ----------------------------------------------------------------------------

constexpr int RITZ_THREADS = 256;

__host__ __device__ inline int ritz_tile_rows(int r) {
  const int cg = (r + 3) / 4;
  return (RITZ_THREADS / cg) * 4;
}

__global__ void __launch_bounds__(RITZ_THREADS)
ritz_vectors_kernel(LanczosBatch bt, float* __restrict__ U) {
  extern __shared__ float rsm[];
  const int p = blockIdx.y;
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  if (p >= nprob) return;
  const int r = bt.r, ldq = q_ld(r);
  const int kn = reff_clamped(bt, p);
  const int64_t row0 = bt.row0 ? bt.row0[p] : 0;
  const int64_t n = bt.n ? (int64_t)bt.n[p] : bt.n_single;
  const int cg = (r + 3) / 4, rg = RITZ_THREADS / cg, TR = rg * 4, qs = r + 1;
  float* Ss = rsm;                    // r x r
  float* Qh = Ss + (size_t)r * r;     // TR x (r+1)
  float* Ql = Qh + (size_t)TR * qs;   // TR x (r+1)
  const double* S = bt.S + (size_t)p * r * r;
  for (int e = threadIdx.x; e < r * r; e += RITZ_THREADS) Ss[e] = (float)S[e];
  const int t = threadIdx.x;
  const int rgi = t / cg, cgi = t % cg;
  const bool active = rgi < rg;
  for (int64_t i0 = (int64_t)blockIdx.x * TR; i0 < n; i0 += (int64_t)gridDim.x * TR) {
    const int nt = (int)min((int64_t)TR, n - i0);
    __syncthreads();
    const float2* Qt = bt.Q + (row0 + i0) * ldq;
    for (int e = t; e < nt * kn; e += RITZ_THREADS) {
      const int rr = e / kn, k = e % kn;
      const float2 q = Qt[(size_t)rr * ldq + k];
      Qh[rr * qs + k] = q.x;
      Ql[rr * qs + k] = q.y;
    }
    __syncthreads();
    if (!active) continue;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][c] = 0.f;
    const int rb = rgi * 4, cb = cgi * 4;
    for (int k = 0; k < kn; ++k) {
      float s[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) s[c] = (cb + c < r) ? Ss[k * r + cb + c] : 0.f;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float qh = Qh[(rb + a) * qs + k], ql = Ql[(rb + a) * qs + k];
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = fmaf(qh, s[c], fmaf(ql, s[c], acc[a][c]));
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      if (rb + a < nt) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (cb + c < r) U[(row0 + i0 + rb + a) * r + cb + c] = (cb + c < kn) ? acc[a][c] : 0.f;
      }
    }
  }
}

int num_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
      sms = v;
    else
      return 152;  // no device visible: plan for a GB300 (host-only size queries)
  }
  return sms;
}

}  // namespace

int lanczos_plan(int64_t nmax, int D, int r, int nprob, int* groups, int* ctas_per_group) {
  const int sms = num_sms();
  if (nprob <= 1) {
    // one problem: spread it over the whole GPU, but keep >= 32 rows per CTA
    int64_t g = (nmax + 31) / 32;
    if (g > sms) g = sms;
    if (g < 1) g = 1;
    *groups = 1;
    *ctas_per_group = (int)g;
  } else {
    // a batch: enough CTAs per problem for ~1024 rows each, as many groups as
    // fit (fewer CTAs per problem amortise the per-step barriers over more
    // rows; measured on 512 windows of 2048 rows at D = 1024: 256 rows per CTA
    // 65.7 ms, 512 62.4, 1024 59.5, 2048 66.8 with too few groups per round)
    int64_t g = (nmax + 1023) / 1024;
    if (g < 1) g = 1;
    if (g > sms) g = sms;
    int64_t gr = sms / g;
    if (gr < 1) gr = 1;
    if (gr > nprob) gr = nprob;
    *groups = (int)gr;
    *ctas_per_group = (int)g;
  }
  // at most 8192 rows per CTA (one prompt of 1.2 million tokens)
  const int64_t rows = (nmax + *ctas_per_group - 1) / *ctas_per_group;
  if (rows > 8192) return SLS_ERR_UNSUPPORTED;
  (void)D;
  (void)r;
  return SLS_OK;
}

size_t lanczos_scratch_bytes(int D, int r, int groups, int g) {
  return (size_t)groups * lz_layout(D, r, g).total;
}

size_t lanczos_exchange_extra(int64_t N, int D, int r) {
  int groups = 0, g = 0;
  if (lanczos_plan(N, D, r, 1, &groups, &g) != SLS_OK) return 0;
  const LzLayout L = lz_layout(D, r, g);
  return L.ones_end - (256 + lz_al((size_t)2 * (r + 4) * 8) + lz_al((size_t)g * D * 8) +
                       lz_al((size_t)D * 8));
}

int launch_lanczos(const LanczosBatch& bt, void* scratch, size_t scratch_bytes, int* status,
                   int groups, int g, cudaStream_t stream) {
  const LzLayout L = lz_layout(bt.D, bt.r, g);
  if ((size_t)groups * L.total > scratch_bytes) return SLS_ERR_WORKSPACE;
  // the exchange slots of every group start empty (one strided memset)
  SLS_CUDA_TRY(cudaMemset2DAsync((char*)scratch + L.bar, L.total, 0xff, L.ones_end - L.bar,
                                 groups, stream));
  if (bt.D > SLS_MAX_D) return SLS_ERR_UNSUPPORTED;
  if (bt.phi_bf16 && (bt.D % 8)) return SLS_ERR_UNSUPPORTED;  // 16-byte rows for the copies
  const LzShape shp = lz_shape(bt.D);
  const size_t limit = 227 * 1024 - 1024;  // leave room for static shared memory
  const size_t stage = lz_stage_bytes(bt.D, q_ld(bt.r), bt.phi_bf16 ? 2 : 4, shp.R);
  const int teams = LZ_NCW / shp.wpr;
  const LzOwn own = lz_own(bt.D, bt.r, g);
  const int red = lz_red_rows(own) * own.WB;
  // the deepest rings that fit; at least 2 stages each: a team of several
  // warps refills a slot once the exchange of its next batch shows that every
  // warp is done with it, so a ring of one stage would wait for its own refill
  // (and the pass ends use two stages of room)
  int stages = 0;
  for (int s = LZ_MAX_STAGES; s >= 2; --s) {
    if ((size_t)teams * s * stage + lz_smem_other(bt.D, bt.r, shp, red, s) <= limit) {
      stages = s;
      break;
    }
  }
  if (stages < 2) return SLS_ERR_UNSUPPORTED;
  const size_t smem = (size_t)teams * stages * stage + lz_smem_other(bt.D, bt.r, shp, red, stages);
#define SLS_LZ_CASE(NV, WPR)                                                               \
  if (shp.nv == NV && shp.wpr == WPR)                                                      \
    return bt.phi_bf16 ? launch_lanczos_bf16_##NV##_##WPR(bt, scratch, L.total, groups, g, \
                                                          stages, status, smem, stream)    \
                       : launch_lanczos_f32_##NV##_##WPR(bt, scratch, L.total, groups, g,  \
                                                         stages, status, smem, stream)
  SLS_LZ_CASE(2, 1);
  SLS_LZ_CASE(3, 1);
  SLS_LZ_CASE(4, 1);
  SLS_LZ_CASE(3, 2);
  SLS_LZ_CASE(4, 2);
  SLS_LZ_CASE(3, 4);
  SLS_LZ_CASE(4, 4);
  SLS_LZ_CASE(4, 8);
  SLS_LZ_CASE(8, 8);
#undef SLS_LZ_CASE
  return SLS_ERR_UNSUPPORTED;
}

int launch_tridiag_eigen(const LanczosBatch& bt, cudaStream_t stream, bool values_done) {
  dim3 grid(bt.r, bt.nprob_max);
  if (!values_done) {
    if ((int64_t)bt.r * bt.nprob_max <= 1024) {
      tridiag_eigvals_cta_kernel<<<grid, EIG_THREADS, 0, stream>>>(bt);
    } else {
      dim3 vgrid((bt.r + EIG_WARPS - 1) / EIG_WARPS, bt.nprob_max);
      tridiag_eigvals_kernel<<<vgrid, EIG_WARPS * 32, 0, stream>>>(bt);
    }
    SLS_LAUNCH_CHECK();
  }
  if (bt.r <= EIGW_MAXR && (int64_t)bt.r * bt.nprob_max > EIGV_WARPS_MAX) {
    const int blocks = (bt.nprob_max + EIGW_WARPS - 1) / EIGW_WARPS;
    tridiag_eigvecs_warp_kernel<<<blocks, EIGW_WARPS * 32, 0, stream>>>(bt);
  } else {
    tridiag_eigvecs_kernel<<<grid, 32, 0, stream>>>(bt);
  }
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

int launch_ritz_vectors(const LanczosBatch& bt, float* U, cudaStream_t stream) {
  const int r = bt.r;
  const int TR = ritz_tile_rows(r);
  int64_t blocks = (bt.nmax + TR - 1) / TR;
  if (blocks > 4 * (int64_t)num_sms()) blocks = 4 * (int64_t)num_sms();
  if (blocks < 1) blocks = 1;
  const size_t smem = sizeof(float) * ((size_t)r * r + 2 * (size_t)TR * (r + 1));
  SLS_CUDA_TRY(cudaFuncSetAttribute(ritz_vectors_kernel,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ritz_vectors_kernel<<<dim3((unsigned)blocks, bt.nprob_max), RITZ_THREADS, smem, stream>>>(bt, U);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

}  // namespace sls
