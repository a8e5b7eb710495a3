// SimHash (Sec. 3.3), clusters and the exact-length adjustment (Sec. 3.3),
// macro-token aggregation with positions (Sec. 3.4) and the window
// redundancy score of the adaptive router (Sec. 3.6, Eq. redundancy).
//
// Work is organised by "problems" (one token set compressed on its own; see
// segment.cuh).  The per-problem bookkeeping -- a stable radix sort of
// (code, token), cluster boundaries, the merge or D'Hondt split to exactly m
// groups, group positions and the ordering of groups by position -- runs in
// one 1024-thread CTA per problem (a cluster of them for one large problem, a
// warp for windows of at most 32 tokens) and touches only integers.  Reading X and
// writing the macro-token embeddings is spread over the whole GPU.
#include <atomic>
#include <climits>

#include "common.cuh"
#include "kernels.cuh"
#include "segment.cuh"

namespace sls {

// ============================================================================
// SimHash: code[i] = sum_l [ fl32 dot(U[i,:k], R[l,:k]) > 0 ] << l
// ============================================================================

namespace {

// cp.async of 16 or 4 bytes (the first `bytes` of them, zeros after), and the
// wait for all but the newest `pending` groups of a thread's copies.
SLS_DEV void cp_async16(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
SLS_DEV void cp_async4(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
SLS_DEV void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
SLS_DEV void cp_async_wait_pending(int pending) {
  switch (pending) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
  }
}

// One tile of SimHash.  A thread forms the dots of RPT rows with eight
// hyperplanes by the fixed float32 chain of the specification (acc = 0; for m =
// 0 .. k-1: acc = fl(acc + fl(U[i,m] * R[l,m])), multiply and add rounded
// separately; two hyperplanes per packed instruction); the 2^lg threads of a row
// are neighbouring lanes and OR their bits.  The rows come through shared memory
// by asynchronous copies in groups of SH_MC columns, all in flight at once, so
// that the first groups' arithmetic hides the later groups' arrival.
//
// Bound by the packed multiplies and adds (N bits k / 2 each at two cycles a
// warp: 6.7 us at N = 131060, k = 64, 16 bits, against 5 us for reading U).  The
// former kernel, a lane per hyperplane with a row's elements read by every lane,
// spent a load and an address per multiply; sls_simhash there 48 -> 18 us a call
// (16 of them the host's, when nothing else runs), N = 32000, 20 bits 24 -> 17.
constexpr int SH_T = 128;   // threads per CTA
constexpr int SH_MC = 16;   // columns per copy group
constexpr int SH_LMAX = 32; // row length of the transposed hyperplanes

__host__ __device__ inline int sh_lg(int bits) { return bits <= 8 ? 0 : bits <= 16 ? 1 : 2; }
__host__ __device__ inline int sh_rows(int bits, int rpt) { return (SH_T >> sh_lg(bits)) * rpt; }
__host__ __device__ inline size_t sh_smem(int bits, int k, int rpt) {
  const size_t k4 = (size_t)((k + 3) & ~3);
  return sizeof(float) * (k4 * SH_LMAX + (size_t)sh_rows(bits, rpt) * (k4 + 4));
}

// R (bits x kk, row stride ldr) transposed into Rt[m][l], zero where there is
// no hyperplane or column
SLS_DEV void simhash_stage_R(const float* __restrict__ R, int ldr, int bits, int kk, float* Rt) {
  const int k4 = (kk + 3) & ~3;
  for (int e = threadIdx.x; e < k4 * SH_LMAX; e += SH_T) {
    const int l = e & (SH_LMAX - 1), m = e / SH_LMAX;
    Rt[e] = (l < bits && m < kk) ? R[(size_t)l * ldr + m] : 0.f;
  }
}

template <int RPT>
SLS_DEV void simhash_tile(const float* __restrict__ U, int64_t n, int64_t r0, int ldu, bool vec,
                          int kk, const float* Rt, float* Us, int bits,
                          uint32_t* __restrict__ codes) {
  const int tid = threadIdx.x;
  const int lg = sh_lg(bits), rows = sh_rows(bits, RPT);
  const int k4 = (kk + 3) & ~3, us = k4 + 4;  // 16-byte rows, no bank conflicts
  const int nch = (k4 + SH_MC - 1) / SH_MC;
  for (int c = 0; c < nch; ++c) {
    for (int e = tid; e < rows * (SH_MC / 4); e += SH_T) {
      const int row = e / (SH_MC / 4), col = c * SH_MC + 4 * (e % (SH_MC / 4));
      if (col < k4) {
        const bool live = r0 + row < n;
        const float* src = U + (live ? r0 + row : 0) * ldu;
        const int left = live ? min(4, kk - col) : 0;  // elements of the quad that exist
        float* dst = Us + row * us + col;
        if (vec) {
          cp_async16(dst, left ? src + col : src, 4 * left);
        } else {
#pragma unroll
          for (int x = 0; x < 4; ++x) cp_async4(dst + x, x < left ? src + col + x : src, x < left ? 4 : 0);
        }
      }
    }
    cp_async_commit_group();
  }
  const int slot = tid >> lg, grp = tid & ((1 << lg) - 1);
  f32x2_t acc[RPT][4];
#pragma unroll
  for (int s = 0; s < RPT; ++s)
#pragma unroll
    for (int h = 0; h < 4; ++h) acc[s][h] = 0ull;
  const float* up = Us + slot * us;
  const float* rp = Rt + grp * 8;
  for (int c = 0; c < nch; ++c) {
    cp_async_wait_pending(nch - 1 - c);
    __syncthreads();
    const int m1 = min(k4, (c + 1) * SH_MC);
#pragma unroll 2
    for (int m = c * SH_MC; m < m1; m += 4) {
      float4 u[RPT];
#pragma unroll
      for (int s = 0; s < RPT; ++s)
        u[s] = *reinterpret_cast<const float4*>(up + s * (SH_T >> lg) * us + m);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float4 ra = *reinterpret_cast<const float4*>(rp + (m + x) * SH_LMAX);
        const float4 rb = *reinterpret_cast<const float4*>(rp + (m + x) * SH_LMAX + 4);
        const f32x2_t r0p = pk2(ra.x, ra.y), r1p = pk2(ra.z, ra.w);
        const f32x2_t r2p = pk2(rb.x, rb.y), r3p = pk2(rb.z, rb.w);
#pragma unroll
        for (int s = 0; s < RPT; ++s) {
          const float ux = x == 0 ? u[s].x : x == 1 ? u[s].y : x == 2 ? u[s].z : u[s].w;
          const f32x2_t uu = pk2(ux, ux);
          acc[s][0] = add2(acc[s][0], mul2(uu, r0p));
          acc[s][1] = add2(acc[s][1], mul2(uu, r1p));
          acc[s][2] = add2(acc[s][2], mul2(uu, r2p));
          acc[s][3] = add2(acc[s][3], mul2(uu, r3p));
        }
      }
    }
  }
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    unsigned code = 0u;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float a, b;
      upk2(acc[s][h], a, b);
      code |= (a > 0.f ? 1u : 0u) << (2 * h);
      code |= (b > 0.f ? 1u : 0u) << (2 * h + 1);
    }
    code <<= 8 * grp;
    if (lg > 0) code |= __shfl_xor_sync(0xffffffffu, code, 1);
    if (lg > 1) code |= __shfl_xor_sync(0xffffffffu, code, 2);
    const int64_t i = r0 + slot + s * (SH_T >> lg);
    if (grp == 0 && i < n) codes[i] = code;
  }
}

SLS_DEV bool simhash_vec(const float* U, int ldu) {
  return (reinterpret_cast<uintptr_t>(U) & 15u) == 0 && (ldu & 3) == 0;
}

template <int RPT>
__global__ void __launch_bounds__(SH_T)
simhash_kernel(const float* __restrict__ U, int64_t N, int k, int ldu,
               const int32_t* __restrict__ k_dev, const float* __restrict__ R, int bits,
               int ldr, uint32_t* __restrict__ codes) {
  extern __shared__ __align__(16) float sh_smem_f[];
  int kk = k;
  if (k_dev) kk = min(kk, max(0, (int)*k_dev));
  simhash_stage_R(R, ldr, bits, kk, sh_smem_f);
  __syncthreads();
  simhash_tile<RPT>(U, N, (int64_t)blockIdx.x * sh_rows(bits, RPT), ldu, simhash_vec(U, ldu), kk,
                    sh_smem_f, sh_smem_f + ((kk + 3) & ~3) * SH_LMAX, bits, codes);
}

// Batched over spectral problems: rows of problem p start at phi_row, k is
// the problem's r_eff, bits its own bit count; tiles of a problem over x.
__global__ void __launch_bounds__(SH_T)
simhash_batched_kernel(const ProbDesc* __restrict__ probs, const int* __restrict__ spec_list,
                       const int* __restrict__ nspec_dev, int nspec_max,
                       const int* __restrict__ r_eff, const float* __restrict__ U, int ldu,
                       const float* __restrict__ R, int ldr, uint32_t* __restrict__ codes) {
  extern __shared__ __align__(16) float sh_smem_f[];
  const int s = blockIdx.y;
  int nspec = nspec_max;
  if (nspec_dev) nspec = min(nspec, *nspec_dev);
  if (s >= nspec) return;
  const ProbDesc P = probs[spec_list ? spec_list[s] : s];
  const int rows = sh_rows(P.bits, 1);
  if ((int64_t)blockIdx.x * rows >= P.n) return;
  const int kk = min(ldu, max(0, r_eff[s]));
  simhash_stage_R(R, ldr, P.bits, kk, sh_smem_f);
  __syncthreads();
  const float* Up = U + (int64_t)P.phi_row * ldu;
  for (int64_t r0 = (int64_t)blockIdx.x * rows; r0 < P.n; r0 += (int64_t)gridDim.x * rows) {
    simhash_tile<1>(Up, P.n, r0, ldu, simhash_vec(Up, ldu), kk, sh_smem_f,
                    sh_smem_f + ((kk + 3) & ~3) * SH_LMAX, P.bits, codes + P.phi_row);
    __syncthreads();
  }
}

// Small problems (windows of at most SH_FLAT_MAX tokens): one thread per
// (problem, row) over all spectral problems, R read through the read-only
// cache (row l of R at R + l * ldr), the same float32 chain as simhash_tile.
constexpr int SH_FLAT_MAX = 64;

__global__ void __launch_bounds__(256)
simhash_flat_kernel(const ProbDesc* __restrict__ probs, const int* __restrict__ spec_list,
                    const int* __restrict__ nspec_dev, int nspec_max, int nmax,
                    const int* __restrict__ r_eff, const float* __restrict__ U, int ldu,
                    const float* __restrict__ R, int ldr, uint32_t* __restrict__ codes) {
  int nspec = nspec_max;
  if (nspec_dev) nspec = min(nspec, *nspec_dev);
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int s = (int)(t / nmax), i = (int)(t % nmax);
  if (s >= nspec) return;
  const ProbDesc P = probs[spec_list ? spec_list[s] : s];
  if (i >= P.n) return;
  const int k = min(ldu, max(0, r_eff[s]));
  const float* __restrict__ u = U + (P.phi_row + i) * ldu;
  float acc[SLS_MAX_BITS];
#pragma unroll
  for (int l = 0; l < SLS_MAX_BITS; ++l) acc[l] = 0.0f;
  for (int m = 0; m < k; ++m) {
    const float um = __ldg(u + m);
#pragma unroll
    for (int l = 0; l < SLS_MAX_BITS; ++l)
      if (l < P.bits) acc[l] = __fadd_rn(acc[l], __fmul_rn(um, __ldg(R + (size_t)l * ldr + m)));
  }
  uint32_t code = 0;
#pragma unroll
  for (int l = 0; l < SLS_MAX_BITS; ++l)
    if (l < P.bits && acc[l] > 0.0f) code |= (1u << l);
  codes[P.phi_row + i] = code;
}

// ============================================================================
// block-level integer primitives (1024 threads)
// ============================================================================

constexpr int SEG_T = 1024;
constexpr int SEG_W = SEG_T / 32;

SLS_DEV unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Exclusive scan of 1024 per-thread values; returns the exclusive prefix of
// the calling thread, *total receives the sum.  sh: SEG_W + 1 ints.
template <typename T>
SLS_DEV T block_excl_scan(T v, T* sh, T* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  if (warp == 0) {
    T w = (lane < SEG_W) ? sh[lane] : (T)0;
    T z = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, z, o);
      if (lane >= o) z += y;
    }
    if (lane < SEG_W) sh[lane] = z - w;
    if (lane == SEG_W - 1) sh[SEG_W] = z;
  }
  __syncthreads();
  const T res = sh[warp] + x - v;
  *total = sh[SEG_W];
  __syncthreads();
  return res;
}

// Exclusive scan of in[0..n) into out (may alias); returns the total.
// Each thread scans a contiguous chunk serially.
template <typename T>
SLS_DEV T block_scan_array(const T* in, T* out, int n, T* sh) {
  const int tid = threadIdx.x;
  const int chunk = (n + SEG_T - 1) / SEG_T;
  const int b = min(n, tid * chunk), e = min(n, b + chunk);
  T s = 0;
  for (int i = b; i < e; ++i) s += in[i];
  T total;
  T off = block_excl_scan<T>(s, sh, &total);
  for (int i = b; i < e; ++i) {
    const T v = in[i];
    out[i] = off;
    off += v;
  }
  __syncthreads();
  return total;
}

template <typename T>
SLS_DEV T block_sum(T v, T* sh) {
  T total;
  block_excl_scan<T>(v, sh, &total);
  return total;
}

// Stable LSD radix sort of (key, val) pairs on the low key_bits bits, one
// 8-bit digit per pass, ping-ponging between the (ka, va) and (kb, vb)
// buffers in global memory.  On return (ka, va) point at the sorted data.
// sh: 256 + 256 + SEG_W * 256 ints.
template <typename K>
SLS_DEV void block_radix_sort(K*& ka, int*& va, K*& kb, int*& vb, int n, int key_bits, int* sh) {
  int* base = sh;
  int* tot = sh + 256;
  int* wc = sh + 512;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int shift = 0; shift < key_bits; shift += 8) {
    if (tid < 256) base[tid] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += SEG_T) atomicAdd(&base[(int)((ka[i] >> shift) & 255)], 1);
    __syncthreads();
    if (tid < 256) {
      // exclusive scan of 256 bins by the first 8 warps
      int v = base[tid];
      int x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) tot[warp] = x;
      __syncwarp();
      x -= v;
      base[tid] = x;  // warp-local exclusive prefix
    }
    __syncthreads();
    if (tid < 256) {
      int add = 0;
      for (int w = 0; w < warp; ++w) add += tot[w];
      base[tid] += add;
    }
    __syncthreads();
    for (int t0 = 0; t0 < n; t0 += SEG_T) {
      for (int e = tid; e < SEG_W * 256; e += SEG_T) wc[e] = 0;
      __syncthreads();
      const int i = t0 + tid;
      const bool valid = i < n;
      K key = 0;
      int val = 0;
      unsigned dg = 256u + (unsigned)lane;
      if (valid) {
        key = ka[i];
        val = va[i];
        dg = (unsigned)((key >> shift) & 255);
      }
      const unsigned peers = __match_any_sync(0xffffffffu, dg);
      const int rank = __popc(peers & lanemask_lt());
      if (valid && rank == 0) wc[warp * 256 + dg] = __popc(peers);
      __syncthreads();
      if (tid < 256) {
        int run = 0;
        for (int w = 0; w < SEG_W; ++w) {
          const int c = wc[w * 256 + tid];
          wc[w * 256 + tid] = run;
          run += c;
        }
        tot[tid] = run;
      }
      __syncthreads();
      if (valid) {
        const int pos = base[dg] + wc[warp * 256 + dg] + rank;
        kb[pos] = key;
        vb[pos] = val;
      }
      __syncthreads();
      if (tid < 256) base[tid] += tot[tid];
      __syncthreads();
    }
    K* tk = ka;
    ka = kb;
    kb = tk;
    int* tv = va;
    va = vb;
    vb = tv;
  }
}

SLS_DEV int bit_length_u64(unsigned long long x) { return x ? 64 - __clzll((long long)x) : 0; }

// Per-problem scratch layout (ints unless noted), identical on host and device.
struct SegLayout {
  size_t ka, kb, va, vb, f, cst, grp, gst, gmax, gmin, gsum, ok_a, ok_b, ov_a, ov_b, oidx, rep,
      seat, gbar, ghist, gcsum, total;
};

__host__ __device__ inline size_t seg_al(size_t x) { return (x + 255) & ~(size_t)255; }

__host__ __device__ inline SegLayout seg_layout(int64_t nmax, int64_t mmax) {
  SegLayout L;
  size_t o = 0;
  const size_t n1 = (size_t)nmax + 1, m1 = (size_t)mmax + 1;
  L.ka = o;   o += seg_al(n1 * 8);   // keys (uint32 for codes, uint64 reused)
  L.kb = o;   o += seg_al(n1 * 8);
  L.va = o;   o += seg_al(n1 * 4);
  L.vb = o;   o += seg_al(n1 * 4);
  L.f = o;    o += seg_al(n1 * 4);
  L.cst = o;  o += seg_al(n1 * 4);
  L.grp = o;  o += seg_al(n1 * 4);
  L.gst = o;  o += seg_al(m1 * 4);
  L.gmax = o; o += seg_al(m1 * 4);
  L.gmin = o; o += seg_al(m1 * 4);
  L.gsum = o; o += seg_al(m1 * 8);
  L.ok_a = o; o += seg_al(m1 * 8);
  L.ok_b = o; o += seg_al(m1 * 8);
  L.ov_a = o; o += seg_al(m1 * 4);
  L.ov_b = o; o += seg_al(m1 * 4);
  L.oidx = o; o += seg_al(m1 * 4);
  L.rep = o;  o += seg_al(m1 * 4);
  L.seat = o; o += seg_al(n1 * 4);
  // grid version (one large problem): barrier words, digit counts per CTA,
  // CTA sums of the scans
  L.gbar = o;  o += 256;
  L.ghist = o; o += seg_al((size_t)256 * 256 * 4);
  L.gcsum = o; o += seg_al((size_t)256 * 4);
  L.total = o;
  return L;
}

// The segment kernel's sort buffers in shared memory (byte offsets): keys
// and values of the (code, token) sort and the 64-bit order keys with their
// values.
constexpr size_t SEG_SMEM_MAX = 180 * 1024;  // beside 35 KB of static shared memory

struct SegSmem {
  size_t ka, kb, va, vb, oka, okb, ova, ovb, total;
};

__host__ __device__ inline SegSmem seg_smem_layout(int64_t nmax, int64_t mmax) {
  SegSmem S;
  const size_t n1 = (size_t)nmax + 1, m1 = (size_t)mmax + 1;
  auto al = [](size_t x) { return (x + 15) & ~(size_t)15; };
  size_t o = 0;
  S.ka = o;  o += al(n1 * 4);
  S.kb = o;  o += al(n1 * 4);
  S.va = o;  o += al(n1 * 4);
  S.vb = o;  o += al(n1 * 4);
  S.oka = o; o += al(m1 * 8);
  S.okb = o; o += al(m1 * 8);
  S.ova = o; o += al(m1 * 4);
  S.ovb = o; o += al(m1 * 4);
  S.total = o;
  return S;
}

// Number of D'Hondt quotients n/m (2 <= m <= n) that are >= a / 2^40.
SLS_DEV long long dhondt_count_ge(long long n, long long a) {
  if (n < 2) return 0;
  long long k = (a == 0) ? n : min(n, (n << 40) / a);
  return k > 1 ? k - 1 : 0;
}

// ============================================================================
// segment kernel: one CTA per problem
// ============================================================================

__global__ void __launch_bounds__(SEG_T, 1)
segment_kernel(const ProbDesc* __restrict__ probs, int nprob, const uint32_t* __restrict__ codes,
               int pos_scheme, int pos_mode, char* scratch, size_t pstride, int64_t nmax,
               int64_t mmax, int* __restrict__ perm, int* __restrict__ mstart,
               int* __restrict__ mlen, int32_t* __restrict__ pos_out,
               int32_t* __restrict__ tok2macro, int chunk_done, int sort_in_smem) {
  __shared__ int sh_sort[512 + SEG_W * 256];
  __shared__ long long sh_ll[SEG_W + 1];
  __shared__ int sh_i[SEG_W + 1];
  extern __shared__ __align__(16) unsigned char seg_dyn[];
  const int tid = threadIdx.x;
  const SegLayout L = seg_layout(nmax, mmax);
  char* sb = scratch + (size_t)blockIdx.x * pstride;
  // the radix sorts' key and value buffers: in shared memory when the launch
  // gave room for them (seg_smem_layout), else in the problem's scratch
  const SegSmem SL = seg_smem_layout(nmax, mmax);
  char* sortb = sort_in_smem ? reinterpret_cast<char*>(seg_dyn) : nullptr;

  for (int p = blockIdx.x; p < nprob; p += gridDim.x) {
    const ProbDesc P = probs[p];
    const int n = P.n, M = P.m;
    if (n <= 0 || M <= 0) continue;
    if (chunk_done && !P.spectral) {
      // outputs already written by the score pass: nothing to aggregate
      for (int t = tid; t < M; t += SEG_T) mlen[P.out0 + t] = 0;
      continue;
    }
    int* va = reinterpret_cast<int*>(sortb ? sortb + SL.va : sb + L.va);
    int* vb = reinterpret_cast<int*>(sortb ? sortb + SL.vb : sb + L.vb);
    int* f = reinterpret_cast<int*>(sb + L.f);
    int* cst = reinterpret_cast<int*>(sb + L.cst);
    int* grp = reinterpret_cast<int*>(sb + L.grp);
    int* gst = reinterpret_cast<int*>(sb + L.gst);
    int* gmax = reinterpret_cast<int*>(sb + L.gmax);
    int* gmin = reinterpret_cast<int*>(sb + L.gmin);
    unsigned long long* gsum = reinterpret_cast<unsigned long long*>(sb + L.gsum);
    int* oidx = reinterpret_cast<int*>(sb + L.oidx);
    int* rep = reinterpret_cast<int*>(sb + L.rep);
    int* seat = reinterpret_cast<int*>(sb + L.seat);
    bool merged = false;

    if (P.spectral) {
      // ---- stable sort of (code, token) ----
      uint32_t* ka = reinterpret_cast<uint32_t*>(sortb ? sortb + SL.ka : sb + L.ka);
      uint32_t* kb = reinterpret_cast<uint32_t*>(sortb ? sortb + SL.kb : sb + L.kb);
      for (int i = tid; i < n; i += SEG_T) {
        ka[i] = codes[P.phi_row + i];
        va[i] = i;
      }
      __syncthreads();
      block_radix_sort<uint32_t>(ka, va, kb, vb, n, P.bits, sh_sort);
      // ---- clusters: runs of equal codes ----
      for (int s = tid; s < n; s += SEG_T) f[s] = (s == 0 || ka[s] != ka[s - 1]) ? 1 : 0;
      __syncthreads();
      const int C = block_scan_array<int>(f, grp, n, sh_i);  // grp[s] = clusters before s
      for (int s = tid; s < n; s += SEG_T)
        if (f[s]) cst[grp[s]] = s;
      if (tid == 0) cst[C] = n;
      __syncthreads();
      if (C >= M) {
        // merge: the cluster of rank t joins group floor(t M / C)
        merged = (C > M);
        for (int t = tid; t < C; t += SEG_T) {
          const int g = (int)(((long long)t * M) / C);
          const int gp = (t == 0) ? -1 : (int)(((long long)(t - 1) * M) / C);
          if (g != gp) gst[g] = cst[t];
        }
      } else {
        // split: D'Hondt seats, one guaranteed per cluster, ties to the lower code
        const long long K = (long long)(M - C);
        int maxn = 0;
        for (int t = tid; t < C; t += SEG_T) maxn = max(maxn, cst[t + 1] - cst[t]);
        // block max via the sum helper on a per-thread max is not valid; use atomics
        if (tid == 0) sh_i[0] = 0;
        __syncthreads();
        atomicMax(&sh_i[0], maxn);
        __syncthreads();
        maxn = sh_i[0];
        __syncthreads();
        long long lo = 0, hi = ((long long)maxn) << 40;
        while (hi - lo > 1) {
          const long long mid = lo + (hi - lo) / 2;
          long long c = 0;
          for (int t = tid; t < C; t += SEG_T) c += dhondt_count_ge(cst[t + 1] - cst[t], mid);
          c = block_sum<long long>(c, sh_ll);
          if (c >= K) lo = mid;
          else hi = mid;
        }
        // seats strictly above the K-th quotient, and ties at it (<= 1 per cluster)
        long long gt_sum = 0;
        for (int t = tid; t < C; t += SEG_T) {
          const long long nt = cst[t + 1] - cst[t];
          const long long ge = dhondt_count_ge(nt, lo);
          const long long gt = dhondt_count_ge(nt, lo + 1);
          seat[t] = (int)gt;
          f[t] = (int)(ge - gt);
          gt_sum += gt;
        }
        gt_sum = block_sum<long long>(gt_sum, sh_ll);
        const int R = (int)(K - gt_sum);
        __syncthreads();
        // exclusive scan of the tie flags in cluster order
        int* eqs = grp;  // reuse as scratch (size >= C)
        block_scan_array<int>(f, eqs, C, sh_i);
        for (int t = tid; t < C; t += SEG_T) {
          const int extra = (f[t] && eqs[t] < R) ? 1 : 0;
          seat[t] = 1 + seat[t] + extra;
        }
        __syncthreads();
        int* so = f;  // seat offsets
        block_scan_array<int>(seat, so, C, sh_i);
        for (int t = tid; t < C; t += SEG_T) {
          const int nt = cst[t + 1] - cst[t], pt = seat[t];
          const int q = nt / pt, rem = nt % pt;
          for (int k = 0; k < pt; ++k) {
            const int off = (k < rem) ? k * (q + 1) : rem * (q + 1) + (k - rem) * q;
            gst[so[t] + k] = cst[t] + off;
          }
        }
      }
      if (tid == 0) gst[M] = n;
      __syncthreads();
    } else {
      // chunk: contiguous groups (array_split into m, or runs of k)
      for (int i = tid; i < n; i += SEG_T) va[i] = i;
      for (int g = tid; g < M; g += SEG_T) {
        int off;
        if (P.chunk_k > 0) {
          off = min(n, g * P.chunk_k);
        } else {
          const int q = n / M, rem = n % M;
          off = (g < rem) ? g * (q + 1) : rem * (q + 1) + (g - rem) * q;
        }
        gst[g] = off;
      }
      if (tid == 0) gst[M] = n;
      __syncthreads();
    }
    const int* perm_l = va;  // sorted position -> local token
    // ---- group id of every sorted position ----
    for (int s = tid; s < n; s += SEG_T) f[s] = 0;
    __syncthreads();
    for (int g = tid; g < M; g += SEG_T) f[gst[g]] = 1;
    __syncthreads();
    block_scan_array<int>(f, grp, n, sh_i);
    for (int s = tid; s < n; s += SEG_T) grp[s] = grp[s] + f[s] - 1;
    for (int g = tid; g < M; g += SEG_T) {
      gmax[g] = -1;
      gmin[g] = INT_MAX;
      gsum[g] = 0ull;
    }
    __syncthreads();
    for (int s = tid; s < n; s += SEG_T) {
      const int g = grp[s], i = perm_l[s];
      atomicMax(&gmax[g], i);
      atomicMin(&gmin[g], i);
      if (pos_scheme == SLS_POS_MEAN) atomicAdd(&gsum[g], (unsigned long long)i);
    }
    __syncthreads();
    // ---- representative positions ----
    if (pos_scheme == SLS_POS_MEDIAN && merged) {
      // members of merged groups are not in token order: sort (group, token)
      uint32_t* ka = reinterpret_cast<uint32_t*>(sortb ? sortb + SL.ka : sb + L.ka);
      uint32_t* kb = reinterpret_cast<uint32_t*>(sortb ? sortb + SL.kb : sb + L.kb);
      int* xa = seat;
      int* xb = cst;
      for (int s = tid; s < n; s += SEG_T) ka[perm_l[s]] = (uint32_t)grp[s];
      for (int i = tid; i < n; i += SEG_T) xa[i] = i;
      __syncthreads();
      block_radix_sort<uint32_t>(ka, xa, kb, xb, n, bit_length_u64((unsigned long long)M), sh_sort);
      for (int g = tid; g < M; g += SEG_T) rep[g] = xa[gst[g] + (gst[g + 1] - gst[g] - 1) / 2];
    } else {
      for (int g = tid; g < M; g += SEG_T) {
        const int len = gst[g + 1] - gst[g];
        int rp;
        if (pos_scheme == SLS_POS_MAX) rp = gmax[g];
        else if (pos_scheme == SLS_POS_MEDIAN) rp = perm_l[gst[g] + (len - 1) / 2];
        else rp = (int)((2ull * gsum[g] + (unsigned long long)len) / (2ull * (unsigned long long)len));
        rep[g] = rp;
      }
    }
    __syncthreads();
    // ---- order groups by (position, first token) ----
    {
      unsigned long long* oka =
          reinterpret_cast<unsigned long long*>(sortb ? sortb + SL.oka : sb + L.ok_a);
      unsigned long long* okb =
          reinterpret_cast<unsigned long long*>(sortb ? sortb + SL.okb : sb + L.ok_b);
      int* ova = reinterpret_cast<int*>(sortb ? sortb + SL.ova : sb + L.ov_a);
      int* ovb = reinterpret_cast<int*>(sortb ? sortb + SL.ovb : sb + L.ov_b);
      for (int g = tid; g < M; g += SEG_T) {
        oka[g] = (unsigned long long)rep[g] * (unsigned long long)n + (unsigned long long)gmin[g];
        ova[g] = g;
      }
      __syncthreads();
      const int kbits = bit_length_u64((unsigned long long)n * (unsigned long long)n);
      block_radix_sort<unsigned long long>(oka, ova, okb, ovb, M, kbits, sh_sort);
      for (int t = tid; t < M; t += SEG_T) {
        const int g = ova[t];
        oidx[g] = t;
        const int64_t mrow = P.out0 + t;
        mstart[mrow] = (int)(P.tok_row + gst[g]);
        mlen[mrow] = gst[g + 1] - gst[g];
        pos_out[mrow] = (pos_mode == SLS_MODE_COMPACT) ? (P.out_local + t) : (P.pos0 + rep[g]);
      }
      __syncthreads();
      for (int s = tid; s < n; s += SEG_T) {
        const int i = perm_l[s];
        perm[P.tok_row + s] = (int)(P.tok_row + i);
        tok2macro[P.tok_row + i] = P.out_local + oidx[grp[s]];
      }
      __syncthreads();
    }
  }
}

// ============================================================================
// segment kernel for one large problem: the same computation spread over a
// cooperative grid (G CTAs of SEG_T threads), for the single-prompt pass
// ============================================================================

constexpr int SEGG_MAX = 256;           // CTAs of the grid segment kernel, at most

// All CTAs of one thread-block cluster meet (arrive: release, wait: acquire, at
// cluster scope, global memory included).
SLS_DEV void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct GridSync {
  GroupBarrier bar;
  unsigned lgen;
  int* status;
  int* sflag;
  volatile int* serr;
  bool cluster;  // the grid is one cluster: its hardware barrier
};

SLS_DEV bool gsync(GridSync& gs) {
  if (gs.cluster) {
    cluster_sync_all();
    return true;
  }
  return group_sync_named(gs.bar, gs.lgen, gs.status, gs.sflag, gs.serr, 1, SEG_T);
}

// Exclusive scan of in[0..n) into out over the grid; CTA b owns the slice
// [b n / G, (b+1) n / G).  On return this CTA's slice of out is final and the
// total is returned; other slices are final after the next gsync.  csum: G
// ints in global memory.
SLS_DEV bool grid_scan(const int* in, int* out, int n, int* csum, GridSync& gs, int* sh,
                       int* total) {
  const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
  const int c0 = (int)((int64_t)b * n / G), c1 = (int)((int64_t)(b + 1) * n / G);
  const int loc = block_scan_array<int>(in + c0, out + c0, c1 - c0, sh);
  if (tid == 0) csum[b] = loc;
  if (!gsync(gs)) return false;
  int pre = 0, tot = 0;
  for (int c = tid; c < G; c += SEG_T) {
    const int v = csum[c];
    tot += v;
    if (c < b) pre += v;
  }
  pre = block_sum<int>(pre, sh);
  tot = block_sum<int>(tot, sh);
  for (int i = c0 + tid; i < c1; i += SEG_T) out[i] += pre;
  *total = tot;
  __syncthreads();
  return true;
}

// One stable LSD pass (8 bits at `shift`) of (key, val) pairs over the grid:
// per-CTA digit counts, the prefix over (digit, CTA), then the CTA's slice is
// scattered in order (stable within the CTA as in block_radix_sort).
// hist: 256 x G ints in global memory.  sh: 256 + 256 + SEG_W * 256 ints.
template <typename K>
SLS_DEV bool grid_radix_pass(const K* ka, const int* va, K* kb, int* vb, int n, int shift,
                             int* hist, GridSync& gs, int* sh) {
  const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int* base = sh;
  int* tot = sh + 256;
  int* wc = sh + 512;
  const int c0 = (int)((int64_t)b * n / G), c1 = (int)((int64_t)(b + 1) * n / G);
  if (tid < 256) base[tid] = 0;
  __syncthreads();
  for (int i = c0 + tid; i < c1; i += SEG_T) atomicAdd(&base[(int)((ka[i] >> shift) & 255)], 1);
  __syncthreads();
  if (tid < 256) hist[tid * G + b] = base[tid];
  if (!gsync(gs)) return false;
  if (tid < 256) {
    int all = 0, part = 0;
    for (int c = 0; c < G; ++c) {
      const int h = hist[tid * G + c];
      all += h;
      if (c < b) part += h;
    }
    // exclusive scan of the digit totals by the first 8 warps
    int x = all;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) tot[warp] = x;
    base[tid] = x - all + part;
  }
  __syncthreads();
  if (tid < 256) {
    int add = 0;
    for (int w = 0; w < warp; ++w) add += tot[w];
    base[tid] += add;
  }
  __syncthreads();
  for (int t0 = c0; t0 < c1; t0 += SEG_T) {
    for (int e = tid; e < SEG_W * 256; e += SEG_T) wc[e] = 0;
    __syncthreads();
    const int i = t0 + tid;
    const bool valid = i < c1;
    K key = 0;
    int val = 0;
    unsigned dg = 256u + (unsigned)lane;
    if (valid) {
      key = ka[i];
      val = va[i];
      dg = (unsigned)((key >> shift) & 255);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, dg);
    const int rank = __popc(peers & lanemask_lt());
    if (valid && rank == 0) wc[warp * 256 + dg] = __popc(peers);
    __syncthreads();
    if (tid < 256) {
      int run = 0;
      for (int w = 0; w < SEG_W; ++w) {
        const int c = wc[w * 256 + tid];
        wc[w * 256 + tid] = run;
        run += c;
      }
      tot[tid] = run;
    }
    __syncthreads();
    if (valid) {
      const int pos = base[dg] + wc[warp * 256 + dg] + rank;
      kb[pos] = key;
      vb[pos] = val;
    }
    __syncthreads();
    if (tid < 256) base[tid] += tot[tid];
    __syncthreads();
  }
  return gsync(gs);
}

template <typename K>
SLS_DEV bool grid_radix_sort(K*& ka, int*& va, K*& kb, int*& vb, int n, int key_bits, int* hist,
                             GridSync& gs, int* sh) {
  for (int shift = 0; shift < key_bits; shift += 8) {
    if (!grid_radix_pass<K>(ka, va, kb, vb, n, shift, hist, gs, sh)) return false;
    K* tk = ka;
    ka = kb;
    kb = tk;
    int* tv = va;
    va = vb;
    vb = tv;
  }
  return true;
}

__global__ void __launch_bounds__(SEG_T, 1)
segment_grid_kernel(const ProbDesc* __restrict__ probs, const uint32_t* __restrict__ codes,
                    int pos_scheme, int pos_mode, char* sb, int64_t nmax, int64_t mmax,
                    int* __restrict__ perm, int* __restrict__ mstart, int* __restrict__ mlen,
                    int32_t* __restrict__ pos_out, int32_t* __restrict__ tok2macro,
                    int* status, int chunk_done, int cluster) {
  __shared__ int sh_sort[512 + SEG_W * 256];
  __shared__ long long sh_ll[SEG_W + 1];
  __shared__ int sh_i[SEG_W + 1];
  __shared__ int sflag;
  __shared__ volatile int serr;
  const int tid = threadIdx.x, G = gridDim.x, b = blockIdx.x;
  const SegLayout L = seg_layout(nmax, mmax);
  if (tid == 0) serr = 0;
  __syncthreads();
  GridSync gs{GroupBarrier{reinterpret_cast<unsigned*>(sb + L.gbar),
                           reinterpret_cast<unsigned*>(sb + L.gbar) + 32, (unsigned)G},
              0u, status, &sflag, &serr, cluster != 0};
  const ProbDesc P = probs[0];
  const int n = P.n, M = P.m;
  if (n <= 0 || M <= 0) return;
  if (chunk_done && !P.spectral) {  // the whole grid leaves before any grid barrier
    for (int t = b * SEG_T + tid; t < M; t += G * SEG_T) mlen[P.out0 + t] = 0;
    return;
  }
  uint32_t* ka = reinterpret_cast<uint32_t*>(sb + L.ka);
  uint32_t* kb = reinterpret_cast<uint32_t*>(sb + L.kb);
  int* va = reinterpret_cast<int*>(sb + L.va);
  int* vb = reinterpret_cast<int*>(sb + L.vb);
  int* f = reinterpret_cast<int*>(sb + L.f);
  int* cst = reinterpret_cast<int*>(sb + L.cst);
  int* grp = reinterpret_cast<int*>(sb + L.grp);
  int* gst = reinterpret_cast<int*>(sb + L.gst);
  int* gmax = reinterpret_cast<int*>(sb + L.gmax);
  int* gmin = reinterpret_cast<int*>(sb + L.gmin);
  unsigned long long* gsum = reinterpret_cast<unsigned long long*>(sb + L.gsum);
  int* oidx = reinterpret_cast<int*>(sb + L.oidx);
  int* rep = reinterpret_cast<int*>(sb + L.rep);
  int* seat = reinterpret_cast<int*>(sb + L.seat);
  int* hist = reinterpret_cast<int*>(sb + L.ghist);
  int* csum = reinterpret_cast<int*>(sb + L.gcsum);
  const int s0 = (int)((int64_t)b * n / G), s1 = (int)((int64_t)(b + 1) * n / G);
  const int m0 = (int)((int64_t)b * M / G), m1 = (int)((int64_t)(b + 1) * M / G);
  bool merged = false;

  if (P.spectral) {
    // ---- stable sort of (code, token) ----
    for (int i = s0 + tid; i < s1; i += SEG_T) {
      ka[i] = codes[P.phi_row + i];
      va[i] = i;
    }
    if (!gsync(gs)) return;
    if (!grid_radix_sort<uint32_t>(ka, va, kb, vb, n, P.bits, hist, gs, sh_sort)) return;
    // ---- clusters: runs of equal codes ----
    for (int s = s0 + tid; s < s1; s += SEG_T) f[s] = (s == 0 || ka[s] != ka[s - 1]) ? 1 : 0;
    __syncthreads();
    int C = 0;
    if (!grid_scan(f, grp, n, csum, gs, sh_i, &C)) return;  // grp[s] = clusters before s
    for (int s = s0 + tid; s < s1; s += SEG_T)
      if (f[s]) cst[grp[s]] = s;
    if (b == 0 && tid == 0) cst[C] = n;
    if (!gsync(gs)) return;
    if (C >= M) {
      // merge: the cluster of rank t joins group floor(t M / C)
      merged = (C > M);
      const int t0 = (int)((int64_t)b * C / G), t1 = (int)((int64_t)(b + 1) * C / G);
      for (int t = t0 + tid; t < t1; t += SEG_T) {
        const int g = (int)(((long long)t * M) / C);
        const int gp = (t == 0) ? -1 : (int)(((long long)(t - 1) * M) / C);
        if (g != gp) gst[g] = cst[t];
      }
    } else {
      // split: D'Hondt seats, one guaranteed per cluster, ties to the lower
      // code.  The K-th quotient by multisection: every CTA counts the
      // quotients at or above its own threshold, one grid barrier per round.
      const long long K = (long long)(M - C);
      int maxn = 0;
      for (int t = tid; t < C; t += SEG_T) maxn = max(maxn, cst[t + 1] - cst[t]);
      if (tid == 0) sh_i[0] = 0;
      __syncthreads();
      atomicMax(&sh_i[0], maxn);
      __syncthreads();
      maxn = sh_i[0];
      __syncthreads();
      long long lo = 0, hi = ((long long)maxn) << 40;
      long long* cnt = reinterpret_cast<long long*>(hist);  // 2 x G counts by round parity
      for (int round = 0; hi - lo > 1; ++round) {
        // threshold x (1 <= x <= G): lo + x (hi - lo) / (G + 1), the quotient and
        // remainder apart so that nothing overflows
        const long long w = hi - lo, wq = w / (G + 1), wr = w % (G + 1);
        auto thr = [&](int x) { return lo + wq * x + wr * x / (G + 1); };
        const long long mine = thr(b + 1);
        long long c = 0;
        for (int t = tid; t < C; t += SEG_T) c += dhondt_count_ge(cst[t + 1] - cst[t], mine);
        c = block_sum<long long>(c, sh_ll);
        if (tid == 0) cnt[(round & 1) * G + b] = c;
        if (!gsync(gs)) return;
        // counts fall with the threshold: the last one still at K or above
        int ok = 0;
        for (int x = tid; x < G; x += SEG_T) ok += cnt[(round & 1) * G + x] >= K ? 1 : 0;
        const int nok = block_sum<int>(ok, sh_i);
        const long long nlo = nok > 0 ? thr(nok) : lo, nhi = nok < G ? thr(nok + 1) : hi;
        lo = nlo;
        hi = nhi;
      }
      if (b == 0) {
        long long gt_sum = 0;
        for (int t = tid; t < C; t += SEG_T) {
          const long long nt = cst[t + 1] - cst[t];
          const long long ge = dhondt_count_ge(nt, lo);
          const long long gt = dhondt_count_ge(nt, lo + 1);
          seat[t] = (int)gt;
          f[t] = (int)(ge - gt);
          gt_sum += gt;
        }
        gt_sum = block_sum<long long>(gt_sum, sh_ll);
        const int R = (int)(K - gt_sum);
        __syncthreads();
        int* eqs = grp;  // scratch (size >= C)
        block_scan_array<int>(f, eqs, C, sh_i);
        for (int t = tid; t < C; t += SEG_T) {
          const int extra = (f[t] && eqs[t] < R) ? 1 : 0;
          seat[t] = 1 + seat[t] + extra;
        }
        __syncthreads();
        int* so = f;
        block_scan_array<int>(seat, so, C, sh_i);
        for (int t = tid; t < C; t += SEG_T) {
          const int nt = cst[t + 1] - cst[t], pt = seat[t];
          const int q = nt / pt, rem = nt % pt;
          for (int k = 0; k < pt; ++k) {
            const int off = (k < rem) ? k * (q + 1) : rem * (q + 1) + (k - rem) * q;
            gst[so[t] + k] = cst[t] + off;
          }
        }
      }
    }
  } else {
    // chunk: contiguous groups (array_split into m, or runs of k)
    for (int i = s0 + tid; i < s1; i += SEG_T) va[i] = i;
    for (int g = m0 + tid; g < m1; g += SEG_T) {
      int off;
      if (P.chunk_k > 0) {
        off = min(n, g * P.chunk_k);
      } else {
        const int q = n / M, rem = n % M;
        off = (g < rem) ? g * (q + 1) : rem * (q + 1) + (g - rem) * q;
      }
      gst[g] = off;
    }
  }
  if (b == 0 && tid == 0) gst[M] = n;
  if (!gsync(gs)) return;
  const int* perm_l = va;  // sorted position -> local token
  // ---- group id of every sorted position ----
  for (int s = s0 + tid; s < s1; s += SEG_T) f[s] = 0;
  if (!gsync(gs)) return;
  for (int g = m0 + tid; g < m1; g += SEG_T) f[gst[g]] = 1;
  if (!gsync(gs)) return;
  int Mchk = 0;
  if (!grid_scan(f, grp, n, csum, gs, sh_i, &Mchk)) return;
  for (int s = s0 + tid; s < s1; s += SEG_T) grp[s] = grp[s] + f[s] - 1;
  for (int g = m0 + tid; g < m1; g += SEG_T) {
    gmax[g] = -1;
    gmin[g] = INT_MAX;
    gsum[g] = 0ull;
  }
  if (!gsync(gs)) return;
  for (int s = s0 + tid; s < s1; s += SEG_T) {
    const int g = grp[s], i = perm_l[s];
    atomicMax(&gmax[g], i);
    atomicMin(&gmin[g], i);
    if (pos_scheme == SLS_POS_MEAN) atomicAdd(&gsum[g], (unsigned long long)i);
  }
  if (!gsync(gs)) return;
  // ---- representative positions ----
  if (pos_scheme == SLS_POS_MEDIAN && merged) {
    // members of merged groups are not in token order: sort (group, token)
    int* xa = seat;
    int* xb = cst;
    uint32_t* ga = ka;
    uint32_t* gb2 = kb;
    for (int s = s0 + tid; s < s1; s += SEG_T) ga[perm_l[s]] = (uint32_t)grp[s];
    for (int i = s0 + tid; i < s1; i += SEG_T) xa[i] = i;
    if (!gsync(gs)) return;
    if (!grid_radix_sort<uint32_t>(ga, xa, gb2, xb, n, bit_length_u64((unsigned long long)M),
                                   hist, gs, sh_sort))
      return;
    for (int g = m0 + tid; g < m1; g += SEG_T) rep[g] = xa[gst[g] + (gst[g + 1] - gst[g] - 1) / 2];
  } else {
    for (int g = m0 + tid; g < m1; g += SEG_T) {
      const int len = gst[g + 1] - gst[g];
      int rp;
      if (pos_scheme == SLS_POS_MAX) rp = gmax[g];
      else if (pos_scheme == SLS_POS_MEDIAN) rp = perm_l[gst[g] + (len - 1) / 2];
      else rp = (int)((2ull * gsum[g] + (unsigned long long)len) / (2ull * (unsigned long long)len));
      rep[g] = rp;
    }
  }
  if (!gsync(gs)) return;
  // ---- order groups by (position, first token) ----
  if (pos_scheme != SLS_POS_MEAN) {
    // max and median positions are member tokens of disjoint groups, hence
    // distinct: the rank of a group is the number of marked positions below
    // its own (one scan over the token positions)
    for (int s = s0 + tid; s < s1; s += SEG_T) f[s] = 0;
    if (!gsync(gs)) return;
    for (int g = m0 + tid; g < m1; g += SEG_T) f[rep[g]] = 1;
    if (!gsync(gs)) return;
    int* rk = cst;  // rank of a marked position
    int tmk = 0;
    if (!grid_scan(f, rk, n, csum, gs, sh_i, &tmk)) return;
    if (!gsync(gs)) return;
    for (int g = m0 + tid; g < m1; g += SEG_T) oidx[g] = rk[rep[g]];
  } else {
    unsigned long long* oka = reinterpret_cast<unsigned long long*>(sb + L.ok_a);
    unsigned long long* okb = reinterpret_cast<unsigned long long*>(sb + L.ok_b);
    int* ova = reinterpret_cast<int*>(sb + L.ov_a);
    int* ovb = reinterpret_cast<int*>(sb + L.ov_b);
    for (int g = m0 + tid; g < m1; g += SEG_T) {
      oka[g] = (unsigned long long)rep[g] * (unsigned long long)n + (unsigned long long)gmin[g];
      ova[g] = g;
    }
    if (!gsync(gs)) return;
    const int kbits = bit_length_u64((unsigned long long)n * (unsigned long long)n);
    if (!grid_radix_sort<unsigned long long>(oka, ova, okb, ovb, M, kbits, hist, gs, sh_sort))
      return;
    for (int t = m0 + tid; t < m1; t += SEG_T) oidx[ova[t]] = t;
  }
  if (!gsync(gs)) return;
  // ---- outputs ----
  for (int g = m0 + tid; g < m1; g += SEG_T) {
    const int t = oidx[g];
    const int64_t mrow = P.out0 + t;
    mstart[mrow] = (int)(P.tok_row + gst[g]);
    mlen[mrow] = gst[g + 1] - gst[g];
    pos_out[mrow] = (pos_mode == SLS_MODE_COMPACT) ? (P.out_local + t) : (P.pos0 + rep[g]);
  }
  for (int s = s0 + tid; s < s1; s += SEG_T) {
    const int i = perm_l[s];
    perm[P.tok_row + s] = (int)(P.tok_row + i);
    tok2macro[P.tok_row + i] = P.out_local + oidx[grp[s]];
  }
}

// ============================================================================
// small problems (windows of at most 32 tokens): one warp per problem
// ============================================================================

// The same clusters, exact-length adjust, positions and causal order as
// segment_kernel for a problem of n <= 32 tokens, held in one warp: lane s
// holds the s-th token of the order the groups are cut from ((code, token)
// order for spectral windows, token order for chunk windows), so every group
// is a run of consecutive lanes.
constexpr int SEGW_WARPS = 8;

SLS_DEV unsigned long long shfl_u64(unsigned long long v, int src) {
  return ((unsigned long long)__shfl_sync(0xffffffffu, (unsigned)(v >> 32), src) << 32) |
         __shfl_sync(0xffffffffu, (unsigned)v, src);
}

__global__ void __launch_bounds__(SEGW_WARPS * 32)
segment_warp_kernel(const ProbDesc* __restrict__ probs, int nprob,
                    const uint32_t* __restrict__ codes, int pos_scheme, int pos_mode,
                    int* __restrict__ perm, int* __restrict__ mstart, int* __restrict__ mlen,
                    int32_t* __restrict__ pos_out, int32_t* __restrict__ tok2macro,
                    int chunk_done) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int w0 = blockIdx.x * SEGW_WARPS + (threadIdx.x >> 5);
  const int nw = gridDim.x * SEGW_WARPS;
  for (int p = w0; p < nprob; p += nw) {
    const ProbDesc P = probs[p];
    const int n = P.n, M = P.m;
    if (n <= 0 || M <= 0) continue;
    if (chunk_done && !P.spectral) {
      for (int t = lane; t < M; t += 32) mlen[P.out0 + t] = 0;
      continue;
    }
    const bool valid = lane < n;
    // ---- order: (code, token) for spectral windows, token order otherwise ----
    unsigned long long key = ~0ull;
    if (valid)
      key = P.spectral ? (((unsigned long long)codes[P.phi_row + lane] << 5) | (unsigned)lane)
                       : (unsigned long long)lane;
    if (P.spectral) {
      // bitonic sort over the 32 lanes, ascending
#pragma unroll
      for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
          const unsigned long long o = shfl_u64(key, lane ^ j);
          const bool up = ((lane & k) == 0);
          const bool lower = (lane & j) == 0;
          // the lower lane of the pair keeps the smaller key when ascending
          const bool keep_min = (lower == up);
          key = keep_min ? (o < key ? o : key) : (o > key ? o : key);
        }
      }
    }
    const int tok = (int)(key & 31u);
    // ---- group of each position ----
    int g = 0;
    if (!P.spectral) {
      const int q = n / M, rem = n % M;
      g = (lane < (q + 1) * rem) ? lane / (q + 1) : rem + (lane - (q + 1) * rem) / max(q, 1);
    } else {
      const unsigned long long code = key >> 5;
      const unsigned long long prevc = shfl_u64(code, max(lane - 1, 0));
      const bool head = valid && (lane == 0 || code != prevc);
      const unsigned hm = __ballot_sync(FULL, head);
      const int C = __popc(hm);
      const int cl = __popc(hm & (0xffffffffu >> (31 - lane))) - 1;  // cluster of this position
      if (C >= M) {
        // merge: the cluster of rank t joins group floor(t M / C)
        g = (int)(((long long)cl * M) / C);
      } else {
        // split: D'Hondt seats, one guaranteed per cluster, ties to the lower
        // code; lane c holds cluster c
        const int cs = (lane < C) ? (int)__fns(hm, 0, lane + 1) : n;
        const int cn = (lane + 1 < C) ? (int)__fns(hm, 0, lane + 2) : n;
        const int size = (lane < C) ? cn - cs : 0;
        int seats = (lane < C) ? 1 : 0;
        for (int it = 0; it < M - C; ++it) {
          bool el = lane < C && seats < size;
          int num = size, den = seats + 1, idx = lane;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const bool el2 = __shfl_xor_sync(FULL, el ? 1 : 0, o) != 0;
            const int num2 = __shfl_xor_sync(FULL, num, o);
            const int den2 = __shfl_xor_sync(FULL, den, o);
            const int idx2 = __shfl_xor_sync(FULL, idx, o);
            const long long a = (long long)num2 * den, b = (long long)num * den2;
            const bool better = el2 && (!el || a > b || (a == b && idx2 < idx));
            if (better) {
              el = el2;
              num = num2;
              den = den2;
              idx = idx2;
            }
          }
          if (lane == idx) ++seats;
        }
        int gfirst = seats;  // exclusive prefix of seats: first group of each cluster
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(FULL, gfirst, o);
          if (lane >= o) gfirst += y;
        }
        gfirst -= seats;
        const int ccl = max(cl, 0);
        const int c_start = __shfl_sync(FULL, cs, ccl);
        const int c_size = __shfl_sync(FULL, size, ccl);
        const int c_seats = __shfl_sync(FULL, seats, ccl);
        const int c_g0 = __shfl_sync(FULL, gfirst, ccl);
        const int j = lane - c_start;
        const int q = c_size / max(c_seats, 1), rem = c_size % max(c_seats, 1);
        g = c_g0 + ((j < (q + 1) * rem) ? j / (q + 1) : rem + (j - (q + 1) * rem) / max(q, 1));
      }
    }
    if (!valid) g = M;  // past every group
    // ---- group runs: start, end, positions ----
    const int gp = __shfl_sync(FULL, g, max(lane - 1, 0));
    const bool ghead = valid && (lane == 0 || g != gp);
    const unsigned gm = __ballot_sync(FULL, ghead);
    const int gs = valid ? (int)__fns(gm, 0, g + 1) : 32;
    const int ge = (valid && g + 1 < M) ? (int)__fns(gm, 0, g + 2) : n;
    int vmax = valid ? tok : -1, vmin = valid ? tok : 1 << 30, vsum = valid ? tok : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ymax = __shfl_down_sync(FULL, vmax, o);
      const int ymin = __shfl_down_sync(FULL, vmin, o);
      const int ysum = __shfl_down_sync(FULL, vsum, o);
      if (lane + o < ge) {
        vmax = max(vmax, ymax);
        vmin = min(vmin, ymin);
      }
      // a sum over [lane, ge) needs the partial of lane + o to cover
      // [lane + o, ge) exactly: doubling steps keep that true
      if (lane + o < ge) vsum += ysum;
    }
    // lower median: the member whose token has (len - 1) / 2 smaller members
    int rank = 0;
#pragma unroll
    for (int o = 0; o < 32; ++o) {
      const int t = __shfl_sync(FULL, tok, o);
      if (o >= gs && o < ge && t < tok) ++rank;
    }
    const int len = ge - gs;
    const bool ismed = valid && rank == (len - 1) / 2;
    const unsigned medm = __ballot_sync(FULL, ismed);
    // group g's summary moves to lane g
    const int src = (lane < M) ? (int)__fns(gm, 0, lane + 1) : 0;
    const int g_start = src;
    const int g_end = __shfl_sync(FULL, ge, src);
    const int g_len = g_end - g_start;
    const int g_max = __shfl_sync(FULL, vmax, src);
    const int g_min = __shfl_sync(FULL, vmin, src);
    const int g_sum = __shfl_sync(FULL, vsum, src);
    const unsigned g_end_mask = (g_end >= 32) ? 0xffffffffu : ((1u << g_end) - 1u);
    const unsigned g_mask = g_end_mask & ~((1u << g_start) - 1u);
    const int med_lane = (lane < M) ? (int)__fns(medm & g_mask, 0, 1) : 0;
    const int g_med = __shfl_sync(FULL, tok, med_lane);
    int rep = g_max;
    if (pos_scheme == SLS_POS_MEDIAN) rep = g_med;
    if (pos_scheme == SLS_POS_MEAN) rep = (2 * g_sum + g_len) / (2 * max(g_len, 1));
    // ---- causal order of the groups: by (position, first token) ----
    int orank = 0;
#pragma unroll
    for (int o = 0; o < 32; ++o) {
      const int r2 = __shfl_sync(FULL, rep, o), m2 = __shfl_sync(FULL, g_min, o);
      if (o < M && lane < M && (r2 < rep || (r2 == rep && m2 < g_min))) ++orank;
    }
    if (lane < M) {
      const int64_t mrow = P.out0 + orank;
      mstart[mrow] = (int)(P.tok_row + g_start);
      mlen[mrow] = g_len;
      pos_out[mrow] = (pos_mode == SLS_MODE_COMPACT) ? (P.out_local + orank) : (P.pos0 + rep);
    }
    const int my_rank = __shfl_sync(FULL, orank, min(g, 31));
    if (valid) {
      perm[P.tok_row + lane] = (int)(P.tok_row + tok);
      tok2macro[P.tok_row + tok] = P.out_local + my_rank;
    }
  }
}

// ============================================================================
// preserved tokens, identity
// ============================================================================

__global__ void preserved_kernel(int64_t B, int64_t N, int64_t M, int pf, int pl, int pos_mode,
                                 int* __restrict__ perm, int* __restrict__ mstart,
                                 int* __restrict__ mlen, int32_t* __restrict__ pos_out,
                                 int32_t* __restrict__ tok2macro) {
  const int per = pf + pl;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < B * per;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = e / per;
    const int k = (int)(e % per);
    int64_t tok, mac;
    if (k < pf) {
      tok = k;
      mac = k;
    } else {
      tok = N - pl + (k - pf);
      mac = M - pl + (k - pf);
    }
    const int64_t trow = b * N + tok, mrow = b * M + mac;
    perm[trow] = (int)trow;
    mstart[mrow] = (int)trow;
    mlen[mrow] = 1;
    pos_out[mrow] = (int32_t)((pos_mode == SLS_MODE_COMPACT) ? mac : tok);
    tok2macro[trow] = (int32_t)mac;
  }
}

template <typename T>
SLS_DEV float to_f32(T v);
template <>
SLS_DEV float to_f32<float>(float v) {
  return v;
}
template <>
SLS_DEV float to_f32<uint16_t>(uint16_t v) {
  return __uint_as_float(((unsigned)v) << 16);
}

template <typename T>
__global__ void identity_kernel(const T* __restrict__ X, int64_t B, int64_t N, int d, int64_t ldx,
                                float* __restrict__ Xt, int32_t* __restrict__ pos,
                                int32_t* __restrict__ tok2macro) {
  const int64_t total = B * N * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / d;
    const int c = (int)(e % d);
    Xt[e] = to_f32<T>(X[row * ldx + c]);
    if (c == 0) {
      pos[row] = (int32_t)(row % N);
      tok2macro[row] = (int32_t)(row % N);
    }
  }
}

// ============================================================================
// token norms and macro-token embeddings (Eq. macro_embed)
// ============================================================================

constexpr int AGG_T = 256;
constexpr int AGG_CH = 64;      // members per work item, at most

// Work items: macro-token m is split into ceil(len / AGG_CH) items, listed in
// macro order.  One cluster of AI_CL CTAs: each thread takes a run of macros and
// adds up its items, the partial-sum slots and the macros that span several
// items; scans over the CTA and (through distributed shared memory) the cluster
// turn the counts into offsets, and the thread writes its items.
constexpr int AI_CL = 8;

// Auxiliary integers of the aggregation: counts (16) and the multi-item macros.
struct AggAux {
  int* counts;  // [0] items, [1] partial slots, [2] multi-item macros, [3] item ticket
  int* multi;
};

__host__ __device__ inline AggAux agg_aux(int* base) { return AggAux{base, base + 16}; }

SLS_DEV int nchunks(int len) { return (len + AGG_CH - 1) / AGG_CH; }

SLS_DEV uint32_t cluster_addr(const void* p, unsigned rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}

__global__ void __cluster_dims__(AI_CL, 1, 1) __launch_bounds__(SEG_T)
agg_items_kernel(const int* __restrict__ mlen, int64_t Mtot, int* __restrict__ aux,
                 int2* __restrict__ items, int* __restrict__ pt_start) {
  __shared__ int sh[SEG_W + 1];
  __shared__ int s_tot[3], s_pre[3];
  const AggAux A = agg_aux(aux);
  const int tid = threadIdx.x, rank = blockIdx.x;
  const int64_t K = (Mtot + (int64_t)AI_CL * SEG_T - 1) / ((int64_t)AI_CL * SEG_T);
  const int64_t b = min(Mtot, ((int64_t)rank * SEG_T + tid) * K), e = min(Mtot, b + K);
  int c0 = 0, c1 = 0, c2 = 0;
  for (int64_t m = b; m < e; ++m) {
    const int nch = nchunks(mlen[m]);
    c0 += nch;
    c1 += nch > 1 ? nch : 0;
    c2 += nch > 1 ? 1 : 0;
  }
  int t0, t1, t2;
  int o0 = block_excl_scan<int>(c0, sh, &t0);
  int o1 = block_excl_scan<int>(c1, sh, &t1);
  int o2 = block_excl_scan<int>(c2, sh, &t2);
  if (tid == 0) {
    s_tot[0] = t0;
    s_tot[1] = t1;
    s_tot[2] = t2;
  }
  cluster_sync_all();
  if (tid < 3) {
    int pre = 0;
    for (int r = 0; r < rank; ++r) {
      int v;
      asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v)
                   : "r"(cluster_addr(&s_tot[tid], (unsigned)r)) : "memory");
      pre += v;
    }
    s_pre[tid] = pre;
    if (rank == AI_CL - 1) A.counts[tid] = pre + s_tot[tid];
  }
  if (rank == 0 && tid == 3) A.counts[3] = 0;
  cluster_sync_all();  // s_pre is ready, and every CTA has read the totals
  o0 += s_pre[0];
  o1 += s_pre[1];
  o2 += s_pre[2];
  for (int64_t m = b; m < e; ++m) {
    const int nch = nchunks(mlen[m]);
    for (int c = 0; c < nch; ++c) items[o0 + c] = make_int2((int)m, c);
    pt_start[m] = nch > 1 ? o1 : -1;
    o0 += nch;
    if (nch > 1) {
      A.multi[o2++] = (int)m;
      o1 += nch;
    }
  }
}

template <typename T>
struct VecOf;
template <>
struct VecOf<float> {
  static constexpr int V = 4;
};
template <>
struct VecOf<uint16_t> {
  static constexpr int V = 8;
};

SLS_DEV float agg_block_sum(float v, float* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum_f(v);
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < AGG_T / 32; ++w) s += sh[w];
  return s;
}

SLS_DEV void store_vec4(float* p, float a, float b, float c, float e) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, e);
}

// Thread `tid` owns the V-wide column groups c0 = (tid + q * AGG_T) * V, q < NV.
template <int V, int NV>
SLS_DEV void store_row(const float (&acc)[NV * V], float scale, int d, float* __restrict__ out) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int c0 = (tid + q * AGG_T) * V;
    if (c0 < d)
#pragma unroll
      for (int v = 0; v < V; v += 4)
        store_vec4(out + c0 + v, acc[q * V + v] * scale, acc[q * V + v + 1] * scale,
                   acc[q * V + v + 2] * scale, acc[q * V + v + 3] * scale);
  }
}

// Member rows loaded per batch, so that about eight 16-byte loads per thread
// are in flight.
template <int NV>
constexpr int agg_batch() {
  return NV >= 8 ? 1 : 8 / NV;
}

// The macro-tokens whose members span several items: sum their partial rows
// and finalise (Eq. macro_embed), a cluster of AF_CL CTAs per macro-token of the
// compact list, each CTA a slice of its columns with the rows split over its
// threads; the slices' |sum|^2 meet through distributed shared memory.  Latency
// bound: one CTA per macro-token summed a frequent token's sixty partial rows
// four at a time (N = 32756, d = 3584: 38 -> 8 us).
constexpr int AF_CL = 8;

SLS_DEV float ld_cluster_f32(const float* p, unsigned rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr(p, rank)) : "memory");
  return v;
}

__global__ void __cluster_dims__(AF_CL, 1, 1) __launch_bounds__(AGG_T)
agg_final_kernel(int d, const int* __restrict__ mlen, const int* __restrict__ pt_start,
                 int renorm, const int* __restrict__ aux, const float* __restrict__ part,
                 const float* __restrict__ part_eta, float* __restrict__ Xt) {
  __shared__ float sh[AGG_T / 32];
  __shared__ float s_sq;
  __shared__ float4 red[AGG_T];
  const int tid = threadIdx.x;
  const AggAux A = agg_aux(const_cast<int*>(aux));
  const int nmulti = A.counts[2];
  const int rank = blockIdx.x % AF_CL;
  const int wq = (d / 4 + AF_CL - 1) / AF_CL;          // float4 columns per slice (<= AGG_T)
  const int q0 = rank * wq, nq = max(0, min(d / 4 - q0, wq));
  const int RG = AGG_T / wq;                           // rows summed side by side
  const int cq = tid % wq, rg = tid / wq;
  for (int t = blockIdx.x / AF_CL; t < nmulti; t += gridDim.x / AF_CL) {
    const int64_t m = A.multi[t];
    const int ps = pt_start[m];
    const int len = mlen[m];
    const int nch = (len + AGG_CH - 1) / AGG_CH;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rg < RG && cq < nq) {
      const float4* src = reinterpret_cast<const float4*>(part + (int64_t)ps * d) + q0 + cq;
#pragma unroll 8
      for (int c = rg; c < nch; c += RG) {
        const float4 v = src[(int64_t)c * (d / 4)];
        acc = make_float4(acc.x + v.x, acc.y + v.y, acc.z + v.z, acc.w + v.w);
      }
    }
    float eta = 0.f;
    for (int c = tid; c < nch; c += AGG_T) eta += part_eta[ps + c];
    red[tid] = acc;
    eta = agg_block_sum(eta, sh);  // (its barriers also publish red)
    float sq = 0.f;
    if (rg == 0 && cq < nq) {
      for (int g = 1; g < RG; ++g) {
        const float4 v = red[g * wq + cq];
        acc = make_float4(acc.x + v.x, acc.y + v.y, acc.z + v.z, acc.w + v.w);
      }
      const float inv = 1.0f / (float)len;
      acc = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
      sq = fmaf(acc.x, acc.x, fmaf(acc.y, acc.y, fmaf(acc.z, acc.z, acc.w * acc.w)));
    }
    float scale = 1.0f;
    if (renorm) {
      sq = agg_block_sum(sq, sh);
      if (tid == 0) s_sq = sq;
      cluster_sync_all();
      float tot = 0.f;
      for (int r = 0; r < AF_CL; ++r) tot += ld_cluster_f32(&s_sq, (unsigned)r);
      const float nrm = sqrtf(tot);
      if (nrm >= 1e-30f) scale = (eta / (float)len) / nrm;
      cluster_sync_all();  // every CTA has read the sums
    }
    if (rg == 0 && cq < nq)
      store_vec4(Xt + m * d + 4 * (q0 + cq), acc.x * scale, acc.y * scale, acc.z * scale,
                 acc.w * scale);
    __syncthreads();
  }
}

// Elements 2 p and 2 p + 1 of a 16-byte word of X as a packed pair.
template <typename T>
SLS_DEV f32x2_t raw_pair(const uint4& r, int p);
template <>
SLS_DEV f32x2_t raw_pair<float>(const uint4& r, int p) {
  return p == 0 ? pk2(__uint_as_float(r.x), __uint_as_float(r.y))
                : pk2(__uint_as_float(r.z), __uint_as_float(r.w));
}
template <>
SLS_DEV f32x2_t raw_pair<uint16_t>(const uint4& r, int p) {
  const unsigned w = (p == 0) ? r.x : (p == 1) ? r.y : (p == 2) ? r.z : r.w;
  return pk2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// Sums over the warp of R values per lane (R a power of two up to 8) by a
// transposed butterfly: lane L gets the sum of value L / (32 / R).
template <int R>
SLS_DEV float warp_sums(float (&v)[R]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int h = 16 >> s;
    const int nv = (R >> s) > 1 ? (R >> s) : 1;
    if (nv > 1) {
      const bool up = (lane & h) != 0;
#pragma unroll
      for (int i = 0; i < nv / 2; ++i) {
        const float send = up ? v[i] : v[i + nv / 2];
        const float keep = up ? v[i + nv / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], h);
    }
  }
  return v[0];
}

// ---------------------------------------------------------------------------
// Member pass: a CTA per work item, its member rows by plain 16-byte loads in
// batches of MB rows per thread (eight or more loads in flight each).  A thread
// owns the column groups c0 = (tid + q * AGG_T) * V, sums them and the rows'
// |x|^2 on packed pairs; one barrier per item publishes the row norms and the
// sum's own, and every thread finalises its columns of the macro-token (Eq.
// macro_embed) or stores them as a partial sum.
//
// Bound by reading X: an SM keeps 100 KB of rows in flight, and an item's chain of
// descriptor, member ids and rows hides behind the other CTAs', unless its members are
// few: then the chain is the time, and the next item's is fetched ahead.  Whole calls,
// us (a bulk copy per row as below / neither / fetched ahead / ahead on twice the CTAs;
// groups of m consecutive tokens):
//   N = 32768, d = 3584 bf16   m = 1  321 / 426 / 370 / 250     m = 2  278 / 266 / 239 / 178
//                              m = 4  246 / 175 / 166 / 148     m = 8  232 / 124 / 121 / 122
//   N = 131072, d = 5120 bf16  m = 2  684 / 920 / 815           m = 4  532 / 640 / 579
// On Zipf-distributed codes fetching ahead costs 2% at rho = 16 (N = 32756, d = 3584:
// 151 -> 154 us), and twice the CTAs draw out a long item (rho = 4, N = 3000: 98 -> 115):
// hence the lines at 6 and 3 members.
// The former pass streamed each row through a shared-memory ring with one bulk
// copy per row; issuing those took a producer warp about 1000 cycles per row
// (N = 32756, d = 3584: 90 -> 58 us, against 35 us for the bytes; N = 8180,
// d = 4096: 43 -> 29).
// ---------------------------------------------------------------------------

// Which items the launch expects, by the members per macro-token.
enum AggItems {
  AGG_LONG,   // 6 members and more
  AGG_FEW,    // fewer: an item's chain of ticket, descriptor and ids outlasts its rows, so
              // the next item's is fetched while this one's rows arrive
  AGG_BRIEF   // fewer than 3, NV = 2: besides, batches of two rows on twice the CTAs
};

// Rows per batch and CTAs per SM.
template <int NV, AggItems K>
constexpr int agg_rows() {
  return NV != 2 ? agg_batch<NV>() : K == AGG_BRIEF ? 2 : 8;
}
template <int NV, AggItems K>
constexpr int agg_ctas() {
  return NV == 1 || K == AGG_BRIEF ? 4 : 2;
}

template <typename T, int NV, AggItems K>
__global__ void __launch_bounds__(AGG_T, agg_ctas<NV, K>())
agg_member_kernel(const T* __restrict__ X, int d, int64_t ldx, const int* __restrict__ perm,
                  const int* __restrict__ mstart, const int* __restrict__ mlen,
                  const int2* __restrict__ items, int* __restrict__ aux,
                  const int* __restrict__ pt_start, int renorm, float* __restrict__ Xt,
                  float* __restrict__ part, float* __restrict__ part_eta, int* status,
                  int64_t ntot) {
  constexpr int V = VecOf<T>::V;
  constexpr int PN = NV * V / 2;  // element pairs per thread
  // NV = 2 (d up to 4096 in bf16): twice the rows in flight on half the CTAs, so
  // that a long item ends sooner (N = 8180, d = 4096: 31 -> 26 us); NV = 1 keeps
  // four CTAs (N = 20000, d = 512: 198 us for the call against 227).
  constexpr int MB = agg_rows<NV, K>();
  constexpr bool AHEAD = K != AGG_LONG;
  constexpr int NW = AGG_T / 32, LPR = 32 / MB;
  __shared__ float shq[2][AGG_CH][NW];  // row |x|^2 by warp
  __shared__ float shm[2][NW];          // |member sum|^2 by warp
  __shared__ int s_next[2];
  (void)status;
  (void)ntot;  // bounds of the member rows (debug-build checks)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int* counts = agg_aux(aux).counts;
  const int nitems = counts[0];
  // An item: its macro-token m (len members, partial slot ps), chunk c of it, the first
  // of its n member ids, and with `id` those of its first 32 rows, a lane each.
  struct Item {
    int m, c, len, ps, first, id;
    __device__ int n() const { return min(len - c * AGG_CH, AGG_CH); }
  };
  auto open_item = [&](Item& I, int2 mc) {
    I.m = mc.x;
    I.c = mc.y;
    I.len = mlen[mc.x];
    I.ps = pt_start[mc.x];
    I.first = mstart[mc.x] + mc.y * AGG_CH;
  };
  auto fetch_ids = [&](Item& I) { I.id = lane < I.n() ? perm[I.first + lane] : 0; };
  Item I{};
  int buf = 0, it = blockIdx.x;
  int nx = it + gridDim.x;  // AHEAD: the item after this one
  if (AHEAD && it < nitems) {
    open_item(I, items[it]);
    fetch_ids(I);
  }
  while (it < nitems) {
    if (!AHEAD) {
      open_item(I, items[it]);
      fetch_ids(I);
    }
    // a later item, handed out by a ticket (read after this one's barrier)
    if (tid == 0) s_next[buf] = (AHEAD ? 2 : 1) * (int)gridDim.x + atomicAdd(&counts[3], 1);
    Item X1{};
    int2 next_mc = make_int2(0, 0);
    if (AHEAD && nx < nitems) next_mc = items[nx];
    const int m = I.m, c = I.c, len = I.len, ps = I.ps, n = I.n();
    const int* ids = perm + I.first;
    f32x2_t acc[PN];
#pragma unroll
    for (int e = 0; e < PN; ++e) acc[e] = 0ull;
    int id = I.id;
    for (int s = 0; s < n; s += MB) {
      if (s != 0 && (s & 31) == 0) id = s + lane < n ? ids[s + lane] : 0;  // MB divides 32
      uint4 raw[MB][NV];
#pragma unroll
      for (int j = 0; j < MB; ++j) {
        int64_t row = __shfl_sync(0xffffffffu, id, (s + j) & 31);
#ifdef SLS_DEBUG
        // a member row outside the token set is not read: row 0 instead, and
        // the status records SLS_ERR_BOUNDS
        if (!(row >= 0 && row < ntot)) {
          atomicExch(status, SLS_ERR_BOUNDS);
          row = 0;
        }
#endif
        const T* x = X + row * ldx;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          const int c0 = (tid + q * AGG_T) * V;
          raw[j][q] = make_uint4(0u, 0u, 0u, 0u);
          if (s + j < n && c0 < d) raw[j][q] = __ldcs(reinterpret_cast<const uint4*>(x + c0));
        }
      }
      // the next item's lengths and offsets while this one's rows are on their way, its
      // ids below
      if (AHEAD && s == 0 && nx < nitems) open_item(X1, next_mc);
      float sq[MB];
#pragma unroll
      for (int j = 0; j < MB; ++j) {
        f32x2_t q2 = 0ull;
#pragma unroll
        for (int e = 0; e < PN; ++e) {
          const f32x2_t x = raw_pair<T>(raw[j][e / (V / 2)], e % (V / 2));
          acc[e] = add2(acc[e], x);
          q2 = fma2(x, x, q2);
        }
        float qa, qb;
        upk2(q2, qa, qb);
        sq[j] = qa + qb;
      }
      const float t = warp_sums<MB>(sq);
      if (lane % LPR == 0 && s + lane / LPR < n) shq[buf][s + lane / LPR][warp] = t;
    }
    if (AHEAD && nx < nitems) fetch_ids(X1);
    float v[NV * V];
    float msq = 0.f;
#pragma unroll
    for (int e = 0; e < PN; ++e) {
      upk2(acc[e], v[2 * e], v[2 * e + 1]);
      msq = fmaf(v[2 * e], v[2 * e], msq);
      msq = fmaf(v[2 * e + 1], v[2 * e + 1], msq);
    }
    msq = warp_sum_f(msq);
    if (lane == 0) shm[buf][warp] = msq;
    __syncthreads();
    // sum of member norms (every warp forms the same total)
    float eta = 0.f;
#pragma unroll
    for (int h = 0; h < AGG_CH / 32; ++h) {
      const int r = lane + 32 * h;
      if (r < n) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) t += shq[buf][r][w];
        eta += sqrtf(t);
      }
    }
    eta = warp_sum_f(eta);
    float scale = 1.0f;
    float* dst;
    if (ps < 0) {
      dst = Xt + (int64_t)m * d;
      if (len > 1) {
        // mean = sum / len, rescaled to the mean member norm
        const float inv = 1.0f / (float)len;
        scale = inv;
        if (renorm) {
          float tot = 0.f;
#pragma unroll
          for (int w = 0; w < NW; ++w) tot += shm[buf][w];
          const float nrm = sqrtf(tot) * inv;
          if (nrm >= 1e-30f) scale = inv * ((eta * inv) / nrm);
        }
      }
    } else {
      dst = part + (int64_t)(ps + c) * d;
      if (tid == 0) part_eta[ps + c] = eta;
    }
    store_row<V, NV>(v, scale, d, dst);
    const int ticket = s_next[buf];
    buf ^= 1;
    it = AHEAD ? nx : ticket;
    nx = ticket;
    if (AHEAD) I = X1;
  }
}

// ============================================================================
// adaptive router: window redundancy score (Eq. redundancy)
// ============================================================================

// score = (1/L) sum_i cos(x_i, c) with c the window centroid; computed in one
// pass over X as (sum_i x_i/|x_i|) . (sum_i x_i) / (L |sum_i x_i|).  Zero rows
// add 0.  Every window is cut into parts; a CTA takes a part, reduces each row's
// |x|^2 (per warp, then across warps through a double-buffered shared array, one
// barrier per batch of agg_batch<NV>() rows) and writes the part's sums of x and
// of x/|x|; window_score_combine_kernel adds a window's parts in order and forms
// the score.  The parts are a function of the window and the row width alone, so a
// window's score, and with it its route, has the same bits alone, in any batch and
// on any number of SMs, and no chain of sums grows with the batch.  About 80 rows
// each (64 of rows wider than 4096).  Pass times in us for 16 prompts of 16384 tokens,
// one of 9000 and two of 12764 (d = 4096, 4096, 3496): parts that fill the GPU evenly for
// the batch at hand 573, 123, 158; 64 rows 626, 122, 167; 80 rows 611, 129, 149; 128 rows
// 600, 144, 179; one part per 256 rows 607 and up to half as long again.

// ---------------------------------------------------------------------------
// The score pass with the chunk path folded in (adaptive backend below rho =
// 16, Sec. 3.6): the windows whose score falls below tau are averaged in
// consecutive groups (numpy array_split of the window's n tokens into its m
// macro-tokens), and those means need the same rows the score reads.  So the
// score pass computes, for every window, the chunk macro-tokens as if it were
// routed to the chunk path -- renormalised means (Eq. macro_embed), their
// positions and the token map -- and the segment and aggregation steps then
// handle the spectral windows only, whose outputs replace these.  Parts are
// cut on group boundaries, so no group spans two CTAs; a batch's shared-memory
// reduction carries, besides the row norms, the squared norms of the group means
// that end in the batch.
// ---------------------------------------------------------------------------

// first token of chunk group g (g <= m; group m starts at n)
__host__ __device__ inline int chunk_gstart(int n, int m, int g) {
  const int q = n / m, rem = n % m;
  return (g < rem) ? g * (q + 1) : rem * (q + 1) + (g - rem) * q;
}
// parts of a window of n tokens, at most, and groups per part
__host__ __device__ inline int score_parts(int64_t n, int d) {
  const int rows = d > 4096 ? 64 : 80;
  return n < rows ? 1 : (int)(n / rows);
}
__host__ __device__ inline int score_gpp(int n, int m, int d) {
  return (m + score_parts(n, d) - 1) / score_parts(n, d);
}

// Rows of a batch staged per thread: slot [buffer][row][column group][thread];
// two batches of MB * NV = 8 words, the next in flight while one is used (a
// third stage measured slower: its registers spill).
constexpr int CHK_RING_BYTES = 2 * 8 * AGG_T * 16;

template <typename T, int NV>
__global__ void __launch_bounds__(AGG_T, 2)
window_score_chunk_kernel(const T* __restrict__ X, int d, int64_t ldx,
                          const ProbDesc* __restrict__ probs, int nprob, int KP,
                          float* __restrict__ part, int pos_scheme, int pos_mode, int renorm,
                          float* __restrict__ Xt, int32_t* __restrict__ pos_out,
                          int32_t* __restrict__ tok2macro) {
  constexpr int V = VecOf<T>::V;
  constexpr int MB = agg_batch<NV>();
  constexpr int NW = AGG_T / 32;
  static_assert(MB * NV == 8, "staging ring sized for eight 16-byte words per thread");
  __shared__ float shq[2][MB][NW];  // row |x|^2 partials
  __shared__ float shg[2][MB][NW];  // |group mean|^2 partials, slot = the group's last row
  extern __shared__ uint4 chk_ring[];  // [2][MB][NV][AGG_T]: each thread reads only its own words
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int units = nprob * KP;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int p = u / KP, k = u % KP;
    const ProbDesc P = probs[p];
    const int n = P.n, m = P.m;
    if (n <= 0 || m <= 0) continue;
    const int gp = score_gpp(n, m, d);
    if (k >= (m + gp - 1) / gp) continue;
    const int g0 = k * gp, g1 = min(m, g0 + gp);
    const int r0 = chunk_gstart(n, m, g0), r1 = chunk_gstart(n, m, g1);
    const int q = n / m, rem = n % m;
    // positions of the part's groups and the token map
    for (int g = g0 + tid; g < g1; g += AGG_T) {
      const int a = chunk_gstart(n, m, g), len = chunk_gstart(n, m, g + 1) - a;
      int rp;
      if (pos_scheme == SLS_POS_MAX) {
        rp = a + len - 1;
      } else if (pos_scheme == SLS_POS_MEDIAN) {
        rp = a + (len - 1) / 2;
      } else {
        const unsigned long long sum =
            (unsigned long long)len * a + (unsigned long long)len * (len - 1) / 2;
        rp = (int)((2ull * sum + (unsigned long long)len) / (2ull * (unsigned long long)len));
      }
      pos_out[P.out0 + g] = (pos_mode == SLS_MODE_COMPACT) ? (P.out_local + g) : (P.pos0 + rp);
    }
    for (int i = r0 + tid; i < r1; i += AGG_T) {
      const int g = (i < rem * (q + 1)) ? i / (q + 1) : rem + (i - rem * (q + 1)) / q;
      tok2macro[P.tok_row + i] = P.out_local + g;
    }
    constexpr int PN = NV * V / 2;  // element pairs per thread
    f32x2_t cs[PN], ns[PN], gs[PN];
#pragma unroll
    for (int e = 0; e < PN; ++e) cs[e] = ns[e] = gs[e] = 0ull;
    int gcur = g0, gend = chunk_gstart(n, m, g0 + 1), gcnt = 0;  // before the barrier
    int pcur = g0, pend = gend, pcnt = 0;                          // after it
    float geta = 0.f;
    // the copies of batch s0 go to ring slot b; the next batch is in flight
    // while this one is processed
    const T* xrow = X + (P.tok_row + r0) * ldx + tid * V;  // of the next batch to issue
    auto issue = [&](int s0, int b) {
#pragma unroll
      for (int j = 0; j < MB; ++j) {
        const bool rl = s0 + j < r1;
#pragma unroll
        for (int qv = 0; qv < NV; ++qv) {
          const bool live = rl && (tid + qv * AGG_T) * V < d;
          cp_async16(&chk_ring[((b * MB + j) * NV + qv) * AGG_T + tid],
                     live ? xrow + j * ldx + qv * AGG_T * V : X, live ? 16 : 0);
        }
      }
      xrow += MB * ldx;
      cp_async_commit_group();
    };
    issue(r0, 0);
    int buf = 0;
    constexpr int LPR = 32 / MB;  // lanes that share a row's scalars
    for (int s0 = r0; s0 < r1; s0 += MB, buf ^= 1) {
      if (s0 + MB < r1) {
        issue(s0 + MB, buf ^ 1);
        cp_async_wait_pending(1);
      } else {
        cp_async_wait_pending(0);
      }
      uint4 raw[MB][NV];
#pragma unroll
      for (int j = 0; j < MB; ++j)
#pragma unroll
        for (int qv = 0; qv < NV; ++qv)
          raw[j][qv] = chk_ring[((buf * MB + j) * NV + qv) * AGG_T + tid];
      // before the barrier: row |x|^2 partials; the group sums, and for every
      // group that ends in this batch its mean (stored unscaled; a singleton is
      // its token) and the |mean|^2 partial
      float sq[MB];
#pragma unroll
      for (int j = 0; j < MB; ++j) {
        f32x2_t q2 = 0ull;
#pragma unroll
        for (int e = 0; e < PN; ++e) {
          const f32x2_t x = raw_pair<T>(raw[j][e / (V / 2)], e % (V / 2));
          q2 = fma2(x, x, q2);
          gs[e] = add2(gs[e], x);  // a row past the part is zero
        }
        float qa, qb;
        upk2(q2, qa, qb);
        sq[j] = qa + qb;
        if (s0 + j < r1) {
          ++gcnt;
          if (s0 + j + 1 == gend) {
            const float ginv = (gcnt > 1) ? 1.0f / (float)gcnt : 1.0f;
            float gq = 0.f, mean[NV * V];
#pragma unroll
            for (int e = 0; e < PN; ++e) {
              cs[e] = add2(cs[e], gs[e]);
              upk2(gs[e], mean[2 * e], mean[2 * e + 1]);
              if (gcnt > 1) {
                mean[2 * e] *= ginv;
                mean[2 * e + 1] *= ginv;
              }
              gq = fmaf(mean[2 * e], mean[2 * e], gq);
              gq = fmaf(mean[2 * e + 1], mean[2 * e + 1], gq);
              gs[e] = 0ull;
            }
            gq = warp_sum_f(gq);
            if (lane == 0) shg[buf][j][warp] = gq;
            store_row<V, NV>(mean, 1.0f, d, Xt + (P.out0 + gcur) * (int64_t)d);
            gcnt = 0;
            ++gcur;
            gend = chunk_gstart(n, m, gcur + 1);
          }
        }
      }
      {
        const float t = warp_sums<MB>(sq);
        if (lane % LPR == 0) shq[buf][lane / LPR][warp] = t;
      }
      __syncthreads();
      // after it: the score sums, and each finished group's mean rescaled in
      // place to the mean member norm (Eq. macro_embed).  LPR lanes add a row's
      // warp sums and form its norm; shuffles hand it to the others.
      float tq = 0.f;
#pragma unroll
      for (int w = lane % LPR; w < NW; w += LPR) tq += shq[buf][lane / LPR][w];
#pragma unroll
      for (int o = 1; o < LPR && o < NW; o <<= 1) tq += __shfl_xor_sync(0xffffffffu, tq, o);
      const float nrm_l = sqrtf(tq), inv_l = (tq > 0.f) ? 1.0f / nrm_l : 0.f;
#pragma unroll
      for (int j = 0; j < MB; ++j) {
        if (s0 + j >= r1) break;
        const float nrm = __shfl_sync(0xffffffffu, nrm_l, j * LPR);
        const float inv = __shfl_sync(0xffffffffu, inv_l, j * LPR);
        const f32x2_t inv2 = pk2(inv, inv);
#pragma unroll
        for (int e = 0; e < PN; ++e)
          ns[e] = fma2(raw_pair<T>(raw[j][e / (V / 2)], e % (V / 2)), inv2, ns[e]);
        geta += nrm;
        ++pcnt;
        if (s0 + j + 1 == pend) {
          if (pcnt > 1 && renorm) {
            float gq = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) gq += shg[buf][j][w];
            const float gn = sqrtf(gq);
            if (gn >= 1e-30f) {
              const float scale = (geta * (1.0f / (float)pcnt)) / gn;
              float* out = Xt + (P.out0 + pcur) * (int64_t)d;
#pragma unroll
              for (int qv = 0; qv < NV; ++qv) {
                const int c0 = (tid + qv * AGG_T) * V;
                if (c0 < d)
#pragma unroll
                  for (int e = 0; e < V; e += 4) {
                    const float4 mv = *reinterpret_cast<const float4*>(out + c0 + e);
                    store_vec4(out + c0 + e, mv.x * scale, mv.y * scale, mv.z * scale,
                               mv.w * scale);
                  }
              }
            }
          }
          geta = 0.f;
          pcnt = 0;
          ++pcur;
          pend = chunk_gstart(n, m, pcur + 1);
        }
      }
    }
    float* dst = part + (size_t)u * 2 * d;
#pragma unroll
    for (int qv = 0; qv < NV; ++qv) {
      const int c0 = (tid + qv * AGG_T) * V;
      if (c0 < d)
#pragma unroll
        for (int e = 0; e < V; e += 4) {
          float a0, a1, a2, a3;
          upk2(cs[(qv * V + e) / 2], a0, a1);
          upk2(cs[(qv * V + e) / 2 + 1], a2, a3);
          store_vec4(dst + c0 + e, a0, a1, a2, a3);
          upk2(ns[(qv * V + e) / 2], a0, a1);
          upk2(ns[(qv * V + e) / 2 + 1], a2, a3);
          store_vec4(dst + d + c0 + e, a0, a1, a2, a3);
        }
    }
    __syncthreads();
  }
}

// score[p] = (sum of the parts' x / |x|) . (sum of the parts' x) / (n |sum x|):
// a cluster of SC_CL CTAs per window, four columns per thread (d % 4 == 0) with
// several parts' loads in flight; latency bound (one CTA per window took twice
// the time).
constexpr int SC_CL = 4;

__global__ void __cluster_dims__(SC_CL, 1, 1) __launch_bounds__(AGG_T)
window_score_combine_kernel(int d, const ProbDesc* __restrict__ probs, int nprob, int KP,
                            const float* __restrict__ part, float* __restrict__ score) {
  __shared__ float sh[AGG_T / 32];
  __shared__ float s_sum[2];
  const int rank = blockIdx.x % SC_CL;
  for (int p = blockIdx.x / SC_CL; p < nprob; p += gridDim.x / SC_CL) {
    const int n = probs[p].n, m = max(probs[p].m, 1);
    const int gp = score_gpp(n, m, d), kp = (m + gp - 1) / gp;
    float dot = 0.f, cc = 0.f;
    for (int c = 4 * (rank * AGG_T + threadIdx.x); c < d; c += 4 * AGG_T * SC_CL) {
      float4 cs = make_float4(0.f, 0.f, 0.f, 0.f), ns = cs;
      const float* src = part + (size_t)p * KP * 2 * d + c;
#pragma unroll 8
      for (int k = 0; k < kp; ++k, src += 2 * d) {
        const float4 a = *reinterpret_cast<const float4*>(src);
        const float4 b = *reinterpret_cast<const float4*>(src + d);
        cs = make_float4(cs.x + a.x, cs.y + a.y, cs.z + a.z, cs.w + a.w);
        ns = make_float4(ns.x + b.x, ns.y + b.y, ns.z + b.z, ns.w + b.w);
      }
      dot = fmaf(ns.x, cs.x, fmaf(ns.y, cs.y, fmaf(ns.z, cs.z, fmaf(ns.w, cs.w, dot))));
      cc = fmaf(cs.x, cs.x, fmaf(cs.y, cs.y, fmaf(cs.z, cs.z, fmaf(cs.w, cs.w, cc))));
    }
    dot = agg_block_sum(dot, sh);
    cc = agg_block_sum(cc, sh);
    if (threadIdx.x == 0) s_sum[0] = dot, s_sum[1] = cc;
    cluster_sync_all();
    if (rank == 0 && threadIdx.x == 0) {
      dot = cc = 0.f;
      for (int r = 0; r < SC_CL; ++r) {
        dot += ld_cluster_f32(&s_sum[0], (unsigned)r);
        cc += ld_cluster_f32(&s_sum[1], (unsigned)r);
      }
      score[p] = (cc > 0.f) ? dot / ((float)n * sqrtf(cc)) : 0.f;
    }
    cluster_sync_all();  // the sums have been read
  }
}

}  // namespace

// ============================================================================
// launchers
// ============================================================================

int launch_simhash(const float* U, int64_t N, int k, int ldu, const int32_t* k_dev,
                   const float* R, int bits, int ldr, uint32_t* codes, cudaStream_t stream) {
  if (N == 0) return SLS_OK;
  int dev = 0, sms = 0;
  SLS_CUDA_TRY(cudaGetDevice(&dev));
  SLS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // two rows per thread (a hyperplane's load feeds both) once that still leaves
  // every SM four tiles
  const int rpt = N / sh_rows(bits, 2) >= 4 * (int64_t)sms ? 2 : 1;
  auto fn = rpt == 2 ? simhash_kernel<2> : simhash_kernel<1>;
  const size_t smem = sh_smem(bits, k, rpt);
  const int64_t blocks = (N + sh_rows(bits, rpt) - 1) / sh_rows(bits, rpt);
  if (blocks > 0x7fffffffLL) return SLS_ERR_UNSUPPORTED;
  if (smem > 48 * 1024)
    SLS_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  fn<<<(unsigned)blocks, SH_T, smem, stream>>>(U, N, k, ldu, k_dev, R, bits, ldr, codes);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

size_t segment_scratch_bytes(int64_t nmax, int64_t mmax, int slots) {
  return (size_t)slots * seg_layout(nmax, mmax).total;
}

int launch_simhash_problems(const ProbDesc* probs, const int* spec_list, const int* nspec_dev,
                            int nspec_max, int64_t nmax, const int* r_eff, const float* U, int ldu,
                            const float* R, int ldr, int bits_max, uint32_t* codes,
                            cudaStream_t stream) {
  if (nspec_max <= 0) return SLS_OK;
  if (nmax <= SH_FLAT_MAX) {
    const int64_t threads = (int64_t)nspec_max * nmax;
    const int64_t blocks = (threads + 255) / 256;
    if (blocks > 0x7fffffffLL) return SLS_ERR_UNSUPPORTED;
    simhash_flat_kernel<<<(unsigned)blocks, 256, 0, stream>>>(
        probs, spec_list, nspec_dev, nspec_max, (int)nmax, r_eff, U, ldu, R, ldr, codes);
    SLS_LAUNCH_CHECK();
    return SLS_OK;
  }
  // shared memory for the widest tile of the problems' bit counts (bits <=
  // bits_max; fewer bits per problem mean more rows per tile)
  const size_t smem = sh_smem(1, ldu, 1);
  int64_t bx = (nmax + sh_rows(bits_max, 1) - 1) / sh_rows(bits_max, 1);
  // at most about 8192 CTAs in all (the CTAs loop over their problem's
  // rows): the launch is sized by the bound on the spectral problems, most
  // of which may be empty at run time
  const int64_t cap = 8192 / (nspec_max > 0 ? nspec_max : 1);
  if (bx > cap) bx = cap;
  if (bx < 1) bx = 1;
  if (smem > 48 * 1024)
    SLS_CUDA_TRY(cudaFuncSetAttribute(simhash_batched_kernel,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  simhash_batched_kernel<<<dim3((unsigned)bx, nspec_max), SH_T, smem, stream>>>(
      probs, spec_list, nspec_dev, nspec_max, r_eff, U, ldu, R, ldr, codes);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

namespace {
// The launch of segment_grid_kernel as one cluster.
cudaLaunchConfig_t segment_cluster_config(cudaLaunchAttribute* at, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(SEG_CL);
  cfg.blockDim = dim3(SEG_T);
  cfg.stream = stream;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = SEG_CL;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// Whether the current device can place that cluster (asked once per device).
cudaError_t segment_cluster_fits(bool* fits) {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];  // 0: not asked yet, 1: no, 2: yes
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int k = dev < kDevices ? known[dev].load() : 0;
  if (k == 0) {
    if ((e = cudaFuncSetAttribute(segment_grid_kernel,
                                  cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) ==
        cudaSuccess) {
      cudaLaunchAttribute at;
      const cudaLaunchConfig_t cfg = segment_cluster_config(&at, nullptr);
      int clusters = 0;
      e = cudaOccupancyMaxActiveClusters(&clusters, segment_grid_kernel, &cfg);
      k = e == cudaSuccess && clusters > 0 ? 2 : 1;
    } else {
      k = 1;
    }
    if (e != cudaSuccess) (void)cudaGetLastError();  // a device without it: the other kernels
    if (dev < kDevices) known[dev].store(k);
  }
  *fits = k == 2;
  return cudaSuccess;
}
}  // namespace

int launch_segment(const ProbDesc* probs, int nprob, const uint32_t* codes, int pos_scheme,
                   int pos_mode, void* scratch, int slots, int64_t nmax, int64_t mmax, int* perm,
                   int* mstart, int* mlen, int32_t* pos_out, int32_t* tok2macro, int* status,
                   cudaStream_t stream, int chunk_done) {
  if (nprob <= 0) return SLS_OK;
  const SegLayout L = seg_layout(nmax, mmax);
  const size_t stride = L.total;
  bool fits = false;
  if (segment_route(nprob, nmax, status != nullptr, true) == SegRoute::cluster)
    SLS_CUDA_TRY(segment_cluster_fits(&fits));
  const SegRoute route = segment_route(nprob, nmax, status != nullptr, fits);
  if (route == SegRoute::warp) {
    // windows of at most 32 tokens: one warp per window
    int64_t blocks = ((int64_t)nprob + SEGW_WARPS - 1) / SEGW_WARPS;
    if (blocks > 65535) blocks = 65535;
    segment_warp_kernel<<<(unsigned)blocks, SEGW_WARPS * 32, 0, stream>>>(
        probs, nprob, codes, pos_scheme, pos_mode, perm, mstart, mlen, pos_out, tok2macro,
        chunk_done);
    SLS_LAUNCH_CHECK();
    return SLS_OK;
  }
  if (route == SegRoute::cluster) {
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = segment_cluster_config(&at, stream);
    SLS_CUDA_TRY(cudaFuncSetAttribute(segment_grid_kernel,
                                      cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    SLS_CUDA_TRY(cudaLaunchKernelEx(&cfg, segment_grid_kernel, probs, codes, pos_scheme, pos_mode,
                                    (char*)scratch, nmax, mmax, perm, mstart, mlen, pos_out,
                                    tok2macro, status, chunk_done, 1));
    count_launch(1);
    return SLS_OK;
  }
  if (route == SegRoute::grid) {
    char* sb = (char*)scratch;
    int dev = 0, sms = 0;
    SLS_CUDA_TRY(cudaGetDevice(&dev));
    SLS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    int G = sms < SEGG_MAX ? sms : SEGG_MAX;
    SLS_CUDA_TRY(cudaMemsetAsync(sb + L.gbar, 0, 256, stream));
    int64_t nm = nmax, mm = mmax;
    int cluster = 0;
    void* args[] = {(void*)&probs, (void*)&codes, (void*)&pos_scheme, (void*)&pos_mode,
                    (void*)&sb, (void*)&nm, (void*)&mm, (void*)&perm, (void*)&mstart,
                    (void*)&mlen, (void*)&pos_out, (void*)&tok2macro, (void*)&status,
                    (void*)&chunk_done, (void*)&cluster};
    SLS_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)segment_grid_kernel, dim3(G), dim3(SEG_T),
                                             args, 0, stream));
    count_launch(1);
    return SLS_OK;
  }
  const int grid = nprob < slots ? nprob : slots;
  // the sort buffers in shared memory when they fit beside the static arrays
  // (the mistral7b prompt's segment step 85 -> 81 us)
  const size_t dyn = seg_smem_layout(nmax, mmax).total;
  const int in_smem = dyn <= SEG_SMEM_MAX ? 1 : 0;
  const size_t dyn_bytes = in_smem ? dyn : 0;
  if (in_smem)
    SLS_CUDA_TRY(cudaFuncSetAttribute(segment_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)dyn_bytes));
  segment_kernel<<<grid, SEG_T, dyn_bytes, stream>>>(probs, nprob, codes, pos_scheme, pos_mode,
                                                     (char*)scratch, stride, nmax, mmax, perm,
                                                     mstart, mlen, pos_out, tok2macro,
                                                     chunk_done, in_smem);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

int launch_preserved(int64_t B, int64_t N, int64_t M, int pf, int pl, int pos_mode, int* perm,
                     int* mstart, int* mlen, int32_t* pos_out, int32_t* tok2macro,
                     cudaStream_t stream) {
  if (pf + pl == 0 || B == 0) return SLS_OK;
  int64_t blocks = (B * (pf + pl) + 255) / 256;
  if (blocks > 1024) blocks = 1024;
  preserved_kernel<<<(unsigned)blocks, 256, 0, stream>>>(B, N, M, pf, pl, pos_mode, perm, mstart,
                                                         mlen, pos_out, tok2macro);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

int launch_identity(const void* X, int x_dtype, int64_t B, int64_t N, int d, int64_t ldx,
                    float* Xt, int32_t* pos, int32_t* tok2macro, cudaStream_t stream) {
  if (B * N == 0) return SLS_OK;
  int64_t blocks = (B * N * d + 255) / 256;
  if (blocks > 65536) blocks = 65536;
  if (x_dtype == SLS_F32)
    identity_kernel<float><<<(unsigned)blocks, 256, 0, stream>>>((const float*)X, B, N, d, ldx,
                                                                  Xt, pos, tok2macro);
  else
    identity_kernel<uint16_t><<<(unsigned)blocks, 256, 0, stream>>>((const uint16_t*)X, B, N, d,
                                                                     ldx, Xt, pos, tok2macro);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

size_t agg_item_capacity(int64_t Mtot, int64_t Ntot) { return (size_t)(Mtot + Ntot / AGG_CH + 2); }
size_t agg_aux_ints(int64_t Mtot, int64_t Ntot) {
  (void)Mtot;
  return (size_t)(16 + Ntot / AGG_CH + 2);
}
size_t agg_part_capacity(int64_t Ntot) { return (size_t)(2 * (Ntot / AGG_CH) + 2); }

namespace {
template <typename T, int NV>
int launch_agg_t(const void* X, int d, int64_t ldx, const int* perm, const int* mstart,
                 const int* mlen, int64_t Mtot, int64_t Ntot, int64_t fblocks, int renorm,
                 float* Xt,
                 int* pt_start, int2* items, int* aux, float* part, float* part_eta,
                 int* status, cudaStream_t stream) {
  int dev = 0, sms = 0;
  SLS_CUDA_TRY(cudaGetDevice(&dev));
  SLS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  agg_items_kernel<<<AI_CL, SEG_T, 0, stream>>>(mlen, Mtot, aux, items, pt_start);
  SLS_LAUNCH_CHECK();
  // CTAs that fit the GPU at once; items by ticket
  int occ = 0;
  auto fn = agg_member_kernel<T, NV, AGG_LONG>;
  if (Ntot < 6 * Mtot) fn = agg_member_kernel<T, NV, AGG_FEW>;
  if constexpr (NV == 2)
    if (Ntot < 3 * Mtot) fn = agg_member_kernel<T, NV, AGG_BRIEF>;
  SLS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, AGG_T, 0));
  int64_t grid = (int64_t)sms * (occ < 1 ? 1 : occ);
  const int64_t most = Mtot + Ntot / AGG_CH;  // items at most
  if (grid > most) grid = most;
  fn<<<(unsigned)grid, AGG_T, 0, stream>>>(
      (const T*)X, d, ldx, perm, mstart, mlen, items, aux, pt_start, renorm, Xt, part, part_eta,
      status, Ntot);
  SLS_LAUNCH_CHECK();
  const int64_t clusters = fblocks < 64 ? fblocks : 64;
  agg_final_kernel<<<(unsigned)(clusters * AF_CL), AGG_T, 0, stream>>>(
      d, mlen, pt_start, renorm, aux, part, part_eta, Xt);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

template <typename T>
int launch_agg_dtype(const void* X, int d, int64_t ldx, const int* perm, const int* mstart,
                     const int* mlen, int64_t Mtot, int64_t Ntot, int64_t fblocks, int renorm,
                     float* Xt,
                     int* pt_start, int2* items, int* aux, float* part, float* part_eta,
                     int* status, cudaStream_t stream) {
  constexpr int V = VecOf<T>::V;
  const int nv = (d / V + AGG_T - 1) / AGG_T;
#define SLS_AGG_NV(N)                                                                       \
  return launch_agg_t<T, N>(X, d, ldx, perm, mstart, mlen, Mtot, Ntot, fblocks, renorm, Xt, \
                            pt_start, items, aux, part, part_eta, status, stream)
  if (nv <= 1) SLS_AGG_NV(1);
  if (nv <= 2) SLS_AGG_NV(2);
  if (nv <= 4) SLS_AGG_NV(4);
  if (nv <= 8) SLS_AGG_NV(8);
#undef SLS_AGG_NV
  return SLS_ERR_UNSUPPORTED;
}
}  // namespace

int launch_aggregate(const void* X, int x_dtype, int d, int64_t ldx, const int* perm,
                     const int* mstart, const int* mlen, int64_t Mtot, int64_t Ntot, int renorm,
                     float* Xt, int* pt_start, int2* items, int* aux, float* part,
                     float* part_eta, int* status, cudaStream_t stream) {
  if (Mtot == 0) return SLS_OK;
  int64_t fblocks = Ntot / AGG_CH + 1;
  if (fblocks > 1024) fblocks = 1024;
  if (x_dtype == SLS_F32)
    return launch_agg_dtype<float>(X, d, ldx, perm, mstart, mlen, Mtot, Ntot, fblocks, renorm,
                                   Xt, pt_start, items, aux, part, part_eta, status, stream);
  return launch_agg_dtype<uint16_t>(X, d, ldx, perm, mstart, mlen, Mtot, Ntot, fblocks, renorm,
                                    Xt, pt_start, items, aux, part, part_eta, status, stream);
}

namespace {
template <typename T, int NV>
int launch_score_chunk_nv(const T* X, int d, int64_t ldx, const ProbDesc* probs, int nprob,
                          int64_t nmax, float* part, float* score, int pos_scheme, int pos_mode,
                          int renorm, float* Xt, int32_t* pos, int32_t* tok2macro,
                          cudaStream_t stream) {
  auto fn = window_score_chunk_kernel<T, NV>;
  SLS_CUDA_TRY(
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, CHK_RING_BYTES));
  const int KP = score_parts(nmax, d);
  const int64_t units = (int64_t)nprob * KP;
  const int blocks = (int)(units < 65535 ? units : 65535);
  fn<<<blocks, AGG_T, CHK_RING_BYTES, stream>>>(X, d, ldx, probs, nprob, KP, part, pos_scheme,
                                                pos_mode, renorm, Xt, pos, tok2macro);
  SLS_LAUNCH_CHECK();
  const int cb = nprob < 4096 ? nprob : 4096;
  window_score_combine_kernel<<<cb * SC_CL, AGG_T, 0, stream>>>(d, probs, nprob, KP, part, score);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

template <typename T>
int launch_score_chunk_dtype(const void* X, int d, int64_t ldx, const ProbDesc* probs, int nprob,
                             int64_t nmax, float* part, float* score, int pos_scheme,
                             int pos_mode, int renorm, float* Xt, int32_t* pos,
                             int32_t* tok2macro, cudaStream_t stream) {
  const int nv = (d / VecOf<T>::V + AGG_T - 1) / AGG_T;
  auto fn = nv <= 1   ? launch_score_chunk_nv<T, 1>
            : nv <= 2 ? launch_score_chunk_nv<T, 2>
            : nv <= 4 ? launch_score_chunk_nv<T, 4>
                      : launch_score_chunk_nv<T, 8>;
  if (nv > 8) return SLS_ERR_UNSUPPORTED;
  return fn((const T*)X, d, ldx, probs, nprob, nmax, part, score, pos_scheme, pos_mode, renorm,
            Xt, pos, tok2macro, stream);
}
}  // namespace

// Part sums go to the aggregation's partial rows, idle at that time; where those are
// too few (windows of fewer than 64 tokens; prompts of hardly more than one window;
// some of wide rows) they have room of their own.
size_t score_part_floats(int64_t nprob, int64_t nmax, int64_t Ntot, int d) {
  const int64_t pairs = nprob * score_parts(nmax, d);
  return 2 * pairs > (int64_t)agg_part_capacity(Ntot) ? (size_t)pairs * 2 * (size_t)d : 0;
}

int launch_window_score_chunk(const void* X, int x_dtype, int d, int64_t ldx,
                              const ProbDesc* probs, int nprob, int64_t nmax, int64_t Ntot,
                              float* agg_part, float* own_part, float* score, int pos_scheme,
                              int pos_mode, int renorm, float* Xt, int32_t* pos,
                              int32_t* tok2macro, cudaStream_t stream) {
  if (nprob <= 0) return SLS_OK;
  float* part = score_part_floats(nprob, nmax, Ntot, d) == 0 ? agg_part : own_part;
  if (x_dtype == SLS_F32)
    return launch_score_chunk_dtype<float>(X, d, ldx, probs, nprob, nmax, part, score,
                                           pos_scheme, pos_mode, renorm, Xt, pos, tok2macro,
                                           stream);
  return launch_score_chunk_dtype<uint16_t>(X, d, ldx, probs, nprob, nmax, part, score,
                                            pos_scheme, pos_mode, renorm, Xt, pos, tok2macro,
                                            stream);
}

}  // namespace sls
