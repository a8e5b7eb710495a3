// Random Fourier feature map, Sec. 3.2 Eq. rff_map:
//   Phi[i, c] = sqrt(2/D) * cos( X[i, :] . W[c, :] + b[c] ),  W = Omega^T (D x d).
//
// The contraction X W^T is GEMM-shaped (M = tokens, N = features, K = d).
// This file holds the fp32 SIMT kernel (shallow or small float32 contractions,
// unaligned or odd shapes); the tcgen05 kernels for bf16 and for deep float32
// inputs live in feature_map_tc.cu.  All fuse the bias, cosine and scale into the epilogue,
// so Phi is written exactly once, as float32 or (opt-in) as bfloat16 rounded
// to nearest even from the float32 value.
#include "common.cuh"
#include "kernels.cuh"

namespace sls {

namespace {

constexpr int FM_BK = 16;   // K slice

SLS_DEV float load_elem(const uint16_t* p) {
  return __uint_as_float(((unsigned)*p) << 16);
}

// Elements k .. k + 3 of a row of d elements (zero past its end); vec: the row
// start and d allow 16-byte (float32) or 8-byte (bf16) loads.
template <typename T>
SLS_DEV float4 load_quad(const T* row, int k, int d, bool vec);

template <>
SLS_DEV float4 load_quad<float>(const float* row, int k, int d, bool vec) {
  if (vec && k + 3 < d) return __ldg(reinterpret_cast<const float4*>(row + k));
  return make_float4(k < d ? row[k] : 0.f, k + 1 < d ? row[k + 1] : 0.f,
                     k + 2 < d ? row[k + 2] : 0.f, k + 3 < d ? row[k + 3] : 0.f);
}

template <>
SLS_DEV float4 load_quad<uint16_t>(const uint16_t* row, int k, int d, bool vec) {
  if (vec && k + 3 < d) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(row + k));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
  }
  return make_float4(k < d ? load_elem(row + k) : 0.f, k + 1 < d ? load_elem(row + k + 1) : 0.f,
                     k + 2 < d ? load_elem(row + k + 2) : 0.f,
                     k + 3 < d ? load_elem(row + k + 3) : 0.f);
}

// G (2 or 4) neighbouring floats of shared memory in one load.
template <int G>
SLS_DEV void load_group(const float* p, float* out) {
  if constexpr (G == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    out[0] = v.x;
    out[1] = v.y;
    out[2] = v.z;
    out[3] = v.w;
  } else {
    const float2 v = *reinterpret_cast<const float2*>(p);
    out[0] = v.x;
    out[1] = v.y;
  }
}

// G (2 or 4) neighbouring features; vec: Phi allows the store of four as one.
template <int G>
SLS_DEV void store_group(float* p, const float* v, bool vec) {
  if (G == 4 && vec) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[G - 2], v[G - 1]);
  } else if (vec) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int e = 0; e < G; ++e) p[e] = v[e];
  }
}
template <int G>
SLS_DEV void store_group(uint16_t* p, const float* v, bool vec) {
  if (vec) {
    __align__(8) __nv_bfloat162 h[2];
#pragma unroll
    for (int e = 0; e < G; e += 2) h[e / 2] = __floats2bfloat162_rn(v[e], v[e + 1]);
    if (G == 4)
      *reinterpret_cast<uint2*>(p) = *reinterpret_cast<const uint2*>(h);
    else
      *reinterpret_cast<unsigned*>(p) = *reinterpret_cast<const unsigned*>(h);
  } else {
#pragma unroll
    for (int e = 0; e < G; ++e) phi_st(p + e, v[e]);
  }
}

// One CTA computes a BM x BN tile, each thread TM x TN of it; every output is
// one chain of fused multiply-adds over k ascending, whatever the tile.  T:
// element type of X and W; OT: of Phi (float, or uint16_t for bfloat16).
//
// Bound by the FP32 pipes (two features per packed instruction).  A K slice is
// loaded as quads along the rows into registers while the previous slice is
// computed, then stored transposed into the other of two shared-memory buffers:
// one barrier per slice, and TM + TN floats read per TM * TN multiply-adds.
// N = 4084, d = 2048, D = 1024: 600 -> 395 us a call against the former kernel
// (64 x 64 tiles, 4 x 4 per thread, scalar loads between two barriers), with the
// same bits.
template <typename T, typename OT, int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), TM * TN >= 64 ? 4 : TM * TN >= 32 ? 6 : 4)
feature_map_simt_kernel(const T* __restrict__ X, int64_t N, int d, int64_t ldx,
                        const T* __restrict__ W, const float* __restrict__ bvec,
                        int D, float scale, OT* __restrict__ Phi, int vecx, int vecw, int vecp) {
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int QA = (BM * FM_BK / 4) / NT, QB = (BN * FM_BK / 4) / NT;  // quads per thread
  static_assert(QA * NT == BM * FM_BK / 4 && QB * NT == BN * FM_BK / 4, "whole quads per thread");
  static_assert(TM % 2 == 0 && TN % 2 == 0, "pairs");
  __shared__ __align__(16) float As[2][FM_BK][BM + 4];
  __shared__ __align__(16) float Bs[2][FM_BK][BN + 4];
  const int tid = threadIdx.x;
  const int64_t row0 = (int64_t)blockIdx.y * BM;
  const int col0 = blockIdx.x * BN;
  const int ty = tid / (BN / TN), tx = tid % (BN / TN);
  f32x2_t acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
  float4 ra[QA], rb[QB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int e = tid + q * NT, r = e / (FM_BK / 4), k = k0 + 4 * (e % (FM_BK / 4));
      ra[q] = row0 + r < N ? load_quad<T>(X + (row0 + r) * ldx, k, d, vecx)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
      const int e = tid + q * NT, r = e / (FM_BK / 4), k = k0 + 4 * (e % (FM_BK / 4));
      rb[q] = col0 + r < D ? load_quad<T>(W + (int64_t)(col0 + r) * d, k, d, vecw)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int e = tid + q * NT, r = e / (FM_BK / 4), k = 4 * (e % (FM_BK / 4));
      As[buf][k][r] = ra[q].x;
      As[buf][k + 1][r] = ra[q].y;
      As[buf][k + 2][r] = ra[q].z;
      As[buf][k + 3][r] = ra[q].w;
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
      const int e = tid + q * NT, r = e / (FM_BK / 4), k = 4 * (e % (FM_BK / 4));
      Bs[buf][k][r] = rb[q].x;
      Bs[buf][k + 1][r] = rb[q].y;
      Bs[buf][k + 2][r] = rb[q].z;
      Bs[buf][k + 3][r] = rb[q].w;
    }
  };
  fetch(0);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < d; k0 += FM_BK, buf ^= 1) {
    const bool more = k0 + FM_BK < d;
    if (more) fetch(k0 + FM_BK);
#pragma unroll
    for (int k = 0; k < FM_BK; ++k) {
      // the thread's rows in groups of two or four spread over the tile (rows
      // ty * G + i of each BM / (TM / G) rows), so that a warp's reads of a
      // group touch neighbouring words
      constexpr int GA = TM % 4 ? 2 : 4, GB = TN % 4 ? 2 : 4;
      float a[TM], bb[TN];
#pragma unroll
      for (int i = 0; i < TM; i += GA)
        load_group<GA>(&As[buf][k][(i / GA) * (BM / (TM / GA)) + ty * GA], a + i);
#pragma unroll
      for (int j = 0; j < TN; j += GB)
        load_group<GB>(&Bs[buf][k][(j / GB) * (BN / (TN / GB)) + tx * GB], bb + j);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f32x2_t aa = pk2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = fma2(aa, pk2(bb[2 * j], bb[2 * j + 1]), acc[i][j]);
      }
    }
    if (more) stage(buf ^ 1);
    __syncthreads();
  }
  // The epilogue is what a shallow contraction spends its time on: biases read once, a
  // group of neighbouring features in one store (D is a multiple of four, so a group
  // lies inside the row or outside it).  N = 60000, d = 64, D = 1500: 600 -> 500 us bf16,
  // 559 -> 471 float32 (478, 473 with the former 64 x 64 tiles).
  constexpr int GA = TM % 4 ? 2 : 4, GB = TN % 4 ? 2 : 4;
  float bias[TN];
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int c = col0 + (j / GB) * (BN / (TN / GB)) + tx * GB + j % GB;
    bias[j] = c < D ? bvec[c] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t gr = row0 + (i / GA) * (BM / (TM / GA)) + ty * GA + i % GA;
    if (gr >= N) continue;
#pragma unroll
    for (int j = 0; j < TN; j += GB) {
      const int c = col0 + (j / GB) * (BN / (TN / GB)) + tx * GB;
      if (c >= D) continue;
      float v[GB];
#pragma unroll
      for (int e = 0; e < GB; e += 2) {
        upk2(acc[i][(j + e) / 2], v[e], v[e + 1]);
        v[e] = scale * cosf(v[e] + bias[j + e]);
        v[e + 1] = scale * cosf(v[e + 1] + bias[j + e + 1]);
      }
      store_group<GB>(Phi + gr * D + c, v, vecp);
    }
  }
}

template <typename T, int BM, int BN, int TM, int TN>
int launch_simt_tile(const void* X, int64_t N, int d, int64_t ldx, const void* W, const float* b,
                     int D, float scale, void* Phi, int phi_bf16, cudaStream_t stream) {
  const uintptr_t al = sizeof(T) == 4 ? 15 : 7;  // a quad of elements
  const int vecx = ((uintptr_t)X & al) == 0 && ldx % 4 == 0;
  const int vecw = ((uintptr_t)W & al) == 0 && d % 4 == 0;
  const int vecp = ((uintptr_t)Phi & (phi_bf16 ? 7 : 15)) == 0;
  const dim3 grid((D + BN - 1) / BN, (unsigned)((N + BM - 1) / BM));
  constexpr int NT = (BM / TM) * (BN / TN);
  if (phi_bf16)
    feature_map_simt_kernel<T, uint16_t, BM, BN, TM, TN><<<grid, NT, 0, stream>>>(
        (const T*)X, N, d, ldx, (const T*)W, b, D, scale, (uint16_t*)Phi, vecx, vecw, vecp);
  else
    feature_map_simt_kernel<T, float, BM, BN, TM, TN><<<grid, NT, 0, stream>>>(
        (const T*)X, N, d, ldx, (const T*)W, b, D, scale, (float*)Phi, vecx, vecw, vecp);
  SLS_LAUNCH_CHECK();
  return SLS_OK;
}

// The tile: 128 x 64 once every SM gets three of them, 64 x 64 from one per SM
// on, else 32 x 32, which keeps more SMs busy on a short prompt.  Measured (us;
// 128 x 128 / 128 x 64 / 64 x 64): N = 4084, d = 2048, D = 1024 391 / 395 / 412;
// 8192, 2048, 1024 750 / 659 / 777; 2000, 1024, 512 121 / 83 / 79.
template <typename T>
int launch_simt_t(const void* X, int64_t N, int d, int64_t ldx, const void* W, const float* b,
                  int D, float scale, void* Phi, int phi_bf16, int sms, cudaStream_t stream) {
  auto tiles = [&](int64_t bm, int64_t bn) { return ((N + bm - 1) / bm) * ((D + bn - 1) / bn); };
  if (tiles(128, 64) >= 3 * (int64_t)sms)
    return launch_simt_tile<T, 128, 64, 8, 8>(X, N, d, ldx, W, b, D, scale, Phi, phi_bf16, stream);
  if (tiles(64, 64) >= (int64_t)sms)
    return launch_simt_tile<T, 64, 64, 8, 4>(X, N, d, ldx, W, b, D, scale, Phi, phi_bf16, stream);
  return launch_simt_tile<T, 32, 32, 4, 2>(X, N, d, ldx, W, b, D, scale, Phi, phi_bf16, stream);
}

}  // namespace

int launch_feature_map_simt(const void* X, int x_dtype, int64_t N, int d, int64_t ldx,
                            const void* W, const float* b, int D, void* Phi,
                            cudaStream_t stream, int phi_bf16) {
  if (N == 0) return SLS_OK;
  const float scale = (float)sqrt(2.0 / (double)D);
  if ((N + 63) / 64 > 65535) return SLS_ERR_UNSUPPORTED;
  int dev = 0, sms = 0;
  SLS_CUDA_TRY(cudaGetDevice(&dev));
  SLS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (x_dtype == SLS_F32)
    return launch_simt_t<float>(X, N, d, ldx, W, b, D, scale, Phi, phi_bf16, sms, stream);
  return launch_simt_t<uint16_t>(X, N, d, ldx, W, b, D, scale, Phi, phi_bf16, sms, stream);
}

}  // namespace sls
