// Implicit Lanczos (Algorithm 2): the persistent kernel.
//
// Lanczos runs as one persistent cooperative kernel.  The grid is split into
// groups of CTAs; a group owns one problem at a time (one prompt, or one
// adaptive window) and every CTA owns a contiguous strip of the problem's rows
// of the feature matrix Phi (N x D, float32 or bfloat16) and of the basis Q.
// The eight warps of a CTA form teams of WPR warps (WPR = 1 up to D = 1024, 2
// up to 2048, 4, 8): a team takes whole rows of the strip, R at a time, and
// every lane keeps its columns of w_j and of the column sums in registers.  A
// team streams its rows through its own shared-memory ring with
// one-dimensional bulk copies (cp.async.bulk + mbarrier): a stage holds R rows
// of Phi and the same rows of Q.
//
// The whole run makes r passes over Phi: a prologue pass Phi^T q1, then one
// fused pass per step but the last.  Step j starts from z' (the new Lanczos
// direction before its re-orthogonalisation; z' = q1 for j = 0; kept in column
// j of Q), the CTA partials of Phi^T z' and the group sums of c = Q^T z' and
// of |z'|^2:
//
//   [barrier 1]
//   slice phase   c from the group sums; each CTA finishes a slice of the D
//                 columns of Phi^T z1 = Phi^T z' - sum_k c_k w_k with
//                 z1 = z' - Q c and w_k = Phi^T q_k kept from earlier steps.
//   [barrier 2]
//                 beta_{j-1} = |z1| = sqrt(|z'|^2 - |c|^2), the break test,
//                 w_j = Phi^T q_j, alpha_j = |w_j|^2.
//   fused pass    per R rows of a team: the implicit matvec rows s = Phi w_j
//                 (Eq. implicit_matvec); z1 = z' - Q c and q_j = z1 / beta;
//                 the three-term recurrence z' = s - alpha_j q_j -
//                 beta_{j-1} q_{j-1} with its partials of c and |z'|^2; and
//                 the columns Phi^T z' of the next step, from the same rows
//                 while they are in shared memory.
//
// The last step only forms q_{r-1}.  This is Algorithm 2 with full
// re-orthogonalisation by one classical Gram-Schmidt pass per step, applied to
// Phi^T z' through the stored w_k so that one pass over Phi per step carries
// both halves of the matvec.  The projection c = Q^T z' of a fully
// re-orthogonalised Lanczos run stays at rounding level, so a second pass
// would change z1 only in the second order of the rounding unit.  Passes
// alternate direction so each starts on the rows the previous one left in
// L2.  Vectors are double-float (two float32) and every sum over N or D is
// compensated.  The column sums of Phi^T z' are added over the CTAs in a fixed
// order; the group sums of the scalars (c, |z'|^2, |Phi^T z1|^2) are float64
// atomic additions, one per CTA, whose order may vary in the last float64 bit.
// Barriers and waits poll without sleeping and give up after about a second
// of clock cycles, reporting SLS_ERR_TIMEOUT through the status word.
//
// Why whole rows per team: a row's scalars (q_j, z', its products with the
// basis) are a serial chain of double-float operations.  When all eight warps
// shared every row, that chain stood between two barriers of the whole CTA for
// every eight rows, and each warp ran it for one row on 32 identical lanes.
// Here 32 / R lanes share a row's chain, R rows at a time, and the teams run
// independently (with WPR = 1 a pass holds no barrier at all), so one team's
// chain is hidden behind the sweeps of the others, and inside a warp behind the
// row dots of the next R rows.  Measured against the CTA-wide form (whole
// sls_lanczos_topr calls, both built and timed alternately): 64 windows of 2048
// rows at D = 1024, r = 32 5.91 -> 4.32 ms; N = 32756, D = 2048, r = 64 4.57 ->
// 4.01 ms; N = 8180, D = 1024, r = 32 0.750 -> 0.731 ms; windows of 1024 rows at
// D = 256 2.95 -> 1.07 ms; N = 12000, D = 1536, r = 48 2.10 -> 1.34 ms.
//
// The kernel is a template over NV (float4 column groups of Phi per lane), WPR,
// KT (32-wide tiles of the basis index k < r), FULLD (D = 128 NV WPR, no ragged
// columns) and the element type of Phi; each lanczos_{f32,bf16}_<NV>_<WPR>.cu
// instantiates one (NV, WPR) and type.
#pragma once

#include <cfloat>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace sls {

namespace {

constexpr int LZ_NCW = 8;                 // warps per CTA
constexpr int LZ_NT = LZ_NCW * 32;        // threads per CTA
constexpr unsigned BAR_ALL = 1;           // named barrier: every warp
constexpr unsigned BAR_TEAM = 2;          // named barriers 2 .. 5: the warps of a team

// Per-group scratch layout (byte offsets), identical on host and device.
//   acc:   2 x (r + 4) float64 group sums by step parity: c_k (k <= r), |z'|^2
//          at r + 1, |Phi^T z1|^2 at r + 2 (float64 atomic additions)
//   wpart: g x D double-float CTA partials of Phi^T z'
//   wred:  D double-float: Phi^T z1, finished slice by slice
//   Wm:    r x D double-float: w_k = Phi^T q_k (each CTA writes its slice)
struct LzLayout {
  size_t bar, acc, zero_end, wpart, wred, Wm, total;
};

__host__ __device__ inline size_t lz_al(size_t x) { return (x + 255) & ~(size_t)255; }
__host__ __device__ inline int lz_acc_stride(int r) { return r + 4; }

__host__ __device__ inline LzLayout lz_layout(int64_t nmax, int D, int r, int g) {
  (void)nmax;
  LzLayout L;
  size_t o = 0;
  L.bar = o;    o += 256;
  L.acc = o;    o += lz_al((size_t)2 * lz_acc_stride(r) * sizeof(double));
  L.zero_end = o;  // [bar, zero_end) starts at zero before the launch
  L.wpart = o;  o += lz_al((size_t)g * D * sizeof(float2));
  L.wred = o;   o += lz_al((size_t)D * sizeof(float2));
  L.Wm = o;     o += lz_al((size_t)D * r * sizeof(float2));
  L.total = o;
  return L;
}

SLS_DEV dfloat shfl_xor_df(dfloat v, int m) {
  v.hi = __shfl_xor_sync(0xffffffffu, v.hi, m);
  v.lo = __shfl_xor_sync(0xffffffffu, v.lo, m);
  return v;
}

// float64 atomic addition whose result is not used (a reduction operation)
SLS_DEV void red_add_f64(double* p, double v) { atomicAdd(p, v); }

// The split of a row over a team: NV float4 column groups per lane, WPR warps
// (NV * 32 * 4 * WPR >= D), R rows at a time.  NV <= 8: a lane keeps w_j, the
// column sums and their offset sums (10 float32 per column pair and group) in
// registers, 160 of 255 at NV = 8.  The narrowest split that holds the row is
// taken: lanes past the row's end would do their share of the arithmetic on
// nothing.  R = 4 up to D = 512, where a row's sweeps are shorter than its row
// work; 2 above, where 3 stages of 2 rows per team fill the shared memory.
struct LzShape {
  int nv, wpr, R;
};

__host__ __device__ constexpr int lz_rows(int nv) { return nv >= 6 ? 2 : 4; }

__host__ __device__ inline LzShape lz_shape(int D) {
  LzShape s{8, 8, lz_rows(8)};
  if (D <= 256) s = LzShape{2, 1, lz_rows(2)};
  else if (D <= 384) s = LzShape{3, 1, lz_rows(3)};
  else if (D <= 512) s = LzShape{4, 1, lz_rows(4)};
  else if (D <= 768) s = LzShape{6, 1, lz_rows(6)};
  else if (D <= 1024) s = LzShape{8, 1, lz_rows(8)};
  else if (D <= 1536) s = LzShape{6, 2, lz_rows(6)};
  else if (D <= 2048) s = LzShape{8, 2, lz_rows(8)};
  else if (D <= 4096) s = LzShape{8, 4, lz_rows(8)};
  return s;
}

// Ring stage: R rows of Phi (esz bytes per element: 4 for float32, 2 for
// bfloat16) followed by the same R rows of the basis Q (ldq float2 each).
constexpr int LZ_MAX_STAGES = 8;

__host__ __device__ inline unsigned lz_stage_bytes(int D, int ldq, int esz, int R) {
  return (unsigned)R * ((unsigned)D * (unsigned)esz + (unsigned)ldq * 8u);
}

// Shared memory besides the rings (bytes), in the order the kernel carves it:
// the row sums the warps of a team exchange, c, then the mbarriers.
__host__ __device__ inline size_t lz_smem_other(int r, LzShape s, int stages) {
  const int teams = LZ_NCW / s.wpr;
  size_t b = sizeof(float4) * (size_t)(teams * 2 * s.R * s.wpr);
  b += sizeof(float2) * (size_t)(r + 1);
  b = (b + 15) & ~(size_t)15;
  b += (size_t)teams * stages * 8;
  return b;
}

// Transposed butterfly over R rows: every lane holds one partial per row; the
// first three steps (lanes 16, 8 and 4 apart) add plainly, after which lane L
// holds the sum over eight lanes of row L / (32 / R).
template <int R>
SLS_DEV float transpose_sum8(float (&v)[R]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
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

// Double-float sum without the second renormalisation (11 operations): the
// error is a few units of the low part, enough for partial sums that are
// combined once.
SLS_DEV dfloat df_add_fast(dfloat a, dfloat b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  float h, l;
  fast_two_sum(s, e, h, l);
  return df_make(h, l);
}

// The last step: z1 = z' - Q c (the re-orthogonalisation with c = Q^T z' of
// the last pass, float32: the coefficients are at rounding level) and
// q_j = z1 / beta_{j-1}, in place in column j of Q, one warp per row.
SLS_DEV void last_row_phase(float2* __restrict__ Qs, int ldq, int nrows, int j,
                            const float2* __restrict__ cs, dfloat invb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = warp; i < nrows; i += LZ_NCW) {
    float2* q = Qs + (size_t)i * ldq;
    float s = 0.f;
    for (int k = lane; k < j; k += 32) {
      const float2 a = q[k], c = cs[k];
      s = fmaf(a.x, c.x, fmaf(a.x, c.y, fmaf(a.y, c.x, s)));
    }
    s = warp_sum_f(s);
    dfloat z1 = dfv(q[j]);
    if (j > 0) z1 = df_add(z1, df_make(-s, 0.f));
    const dfloat qj = df_mul(z1, invb);
    __syncwarp();
    if (lane == 0) q[j] = f2(qj);
  }
}

// A wait of this CTA gave up: report it and leave at the next group barrier.
SLS_DEV void lz_fail(int* status, volatile int* err) {
  atomicExch(status, SLS_ERR_TIMEOUT);
  *err = 1;
}

SLS_DEV int nprob_of(const LanczosBatch& bt) {
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  return nprob;
}

// Slice phase of step j for the CTA's columns [cbeg, cend): the sum of the g
// CTA partials of Phi^T z' minus sum_{k < j} c_k w_k, into wred, and the
// CTA's part of |Phi^T z1|^2 (each thread returns its own columns' share).
// A column is summed by a segment of G lanes of one warp (G a power of two,
// as many as the compute threads allow), each lane over every G-th partial
// and every G-th basis index, then a butterfly within the segment.  The loads
// of the first column batch are issued before the named barrier after which
// c is ready (warp 0 fills it meanwhile); `synced` records that barrier.
// True when the last warp of the CTA sums no column in the slice phase (the
// column split of slice_columns below): it is free then for beta.
template <int NCW>
SLS_DEV bool slice_last_warp_idle(int ncol) {
  constexpr int NCT = NCW * 32;
  int G = 1;
  while (G < 32 && G * 2 * ncol <= NCT) G *= 2;
  return (NCW - 1) * (32 / G) >= ncol;
}

// c itself (cs[k] = the group sum accj[k], k < j) is loaded by warp cwarp:
// after it has issued its first batch when it sums columns, so that both
// round trips to L2 overlap, else before it reaches the named barrier.
template <int NCW>
SLS_DEV void load_c(float2* __restrict__ cs, const double* __restrict__ accj, int j) {
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < j; k += 32) cs[k] = f2(df_from_double(accj[k]));
}

template <int NCW>
SLS_DEV dfloat slice_columns(const float2* __restrict__ wpart, const float2* __restrict__ Wm,
                             float2* __restrict__ wred, float2* __restrict__ cs,
                             const double* __restrict__ accj, int cwarp, int g, int D, int j,
                             int cbeg, int cend, bool& synced) {
  constexpr int NCT = NCW * 32;
  constexpr int BATCH = 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ncol = cend - cbeg;
  int G = 1;
  while (G < 32 && G * 2 * ncol <= NCT) G *= 2;
  const int cpw = 32 / G;
  const int sub = lane & (G - 1), slot = lane / G;
  dfloat sq = df_make(0.f, 0.f);
  for (int cb = warp * cpw; cb < ncol; cb += NCW * cpw) {
    const int cl = cb + slot;
    const bool valid = cl < ncol;
    const int c = cbeg + (valid ? cl : 0);
    // partials of Phi^T z' and basis columns: the first batches in flight together
    float2 pv[BATCH], wv[BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int b = sub + G * u;
      pv[u] = (valid && b < g) ? wpart[(size_t)b * D + c] : make_float2(0.f, 0.f);
      wv[u] = (valid && b < j) ? Wm[(size_t)b * D + c] : make_float2(0.f, 0.f);
    }
    if (!synced && warp == cwarp) load_c<NCW>(cs, accj, j);
    dfloat s = df_make(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < BATCH; ++u) s = df_add_fast(s, dfv(pv[u]));
    for (int b0 = sub + G * BATCH; b0 < g; b0 += G * BATCH) {
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int b = b0 + G * u;
        pv[u] = (valid && b < g) ? wpart[(size_t)b * D + c] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) s = df_add_fast(s, dfv(pv[u]));
    }
    if (!synced) {
      named_sync(BAR_ALL, NCT);  // c is in shared memory
      synced = true;
    }
    // sum_k c_k w_k (Dot2), subtracted from the lane's part of the column sum
    float ch = 0.f, cl2 = 0.f;
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int k = sub + G * u;
      if (k < j) dot2_acc_df(ch, cl2, dfv(wv[u]), dfv(cs[k]));
    }
    for (int k0 = sub + G * BATCH; k0 < j; k0 += G * BATCH) {
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int k = k0 + G * u;
        wv[u] = (valid && k < j) ? Wm[(size_t)k * D + c] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int k = k0 + G * u;
        if (k < j) dot2_acc_df(ch, cl2, dfv(wv[u]), dfv(cs[k]));
      }
    }
    s = df_sub(s, df_norm(ch, cl2));
    for (int o = 1; o < G; o <<= 1) s = df_add_fast(s, shfl_xor_df(s, o));
    if (sub == 0 && valid) {
      wred[c] = f2(s);
      dot2_acc_df(sq.hi, sq.lo, s, s);
    }
  }
  if (!synced && warp == cwarp) load_c<NCW>(cs, accj, j);  // a warp without columns
  return sq;
}

// Rows of one team in a ring: batches of R rows are numbered over the CTA's
// whole run; batch cnt goes to slot cnt % S, whose mbarrier completes one phase
// per batch.  Every warp of the team consumes every batch in order, and only
// lane 0 of the team's first warp issues them, each after the team has consumed
// the slot's previous batch, so phase parities are unambiguous.
struct RingPos {
  unsigned slot, par;
};

SLS_DEV void ring_next(RingPos& q, unsigned S) {
  if (++q.slot == S) {
    q.slot = 0u;
    q.par ^= 1u;
  }
}

struct TeamRing {
  unsigned char* base;   // S stages
  uint64_t* full;        // S mbarriers
  unsigned S;
  RingPos in;            // next batch to issue (lane 0 of the team's first warp)
  RingPos out;           // next batch to consume
};

// Issue the next batch: rows [i0, i0 + nr) of the strip, Phi and (from the
// first fused pass on) the same rows of Q.
template <typename PT>
SLS_DEV void ring_issue(TeamRing& T, int i0, int nr, int D, int ldq, unsigned stage,
                        unsigned phib, bool with_q, const PT* __restrict__ Phi,
                        const float2* __restrict__ Qs, uint64_t pol) {
  const unsigned b1 = (unsigned)(nr * D * (int)sizeof(PT));
  const unsigned b2 = with_q ? (unsigned)(nr * ldq * 8) : 0u;
  unsigned char* dst = T.base + (size_t)T.in.slot * stage;
  uint64_t* bar = &T.full[T.in.slot];
  mbar_expect_tx(bar, b1 + b2);
  bulk_g2s(dst, Phi + (int64_t)i0 * D, b1, bar, pol);
  if (b2) bulk_g2s(dst + phib, Qs + (int64_t)i0 * ldq, b2, bar, pol);
  ring_next(T.in, T.S);
}

// z' = s - alpha q - beta qp, all double-float: the two products are split
// exactly, their high parts subtracted by TwoSum, and every error term is
// gathered in the low part.
SLS_DEV dfloat df_recur(dfloat s, dfloat alpha, dfloat q, dfloat beta, dfloat qp) {
  float p1, e1, p2, e2, t1, f1, t2, f2_;
  two_prod(alpha.hi, q.hi, p1, e1);
  two_prod(beta.hi, qp.hi, p2, e2);
  e1 = __fmaf_rn(alpha.hi, q.lo, e1);
  e2 = __fmaf_rn(beta.hi, qp.lo, e2);
  e1 = __fmaf_rn(alpha.lo, q.hi, e1);
  e2 = __fmaf_rn(beta.lo, qp.hi, e2);
  two_sum(s.hi, -p1, t1, f1);
  two_sum(t1, -p2, t2, f2_);
  const float lo = __fadd_rn(__fadd_rn(__fsub_rn(f1, e1), __fsub_rn(f2_, e2)), s.lo);
  return df_norm(t2, lo);
}

// One step of the sweeps on a pair of columns: (s, lo) += x * (yh + yl).
// PK: one packed instruction per operation, else two scalar ones.
template <bool PK>
SLS_DEV void ofs_step(f32x2_t& s, f32x2_t& lo, f32x2_t x, f32x2_t yh, f32x2_t yl) {
  if constexpr (PK) {
    ofs_fma_acc2(s, lo, x, yh, yl);
  } else {
    float s0, s1, l0, l1, x0, x1, h0, h1, m0, m1;
    upk2(s, s0, s1);
    upk2(lo, l0, l1);
    upk2(x, x0, x1);
    upk2(yh, h0, h1);
    upk2(yl, m0, m1);
    ofs_fma_acc(s0, l0, x0, h0, m0);
    ofs_fma_acc(s1, l1, x1, h1, m1);
    s = pk2(s0, s1);
    lo = pk2(l0, l1);
  }
}

// The sweeps run on packed float32 pairs: against scalar steps the packed form
// halves the issue slots of the same arithmetic (lanczos 32k 4434 -> 4054 us,
// windows of 2048 rows 4693 -> 4270 us, 8k 771 -> 733 us).
constexpr bool LZ_PK = true;

// One float per row of a batch.
template <int R>
struct RowVals {
  float v[R];
};

template <int NV, int WPR, int KT, bool FULLD, typename PT>
__global__ void __launch_bounds__(LZ_NT, 1)
lanczos_kernel(LanczosBatch bt, char* scratch, size_t gstride, int g, int ngroups,
               int ring_stages, int* status) {
  constexpr int NCW = LZ_NCW, NCT = LZ_NT;
  constexpr int R = lz_rows(NV);
  constexpr int LPR = 32 / R;               // lanes per row in the row work
  constexpr int TEAMS = NCW / WPR;
  constexpr int NC = 4 * NV;                // columns per lane
  using RV = RowVals<R>;
  // basis coefficients per lane: k = sub + LPR * (t * WPR + tw), t < KC
  constexpr int KC = (KT * 32 + LPR * WPR - 1) / (LPR * WPR);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ float2 tmpw[NCW];
  __shared__ float s_red1[NCW];  // per-warp max |Phi| (offset bounds)
  __shared__ double shd[4];
  __shared__ float2 sdf[3];  // 1 / beta, alpha, beta of the step as double-float
  __shared__ int sflag, sbreak;
  __shared__ volatile int s_err;      // a wait of this CTA gave up

  const int D = bt.D, r = bt.r, ldq = q_ld(bt.r);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int team = warp / WPR, tw = warp % WPR;
  const int ri = lane / LPR, sub = lane % LPR;
  const int gi = blockIdx.x / g, rank = blockIdx.x % g;
  const int C4 = D >> 2;
  const unsigned bar_team = BAR_TEAM + (unsigned)team;
  const bool leader = lane == 0 && tw == 0;  // issues the team's copies

  const unsigned phib = (unsigned)R * (unsigned)D * (unsigned)sizeof(PT);
  const unsigned stage = lz_stage_bytes(D, ldq, (int)sizeof(PT), R);
  TeamRing ring{smem_raw + (size_t)team * ring_stages * stage, nullptr, (unsigned)ring_stages,
                RingPos{0u, 0u}, RingPos{0u, 0u}};
  float4* exch = reinterpret_cast<float4*>(smem_raw + (size_t)TEAMS * ring_stages * stage);
  float2* cs = reinterpret_cast<float2*>(exch + TEAMS * 2 * R * WPR);  // r + 1 (c = Q^T z')
  uint64_t* fullb = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(cs + (r + 1)) + 15) & ~(uintptr_t)15);
  ring.full = fullb + team * ring_stages;
  exch += team * 2 * R * WPR;
  // scratch of the pass ends, in the team's ring (idle then): its column sums,
  // its coefficient partials (k < r) and, at r, its part of |z'|^2
  const size_t tstride = (size_t)ring_stages * stage;
  auto tcol = [&](int t) { return reinterpret_cast<float2*>(smem_raw + (size_t)t * tstride); };
  auto tco = [&](int t) { return tcol(t) + D; };

  const LzLayout L = lz_layout(bt.nmax, D, r, g);
  char* gb = scratch + (size_t)gi * gstride;
  unsigned* barw = reinterpret_cast<unsigned*>(gb + L.bar);
  double* acc = reinterpret_cast<double*>(gb + L.acc);
  float2* wpart = reinterpret_cast<float2*>(gb + L.wpart);
  float2* wred = reinterpret_cast<float2*>(gb + L.wred);
  float2* Wm = reinterpret_cast<float2*>(gb + L.Wm);
  const GroupBarrier bar{barw, barw + 32, (unsigned)g};
  const int accs = lz_acc_stride(r);
  const uint64_t pol = l2_policy_evict_first();

  if (tid == 0) {
    for (int s = 0; s < TEAMS * ring_stages; ++s) mbar_init(&fullb[s], 1);
    mbar_fence_init();
    s_err = 0;
  }
  __syncthreads();

  // Before the CTA leaves: every batch issued has landed.  The slots after the
  // issue position hold the oldest batches; a slot that was never issued to is
  // in the first phase, whose predecessor parity reads as complete.
  auto drain = [&]() {
    if (leader) {
      RingPos q = ring.in;
      for (unsigned c = 0; c < ring.S; ++c) {
        mbar_wait(&ring.full[q.slot], q.par ^ 1u);
        ring_next(q, ring.S);
      }
    }
  };
  // Wait (bounded) for the team's next batch; its stage.
  auto next_stage = [&]() -> const unsigned char* {
    const RingPos q = ring.out;
    // once a wait has given up no further batch is issued: nothing to wait for
    if (!mbar_try_wait(&ring.full[q.slot], q.par) && !s_err && !mbar_wait(&ring.full[q.slot], q.par))
      lz_fail(status, &s_err);
    ring_next(ring.out, ring.S);
    return ring.base + (size_t)q.slot * stage;
  };

  const int nprob = nprob_of(bt);
  unsigned lgen = 0;
  unsigned gstep = 0;  // steps run by this group so far (parity of the group sums)
  for (int p = gi; p < nprob; p += ngroups) {
    const int64_t row0 = bt.row0 ? bt.row0[p] : 0;
    const int64_t n = bt.n ? (int64_t)bt.n[p] : bt.n_single;
    const int64_t q1o = bt.q1off ? bt.q1off[p] : row0;
    const double* q1 = bt.q1 + q1o;
    const int64_t rs = (int64_t)rank * n / g, re = (int64_t)(rank + 1) * n / g;
    const PT* Phis = reinterpret_cast<const PT*>(bt.Phi) + (row0 + rs) * D;  // this CTA's rows
    float2* Qs = bt.Q + (row0 + rs) * ldq;  // this CTA's rows of the basis
    const int nrows = (int)(re - rs);
    // batches of the strip, and of this team (batch b of the team: team + b * TEAMS)
    const int nball = (nrows + R - 1) / R;
    const int nb = nball > team ? (nball - team + TEAMS - 1) / TEAMS : 0;
    double* alpha_out = bt.alpha + (size_t)p * r;
    double* beta_out = bt.beta + (size_t)p * r;
    const int cbeg = (int)((int64_t)rank * D / g), cend = (int)((int64_t)(rank + 1) * D / g);

    double scale = 0.0, alpha_prev = 0.0;
    // beta_{j-1} = 1 / e_inv and the break test of the step, in lane 0 of
    // warp bw: the last warp during the slice phase when that warp sums no
    // column there (measured 2% faster at the qwen7b shape), else warp 0
    // after group barrier 2
    double e_inv = 0.0, e_bnew = 0.0;
    int e_brk = 0;
    const bool beta_early = slice_last_warp_idle<NCW>(cend - cbeg);
    const int bw = beta_early ? NCW - 1 : 0;
    dfloat alpha_df = df_make(0.f, 0.f), beta_df = df_make(0.f, 0.f), invb_df;
    float phimax = 0.f;  // max |Phi| over this CTA's strip (prologue pass)
    int reff = 0;
    sbreak = 0;

    // Row range of the team's batch b in pass `pass` (0 = the prologue;
    // passes alternate direction).
    auto batch_row = [&](int pass, int b) {
      return (team + ((pass & 1) ? nb - 1 - b : b) * TEAMS) * R;
    };
    // Issue the team's batch b of a pass.  No batch is issued once a wait of
    // this CTA has given up (s_err): a slot then never receives a batch whose
    // predecessor in the slot was not seen to land.
    auto issue = [&](int pass, int b) {
      if (b < nb && !s_err) {
        const int i0 = batch_row(pass, b);
        SLS_DBG_CHECK(status, i0 >= 0 && i0 < nrows);
        ring_issue<PT>(ring, i0, min(R, nrows - i0), D, ldq, stage, phib, pass > 0, Phis, Qs, pol);
      }
    };
    auto issue_pass_head = [&](int pass) {
      if (leader)
        for (int b = 0; b < (int)ring.S; ++b) issue(pass, b);
    };

    // pass end: the column sums of the teams are added through their rings
    // (idle now) and stored as the CTA's partials of Phi^T z'; the coefficient
    // partials (k < K) and |z'|^2 join the group sums of parity `par` (float64
    // atomics)
    auto pass_end = [&](f32x2_t (&ah)[NC / 2], f32x2_t (&al)[NC / 2], dfloat (&cacc)[KC], int K,
                        dfloat nacc,
                        unsigned par) {
      if constexpr (WPR > 1) named_sync(bar_team, WPR * 32);  // the team is done with its ring
      else __syncwarp();
      {
        float4* d4 = reinterpret_cast<float4*>(tcol(team));
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          const int cg = lane + 32 * (q * WPR + tw);
          if (cg < C4) {
            float h0, h1, h2, h3, l0, l1, l2, l3;
            upk2(ah[2 * q], h0, h1);
            upk2(ah[2 * q + 1], h2, h3);
            upk2(al[2 * q], l0, l1);
            upk2(al[2 * q + 1], l2, l3);
            const dfloat n0 = df_norm(h0, l0), n1 = df_norm(h1, l1);
            const dfloat n2 = df_norm(h2, l2), n3 = df_norm(h3, l3);
            d4[2 * cg] = make_float4(n0.hi, n0.lo, n1.hi, n1.lo);
            d4[2 * cg + 1] = make_float4(n2.hi, n2.lo, n3.hi, n3.lo);
          }
        }
      }
      // coefficients and |z'|^2: the R row groups of the warp hold the same k
      float2* cw = tco(team);
#pragma unroll
      for (int t = 0; t < KC; ++t) {
        if (LPR * (t * WPR + tw) >= K) break;
        dfloat v = df_norm(cacc[t].hi, cacc[t].lo);
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) v = df_add_fast(v, shfl_xor_df(v, o));
        const int k = sub + LPR * (t * WPR + tw);
        if (ri == 0 && k < K) cw[k] = f2(v);
      }
      if (tw == 0) {
        dfloat nv = df_norm(nacc.hi, nacc.lo);
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) nv = df_add_fast(nv, shfl_xor_df(nv, o));
        if (lane == 0) cw[r] = f2(nv);
      }
      // the columns of Q written in this pass reach the bulk reads of the next
      // one, and the ring writes above are ordered before its bulk writes
      // (async proxy)
      asm volatile("fence.proxy.async;" ::: "memory");
      named_sync(BAR_ALL, NCT);
      {
        float4* dst = reinterpret_cast<float4*>(wpart + (size_t)rank * D);
        for (int c = tid; c < (D >> 1); c += NCT) {
          float4 v[TEAMS];
#pragma unroll
          for (int t = 0; t < TEAMS; ++t) v[t] = reinterpret_cast<const float4*>(tcol(t))[c];
#pragma unroll
          for (int w = 1; w < TEAMS; w *= 2)
#pragma unroll
            for (int t = 0; t + w < TEAMS; t += 2 * w) {
              const dfloat a = df_add_fast(df_make(v[t].x, v[t].y), df_make(v[t + w].x, v[t + w].y));
              const dfloat b = df_add_fast(df_make(v[t].z, v[t].w), df_make(v[t + w].z, v[t + w].w));
              v[t] = make_float4(a.hi, a.lo, b.hi, b.lo);
            }
          dst[c] = v[0];
        }
      }
      // coefficient k (|z'|^2 at r): the TEAMS partials summed by two lanes
      double* accn = acc + (size_t)(par & 1u) * accs;
      for (int k0 = 0; k0 < K + 1; k0 += NCT / 2) {
        const int e = k0 + tid / 2, part = tid & 1;
        const int k = (e < K) ? e : r;
        dfloat s = df_make(0.f, 0.f);
        if (e <= K)
          for (int t = part; t < TEAMS; t += 2) s = df_add(s, dfv(tco(t)[k]));
        s = df_add_fast(s, shfl_xor_df(s, 1));
        if (part == 0 && e <= K) red_add_f64(accn + (e < K ? e : r + 1), df_to_double(s));
      }
      named_sync(BAR_ALL, NCT);
    };

    issue_pass_head(0);

    // ---------------- prologue: z' = q1, |z'|^2 and Phi^T z' (pass 0) ------------
    {
      f32x2_t ah[NC / 2], al[NC / 2];
#pragma unroll
      for (int c = 0; c < NC / 2; ++c) ah[c] = al[c] = 0ull;
      dfloat nacc = df_make(0.f, 0.f);
      float mx = 0.f;
      for (int b = 0; b < nb; ++b) {
        const int i0 = batch_row(0, b), nr = min(R, nrows - i0);
        dfloat z = df_make(0.f, 0.f);
        if (ri < nr) {
          z = df_from_double(q1[rs + i0 + ri]);
          if (tw == 0 && sub == 0) {
            SLS_DBG_GUARD(status, i0 + ri < nrows) Qs[(size_t)(i0 + ri) * ldq] = f2(z);
          }
        }
        dot2_acc_df(nacc.hi, nacc.lo, z, z);
        const PT* phi = reinterpret_cast<const PT*>(next_stage());
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float uh = __shfl_sync(0xffffffffu, z.hi, i * LPR);
          const float ul = __shfl_sync(0xffffffffu, z.lo, i * LPR);
          const f32x2_t uhp = pk2(uh, uh), nuh = pk2(-uh, -uh), ulp = pk2(ul, ul);
          if (i < nr) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
              const int cg = lane + 32 * (q * WPR + tw);
              if (cg < C4) {
                const float4 f = phi_ld4(phi, (size_t)i * C4 + cg);
                dot2_acc2n(ah[2 * q], al[2 * q], pk2(f.x, f.y), uhp, nuh, ulp);
                dot2_acc2n(ah[2 * q + 1], al[2 * q + 1], pk2(f.z, f.w), uhp, nuh, ulp);
                mx = fmaxf(mx, fmaxf(fmaxf(fabsf(f.x), fabsf(f.y)), fmaxf(fabsf(f.z), fabsf(f.w))));
              }
            }
          }
        }
        if constexpr (WPR > 1) named_sync(bar_team, WPR * 32);
        else __syncwarp();
        if (leader) issue(0, b + (int)ring.S);
      }
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0) s_red1[warp] = mx;
      dfloat cacc0[KC];
#pragma unroll
      for (int t = 0; t < KC; ++t) cacc0[t] = df_make(0.f, 0.f);
      // |q1|^2 is the group sum of the first step
      pass_end(ah, al, cacc0, 0, nacc, gstep);
      if (r >= 2) issue_pass_head(1);
    }

    if (bt.inject_fail && rank == 0 && tid == 0) lz_fail(status, &s_err);
    for (int j = 0; j < r; ++j, ++gstep) {
      if (!group_sync_named(bar, lgen, status, &sflag, &s_err, BAR_ALL, NCT)) {
        drain();
        return;
      }
      const double* accj = acc + (size_t)(gstep & 1u) * accs;
      // |z1|^2 = |z'|^2 - |c|^2 (Q orthonormal): beta_{j-1} and the break
      // test (warp bw, once c is in shared memory)
      auto beta_phase = [&]() {
        const double zs = accj[r + 1];
        dfloat cn = df_make(0.f, 0.f);
#pragma unroll
        for (int t2 = 0; t2 < KT; ++t2) {
          const int k = lane + 32 * t2;
          if (k < j) dot2_acc_df(cn.hi, cn.lo, dfv(cs[k]), dfv(cs[k]));
        }
        cn = df_norm(cn.hi, cn.lo);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cn = df_add_fast(cn, shfl_xor_df(cn, o));
        if (lane == 0) {
          const double nrm2 = zs - df_to_double(cn);  // |z1|^2
          // one reciprocal square root instead of a square root and two
          // divides (float64 runs at a fraction of the float32 rate here)
          e_inv = (nrm2 > 0.0) ? rsqrt(nrm2) : 0.0;  // 1 / beta
          e_bnew = (nrm2 > 0.0) ? nrm2 * e_inv : 0.0;
          e_brk = 0;
          if (j > 0) {
            scale = fmax(scale, fabs(alpha_prev) + e_bnew);
            if (!(e_bnew > bt.tol * scale)) e_brk = 1;
            else if (rank == 0) beta_out[j - 1] = e_bnew;
          } else if (!(e_bnew > 0.0)) {
            e_brk = 1;
          }
        }
      };

      // ---------------- slice phase: c, Phi^T z1 for this CTA's columns ----------
      // c = Q^T z' (k < j) from the group sums; Phi^T z1 = Phi^T z' - sum_k
      // c_k w_k with w_k = Phi^T q_k kept in Wm.  The group sums of the other
      // parity were read in the previous step by every CTA (all of them have
      // passed barrier 1 since): the first CTA clears them for the next step.
      if (rank == 0) {
        double* accz = acc + (size_t)((gstep + 1u) & 1u) * accs;
        for (int k = tid; k < accs; k += NCT) accz[k] = 0.0;
      }
      {
        // c is loaded by the last warp when it sums no column (it waits for
        // beta there anyway), else by warp 0
        bool synced = false;
        dfloat sq = slice_columns<NCW>(wpart, Wm, wred, cs, accj, beta_early ? NCW - 1 : 0, g, D,
                                       j, cbeg, cend, synced);
        if (!synced) named_sync(BAR_ALL, NCT);
        if (beta_early && warp == NCW - 1) beta_phase();
        sq = df_norm(sq.hi, sq.lo);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq = df_add_fast(sq, shfl_xor_df(sq, o));
        if (lane == 0) tmpw[warp] = f2(sq);
        named_sync(BAR_ALL, NCT);
        if (warp == 0) {
          // the NCW warp sums by a butterfly over the first NCW lanes
          dfloat t = (lane < NCW) ? dfv(tmpw[lane]) : df_make(0.f, 0.f);
#pragma unroll
          for (int o = 1; o < NCW; o <<= 1) t = df_add_fast(t, shfl_xor_df(t, o));
          if (lane == 0) red_add_f64(const_cast<double*>(accj) + r + 2, df_to_double(t));
        }
      }
      if (!group_sync_named(bar, lgen, status, &sflag, &s_err, BAR_ALL, NCT)) {
        drain();
        return;
      }

      // ---------------- beta_{j-1}, alpha_j, break test; w_j gather ---------------
      // this lane's columns of Phi^T z1 (loads in flight while the scalars are formed)
      float4 wv[NV][2];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        const int cg = lane + 32 * (q * WPR + tw);
        wv[q][0] = wv[q][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (cg < C4) {
          wv[q][0] = reinterpret_cast<const float4*>(wred)[2 * cg];
          wv[q][1] = reinterpret_cast<const float4*>(wred)[2 * cg + 1];
        }
      }
      if (!beta_early && warp == 0) beta_phase();
      if (warp == bw && lane == 0) {
        const double q = accj[r + 2];  // |Phi^T z1|^2
        const double a = e_brk ? 0.0 : (q * e_inv) * e_inv;
        if (!e_brk && rank == 0) alpha_out[j] = a;
        shd[1] = e_brk ? 0.0 : e_inv;
        shd[2] = a;
        shd[3] = (j > 0) ? e_bnew : 0.0;
        // converted once here: float64 runs at a small fraction of the
        // float32 rate on this part, and every thread needs these
        sdf[0] = f2(df_from_double(shd[1]));
        sdf[1] = f2(df_from_double(a));
        sdf[2] = f2(df_from_double(shd[3]));
        sbreak = e_brk;
      }
      named_sync(BAR_ALL, NCT);
      if (sbreak) {
        reff = j;
        break;
      }
      invb_df = dfv(sdf[0]);
      alpha_prev = shd[2];
      alpha_df = dfv(sdf[1]);
      beta_df = dfv(sdf[2]);
      if (j == 0) {
#pragma unroll
        for (int w = 0; w < NCW; ++w) phimax = fmaxf(phimax, s_red1[w]);
      }

      if (j == r - 1) {
        // the last step needs no pass over Phi: q_{r-1} = z1 / beta_{r-2}
        last_row_phase(Qs, ldq, nrows, j, cs, invb_df);
        reff = r;
        break;
      }

      // w_j = (Phi^T z1) / beta in registers; the CTA's slice of it is kept for
      // the correction of later steps
      for (int c = cbeg + tid; c < cend; c += NCT)
        Wm[(size_t)j * D + c] = f2(df_mul(dfv(wred[c]), invb_df));
      f32x2_t wh[NC / 2], wl[NC / 2];
      float wt1 = 0.f;  // l1 norm of this lane's part of w_j
#pragma unroll
      for (int c = 0; c < NC / 2; ++c) {
        const float4 v = wv[c / 2][c & 1];
        const dfloat w0 = df_mul(df_make(v.x, v.y), invb_df);
        const dfloat w1 = df_mul(df_make(v.z, v.w), invb_df);
        wh[c] = pk2(w0.hi, w1.hi);
        wl[c] = pk2(w0.lo, w1.lo);
        wt1 += fabsf(w0.hi) + fabsf(w1.hi);
      }
      // Offset of the row dots: a power of two above eight times the largest
      // part a lane can hold, so that the sums of eight lanes' parts are exact
      // multiples of its last place below it (see the row dots)
      float wtm = wt1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) wtm = fmaxf(wtm, __shfl_xor_sync(0xffffffffu, wtm, o));
      const float Ct = ofs_pow2(4.f * (phimax * wtm));

      // ---------------- fused pass j+1 over Phi ----------------------------------
      // The team's batches run as a pipeline inside each warp: while a batch's
      // row work (a serial chain of double-float operations on few lanes'
      // worth of data) is under way, the row dots of the next batch fill the
      // issue slots, and the butterfly of those dots runs beside the column
      // sums of the batch before.
      const int pass = j + 1;
      f32x2_t ah[NC / 2], al[NC / 2], sa[NC / 2];
#pragma unroll
      for (int c = 0; c < NC / 2; ++c) ah[c] = al[c] = sa[c] = 0ull;
      float Ca = 0.f;    // offset of the column sums (0: none yet)
      float room = 0.f;  // what the partial sums may still grow by under Ca
      dfloat cacc[KC];
#pragma unroll
      for (int t = 0; t < KC; ++t) cacc[t] = df_make(0.f, 0.f);
      dfloat nacc = df_make(0.f, 0.f);
      int next_b = min(nb, (int)ring.S);  // next batch to issue (leader)
      bool freed = false;                 // the batch before the last barrier is done with
      unsigned xp = 0u;                   // half of the exchange buffer in use
      auto refill = [&]() {
        if (leader && next_b < nb) issue(pass, next_b);
        ++next_b;
      };
      // (sa - Ca), exact, joins the column sums by one TwoSum
      auto flush = [&]() {
        const f32x2_t Cp = pk2(Ca, Ca);
#pragma unroll
        for (int c = 0; c < NC / 2; ++c) {
          const f32x2_t x = sub2(sa[c], Cp);
          const f32x2_t t = add2(ah[c], x);
          const f32x2_t bb = sub2(t, ah[c]);
          const f32x2_t e = add2(sub2(ah[c], sub2(t, bb)), sub2(x, bb));
          ah[c] = t;
          al[c] = add2(al[c], e);
        }
      };
      // This lane's column group q.  When the row is narrower than NV * WPR * 32
      // groups (FULLD = false), the lanes past its end read its last group
      // instead: w_j is 0 there, and their column sums are never stored.
      auto colgroup = [&](int q) {
        const int cg = lane + 32 * (q * WPR + tw);
        return FULLD ? cg : min(cg, C4 - 1);
      };
      // Row dots s = Phi w_j of a batch: a lane's part of a row accumulates
      // against the offset Ct (5 operations per element, common.cuh).  Every
      // part and every sum of up to eight lanes' parts is a multiple of
      // Ct 2^-24 below Ct, so the first three butterfly steps are exact; the
      // rounding errors travel in the low parts.  And this warp's part of
      // the re-orthogonalisation (Q c)_i of the lane's row.
      auto front = [&](auto rows_c, const unsigned char* st, int nr, RV& vh, RV& vl, float& corr) {
        constexpr bool FULL = decltype(rows_c)::value;
        const PT* phi = reinterpret_cast<const PT*>(st);
        const f32x2_t Cp = pk2(Ct, Ct);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          f32x2_t s0 = Cp, l0 = 0ull;
          if (FULL || i < nr) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
              const float4 f = phi_ld4(phi, (size_t)i * C4 + colgroup(q));
              ofs_step<LZ_PK>(s0, l0, pk2(f.x, f.y), wh[2 * q], wl[2 * q]);
              ofs_step<LZ_PK>(s0, l0, pk2(f.z, f.w), wh[2 * q + 1], wl[2 * q + 1]);
            }
          }
          float sx, sy, lx, ly;
          upk2(s0, sx, sy);
          upk2(l0, lx, ly);
          vh.v[i] = (sx - Ct) + (sy - Ct);
          vl.v[i] = lx + ly;
        }
        const float2* qrow = reinterpret_cast<const float2*>(st + phib) + (size_t)ri * ldq;
        corr = 0.f;
        if (FULL || ri < nr) {
#pragma unroll
          for (int t = 0; t < KC; ++t) {
            const int k = sub + LPR * (t * WPR + tw);
            if (k < j) {
              const float2 q = qrow[k], c = cs[k];
              corr = fmaf(q.x, c.x, fmaf(q.x, c.y, fmaf(q.y, c.x, corr)));
            }
          }
        }
      };
      // the butterflies of front's values: the row's dot (this warp's columns)
      // and correction on every lane of the row; exchanged with the team's
      // other warps (the half of the buffer in use was read before the last
      // team barrier)
      auto middle = [&](RV& vh, RV& vl, float& corr, dfloat& s) {
        const float th = transpose_sum8<R>(vh.v);
        const float tl = transpose_sum8<R>(vl.v);
        two_sum(th, tl, s.hi, s.lo);
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) s = df_add_fast(s, shfl_xor_df(s, o));
#pragma unroll
        for (int o = 1; o < LPR; o <<= 1) corr += __shfl_xor_sync(0xffffffffu, corr, o);
        if constexpr (WPR > 1) {
          if (sub == 0) exch[(xp * R + ri) * WPR + tw] = make_float4(s.hi, s.lo, corr, 0.f);
        }
      };
      // row work of a batch: q_j, z' and its partials of c and |z'|^2; z' of
      // the R rows on every lane
      auto back = [&](auto full_c, const unsigned char* st, int i0, int nr, dfloat s, float corr,
                      RV& uh, RV& ul) {
        constexpr bool FULL = decltype(full_c)::value;
        const bool live = FULL || ri < nr;  // the row of this lane
        const float2* qrow = reinterpret_cast<const float2*>(st + phib) + (size_t)ri * ldq;
        if constexpr (WPR > 1) {
          float4 v[WPR];
#pragma unroll
          for (int w = 0; w < WPR; ++w) v[w] = exch[(xp * R + ri) * WPR + w];
          corr = 0.f;
          dfloat d[WPR];
#pragma unroll
          for (int w = 0; w < WPR; ++w) {
            corr += v[w].z;
            d[w] = df_make(v[w].x, v[w].y);
          }
#pragma unroll
          for (int w = 1; w < WPR; w *= 2)
#pragma unroll
            for (int t = 0; t + w < WPR; t += 2 * w) d[t] = df_add_fast(d[t], d[t + w]);
          s = d[0];
        }
        dfloat z1 = df_make(0.f, 0.f), qp = df_make(0.f, 0.f);
        if (live) {
          z1 = dfv(qrow[j]);
          qp = dfv(qrow[j > 0 ? j - 1 : 0]);  // beta = 0 at j = 0
        }
        {
          float t, e;
          two_sum(z1.hi, -corr, t, e);
          z1 = df_norm(t, __fadd_rn(e, z1.lo));
        }
        const dfloat qj = df_mul(z1, invb_df);
        dfloat zp = df_recur(s, alpha_df, qj, beta_df, qp);
        if (!live) zp = df_make(0.f, 0.f);
        if (live && tw == 0 && sub < 2) {
          SLS_DBG_GUARD(status, i0 + ri < nrows)
          Qs[(size_t)(i0 + ri) * ldq + j + sub] = f2(sub == 0 ? qj : zp);
        }
        dot2_acc_df(nacc.hi, nacc.lo, zp, zp);
#pragma unroll
        for (int t = 0; t < KC; ++t) {
          const int k = sub + LPR * (t * WPR + tw);
          dfloat qk = df_make(0.f, 0.f);
          if (live && k < j) qk = dfv(qrow[k]);
          if (k == j) qk = qj;
          dot2_acc_df(cacc[t].hi, cacc[t].lo, qk, zp);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
          uh.v[i] = __shfl_sync(0xffffffffu, zp.hi, i * LPR);
          ul.v[i] = __shfl_sync(0xffffffffu, zp.lo, i * LPR);
        }
      };
      // the offset for a batch's column sums: kept for as long as max|Phi|
      // times the l1 norm of the z' accumulated under it stays below Ca / 2
      // (about eight rows of like size)
      auto offset = [&](const RV& uh) {
        float l1 = 0.f;
#pragma unroll
        for (int i = 0; i < R; ++i) l1 += fabsf(uh.v[i]);
        const float grow = phimax * l1;
        if (!(grow <= room)) {
          if (Ca != 0.f) flush();
          Ca = ofs_pow2((8.f / R) * grow);
          room = Ca * (0.5f / 1.00390625f);
#pragma unroll
          for (int c = 0; c < NC / 2; ++c) sa[c] = pk2(Ca, Ca);
        }
        room -= grow * 1.0000003f;
      };
      // column sums Phi^T z' of a batch
      auto columns = [&](auto rows_c, const unsigned char* st, int nr, const RV& uh,
                         const RV& ul) {
        constexpr bool FULL = decltype(rows_c)::value;
        const PT* phi = reinterpret_cast<const PT*>(st);
        f32x2_t uhp[R], ulp[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
          uhp[i] = pk2(uh.v[i], uh.v[i]);
          ulp[i] = pk2(ul.v[i], ul.v[i]);
        }
#pragma unroll
        for (int q = 0; q < NV; ++q) {
#pragma unroll
          for (int i = 0; i < R; ++i) {
            if (FULL || i < nr) {
              const float4 f = phi_ld4(phi, (size_t)i * C4 + colgroup(q));
              ofs_step<LZ_PK>(sa[2 * q], al[2 * q], pk2(f.x, f.y), uhp[i], ulp[i]);
              ofs_step<LZ_PK>(sa[2 * q + 1], al[2 * q + 1], pk2(f.z, f.w), uhp[i], ulp[i]);
            }
          }
        }
      };
      // start of a batch's row work: its exchanged sums are complete, and every
      // warp of the team is past the batch before: its slot is refilled
      auto team_barrier = [&]() {
        if constexpr (WPR > 1) {
          named_sync(bar_team, WPR * 32);
          if (freed) refill();
          freed = true;
        }
      };
      auto batch_done = [&]() {
        if constexpr (WPR == 1) {
          __syncwarp();
          refill();
        } else {
          xp ^= 1u;
        }
      };
      // one batch by itself (fewer than R rows)
      auto lone_batch = [&](int b) {
        const std::false_type F{};
        const int i0 = batch_row(pass, b), nr = min(R, nrows - i0);
        const unsigned char* st = next_stage();
        RV vh, vl, uh, ul;
        float corr;
        dfloat s;
        front(F, st, nr, vh, vl, corr);
        middle(vh, vl, corr, s);
        team_barrier();
        back(F, st, i0, nr, s, corr, uh, ul);
        offset(uh);
        columns(F, st, nr, uh, ul);
        batch_done();
      };
      // batches [b0, b1) of the pass, R rows each, as a pipeline
      auto full_batches = [&](int b0, int b1) {
        const std::true_type T{};
        const unsigned char* st = next_stage();
        RV vh, vl;
        float corr;
        dfloat s;
        front(T, st, R, vh, vl, corr);
        middle(vh, vl, corr, s);
        for (int b = b0; b < b1 - 1; ++b) {
          RV uh, ul;
          float corr2;
          team_barrier();
          const unsigned char* st2 = next_stage();
          front(T, st2, R, vh, vl, corr2);
          back(T, st, batch_row(pass, b), R, s, corr, uh, ul);
          offset(uh);
          if constexpr (WPR > 1) xp ^= 1u;
          middle(vh, vl, corr2, s);
          columns(T, st, R, uh, ul);
          if constexpr (WPR == 1) batch_done();
          st = st2;
          corr = corr2;
        }
        RV uh, ul;
        team_barrier();
        back(T, st, batch_row(pass, b1 - 1), R, s, corr, uh, ul);
        offset(uh);
        columns(T, st, R, uh, ul);
        batch_done();
      };
      // the strip's last batch may hold fewer than R rows; it is the first of
      // the passes that run backwards
      const bool ragged = nb > 0 && batch_row(0, nb - 1) + R > nrows;
      const int b0 = (ragged && (pass & 1)) ? 1 : 0, b1 = (ragged && !(pass & 1)) ? nb - 1 : nb;
      if (b0 > 0) lone_batch(0);
      if (b0 < b1) full_batches(b0, b1);
      if (b1 < nb) lone_batch(nb - 1);
      if (Ca != 0.f) flush();
      // partials for step j+1 (read after its barrier 1): Phi^T z', c, |z'|^2
      pass_end(ah, al, cacc, j + 1, nacc, gstep + 1u);
      if (pass + 1 <= r - 1) issue_pass_head(pass + 1);
    }
    // the loop always ends in a break (the break test, or the last step) with
    // gstep at that step; the slice phase of that step cleared the group sums
    // of the next parity, where the next problem's prologue starts
    ++gstep;
    // a break leaves the head of the next pass issued: wait for it to land and
    // count it as consumed
    if (sbreak && !s_err && reff < r - 1)
      for (int b = 0; b < min(nb, (int)ring.S); ++b) next_stage();
    if (rank == 0 && tid == 0) {
      bt.r_eff[p] = reff;
      for (int k = reff; k < r; ++k) alpha_out[k] = 0.0;
      for (int k = (reff > 0 ? reff - 1 : 0); k < r; ++k) beta_out[k] = 0.0;
    }
    // problems on the same group run back to back; keep them apart
    if (!group_sync_named(bar, lgen, status, &sflag, &s_err, BAR_ALL, NCT)) {
      drain();
      return;
    }
  }
  drain();
}

template <int NV, int WPR, int KT, bool FULLD, typename PT>
int launch_lanczos_t(const LanczosBatch& bt, void* scratch, size_t gstride, int groups, int g,
                     int stages, int* status, size_t smem, cudaStream_t stream) {
  auto fn = lanczos_kernel<NV, WPR, KT, FULLD, PT>;
  SLS_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  char* sc = (char*)scratch;
  void* args[] = {(void*)&bt, (void*)&sc, (void*)&gstride, (void*)&g,
                  (void*)&groups, (void*)&stages, (void*)&status};
  SLS_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)fn, dim3(groups * g), dim3(LZ_NT), args,
                                           smem, stream));
  count_launch(1);
  return SLS_OK;
}

// One (NV, WPR) and element type: KT = 1, 2 or 4 basis tiles when the rows fill
// the lanes, KT = 2 or 4 for ragged widths.  A ragged width in its own kernel:
// both forms in one took registers from the full one (windows of 2048 rows at
// D = 1024 4500 us against 4270).
template <int NV, int WPR, typename PT>
int launch_lanczos_kt(const LanczosBatch& bt, void* scratch, size_t gstride, int groups, int g,
                      int stages, int* status, size_t smem, cudaStream_t stream) {
#define SLS_LZ_KT(KT, FULLD)                                                                  \
  launch_lanczos_t<NV, WPR, KT, FULLD, PT>(bt, scratch, gstride, groups, g, stages, status, smem, \
                                           stream)
  if (bt.D == 128 * NV * WPR)
    return bt.r <= 32 ? SLS_LZ_KT(1, true) : bt.r <= 64 ? SLS_LZ_KT(2, true) : SLS_LZ_KT(4, true);
  return bt.r <= 64 ? SLS_LZ_KT(2, false) : SLS_LZ_KT(4, false);
#undef SLS_LZ_KT
}

}  // namespace

// Launch the Lanczos kernel for one (NV, WPR) of lz_shape, Phi in float32
// (lanczos_f32_<NV>_<WPR>.cu) or bfloat16 (lanczos_bf16_<NV>_<WPR>.cu).
#define SLS_LZ_LAUNCH_ARGS                                                                 \
  const LanczosBatch &bt, void *scratch, size_t gstride, int groups, int g, int stages,    \
      int *status, size_t smem, cudaStream_t stream
#define SLS_LZ_PASS_ARGS bt, scratch, gstride, groups, g, stages, status, smem, stream
int launch_lanczos_f32_2_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_2_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_3_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_3_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_4_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_4_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_6_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_6_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_8_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_8_1(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_6_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_6_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_8_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_8_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_8_4(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_8_4(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_8_8(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_8_8(SLS_LZ_LAUNCH_ARGS);

}  // namespace sls
