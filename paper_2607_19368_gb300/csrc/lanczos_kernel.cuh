// Implicit Lanczos (Algorithm 2): the persistent kernel.
//
// Lanczos runs as one persistent cooperative kernel.  The grid is split into
// groups of CTAs; a group owns one problem at a time (one prompt, or one
// adaptive window) and every CTA owns a contiguous strip of the problem's rows
// of the feature matrix Phi (N x D, float32 or bfloat16) and of the basis Q.
// The eight warps of a CTA form teams of WPR warps (WPR = 1 up to D = 512, 2 up
// to 1024, 4 up to 2048, then 8): a team takes whole rows of the strip, R at a time, and
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
//   exchange 1    every CTA publishes its partials of Phi^T z', c and |z'|^2;
//                 the owner of a coefficient or column adds the CTAs' partials.
//   exchange 2    the owners publish c and |z'|^2; column owners subtract
//                 sum_k c_k w_k: Phi^T z1 with z1 = z' - Q c and w_k =
//                 Phi^T q_k kept from earlier steps.
//   exchange 3    the owners publish Phi^T z1; every CTA forms
//                 beta_{j-1} = |z1| = sqrt(|z'|^2 - |c|^2), the break test,
//                 w_j = Phi^T q_j = Phi^T z1 / beta and alpha_j = |w_j|^2.
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
// L2.  Vectors are double-float (two float32), every sum over N or D is
// compensated, and the sums over the CTAs are double-float in a fixed order;
// |z1|^2 = |z'|^2 - |c|^2, beta, its reciprocal, alpha and the break test are
// float64.  Waits poll without sleeping and give up after about a second of
// clock cycles, reporting SLS_ERR_TIMEOUT through the status word.
//
// The exchanges.  The CTAs of a group hold no barrier: a value is published as
// one 64-bit store into a slot that holds the all-ones pattern until then (a
// NaN the arithmetic cannot produce), and a reader polls the value itself, so
// an exchange costs one store and one load through L2.  Readers put the
// pattern back: the partials' slots (two buffers, by exchange parity) by the
// one CTA that reads them, as it reads them; the totals' slots (three buffers)
// by their owner, one exchange later, when the partials of every CTA show that
// all have read them.  A slot is written again only after its writer has seen
// a later value from the CTA that put the pattern back, with one GPU-scope
// fence per thread and step (before a pass's partials are published) between
// the two on either side.
//
// A one-way trip through L2 takes 525 cycles within a die and 850 across (ping-
// pong of two CTAs).  Two barriers of the group with the sums in between
// (float64 atomics for the scalars, each phase behind its own round trips) took
// 22000 cycles per step at N = 8180, D = 1024 on 152 CTAs, more than the pass
// over Phi; the exchanges take 16000.  What is left is mostly their own
// instructions: they run once per step, cold after the row loop.  A slot block
// is contiguous per owner: polling partials spread by source (a sector per
// value) saturated L2 and was slower than the barriers.
//
// Why whole rows per team: a row's scalars (q_j, z', its products with the
// basis) are a serial chain of double-float operations.  When all eight warps
// shared every row, that chain stood between two barriers of the whole CTA for
// every eight rows, and each warp ran it for one row on 32 identical lanes.
// Here 32 / R lanes share a row's chain, R rows at a time, and the teams run
// independently (with WPR = 1 a pass holds no barrier at all), so one team's
// chain is hidden behind the sweeps of the others, and inside a warp behind the
// row dots of the next R rows.  Measured against the CTA-wide form with two
// group barriers per step (whole sls_lanczos_topr calls, both built and timed
// alternately): 64 windows of 2048 rows at D = 1024, r = 32 5.92 -> 3.93 ms;
// N = 32756, D = 2048, r = 64 4.58 -> 3.90 ms; N = 8180, D = 1024, r = 32 0.750 ->
// 0.596 ms; 64 windows of 1024 rows at D = 256, r = 16 2.99 -> 1.22 ms; N = 488,
// D = 256, r = 16 0.308 -> 0.231 ms.
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

// Who owns what in the exchanges of a group of g CTAs: CTA i the columns
// [i cw, (i + 1) cw) and, counted from the last CTA, the coefficients
// [i' kw, (i' + 1) kw) of the r + 1 (c_0 .. c_{r-1}, |z'|^2), i' = g - 1 - i.
// WB: slots of a block (one CTA's partials for one owner): kw coefficients,
// then cw columns.  The form of the owner's sums (mode):
//   0  blocks of at most 16 slots (large groups), padded to a power of two: the
//      threads split over (source, slot pair), then a warp per sum
//   1  at most 256 slots, padded likewise: the same, then a thread per sum
//   2  wider (a few CTAs): a thread per column pair adds the sources
struct LzOwn {
  int cw, kw, WB, mode;
};

__host__ __device__ inline LzOwn lz_own(int D, int r, int g) {
  LzOwn o;
  o.cw = (D + g - 1) / g;
  o.kw = (r + 1 + g - 1) / g;
  o.WB = 2;
  while (o.WB < o.cw + o.kw) o.WB *= 2;
  o.mode = o.WB <= 16 ? 0 : o.WB <= 256 ? 1 : 2;
  if (o.mode == 2) {
    o.cw = (o.cw + 1) & ~1;
    o.kw = (o.kw + 1) & ~1;
    o.WB = o.cw + o.kw;
  }
  return o;
}

// Rows of WB sums that the warps leave in shared memory (modes 0 and 1): one
// per warp, or per set of warps that spans the WB / 2 slot pairs.
__host__ __device__ inline int lz_red_rows(LzOwn o) {
  return o.mode == 2 ? 0 : o.WB <= 64 ? LZ_NCW : 2 * LZ_NT / o.WB;
}

// Per-group scratch layout (byte offsets), identical on host and device.
//   bar:  word 0: all ones, 0 once a CTA of the group has given up
//   part: 2 x g owners x g sources x WB values: the sources' partials of
//         c, |z'|^2 and the columns of Phi^T z', double-float
//   tot:  3 x E values: Phi^T z1 (D), c (r) and |z'|^2, double-float
//   Wm:   r x D double-float: w_k = Phi^T q_k (each CTA its columns; by column
//         in mode 0, else by k)
// [bar, ones_end) is set to all ones before the launch.
struct LzLayout {
  size_t bar, part, tot, ones_end, Wm, total;
};

__host__ __device__ inline size_t lz_al(size_t x) { return (x + 255) & ~(size_t)255; }
__host__ __device__ inline int lz_exch_len(int D, int r) { return (D + r + 2) & ~1; }

__host__ __device__ inline LzLayout lz_layout(int D, int r, int g) {
  LzLayout L;
  const size_t E = (size_t)lz_exch_len(D, r);
  size_t o = 0;
  L.bar = o;    o += 256;
  L.part = o;   o += lz_al(2 * (size_t)g * g * lz_own(D, r, g).WB * 8);
  L.tot = o;    o += lz_al(3 * E * 8);
  L.ones_end = o;
  L.Wm = o;     o += lz_al((size_t)D * r * sizeof(float2));
  L.total = o;
  return L;
}

// ---- exchange slots ---------------------------------------------------------

constexpr unsigned long long LZ_EMPTY = ~0ull;

SLS_DEV unsigned long long x_ld(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
SLS_DEV void x_ld2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
SLS_DEV void x_st(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
SLS_DEV void x_st2(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
// A double-float as a slot's value, never the empty pattern.
SLS_DEV unsigned long long x_pack(dfloat v) {
  const unsigned long long u =
      ((unsigned long long)__float_as_uint(v.lo) << 32) | (unsigned long long)__float_as_uint(v.hi);
  return u == LZ_EMPTY ? 0x7fffffff7fffffffull : u;
}
SLS_DEV dfloat x_unpack(unsigned long long u) {
  return df_make(__uint_as_float((unsigned)u), __uint_as_float((unsigned)(u >> 32)));
}

SLS_DEV dfloat shfl_xor_df(dfloat v, int m) {
  v.hi = __shfl_xor_sync(0xffffffffu, v.hi, m);
  v.lo = __shfl_xor_sync(0xffffffffu, v.lo, m);
  return v;
}

// The split of a row over a team: NV float4 column groups per lane, WPR warps
// (NV * 32 * 4 * WPR >= D), R rows at a time.  A lane keeps w_j, the column sums
// and their offset sums (10 float32 per column pair and group) in registers:
// at NV = 4 with R = 4 the row loop runs without spills.  Measured at D = 1024 /
// 2048 (N = 8180 / 32756; 64 windows of 2048 rows): NV = 8 with half the warps
// and R = 2, whose 160 registers of state spill, 690 / 3937 / 4300 us; NV = 4
// 630 / 3825 / 3863; NV = 2 with twice the warps and R = 8 668 / 4217 / 4283.
// The narrowest split that holds the row is taken: lanes past the row's end
// would do their share of the arithmetic on nothing.
struct LzShape {
  int nv, wpr, R;
};

__host__ __device__ constexpr int lz_rows(int nv) { return nv >= 8 ? 2 : 4; }

__host__ __device__ inline LzShape lz_shape(int D) {
  LzShape s{8, 8, lz_rows(8)};
  if (D <= 256) s = LzShape{2, 1, lz_rows(2)};
  else if (D <= 384) s = LzShape{3, 1, lz_rows(3)};
  else if (D <= 512) s = LzShape{4, 1, lz_rows(4)};
  else if (D <= 768) s = LzShape{3, 2, lz_rows(3)};
  else if (D <= 1024) s = LzShape{4, 2, lz_rows(4)};
  else if (D <= 1536) s = LzShape{3, 4, lz_rows(3)};
  else if (D <= 2048) s = LzShape{4, 4, lz_rows(4)};
  else if (D <= 4096) s = LzShape{4, 8, lz_rows(4)};
  return s;
}

// Ring stage: R rows of Phi (esz bytes per element: 4 for float32, 2 for
// bfloat16) followed by the same R rows of the basis Q (ldq float2 each).
constexpr int LZ_MAX_STAGES = 8;

__host__ __device__ inline unsigned lz_stage_bytes(int D, int ldq, int esz, int R) {
  return (unsigned)R * ((unsigned)D * (unsigned)esz + (unsigned)ldq * 8u);
}

// w_j passes through shared memory when several teams need each column.
__host__ __device__ constexpr bool lz_stage_w(int wpr) { return wpr <= 2; }

// What the exchanges of a CTA share, at the start of its shared memory: they
// are functions of their own (not inlined), so that the compiler gives the row
// loops of the kernel all registers.
struct LzXch {
  unsigned long long *part, *tot;
  float2* Wm;
  unsigned* poison;
  int* status;
  double *alpha_out, *beta_out;  // of the problem (rank 0)
  LzOwn own;
  int g, rank, D, r, E;
  int cbeg, cend, kbeg, kend;   // this CTA's columns and coefficients
  unsigned cw_magic;            // c / cw = umulhi(c, cw_magic)
  unsigned rings, ring_bytes;   // offsets: the teams' rings (column sums, coefficients),
  unsigned whs, wls, red, cs;   // w_j, sums of a block, c
  double tol, scale;            // of the break test
  double nrm2, inv64, alpha64;  // |z1|^2, 1 / beta and alpha of the step
  float2 invb, beta;            // 1 / beta and beta as double-float
  float2 q2;                    // |Phi^T z1|^2 of the step
  float2 tmpw[LZ_NCW];
  int brk;
  volatile int err;             // a wait of this CTA gave up
};

constexpr unsigned LZ_RING0 = (sizeof(LzXch) + 127) / 128 * 128;  // offset of the first ring

// Shared memory besides the rings (bytes), in the order the kernel carves it:
// the exchanges' state (before the rings); w_j (high parts, low parts), the
// warps' sums of an exchange block (red slots), the row sums the warps of a
// team exchange, c, then the mbarriers.
__host__ __device__ inline size_t lz_smem_other(int D, int r, LzShape s, int red, int stages) {
  const int teams = LZ_NCW / s.wpr;
  size_t b = LZ_RING0;
  b += lz_stage_w(s.wpr) ? 2 * sizeof(float) * (size_t)D : 0;
  b += sizeof(float2) * (size_t)red;
  b += sizeof(float4) * (size_t)(teams * 2 * s.R * s.wpr);
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

// Whether the sweeps add by Dot2 (10 operations per element) instead of against an
// offset (5).  An offset is several times the largest sum it may carry, and the low
// parts round at its scale: over rows of up to 512 columns the plain Dot2 sums leave
// alpha and beta ten times closer to float64 (N = 1000, D = 256, r = 24: 3e-15 of |T|
// against 7e-14; 64 windows of 1024 rows there 1.03 -> 1.21 ms).  From D = 1024 on the
// kernel has always added against offsets (of 512 < D < 1024 a former one lost rows).
__host__ __device__ constexpr bool lz_dot2(int wpr) { return wpr == 1; }

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

// The butterfly of transpose_sum8 on double-floats (any values).
template <int R>
SLS_DEV dfloat transpose_sum8_df(float (&h)[R], float (&l)[R]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int m = 16 >> s;
    const int nv = (R >> s) > 1 ? (R >> s) : 1;
    const bool up = (lane & m) != 0;
#pragma unroll
    for (int i = 0; i < (nv > 1 ? nv / 2 : 1); ++i) {
      const int k = nv > 1 ? i + nv / 2 : i;
      const dfloat send = nv > 1 && !up ? df_make(h[k], l[k]) : df_make(h[i], l[i]);
      const dfloat keep = nv > 1 && up ? df_make(h[k], l[k]) : df_make(h[i], l[i]);
      const dfloat t = df_add_fast(keep, shfl_xor_df(send, m));
      h[i] = t.hi;
      l[i] = t.lo;
    }
  }
  return df_make(h[0], l[0]);
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

// A wait of this CTA gave up: report it; the CTA leaves at its next barrier that
// reads the flag.
SLS_DEV void lz_fail(int* status, volatile int* err) {
  atomicExch(status, SLS_ERR_TIMEOUT);
  *err = 1;
}

SLS_DEV int nprob_of(const LanczosBatch& bt) {
  int nprob = bt.nprob_max;
  if (bt.nprob_dev) nprob = min(nprob, *bt.nprob_dev);
  return nprob;
}

// Polls of exchange slots by a warp, bounded: `more` is called by every lane
// for each repetition and returns false once this CTA or another of the group
// has given up.
struct XWait {
  unsigned* poison;   // word of the group: all ones until a CTA gives up
  int* status;
  volatile int* err;  // this CTA's flag
  long long t0;
  unsigned it;

  __device__ __noinline__ bool more() {
    bool bad = false;
    if ((++it & 31u) == 0u) {
      if (it == 32u) t0 = clock64();
      if (*err) {
        bad = true;
      } else if (ld_relaxed_gpu(poison) != ~0u) {
        *err = 1;
        bad = true;
      } else if (clock64() - t0 > SLS_WAIT_CYCLES) {
        lz_fail(status, err);
        atomicExch(poison, 0u);
        bad = true;
      }
    }
    return !__any_sync(0xffffffffu, bad);
  }
};

// One slot per lane (where `need`), polled until full.
SLS_DEV unsigned long long x_poll(const unsigned long long* p, bool need, XWait& w) {
  unsigned long long v = need ? x_ld(p) : 0ull;
  w.it = 0u;
  while (__any_sync(0xffffffffu, v == LZ_EMPTY) && w.more())
    if (v == LZ_EMPTY) v = x_ld(p);
  return v;
}

// B pairs of slots p + u * step (those with need bit u) per lane; wa, wb: which
// slots of a pair are ever written.
template <int B>
SLS_DEV void x_poll2(const unsigned long long* p, size_t step, unsigned need, bool wa, bool wb,
                     unsigned long long (&a)[B], unsigned long long (&b)[B], XWait& w) {
#pragma unroll
  for (int u = 0; u < B; ++u) {
    a[u] = b[u] = 0ull;
    if (need >> u & 1u) x_ld2(p + u * step, a[u], b[u]);
  }
  w.it = 0u;
  for (;;) {
    bool miss = false;
#pragma unroll
    for (int u = 0; u < B; ++u) miss |= (wa && a[u] == LZ_EMPTY) || (wb && b[u] == LZ_EMPTY);
    if (!__any_sync(0xffffffffu, miss) || !w.more()) break;
#pragma unroll
    for (int u = 0; u < B; ++u)
      if ((need >> u & 1u) && ((wa && a[u] == LZ_EMPTY) || (wb && b[u] == LZ_EMPTY)))
        x_ld2(p + u * step, a[u], b[u]);
  }
}

SLS_DEV bool named_sync_any(unsigned id, unsigned nthreads, bool pred) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n"
      " bar.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((unsigned)pred), "r"(id), "r"(nthreads)
      : "memory");
  return r != 0;
}

// The kernel's dynamic shared memory.  Functions that are not inlined address
// it from here by offsets: a pointer handed to them would lose its address
// space.
SLS_DEV unsigned char* lz_smem() {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  return smem_raw;
}

SLS_DEV LzXch& lz_xch() { return *reinterpret_cast<LzXch*>(lz_smem()); }

// After a pass: the column sums and coefficient partials (k < K) the teams left
// in their rings are added and published as exchange xpar; false when a wait of
// this CTA has given up (nothing is published then).
template <int TEAMS>
__device__ __noinline__ bool lz_publish(int K, unsigned xpar) {
  constexpr int NCT = LZ_NT;
  LzXch& X = lz_xch();
  const int tid = threadIdx.x;
  if (named_sync_any(BAR_ALL, NCT, X.err != 0)) {
    if (tid == 0) atomicExch(X.poison, 0u);
    return false;
  }
  const LzOwn own = X.own;
  const int g = X.g, rank = X.rank, D = X.D, r = X.r;
  unsigned long long* part = X.part;
  const unsigned cw_magic = X.cw_magic;
  auto tcol = [&](int t) {
    return reinterpret_cast<float2*>(lz_smem() + X.rings + (size_t)t * X.ring_bytes);
  };
  auto tco = [&](int t) { return tcol(t) + D; };
  // slot i of this CTA's block for owner d
  auto slot = [&](unsigned d, unsigned i) {
    return part + (((size_t)xpar * g + d) * g + rank) * own.WB + i;
  };
  // coefficient e (|z'|^2 at r): the TEAMS partials summed by two lanes
#pragma unroll 1
  for (int e0 = 0; e0 <= r; e0 += NCT / 2) {
    const int e = e0 + tid / 2, h = tid & 1;
    dfloat s = df_make(0.f, 0.f);
    if (e < K || e == r)
      for (int t = h; t < TEAMS; t += 2) s = df_add(s, dfv(tco(t)[e]));
    s = df_add_fast(s, shfl_xor_df(s, 1));
    if (h == 0 && e <= r) x_st(slot(g - 1 - e / own.kw, e % own.kw), x_pack(s));
  }
#pragma unroll 1
  for (int c = 2 * tid; c < D; c += 2 * NCT) {
    float4 v[TEAMS];
#pragma unroll
    for (int t = 0; t < TEAMS; ++t) v[t] = reinterpret_cast<const float4*>(tcol(t) + c)[0];
#pragma unroll
    for (int w = 1; w < TEAMS; w *= 2)
#pragma unroll
      for (int t = 0; t + w < TEAMS; t += 2 * w) {
        const dfloat a = df_add_fast(df_make(v[t].x, v[t].y), df_make(v[t + w].x, v[t + w].y));
        const dfloat b = df_add_fast(df_make(v[t].z, v[t].w), df_make(v[t + w].z, v[t + w].w));
        v[t] = make_float4(a.hi, a.lo, b.hi, b.lo);
      }
    const unsigned long long v0 = x_pack(df_make(v[0].x, v[0].y));
    const unsigned long long v1 = x_pack(df_make(v[0].z, v[0].w));
    const unsigned d0 = own.cw == 1 ? (unsigned)c : __umulhi((unsigned)c, cw_magic);
    const unsigned i0 = (unsigned)c - d0 * own.cw;
    if (own.mode == 2) {  // cw and kw are even: the pair has one owner
      x_st2(slot(d0, own.kw + i0), v0, v1);
    } else {
      x_st(slot(d0, own.kw + i0), v0);
      if (i0 + 1 < (unsigned)own.cw) x_st(slot(d0, own.kw + i0 + 1), v1);
      else x_st(slot(d0 + 1, own.kw), v1);
    }
  }
  named_sync(BAR_ALL, NCT);  // the rings are free
  return true;
}

// c (into shared memory) and beta_{j-1} = |z1|, by one warp: |z1|^2 = |z'|^2 -
// |c|^2 (Q orthonormal; |c|^2 is below the rounding of |z'|^2 until a
// breakdown, so its sum over the lanes is plain).  The difference, beta and its
// reciprocal are float64: q_j is scaled by that reciprocal, and a double-float
// reciprocal square root, off by up to 2^-46, left that error in every alpha and
// beta (N = 1000, D = 256: alpha off by 7e-15 of |T| instead of 2e-15).
SLS_DEV void lz_beta(LzXch& X, const unsigned long long* now, XWait& xw) {
  const int lane = threadIdx.x & 31;
  const int D = X.D, r = X.r;
  float2* cs = reinterpret_cast<float2*>(lz_smem() + X.cs);
  dfloat cn = df_make(0.f, 0.f);
  unsigned long long n0 = x_ld(now + D + r);
#pragma unroll 1
  for (int k0 = 0; k0 < r; k0 += 32) {  // (0 from k = j on)
    const int k = k0 + lane;
    const dfloat c = x_unpack(x_poll(now + D + k, k < r, xw));
    if (k < r) cs[k] = f2(c);
    dot2_acc_df(cn.hi, cn.lo, c, c);
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    cn.hi += __shfl_xor_sync(0xffffffffu, cn.hi, o);
    cn.lo += __shfl_xor_sync(0xffffffffu, cn.lo, o);
  }
  if (__any_sync(0xffffffffu, n0 == LZ_EMPTY)) n0 = x_poll(now + D + r, true, xw);
  if (lane == 0) {
    const double nrm2 = df_to_double(x_unpack(n0)) - df_to_double(cn);  // |z1|^2
    const double inv = nrm2 > 0.0 ? rsqrt(nrm2) : 0.0;
    X.nrm2 = nrm2;
    X.inv64 = inv;
    X.invb = f2(df_from_double(inv));
  }
}

// alpha_j = |Phi^T z1|^2 / beta^2, by the lane that formed 1 / beta.
SLS_DEV void lz_alpha(LzXch& X, int j) {
  X.alpha64 = df_to_double(dfv(X.q2)) * X.inv64 * X.inv64;
  if (X.rank == 0) X.alpha_out[j] = X.alpha64;
}

// beta_{j-1} and the break test of step j, by one lane of the warp that formed
// 1 / beta, while the columns of exchange 3 travel.
SLS_DEV void lz_break_test(LzXch& X, int j) {
  if ((threadIdx.x & 31) == 0) {
    const double bnew = X.nrm2 > 0.0 ? X.nrm2 * X.inv64 : 0.0;
    bool brk = !(bnew > 0.0);
    if (j > 0) {
      X.scale = fmax(X.scale, fabs(X.alpha64) + bnew);  // (alpha of step j - 1)
      brk = !(bnew > X.tol * X.scale);
    }
    X.brk = brk;
    X.beta = f2(df_from_double(bnew));
    if (X.rank == 0 && j > 0 && !brk) X.beta_out[j - 1] = bnew;
  }
}

// Exchanges 1 and 2 of step j: this CTA's coefficients and columns of
// Phi^T z1 are published, c and beta_{j-1} formed.
__device__ __noinline__ void lz_exchange12(int j, unsigned xpar, unsigned x3) {
  constexpr int NCW = LZ_NCW, NCT = LZ_NT;
  LzXch& X = lz_xch();
  const LzOwn own = X.own;
  const int g = X.g, D = X.D, r = X.r;
  const int cbeg = X.cbeg, ncol = X.cend - X.cbeg, kbeg = X.kbeg, ncoef = X.kend - X.kbeg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int red_rows = lz_red_rows(own);
  float2* red = reinterpret_cast<float2*>(lz_smem() + X.red);
  const float2* cs = reinterpret_cast<const float2*>(lz_smem() + X.cs);
  const float2* Wm = X.Wm;
  XWait xw{X.poison, X.status, &X.err, 0ll, 0u};
  if (tid == (NCW - 1) * 32 && j > 0) lz_alpha(X, j - 1);
  unsigned long long* src = X.part + ((size_t)xpar * g + X.rank) * g * own.WB;  // my block
  unsigned long long* now = X.tot + (size_t)x3 * X.E;
  unsigned long long* old = X.tot + (size_t)(x3 == 0u ? 2u : x3 - 1u) * X.E;
  // the g partials of this CTA's coefficients and columns; the columns less
  // sum_{k < j} c_k w_k.  Slots are emptied as they are read.
  if (own.mode < 2) {
    // thread t: the slot pair t % P of the sources t / P, t / P + NCT / P, ...;
    // the lanes and then (through red) the warps that share a pair are added
    const int P = own.WB >> 1, SP = NCT / P;
    const int pr = tid & (P - 1), s0 = tid / P, i0 = 2 * pr;
    const bool wa = i0 < own.kw ? i0 < ncoef : i0 - own.kw < ncol;
    const bool wb = i0 + 1 < own.kw ? i0 + 1 < ncoef : i0 + 1 - own.kw < ncol;
    dfloat a = df_make(0.f, 0.f), b = a;
    constexpr int B = 5;
#pragma unroll 1
    for (int b0 = 0; b0 < g; b0 += B * SP) {
      unsigned need = 0u;
#pragma unroll
      for (int u = 0; u < B; ++u)
        if (b0 + s0 + u * SP < g) need |= 1u << u;
      unsigned long long va[B], vb[B];
      unsigned long long* p0 = src + (size_t)(b0 + s0) * own.WB + i0;
      const size_t step = (size_t)SP * own.WB;
      x_poll2<B>(p0, step, need, wa, wb, va, vb, xw);
#pragma unroll
      for (int u = 0; u < B; ++u)
        if (need >> u & 1u) {
          x_st2(p0 + u * step, LZ_EMPTY, LZ_EMPTY);
          if (wa) a = df_add_fast(a, x_unpack(va[u]));
          if (wb) b = df_add_fast(b, x_unpack(vb[u]));
        }
    }
#pragma unroll 1
    for (int o = P; o < 32; o <<= 1) {
      a = df_add_fast(a, shfl_xor_df(a, o));
      b = df_add_fast(b, shfl_xor_df(b, o));
    }
    if (lane < P) {
      float2* rp = red + (P <= 32 ? warp : warp / (P / 32)) * own.WB + i0;
      rp[0] = f2(a);
      rp[1] = f2(b);
    }
    named_sync(BAR_ALL, NCT);
  }
  if (own.mode == 0) {
    // sum i of the block by warp i % NCW: coefficients first
#pragma unroll 1
    for (int i = warp; i < own.kw + ncol; i += NCW) {
      dfloat v = (lane < red_rows) ? dfv(red[lane * own.WB + i]) : df_make(0.f, 0.f);
      size_t at;
      if (i < own.kw) {
        if (i >= ncoef) continue;
        at = D + kbeg + i;
      } else {
        at = cbeg + i - own.kw;
        float ch = 0.f, cl = 0.f;
#pragma unroll 1
        for (int k0 = 0; k0 < j; k0 += 32) {
          const int k = k0 + lane;
          const float2 w = k < j ? Wm[at * r + k] : make_float2(0.f, 0.f);
          dot2_acc_df(ch, cl, dfv(w), x_unpack(x_poll(now + D + k, k < j, xw)));
        }
        v = df_sub(v, df_norm(ch, cl));
      }
#pragma unroll 1
      for (int o = 16; o > 0; o >>= 1) v = df_add_fast(v, shfl_xor_df(v, o));
      if (lane == 0) {
        x_st(now + at, x_pack(v));
        x_st(old + at, LZ_EMPTY);
      }
    }
    if (warp == NCW - 1) lz_beta(X, now, xw);
  } else {
    dfloat a = df_make(0.f, 0.f), b = a;
    if (own.mode == 1) {
      // a thread per sum
      if (tid < own.WB)
#pragma unroll 1
        for (int w = 0; w < red_rows; ++w) a = df_add(a, dfv(red[w * own.WB + tid]));
      if (tid < ncoef) {
        x_st(now + D + kbeg + tid, x_pack(a));
        x_st(old + D + kbeg + tid, LZ_EMPTY);
      }
    } else if (warp == NCW - 1) {
      // coefficients by the last warp
#pragma unroll 1
      for (int i = lane; i - lane < ncoef; i += 32) {
        dfloat v = df_make(0.f, 0.f);
#pragma unroll 1
        for (int sI = 0; sI < g; ++sI) {
          unsigned long long* p0 = src + (size_t)sI * own.WB + i;
          v = df_add(v, x_unpack(x_poll(p0, i < ncoef, xw)));
          if (i < ncoef) x_st(p0, LZ_EMPTY);
        }
        if (i < ncoef) {
          x_st(now + D + kbeg + i, x_pack(v));
          x_st(old + D + kbeg + i, LZ_EMPTY);
        }
      }
    }
    if (warp == NCW - 1) lz_beta(X, now, xw);
    named_sync(BAR_ALL, NCT);  // c is in shared memory
    if (own.mode == 1) {
      const int q = tid - own.kw;
      if (q >= 0 && q < ncol) {
        float ch = 0.f, cl = 0.f;
#pragma unroll 8
        for (int k = 0; k < j; ++k)
          dot2_acc_df(ch, cl, dfv(Wm[(size_t)k * D + cbeg + q]), dfv(cs[k]));
        a = df_sub(a, df_norm(ch, cl));
        x_st(now + cbeg + q, x_pack(a));
        x_st(old + cbeg + q, LZ_EMPTY);
      }
    } else {
#pragma unroll 1
      for (int q0 = 0; q0 < ncol; q0 += 2 * NCT) {
        const int q = q0 + 2 * tid;  // this thread's columns cbeg + q, cbeg + q + 1
        const bool live = q < ncol;
        a = b = df_make(0.f, 0.f);
#pragma unroll 1
        for (int b0 = 0; b0 < g; b0 += 4) {
          unsigned need = 0u;
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (live && b0 + u < g) need |= 1u << u;
          unsigned long long va[4], vb[4];
          unsigned long long* p0 = src + (size_t)b0 * own.WB + own.kw + q;
          x_poll2<4>(p0, (size_t)own.WB, need, true, true, va, vb, xw);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (need >> u & 1u) {
              x_st2(p0 + (size_t)u * own.WB, LZ_EMPTY, LZ_EMPTY);
              a = df_add(a, x_unpack(va[u]));
              b = df_add(b, x_unpack(vb[u]));
            }
        }
        if (live) {
          float ch = 0.f, cl = 0.f, dh = 0.f, dl = 0.f;
          const float4* wrow = reinterpret_cast<const float4*>(Wm + cbeg + q);
#pragma unroll 8
          for (int k = 0; k < j; ++k) {
            const float4 w = wrow[(size_t)k * (D >> 1)];
            const dfloat c = dfv(cs[k]);
            dot2_acc_df(ch, cl, df_make(w.x, w.y), c);
            dot2_acc_df(dh, dl, df_make(w.z, w.w), c);
          }
          a = df_sub(a, df_norm(ch, cl));
          b = df_sub(b, df_norm(dh, dl));
          x_st2(now + cbeg + q, x_pack(a), x_pack(b));
          x_st2(old + cbeg + q, LZ_EMPTY, LZ_EMPTY);
        }
      }
    }
  }
}

// Exchange 3 of step j: Phi^T z1 of every CTA; w_j = Phi^T z1 / beta (into shared
// memory when STAGE_W; this CTA's columns kept for the correction of later
// steps) and alpha_j = |w_j|^2 = |Phi^T z1|^2 / beta^2, returned packed; LZ_EMPTY when a wait of this CTA
// has given up.
template <bool STAGE_W>
__device__ __noinline__ unsigned long long lz_exchange3(int j, unsigned x3) {
  constexpr int NCW = LZ_NCW, NCT = LZ_NT;
  LzXch& X = lz_xch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (named_sync_any(BAR_ALL, NCT, X.err != 0)) {
    if (tid == 0) atomicExch(X.poison, 0u);
    return LZ_EMPTY;
  }
  if (warp == NCW - 1) lz_break_test(X, j);
  const int D = X.D, cbeg = X.cbeg, cend = X.cend;
  const dfloat invb = dfv(X.invb);
  const unsigned long long* now = X.tot + (size_t)x3 * X.E;
  float2* whs = reinterpret_cast<float2*>(lz_smem() + X.whs);
  float2* wls = reinterpret_cast<float2*>(lz_smem() + X.wls);
  XWait xw{X.poison, X.status, &X.err, 0ll, 0u};
  dfloat sq = df_make(0.f, 0.f);
  constexpr int B = 4;
#pragma unroll 1
  for (int p0 = 0; p0 < (D >> 1); p0 += B * NCT) {
    unsigned need = 0u;
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (p0 + tid + u * NCT < (D >> 1)) need |= 1u << u;
    unsigned long long va[B], vb[B];
    x_poll2<B>(now + 2 * (p0 + tid), 2 * NCT, need, true, true, va, vb, xw);
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (need >> u & 1u) {
        const int c = 2 * (p0 + tid + u * NCT);
        const dfloat z0 = x_unpack(va[u]), z1 = x_unpack(vb[u]);
        const dfloat w0 = df_mul(z0, invb), w1 = df_mul(z1, invb);
        dot2_acc_df(sq.hi, sq.lo, z0, z0);
        dot2_acc_df(sq.hi, sq.lo, z1, z1);
        if (STAGE_W) {
          whs[c >> 1] = make_float2(w0.hi, w1.hi);
          wls[c >> 1] = make_float2(w0.lo, w1.lo);
        }
        if (c + 1 >= cbeg && c < cend) {
          const bool by_col = X.own.mode == 0;
          if (c >= cbeg) X.Wm[by_col ? (size_t)c * X.r + j : (size_t)j * D + c] = f2(w0);
          if (c + 1 < cend) X.Wm[by_col ? (size_t)(c + 1) * X.r + j : (size_t)j * D + c + 1] = f2(w1);
        }
      }
  }
  sq = df_norm(sq.hi, sq.lo);
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) sq = df_add_fast(sq, shfl_xor_df(sq, o));
  if (lane == 0) X.tmpw[warp] = f2(sq);
  if (named_sync_any(BAR_ALL, NCT, X.err != 0)) {
    if (tid == 0) atomicExch(X.poison, 0u);
    return LZ_EMPTY;
  }
  dfloat a = (lane < NCW) ? dfv(X.tmpw[lane]) : df_make(0.f, 0.f);
#pragma unroll 1
  for (int o = 1; o < NCW; o <<= 1) a = df_add_fast(a, shfl_xor_df(a, o));
  a.hi = __shfl_sync(0xffffffffu, a.hi, 0);
  a.lo = __shfl_sync(0xffffffffu, a.lo, 0);
  // alpha_j: double-float for the recurrence (whose z' is orthogonalised against q_j
  // again), float64 as the result and for the break test, formed while the partials
  // of the next step travel
  if (tid == (NCW - 1) * 32) X.q2 = f2(a);
  return x_pack(df_mul(df_mul(a, invb), invb));
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

// The sweeps run on packed float32 pairs, one instruction per operation of two
// columns: scalar steps take twice the issue slots of the same arithmetic (lanczos
// 32k 4434 -> 4054 us, windows of 2048 rows 4693 -> 4270 us, 8k 771 -> 733 us).

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
  constexpr bool DOT2 = lz_dot2(WPR);
  using RV = RowVals<R>;
  // basis coefficients per lane: k = sub + LPR * (t * WPR + tw), t < KC
  constexpr int KC = (KT * 32 + LPR * WPR - 1) / (LPR * WPR);
  unsigned char* smem_raw = lz_smem();
  LzXch& X = lz_xch();
  volatile int& s_err = X.err;
  __shared__ float s_red1[NCW];  // per-warp max |Phi| (offset bounds)

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
  TeamRing ring{smem_raw + LZ_RING0 + (size_t)team * ring_stages * stage, nullptr,
                (unsigned)ring_stages, RingPos{0u, 0u}, RingPos{0u, 0u}};
  float* whs = reinterpret_cast<float*>(smem_raw + LZ_RING0 + (size_t)TEAMS * ring_stages * stage);
  float* wls = whs + D;
  const LzOwn own = lz_own(D, r, g);
  float2* red = reinterpret_cast<float2*>(lz_stage_w(WPR) ? wls + D : whs);
  float4* exch = reinterpret_cast<float4*>(red + lz_red_rows(own) * (own.mode < 2 ? own.WB : 0));
  float2* cs = reinterpret_cast<float2*>(exch + TEAMS * 2 * R * WPR);  // r + 1 (c = Q^T z')
  uint64_t* fullb = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(cs + (r + 1)) + 15) & ~(uintptr_t)15);
  ring.full = fullb + team * ring_stages;
  exch += team * 2 * R * WPR;
  // scratch of the pass ends, in the team's ring (idle then): its column sums,
  // its coefficient partials (k < r) and, at r, its part of |z'|^2
  const size_t tstride = (size_t)ring_stages * stage;
  auto tcol = [&](int t) {
    return reinterpret_cast<float2*>(smem_raw + LZ_RING0 + (size_t)t * tstride);
  };
  auto tco = [&](int t) { return tcol(t) + D; };
  const uint64_t pol = l2_policy_evict_first();

  if (tid == 0) {
    for (int s = 0; s < TEAMS * ring_stages; ++s) mbar_init(&fullb[s], 1);
    mbar_fence_init();
    const LzLayout L = lz_layout(D, r, g);
    char* gb = scratch + (size_t)gi * gstride;
    auto offset = [&](const void* p) {
      return (unsigned)(reinterpret_cast<const unsigned char*>(p) - smem_raw);
    };
    X.part = reinterpret_cast<unsigned long long*>(gb + L.part);
    X.tot = reinterpret_cast<unsigned long long*>(gb + L.tot);
    X.Wm = reinterpret_cast<float2*>(gb + L.Wm);
    X.poison = reinterpret_cast<unsigned*>(gb + L.bar);
    X.status = status;
    X.own = own;
    X.g = g;
    X.rank = rank;
    X.D = D;
    X.r = r;
    X.E = lz_exch_len(D, r);
    X.cbeg = min(D, rank * own.cw);
    X.cend = min(D, X.cbeg + own.cw);
    X.kbeg = min(r + 1, (g - 1 - rank) * own.kw);
    X.kend = min(r + 1, X.kbeg + own.kw);
    X.cw_magic = 0xffffffffu / (unsigned)own.cw + 1u;
    X.rings = LZ_RING0;
    X.ring_bytes = (unsigned)tstride;
    X.whs = offset(whs);
    X.wls = offset(wls);
    X.red = offset(red);
    X.cs = offset(cs);
    X.tol = bt.tol;
    X.err = 0;
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
  // exchanges run by this group so far: the partials' buffer (parity) and the
  // totals' buffer (modulo 3) of the current one
  unsigned xpar = 0u, x3 = 0u;
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
    if (tid == 0) {  // read after the barriers of the prologue's end
      X.alpha_out = alpha_out;
      X.beta_out = beta_out;
      X.scale = 0.0;
    }
    dfloat alpha_df = df_make(0.f, 0.f), beta_df = df_make(0.f, 0.f), invb_df;
    float phimax = 0.f;  // max |Phi| over this CTA's strip (prologue pass)
    int reff = 0;

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
    // the batches [b0, min(b1, stages)) of a pass's head
    auto issue_pass_head = [&](int pass, int b0, int b1) {
      if (leader)
        for (int b = b0; b < min(b1, (int)ring.S); ++b) issue(pass, b);
    };

    // The end of a pass: the team's column sums and coefficient partials (k < K)
    // into its ring.
    auto team_sums = [&](f32x2_t (&ah)[NC / 2], f32x2_t (&al)[NC / 2], dfloat (&cacc)[KC], int K,
                         dfloat nacc) {
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
      // one, the ring writes above are ordered before its bulk writes (async
      // proxy), and the slots emptied in the exchange before this pass before
      // what is published after it
      asm volatile("fence.proxy.async;" ::: "memory");
      __threadfence();
    };

    issue_pass_head(0, 0, (int)ring.S);

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
      team_sums(ah, al, cacc0, 0, nacc);
      if (bt.inject_fail && rank == 0 && tid == 0) lz_fail(status, &s_err);
      // |q1|^2 is the sum of the first step
      if (!lz_publish<TEAMS>(0, xpar)) {
        drain();
        return;
      }
      if (r >= 2) issue_pass_head(1, 0, 1);
    }

    for (int j = 0; j < r; ++j) {
      lz_exchange12(j, xpar, x3);
      // the rest of the next pass's first batches, while the columns travel
      if (j + 1 <= r - 1) issue_pass_head(j + 1, 1, (int)ring.S);
      const unsigned long long alpha = lz_exchange3<lz_stage_w(WPR)>(j, x3);
      if (alpha == LZ_EMPTY) {
        drain();
        return;
      }
      const unsigned long long* now = X.tot + (size_t)x3 * X.E;
      xpar ^= 1u;
      x3 = x3 == 2u ? 0u : x3 + 1u;
      if (X.brk) {
        reff = j;
        break;
      }
      invb_df = dfv(X.invb);
      alpha_df = x_unpack(alpha);
      beta_df = j > 0 ? dfv(X.beta) : df_make(0.f, 0.f);
      if (j == 0) {
#pragma unroll
        for (int w = 0; w < NCW; ++w) phimax = fmaxf(phimax, s_red1[w]);
      }

      if (j == r - 1) {
        // the last step needs no pass over Phi: q_{r-1} = z1 / beta_{r-2}
        if (tid == (NCW - 1) * 32) lz_alpha(X, j);
        last_row_phase(Qs, ldq, nrows, j, cs, invb_df);
        reff = r;
        break;
      }

      // this lane's columns of w_j
      f32x2_t wh[NC / 2], wl[NC / 2];
      float wt1 = 0.f;  // l1 norm of this lane's part of w_j
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        const int cg = lane + 32 * (q * WPR + tw);
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
        if (FULLD || cg < C4) {
          if constexpr (lz_stage_w(WPR)) {
            h = reinterpret_cast<const float4*>(whs)[cg];
            l = reinterpret_cast<const float4*>(wls)[cg];
          } else {
            unsigned long long v[4];
            x_ld2(now + 4 * cg, v[0], v[1]);
            x_ld2(now + 4 * cg + 2, v[2], v[3]);
            const dfloat w0 = df_mul(x_unpack(v[0]), invb_df), w1 = df_mul(x_unpack(v[1]), invb_df);
            const dfloat w2 = df_mul(x_unpack(v[2]), invb_df), w3 = df_mul(x_unpack(v[3]), invb_df);
            h = make_float4(w0.hi, w1.hi, w2.hi, w3.hi);
            l = make_float4(w0.lo, w1.lo, w2.lo, w3.lo);
          }
        }
        wh[2 * q] = pk2(h.x, h.y);
        wh[2 * q + 1] = pk2(h.z, h.w);
        wl[2 * q] = pk2(l.x, l.y);
        wl[2 * q + 1] = pk2(l.z, l.w);
        wt1 += (fabsf(h.x) + fabsf(h.y)) + (fabsf(h.z) + fabsf(h.w));
      }
      // Offset of the row dots: a power of two above eight times the largest
      // part a lane can hold, so that the sums of eight lanes' parts are exact
      // multiples of its last place below it (see the row dots)
      float wtm = wt1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) wtm = fmaxf(wtm, __shfl_xor_sync(0xffffffffu, wtm, o));
      const float Ct = DOT2 ? 0.f : ofs_pow2(4.f * (phimax * wtm));

      // ---------------- fused pass j+1 over Phi ----------------------------------
      // The team's batches run as a pipeline inside each warp: while a batch's
      // row work (a serial chain of double-float operations on few lanes'
      // worth of data) is under way, the row dots of the next batch fill the
      // issue slots, and the butterfly of those dots runs beside the column
      // sums of the batch before.
      const int pass = j + 1;
      f32x2_t ah[NC / 2], al[NC / 2], sa[NC / 2];  // (sa, Ca, room: not with DOT2)
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
      // rounding errors travel in the low parts.  (DOT2: both are double-float
      // sums.)  And this warp's part of the re-orthogonalisation (Q c)_i of the
      // lane's row.
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
              if constexpr (DOT2) {
                dot2_acc2(s0, l0, pk2(f.x, f.y), wh[2 * q], wl[2 * q]);
                dot2_acc2(s0, l0, pk2(f.z, f.w), wh[2 * q + 1], wl[2 * q + 1]);
              } else {
                ofs_fma_acc2(s0, l0, pk2(f.x, f.y), wh[2 * q], wl[2 * q]);
                ofs_fma_acc2(s0, l0, pk2(f.z, f.w), wh[2 * q + 1], wl[2 * q + 1]);
              }
            }
          }
          float sx, sy, lx, ly;
          upk2(s0, sx, sy);
          upk2(l0, lx, ly);
          if constexpr (DOT2) {
            float e;
            two_sum(sx, sy, sx, e);
            const dfloat t = df_norm(sx, e + (lx + ly));
            vh.v[i] = t.hi;
            vl.v[i] = t.lo;
          } else {
            vh.v[i] = (sx - Ct) + (sy - Ct);
            vl.v[i] = lx + ly;
          }
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
        if constexpr (DOT2) {
          s = transpose_sum8_df<R>(vh.v, vl.v);
        } else {
          const float th = transpose_sum8<R>(vh.v);
          const float tl = transpose_sum8<R>(vl.v);
          two_sum(th, tl, s.hi, s.lo);
        }
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
        if constexpr (DOT2) return;
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
              if constexpr (DOT2) {
                dot2_acc2(ah[2 * q], al[2 * q], pk2(f.x, f.y), uhp[i], ulp[i]);
                dot2_acc2(ah[2 * q + 1], al[2 * q + 1], pk2(f.z, f.w), uhp[i], ulp[i]);
              } else {
                ofs_fma_acc2(sa[2 * q], al[2 * q], pk2(f.x, f.y), uhp[i], ulp[i]);
                ofs_fma_acc2(sa[2 * q + 1], al[2 * q + 1], pk2(f.z, f.w), uhp[i], ulp[i]);
              }
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
      // partials for step j+1: Phi^T z', c, |z'|^2
      team_sums(ah, al, cacc, j + 1, nacc);
      if (!lz_publish<TEAMS>(j + 1, xpar)) {
        drain();
        return;
      }
      if (pass + 1 <= r - 1) issue_pass_head(pass + 1, 0, 1);
    }
    // a break leaves the head of the next pass issued: wait for it to land and
    // count it as consumed
    if (reff < r - 1)
      for (int b = 0; b < min(nb, (int)ring.S); ++b) next_stage();
    named_sync(BAR_ALL, NCT);  // every warp is done with the step's shared state
    if (rank == 0 && tid == 0) {
      bt.r_eff[p] = reff;
      for (int k = reff; k < r; ++k) alpha_out[k] = 0.0;
      for (int k = (reff > 0 ? reff - 1 : 0); k < r; ++k) beta_out[k] = 0.0;
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
int launch_lanczos_f32_3_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_3_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_4_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_4_2(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_3_4(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_3_4(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_4_4(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_4_4(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_4_8(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_4_8(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_f32_8_8(SLS_LZ_LAUNCH_ARGS);
int launch_lanczos_bf16_8_8(SLS_LZ_LAUNCH_ARGS);

}  // namespace sls
