// Problem table shared by the SimHash, segment and aggregation kernels and
// by the compress driver.  A "problem" is one token set that is compressed
// independently: the compressible region of a prompt (global backend) or one
// window (adaptive backend).
#pragma once

#include <cstdint>

namespace sls {

struct ProbDesc {
  int64_t tok_row;   // first token row (b * N + pos0); also its Phi/Q/U row base
  int64_t q1off;     // offset of its Lanczos start vector in q1
  int64_t out0;      // first output macro row (b * M + ...)
  int64_t phi_row;   // first row in Phi / Q / U (spectral problems)
  int pos0;          // position of its first token inside the prompt
  int n;             // tokens
  int m;             // macro-tokens to produce (exact budget)
  int bits;          // SimHash bits
  int spectral;      // 1 = Spectral-LSH, 0 = chunk
  int chunk_k;       // chunk backend group size k (0 = m array_split groups)
  int spec_idx;      // index in the compacted spectral list (or -1)
  int out_local;     // first output macro index inside its prompt
};

// Which kernel segments the problems of a launch.
enum class SegRoute {
  warp,     // a warp per problem of at most 32 tokens
  cluster,  // one problem on a thread-block cluster of SEG_CL CTAs
  grid,     // one problem on a cooperative grid
  cta       // a CTA per problem
};

// A cluster of 16 CTAs of 1024 threads is more than every device must place (the
// portable size is 8): cluster_fits says whether this one does.  Its hardware
// barrier costs 0.2 us, the grid's 2.5 us, and the computation holds about thirty
// (N = 8180: 82 -> 50 us, N = 32756: 132 -> 70); below 4096 tokens a CTA by itself,
// its sort in shared memory, is faster (N = 1500: 124 us against 148), above 81920
// the grid's SMs are worth their barriers.  Calls on Zipf-distributed codes, us, cluster
// / grid, 16 bits and rho = 16, 16 and 4, 8 and 8: N = 65536 155 / 191, 363 / 361, 223 /
// 249; 81920 181 / 202, 430 / 409, 247 / 262; 98304 204 / 213, 530 / 481, 283 / 282;
// 131060 458 / 378, 623 / 544, 342 / 317; 262144 633 / 467, 1029 / 862, 581 / 480.
// Without the cluster the grid starts where it beats one CTA.
constexpr int SEG_CL = 16;
constexpr int64_t SEG_CLUSTER_MIN_N = 4096, SEG_CLUSTER_MAX_N = 81920, SEG_GRID_MIN_N = 8192;

inline SegRoute segment_route(int nprob, int64_t nmax, bool has_status, bool cluster_fits) {
  if (nmax <= 32) return SegRoute::warp;
  if (nprob == 1 && has_status) {
    if (cluster_fits && nmax >= SEG_CLUSTER_MIN_N && nmax <= SEG_CLUSTER_MAX_N)
      return SegRoute::cluster;
    if (nmax >= SEG_GRID_MIN_N) return SegRoute::grid;
  }
  return SegRoute::cta;
}

}  // namespace sls
