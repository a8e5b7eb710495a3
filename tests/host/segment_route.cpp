// segment_route for lines of "nprob nmax has_status cluster_fits" on stdin.
#include <cstdio>

#include "../../paper_2607_19368_gb300/csrc/segment.cuh"

int main() {
  int nprob, status, fits;
  long long nmax;
  while (std::scanf("%d %lld %d %d", &nprob, &nmax, &status, &fits) == 4)
    std::printf("%d\n", (int)sls::segment_route(nprob, nmax, status != 0, fits != 0));
  return 0;
}
