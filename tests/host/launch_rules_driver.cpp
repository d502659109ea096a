// Test driver for the launch rules (launch_rules.h): one query per line of
// stdin, the answer on stdout.
//   gram n3 m -> row chunks of the overlap products
//   zchunk n M cols halo fill -> planes per z-chunk of a stage launch
//   split pairs cap -> CTAs per (projector, orbital block) of a gather
#include <cstdio>
#include <cstring>
#include "launch_rules.h"

int main() {
  char what[32];
  while (std::scanf("%31s", what) == 1) {
    if (!std::strcmp(what, "gram")) {
      int n3, m;
      if (std::scanf("%d %d", &n3, &m) != 2) return 2;
      std::printf("%d\n", emd_gram_chunks(n3, m));
    } else if (!std::strcmp(what, "zchunk")) {
      int n, M, cols, fill;
      double halo;
      if (std::scanf("%d %d %d %lf %d", &n, &M, &cols, &halo, &fill) != 5) return 2;
      std::printf("%d\n", emd_zchunk(n, M, cols, halo, fill));
    } else if (!std::strcmp(what, "split")) {
      int pairs, cap;
      if (std::scanf("%d %d", &pairs, &cap) != 2) return 2;
      std::printf("%d\n", emd_gather_split(pairs, cap));
    } else {
      return 2;
    }
  }
  return 0;
}
