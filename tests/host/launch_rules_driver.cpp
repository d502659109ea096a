// Test driver for the launch rules (launch_rules.h): one query per line of
// stdin, the answer on stdout.
//   gram n3 m -> row chunks of the overlap products
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
    } else {
      return 2;
    }
  }
  return 0;
}
