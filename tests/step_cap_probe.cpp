// Test driver (CPU): pdds::below_cap for the triples "n more kmax" on stdin.
#include <cstdio>

#include "pdds_internal.h"

int main() {
  int n, more, kmax;
  while (std::scanf("%d %d %d", &n, &more, &kmax) == 3)
    std::printf("%d\n", pdds::below_cap(n, more, kmax) ? 1 : 0);
}
