// csrc/roots.h on the host: per input line "x seed" (hexadecimal floats) the
// reciprocal square root and the square root of x.
#include <cstdio>

#include "roots.h"

int main() {
  double x, y;
  while (std::scanf("%la %la", &x, &y) == 2)
    std::printf("%a %a\n", etdm::root_rsqrt(x, y), etdm::root_sqrt(x, y));
}
