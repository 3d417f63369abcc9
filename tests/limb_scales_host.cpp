// Prints the scales that the library chooses for a law's tables (sfm_limbs.h),
// or "refused".  Arguments: crowd r k a gamma, or cells r k0 a0 k1 a1.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "sfm_limbs.h"

int main(int argc, char** argv) {
  if (argc < 6) return 2;
  sfm::ProductScales s;
  const int r = atoi(argv[2]);
  const double a = atof(argv[3]), b = atof(argv[4]), c = atof(argv[5]);
  const bool ok = !strcmp(argv[1], "crowd") ? sfm::crowd_limb_scales(r, a, b, c, &s)
                                            : sfm::cell_limb_scales(r, a, b, c, atof(argv[6]), &s);
  if (ok)
    printf("%.17g %.17g\n", s.s0, s.s1);
  else
    puts("refused");
  return 0;
}
