// Host build of the selection's cuts (paper_2312_02756_gb300/csrc/select_cuts.cuh) against the comparisons
// they stand for; built with undefined behaviour trapped.  Prints the number of cases.
#include <stdio.h>

#include "../paper_2312_02756_gb300/csrc/select_cuts.cuh"

int main() {
  const double v[] = {0.0,   -0.0,   5e-324, -5e-324, 1e-310, -1e-310, 1.0,      -1.0,      2.5,
                      -2.5,  20.0,   -20.0,  1e308,   -1e308, 1.7e308, -1.7e308, INFINITY,  -INFINITY,
                      NAN,   -NAN,   2.2250738585072014e-308, -2.2250738585072014e-308, 19.999999999999996};
  const int n = sizeof v / sizeof *v;
  long cases = 0;
  for (int a = 0; a < n; a++)
    for (int b = 0; b < n; b++) {
      const gvx::Cuts c = gvx::make_cuts(v[a], v[b]);
      for (int i = 0; i < n; i++)
        for (int j = 0; j < n; j++, cases++)
          if (gvx::passes(v[i], v[j], c) != (v[i] >= v[a] && fabs(v[j]) <= v[b])) {
            printf("pt_min %g eta_max %g pt %g eta %g\n", v[a], v[b], v[i], v[j]);
            return 1;
          }
    }
  printf("%ld\n", cases);
  return 0;
}
