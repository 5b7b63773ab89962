// Host check of csrc/roots.h: the largest error of the roots of the transform tables
// against long double, in units of 1e-19, and of the symmetries that hold exactly.
#include <cmath>
#include <cstdio>
#include <initializer_list>

#include "roots.h"

int main() {
  long double worst = 0;
  long bad = 0;
  for (const int n : {16, 32, 64, 96, 128, 192, 256, 512}) {
    for (int k = 0; k < 2 * n; ++k) {
      double re, im, re2, im2;
      kfbim::unit_root(k, n, &re, &im);
      const long double a = 4 * std::atan(1.0L) * k / n;
      worst = std::fmax(worst, std::fmax(std::fabs(re - std::cos(a)), std::fabs(im + std::sin(a))));
      kfbim::unit_root((2 * n - k) % (2 * n), n, &re2, &im2);   // the conjugate
      bad += re2 != re || im2 != -im;
      kfbim::unit_root((k + n) % (2 * n), n, &re2, &im2);       // minus it
      bad += re2 != -re || im2 != -im;
    }
  }
  std::printf("worst %ld\nbad %ld\n", (long)(worst * 1e19L), bad);
  return 0;
}
