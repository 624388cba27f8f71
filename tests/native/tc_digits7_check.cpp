// Host driver for the seven-digit arithmetic of the tensor-core row stages above degree 39 (tc_digits.cuh). One request
// per line on stdin, one answer per line on stdout; floating-point values travel as hexadecimal (%a):
//   D yh yl        -> the seven digits d0..d6 of digits_n<7>(yh, yl)   (FP32 operands)
//   H x e          -> the seven digits d0..d6 of digits_host_n(x, e, 7) (FP64 operand)
//   C a6 .. a0     -> hi lo of combine_n<7>                             (FP32 operands)
#include <cstdio>
#include <cstdlib>

#include "tc_digits.cuh"

int main() {
  char op[4];
  char s[7][64];
  while (std::scanf("%3s", op) == 1) {
    if (op[0] == 'D') {
      if (std::scanf("%63s %63s", s[0], s[1]) != 2) return 1;
      float d[shbim::tc::kDig7];
      shbim::tc::digits_n<shbim::tc::kDig7>(std::strtof(s[0], nullptr), std::strtof(s[1], nullptr), d);
      for (int j = 0; j < 7; ++j) std::printf("%d ", (int)d[j]);
      std::printf("\n");
    } else if (op[0] == 'H') {
      int e = 0, d[shbim::tc::kDig7];
      if (std::scanf("%63s %d", s[0], &e) != 2) return 1;
      shbim::tc::digits_host_n(std::strtod(s[0], nullptr), e, shbim::tc::kDig7, d);
      for (int j = 0; j < 7; ++j) std::printf("%d ", d[j]);
      std::printf("\n");
    } else if (op[0] == 'C') {
      float a[shbim::tc::kDig7];
      for (int j = 6; j >= 0; --j) {
        if (std::scanf("%63s", s[0]) != 1) return 1;
        a[j] = std::strtof(s[0], nullptr);
      }
      const dfl::df r = shbim::tc::combine_n<shbim::tc::kDig7>(a);
      std::printf("%a %a\n", (double)r.hi, (double)r.lo);
    } else {
      return 1;
    }
  }
  return 0;
}
