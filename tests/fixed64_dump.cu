// Host evaluation of the FP64 form's fixed-point trial direction: reads pairs
// of words from standard input, prints the three components as integers.
#include <cstdio>

#include "fixed64.cuh"

int main() {
  static constexpr mpk::SineTable table = mpk::make_sine_table();
  unsigned r0, r1;
  while (std::scanf("%u %u", &r0, &r1) == 2) {
    const mpk::Fix3 t = mpk::fix_trial(r0, r1, mpk::fix_root(r0), table.s);
    std::printf("%lld %lld %lld\n", static_cast<long long>(t.x), static_cast<long long>(t.y),
                static_cast<long long>(t.z));
  }
  return 0;
}
