// parts_cuts K bytes...: the cuts of the pieces into K parts (csrc/parts.h).
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "parts.h"

int main(int argc, char** argv) {
  const int K = std::atoi(argv[1]), P = argc - 2;
  std::vector<uint32_t> off(1, 0u), cut(K + 1);
  for (int p = 0; p < P; ++p) off.push_back(off.back() + (uint32_t)std::atoll(argv[2 + p]));
  gocp::tiled_cuts(off.data(), P, K, cut.data());
  for (uint32_t c : cut) std::printf("%u ", c);
  std::printf("\n");
  return 0;
}
