// Checks that touching output pages (paper_1608_04472_gb300/csrc/bc_pages.h)
// leaves every byte as it was, over array sizes around the thresholds and at
// unaligned addresses. Exit status 1 if a byte changed.
#include "../paper_1608_04472_gb300/csrc/bc_pages.h"

#include <cstdio>
#include <vector>

int main() {
  const size_t MB = (size_t)1 << 20;
  long bad = 0;
  for (size_t first : {MB, 4 * MB, 5 * MB + 3, 70 * MB + 1})
    for (size_t second : {(size_t)0, (size_t)1, 4 * MB - 4097}) {
      std::vector<unsigned char> a(first + 1), b(second + 1);
      for (size_t i = 0; i < a.size(); ++i) a[i] = (unsigned char)(i * 7 + 13);
      for (size_t i = 0; i < b.size(); ++i) b[i] = (unsigned char)(i * 5 + 1);
      {
        bcg::PageTouch pages;
        pages.add(a.data() + 1, first);
        pages.add(nullptr, 99);
        pages.add(b.data(), second);
        pages.start();
      }
      for (size_t i = 0; i < a.size(); ++i) bad += a[i] != (unsigned char)(i * 7 + 13);
      for (size_t i = 0; i < b.size(); ++i) bad += b[i] != (unsigned char)(i * 5 + 1);
    }
  std::printf("changed %ld\n", bad);
  return bad != 0;
}
