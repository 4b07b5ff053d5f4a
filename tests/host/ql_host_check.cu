// Host check of the QL rotation (test infrastructure): reads pairs f g of hexadecimal
// doubles from stdin, writes r s c of ql_rotation (ql.cuh) for each.
#include <cstdio>

#include "../../paper_2203_09732_gb300/csrc/ql.cuh"

int main() {
  double f, g, r, s, c;
  while (std::scanf("%la %la", &f, &g) == 2) {
    hs::ql_rotation(f, g, r, s, c);
    std::printf("%a %a %a\n", r, s, c);
  }
  return 0;
}
