// Prints what the exact scan's dispatch rules answer, one line per input line
// "dtype nA nB d T alignA alignB": "cert chain" (1: the form is taken).  Host code only.
#include <cstdio>

#include "../../paper_2307_03043_gb300/csrc/common.cuh"

int main() {
  int dtype, d, aA, aB;
  long long nA, nB, T;
  while (std::scanf("%d %lld %lld %d %lld %d %d", &dtype, &nA, &nB, &d, &T, &aA, &aB) == 7) {
    ch_set A, B;
    A.dtype = B.dtype = dtype;
    A.d = B.d = d;
    A.n = nA;
    B.n = nB;
    A.data = reinterpret_cast<void*>(size_t(4096) + aA);
    B.data = reinterpret_cast<void*>(size_t(8192) + aB);
    std::printf("%d %d\n", int(chx::exact_tc_supported(&A, &B, T)), int(chx::exact_chain_pays(&A, &B, T)));
  }
  return 0;
}
