// Host logic of the CUDA-core products, without a GPU: which kernel and split a size
// takes on 152 SMs.  Arguments: fp64 (0/1), then M N K batch of each size.
#include <cstdio>
#include <cstdlib>

#include "gemm_simt.cu"

int main(int argc, char** argv) {
  for (int i = 2; i + 3 < argc; i += 4) {
    dmrgc::GemmArgs g;
    g.M = std::atoi(argv[i]);
    g.N = std::atoi(argv[i + 1]);
    g.K = std::atoi(argv[i + 2]);
    std::printf("%d\n", dmrgc::small_split(g, std::atoi(argv[i + 3]), std::atoi(argv[1]) != 0, 152));
  }
  return 0;
}
