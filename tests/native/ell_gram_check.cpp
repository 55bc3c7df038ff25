// Host-side check of the launch rule of the sparse FP32 product with its Gram
// sums (kernels.cuh): for slice counts and SM counts given in pairs on the
// command line, prints the blocks and the most slices a warp of them meets.
#include <stdio.h>
#include <stdlib.h>

#include "kernels.cuh"

int main(int argc, char** argv) {
  for (int i = 1; i + 1 < argc; i += 2) {
    const long long nslices = atoll(argv[i]);
    const int blocks = mpcg::ell_gram_blocks(nslices, atoi(argv[i + 1]));
    const long long warps = (long long)blocks * (mpcg::kBlock / 32);
    printf("%d %lld\n", blocks, (nslices + warps - 1) / warps);
  }
  return 0;
}
