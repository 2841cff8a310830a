// csrc/route.cuh without CUDA: the blocks that placements of more than 32 instances get beside smaller ones.
#include "../paper_2509_06362_b200/csrc/route.cuh"

extern "C" uint32_t big_share(uint64_t big, uint64_t small, uint32_t warps, uint32_t grid) { return maaso::walk_big_share(big, small, warps, grid); }
