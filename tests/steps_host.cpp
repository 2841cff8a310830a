// csrc/steps.cuh without CUDA.
#include "../paper_2509_06362_b200/csrc/steps.cuh"

using namespace maaso;

extern "C" uint32_t exact_steps(int64_t dt, uint32_t s) {
    const ExactEntry e = walk_exact_entry(s);
    return e.step >> 5 == s ? walk_exact_steps((int32_t)dt, s, e.step, e.m) : 0xFFFFFFFFu;
}
extern "C" uint32_t corrected_steps(int64_t dt, uint32_t s) { return walk_steps((int32_t)dt, s, walk_rcp(s)); }
extern "C" uint32_t corrected_steps64(int64_t dt, uint32_t s) { return walk_steps(dt, s, walk_rcp(s)); }
