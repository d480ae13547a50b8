// node_stack.cuh -- the step from one wide node to the next of a line that a
// group of lanes follows together, on one traversal stack for the group.
// Compiles as plain C++ for the host tests.
#pragma once

#include <cstdint>
#if defined(__CUDACC__)
#include <cuda_runtime.h>
#define WOB_STACK_FN __device__ __forceinline__
#else
#define WOB_STACK_FN inline
#endif

namespace wob {

// base, im: first interior child of the node just tested and the mask of those
// the line meets (the same in every lane of the group).  Takes the next node --
// the first of these, or of the entry popped when there is none -- and pushes
// the siblings that are left; false: the traversal is complete.  Every lane
// reads the popped entry and the leader may write the same slot again in the
// same turn, so sync() (a barrier of the group's lanes, ordering memory) stands
// between the two: lanes that have branched apart need not be back together.
// The caller has such a barrier before the next turn, whose lanes read what the
// leader pushed here.
template <class Sync>
WOB_STACK_FN bool next_node(volatile int* stack, int stride, int levels, bool leader, int base,
                            uint32_t im, int& sp, int& node, int& err, Sync sync)
{
    if (!im) {
        if (sp == 0) return false;
        const uint32_t e = (uint32_t)stack[--sp * stride];
        base = (int)(e & 0xFFFFFFu);
        im = e >> 24;
        sync();
    }
#if defined(__CUDA_ARCH__)
    node = base + __ffs(im) - 1;
#else
    node = base + __builtin_ctz(im);
#endif
    im &= im - 1;
    if (im) {
        if (sp < levels) {
            if (leader) stack[sp * stride] = base | (int)(im << 24);
            ++sp;
        } else {
            err |= 1;
        }
    }
    return true;
}

}  // namespace wob
