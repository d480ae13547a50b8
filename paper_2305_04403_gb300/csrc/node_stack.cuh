// node_stack.cuh -- the step of a line's traversal from one wide node to the
// next.  Compiles as plain C++ for the host tests.
#pragma once

#include <cstdint>
#if defined(__CUDACC__)
#include <cuda_runtime.h>
#define WOB_STACK_FN __device__ __forceinline__
#else
#define WOB_STACK_FN inline
#endif

namespace wob {

// base, mask: first interior child of the node just tested and those of them
// that the line meets (base is a leaf's reference, below zero, in a node that has
// no interior child, and counts only with a mask).  Takes the next node -- the
// first of these, or of the entry popped when there is none -- and pushes the
// siblings that are left; false: the traversal is complete.  The stack is the
// calling lane's own, entry i at stack[i * stride]: lanes that follow one line
// together each keep a copy, since within a turn nothing orders one lane's push
// against another's pop.
WOB_STACK_FN bool next_node(volatile int* stack, int stride, int levels, int base, uint32_t mask,
                            int& sp, int& node, int& err)
{
    if (!mask && sp > 0) {
        const uint32_t e = (uint32_t)stack[--sp * stride];
        base = (int)(e & 0xFFFFFFu);
        mask = e >> 24;
    }
    if (!mask) return false;
#if defined(__CUDA_ARCH__)
    node = base + __ffs(mask) - 1;
#else
    node = base + __builtin_ctz(mask);
#endif
    mask &= mask - 1;
    if (mask) {
        if (sp < levels) {
            stack[sp * stride] = base | (int)(mask << 24);
            ++sp;
        } else {
            err |= 1;
        }
    }
    return true;
}

}  // namespace wob
