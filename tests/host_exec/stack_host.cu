// Host execution of the node stacks' step rule (stack_take of gwn_internal.h), test harness.
#include <vector>

#include "../../paper_2605_19200_gb300/csrc/gwn_internal.h"

using namespace gwn;

// Walks a tree whose nodes are all near, as a warp or block with a stack of `cap` entries does that
// takes `width` nodes a step.  The tree: a spine of `spine` nodes, each with a balanced subtree of
// `depth` levels as one child (the first if `first`), ending in such a subtree.  Returns the leaves
// reached, or -1 where the stack is full.
extern "C" long long hx_stack_walk(int spine, int depth, int first, int width, int cap) {
    std::vector<int> stk(cap), taken(width);
    long long leaves = 0;
    int sp = 0;
    stk[sp++] = -1 - spine;  // below 0: -1 - (spine nodes left); else levels of a balanced subtree
    while (sp > 0) {
        const int take = stack_take(sp, width, cap);
        if (take <= 0) return -1;
        for (int j = 0; j < take; ++j) taken[j] = stk[sp - 1 - j];
        sp -= take;
        for (int j = 0; j < take; ++j) {
            const int v = taken[j];
            int a, b;  // first and second child
            if (v == 0) {
                ++leaves;
                continue;
            }
            if (v > 0) {
                a = b = v - 1;
            } else if (v == -1) {
                a = b = depth;
            } else {
                a = first ? depth : v + 1;
                b = first ? v + 1 : depth;
            }
            if (sp + 2 > cap) return -1;
            stk[sp++] = b;
            stk[sp++] = a;
        }
    }
    return leaves;
}
