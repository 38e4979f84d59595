// The library's launch rules as a host program (no GPU): each argument is one
// query, answered by one line.
//   priority,P,G       priority of a batch's second branch for a stream of priority P (greatest G)
//   ahead,T,N,C        FP32 D3Q27 step over T tiles of N planes with LBMP_OPT_CHUNK = C: planes per
//                      item, and whether the kernel that loads f' one plane ahead is chosen
#include <stdio.h>
#include <string.h>

#include "lbmp_internal.h"

int main(int argc, char** argv)
{
    for (int k = 1; k < argc; ++k) {
        int a, b, c;
        if (sscanf(argv[k], "priority,%d,%d", &a, &b) == 2)
            printf("%d\n", lbmp::branch_priority(a, b));
        else if (sscanf(argv[k], "ahead,%d,%d,%d", &a, &b, &c) == 3) {
            lbmp_handle h;
            memset(&h, 0, sizeof h);
            h.opt_chunk = c;
            const int per_sm[2] = {4, 3};  // what the two kernels are built for
            bool ahead;
            const lbmp::LaunchShape L = lbmp::launch_shape_ahead(&h, a, b, per_sm, 152, ahead);
            printf("%d %d\n", L.chunk, ahead ? 1 : 0);
        } else
            return 1;
    }
    return 0;
}
