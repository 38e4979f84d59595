// The library's launch rules as a host program (no GPU): each argument is one
// query, answered by one line.
//   priority,P,G       priority of a batch's second branch for a stream of priority P (greatest G)
#include <stdio.h>

#include "lbmp_internal.h"

int main(int argc, char** argv)
{
    for (int k = 1; k < argc; ++k) {
        int a, b;
        if (sscanf(argv[k], "priority,%d,%d", &a, &b) == 2)
            printf("%d\n", lbmp::branch_priority(a, b));
        else
            return 1;
    }
    return 0;
}
