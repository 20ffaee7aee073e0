// Prints pic::maxwell_planes, the planes per z chunk of the fused Yee update, of a launch of one
// grid: arguments ndim n0 n1 n2 fp64, any number of such groups of five.
#include <cstdio>
#include <cstdlib>

#include "../../paper_0909_5603_gb300/csrc/pic_internal.h"

int main(int argc, char **argv)
{
    for (int i = 1; i + 4 < argc; i += 5) {
        const int n[1][3] = {{atoi(argv[i + 1]), atoi(argv[i + 2]), atoi(argv[i + 3])}};
        printf("%d\n", pic::maxwell_planes(n, 1, atoi(argv[i]), atoi(argv[i + 4])));
    }
    return 0;
}
