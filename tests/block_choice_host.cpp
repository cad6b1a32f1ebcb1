// The autotuner's choice among its candidates (csrc/lbm_internal.h), compiled
// for the host.  Arguments: the times of the candidates (0: not tried).
// Prints the choice and the fastest of the fixed sizes.
#include <cstdio>
#include <cstdlib>

#include "../include/lbm.h"
#include "../paper_2101_01702_gb300/csrc/lbm_internal.h"

int main(int argc, char **argv)
{
    float ms[LBMK_NBLOCKS] = {0.f};
    for (int j = 0; j + 1 < argc && j < LBMK_NBLOCKS; ++j) ms[j] = (float)atof(argv[j + 1]);
    int fixed = -1;
    const int bs = lbmk_choose_block(ms, &fixed);
    printf("%d %d\n", bs, fixed);
    return 0;
}
