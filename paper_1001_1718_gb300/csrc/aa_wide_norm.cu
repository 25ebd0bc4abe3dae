// Part 1 of aa_wide.cu: the fused pre-process's kernels.
#define AA_WIDE_PART 1
#include "aa_wide.cu"
