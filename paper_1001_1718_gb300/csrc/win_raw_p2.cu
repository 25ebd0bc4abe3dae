// Part 2 of win_raw.cu: the fused pre-process, bilinear.
#define WIN_RAW_PART 2
#include "win_raw.cu"
