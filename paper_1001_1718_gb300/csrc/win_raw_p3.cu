// Part 3 of win_raw.cu: the fused pre-process, bicubic.
#define WIN_RAW_PART 3
#include "win_raw.cu"
