// Part 1 of win_raw.cu: resize, bicubic.
#define WIN_RAW_PART 1
#include "win_raw.cu"
