// decode_pattern.cu for Strassen's algorithm as it is: 7 products, 2 x 2 cells.
#define FMM_LEVELS 1
#include "decode_pattern.cu"
