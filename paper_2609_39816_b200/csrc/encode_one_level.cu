// encode_pattern.cu for Strassen's algorithm as it is: 7 products of 2 x 2 cells.
#define FMM_LEVELS 1
#include "encode_pattern.cu"
