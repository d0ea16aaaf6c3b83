// The lean H kernels for rows that are no multiple of four (kern_lean.cu), compiled beside the others.
#define CSEM_LEAN_UNIT 1
#include "kern_lean.cu"
