#define LBA_RNE 1
#include "lba_small.inc"
