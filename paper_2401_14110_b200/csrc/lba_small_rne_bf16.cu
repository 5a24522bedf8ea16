#define LBA_RNE 2
#include "lba_small.inc"
