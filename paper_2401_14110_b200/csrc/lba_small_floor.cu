#define LBA_RNE 0
#include "lba_small.inc"
