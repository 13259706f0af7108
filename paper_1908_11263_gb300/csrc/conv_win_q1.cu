// Window-kernel instantiations for INT-1 layers (e4m3 staging).
#define QNN_WIN_BITS 1
#include "conv_win_inst.cuh"
