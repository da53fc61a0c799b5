// attend_split.cu compiled for IEEE-half tensors; see attend_f16.cu.
#define SENTRY_ATT_F16 1
#define attend_split_ws_bytes attend_split_f16_ws_bytes
#define launch_attend_split launch_attend_split_f16
#include "attend_split.cu"
