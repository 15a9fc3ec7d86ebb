// FP64 instances of the stage kernel (see k_stage.cu)
#define STAGE_FP64
#include "k_stage.cu"
