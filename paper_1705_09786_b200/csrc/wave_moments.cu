// The scheduled engine's kernel for training with momentum or Adam.  Plain SGD has one without their code: the accumulators hold forty sums
// in registers, and every call beside them costs spills.
#define WAVE_MOMENTS
#include "wave_engine.cu"
