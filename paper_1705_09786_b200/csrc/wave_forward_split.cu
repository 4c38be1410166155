// The scheduled engine's kernel for evaluation whose cells multiply 32-bit operands on the tensor cores (tc_split.cuh).
#define WAVE_FORWARD
#define WAVE_SPLIT
#include "wave_engine.cu"
