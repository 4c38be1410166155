// The scheduled engine's kernel for training whose cells multiply 32-bit operands on the tensor cores (tc_split.cuh).  The kernel without them
// keeps its registers for the others: with their code in it the small models lose 1-3 %.
#define WAVE_SPLIT
#include "wave_engine.cu"
