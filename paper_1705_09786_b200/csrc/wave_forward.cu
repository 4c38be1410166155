// The scheduled engine's kernel for evaluation: forward cells and loss heads alone, without the branches of training, so that its products
// can use registers that the training kernel's accumulators need.
#define WAVE_FORWARD
#include "wave_engine.cu"
