// The real-operator on-chip kernels in FP32 (mixed precision).
#define OCR_KERNELS
#include "onchip_real.cuh"

int ocr_fwd_f32(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st) { return ocr_dl<float>(o, bt, dt, st); }
int ocr_dens_f32(const OcrPlan* o, const OcdArgs& g, const OcdJob& j, cudaStream_t st) { return dens_dl<float>(o, g, j, st); }
