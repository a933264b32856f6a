// The real-operator on-chip kernels in FP64.
#define OCR_KERNELS
#include "onchip_real.cuh"

int ocr_fwd_f64(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st) { return ocr_dl<double>(o, bt, dt, st); }
int ocr_dens_f64(const OcrPlan* o, const OcdArgs& g, const OcdJob& j, cudaStream_t st) { return dens_dl<double>(o, g, j, st); }
