// The strip kernel's FP16 instances (a translation unit of their own: the
// formats compile in parallel).
#include "strip.cuh"

namespace tts {
namespace strip {
KernelFn kernel_fp16(int nt, int ncol) { return kernel_of<kFmtFP16>(nt, ncol); }
BatchFn batched_fp16(int nt) { return batched_of<kFmtFP16>(nt); }
}  // namespace strip
}  // namespace tts
