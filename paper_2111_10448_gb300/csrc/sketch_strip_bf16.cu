// The strip kernel's BF16 instances (a translation unit of their own: the
// formats compile in parallel).
#include "strip.cuh"

namespace tts {
namespace strip {
KernelFn kernel_bf16(int nt, int ncol) { return kernel_of<kFmtBF16>(nt, ncol); }
BatchFn batched_bf16(int nt) { return batched_of<kFmtBF16>(nt); }
}  // namespace strip
}  // namespace tts
