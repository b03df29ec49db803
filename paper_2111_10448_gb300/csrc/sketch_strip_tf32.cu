// The strip kernel's TF32 instances (a translation unit of their own: the
// formats compile in parallel).
#include "strip.cuh"

namespace tts {
namespace strip {
KernelFn kernel_tf32(int nt, int ncol) { return kernel_of<kFmtTF32>(nt, ncol); }
BatchFn batched_tf32(int nt) { return batched_of<kFmtTF32>(nt); }
}  // namespace strip
}  // namespace tts
