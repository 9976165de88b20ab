// The single-precision network path: the tensor-core kernel of mlp_f32.cu and the SIMT kernel
// that evaluates again the samples it marks (operands beyond the range of its FP16 parts).
#pragma once
#include "common.cuh"

namespace tsdfs {

// head of the path's scratch (the rest holds the split weights): word 0 is set when a sample is marked by
// the network kernel, word 1 when samples are marked for a ray of almost no weight
constexpr size_t kRedoBytes = 256;
// word of that head from which on a word per layer tells that its weights are below the parts' range
constexpr int kLowWord = 8;
// result of a marked sample of a value pass
constexpr uint32_t kRedoBits = 0x7fc5a5a5u;

size_t mlp_f32_stash_bytes(int arch);
int launch_mlp_full_f32(const tsdfs_mlp* m, const SampleSource& src, SampleRec* rec, int64_t max_samples,
                        Scratch stash, cudaStream_t st);
int launch_mlp_value_f32(const tsdfs_mlp* m, const SampleSource& src, float* f_out, Scratch stash, cudaStream_t st);

// redo: NULL (every sample) or the word above (the marked samples only; none when it is 0)
template <int ARCH>
int launch_mlp_full_simt(const NetParams& np, const SampleSource& src, SampleRec* rec, int64_t max_samples,
                         const uint32_t* redo, cudaStream_t st);
template <int ARCH>
int launch_mlp_value_simt(const NetParams& np, const SampleSource& src, float* f_out, const uint32_t* redo,
                          cudaStream_t st);

}  // namespace tsdfs
