// Launchers shared between the encoder's translation units.  Every one queues work on `s` and returns the launch's error.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace xq {

// Per-channel Lloyd (xfp_quant_lloyd.cu).  cosv and rowcnt may be null; where the kernel can, it also writes the cosine
// of every channel against its reconstruction (V2) and the number of extracted weights of every channel.
bool lloyd_fuses_cosine(int cols);
size_t lloyd_scratch_bytes(int rows, int cols);      // global scratch of channels too long for shared memory (0: none)
cudaError_t launch_lloyd(const float* W, const uint8_t* mask, const double* ms, int rows, int cols, int bits, int iters,
                         uint16_t* codebook, uint8_t* idx, double* cosv, int* rowcnt, void* scratch, cudaStream_t s);

}  // namespace xq
