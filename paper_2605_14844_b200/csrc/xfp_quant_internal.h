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

// LibFit (xfp_quant_libfit.cu): the library from the per-channel codebooks, then the groups' assignment; cosv may be null.
cudaError_t launch_libfit_library(const uint16_t* codebook, int rows, int E, int L, int iters, double* u, double* nn,
                                  int* order, int* asg, double* cen, int* flags, uint16_t* lib, cudaStream_t s);
cudaError_t launch_libfit_assign(const float* W, const uint8_t* mask, const double* ms, int rows, int cols, int bits, int L,
                                 int group_size, const uint16_t* lib, uint8_t* idx, uint8_t* gid, uint16_t* gscale,
                                 uint16_t* gmid, double* cosv, cudaStream_t s);

}  // namespace xq
