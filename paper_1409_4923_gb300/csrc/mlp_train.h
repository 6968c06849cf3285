// mlp_train.h -- launchers of the surrogate network's training kernels (internal header).
#pragma once
#include <cstddef>
#include <cstdint>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "sde_mlp.h"

namespace sde_train {

constexpr int kIn = SDE_MLP_IN, kInPad = 16, kH = SDE_MLP_HIDDEN, kOut = SDE_MLP_OUT, kOutPad = 8;

// Offsets in the flat parameter vector.
constexpr size_t oW1 = 0, oB1 = oW1 + kH * kInPad, oW2 = oB1 + kH, oB2 = oW2 + kH * kH,
                 oW3 = oB2 + kH, oB3 = oW3 + kH * kH, oW4 = oB3 + kH, oB4 = oW4 + kOutPad * kH,
                 kNParams = oB4 + kOutPad;
static_assert(kNParams == SDE_MLP_NPARAMS, "parameter layout");

// A minibatch: rows 0 .. M - 1 of x, t as they stand (N == 0), or the rows of
// positions [pos0, pos0 + M) of one epoch's shuffled order of N labels.
struct Batch {
    const float* x;              // [.][7] raw inputs
    const float* t;              // [.][2] raw targets
    uint32_t M;
    uint32_t N, pos0, bits;      // labels, first position, Feistel width (shuffled minibatches)
    unsigned long long seed, epoch;
    uint32_t settled;            // x, t and the maps were complete before the kernel before this step's began
};

constexpr uint32_t kDefaultPolls = 1u << 24;

// Loss sums: blocks of 256 rows, at most 65536 rows.
constexpr int kLossBlocks = 256;

// The network's parameters and the training workspace for up to cap rows
// (cap a multiple of 64).
struct Net {
    CUtensorMap w2, w3;          // the BF16 copies of W2 and W3 as column blocks of 64 (weight_maps)
    float* w;                    // FP32 master parameters
    __nv_bfloat16* wb;           // BF16 copies
    float* m1;                   // Adam moments
    float* m2;
    const float* maps;           // input shift[7], scale[7], output shift[2], scale[2]
    uint32_t log_mask;
    __nv_bfloat16* X;            // [cap][16] mapped inputs
    __nv_bfloat16* A[3];         // [cap][256] activations
    __nv_bfloat16* dH[3];        // [cap][256] gradients of the pre-activations
    __nv_bfloat16* dY;           // [cap][8] gradient of the standardised outputs
    float* res;                  // [cap][2] residuals y' - t'
    double* loss_part;           // [kLossBlocks] partial losses
    uint32_t* loss_done;         // blocks that have written theirs (0 between steps)
    int* error;                  // set when a wait for a copy ran out: no later step changes the parameters
    volatile int* report;        // the same in pinned host memory, for the host to read without a copy
    uint32_t polls;              // of a wait for a copy, before it gives up
    uint32_t sm_count;
};

// What to do with the gradients: write them (grad != NULL) or take one Adam
// step with them.
struct Update {
    float* grad;
    float lr, b1, b2, eps, c1, c2;
    float* loss;                 // the batch loss (may be NULL)
    double* loss64;              // the same in FP64 (may be NULL)
};

// Tensor maps of the BF16 parameter copies wb, for Net.w2 and Net.w3.
cudaError_t weight_maps(const __nv_bfloat16* wb, CUtensorMap* w2, CUtensorMap* w3);

// The kernels' shared-memory limits on the current device; once per network,
// which stays on its device (on every launch they were two more runtime calls
// a step from a host that the steps wait for).
cudaError_t prepare();

// Loss and gradients of the batch, then the update; two kernels on `st`.
cudaError_t step(const Net& n, const Batch& b, const Update& u, cudaStream_t st);

}  // namespace sde_train
