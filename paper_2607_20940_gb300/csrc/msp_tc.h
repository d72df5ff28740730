// Fused MSP kernels (patchify + tier embedding, de-embedding + unpatchify) on
// the sm_103a tensor cores; see msp_tc.cu.
#pragma once
#include <cuda_runtime.h>

#include "kernels.h"

namespace msf {

// One run of consecutive window states of one tier (same patch edge, same
// weight): their tokens are contiguous in the output.
struct MspEmbedRun {
    const void* w;  // [w_rows, K] bf16 tier weight, K = C * P * P contiguous
    int M;          // tokens of the run per stream
    int l0;         // first state
    int n_l;        // tokens per state
    int gw;         // tokens per grid row (Wl / P)
    int P;          // patch edge in latent pixels
    int K;          // C * P * P
    int tok_off;    // first token row of the run
    // LoRA adapter of the tier (Sec. 4.1): tokens += up * bf16(lora_scale *
    // down x) for the patch vector x, with the down projection [rank, K] and
    // the up projection [E, rank] (rank 8..64, a multiple of 8).
    const void* lora_down = nullptr;
    const void* lora_up = nullptr;
    int rank = 0;
    float lora_scale = 1.0f;
};

bool msp_embed_supported(const MspEmbedRun* runs, int n, int E);
// Up to kMaxGemmProblems runs in one launch. With `pool` (bf16 jobs) the
// same launch also runs those K/V pyramid jobs, on more CTAs after the
// embedding tiles and on the tiles' idle warps: they read and write buffers
// the embedding does not touch, so the two share the SMs of one launch.
cudaError_t launch_msp_embed(const MspEmbedRun* runs, int n, const MspShape& sh, int E, const void* latent,
                             void* tokens, long long tok_bstride, int batch, unsigned int* status,
                             cudaStream_t st, const PoolBatch* pool = nullptr);

// The coarse tier's extras of a de-embedding (Sec. 4.1), computed in the same
// launch.
struct DeembedTier {
    // LoRA: up [F, rank] times bf16(scale * down h), down [rank, E]. NULL up: none.
    const void* down = nullptr;
    const void* up = nullptr;
    int rank = 0;
    float scale = 1.0f;
    // Latent residual: residual [F, F] times the raw patch vectors of the
    // position's input latent (stream b at latent + b * latent_bstride).
    // NULL residual: none.
    const void* latent = nullptr;
    long long latent_bstride = 0;  // elements
    const void* residual = nullptr;
};

// De-embedding + unpatchify of M tokens (F = C*P*P features, E = K) of one
// window position; the split-K reduction stays inside a thread-block cluster.
bool msp_deembed_supported(int M, int F, int E);
cudaError_t launch_msp_deembed(const void* tokens, long long tok_bstride_elems, int tok_rows, int tok_row0,
                               const void* w_out, int M, int F, int E, const MspShape& sh, int P, void* latent,
                               int batch, unsigned int* status, cudaStream_t st,
                               const DeembedTier* tier = nullptr);

}  // namespace msf
