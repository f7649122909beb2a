// ts_wide.h -- launch block of the wide-pass kernels (ts_wide.cu): passes of
// 9-64 tokens of a bf16 FFN as gathered tensor-core GEMMs.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace tsffn {

constexpr int kWideMaxRows = 65536;

struct WideLaunch {
    int d, m, n_rows, batch;      // batch: 9 .. 64 tokens
    const int32_t* rows;          // predictor list (ascending neuron ids) or nullptr
    const __nv_bfloat16* x;       // [batch][d] activations
    const __nv_bfloat16* wg;      // [m][d]
    const __nv_bfloat16* wu;
    const __nv_bfloat16* wd;
    // both-active rows listed by the gate+up tiles: tile i's from entry i * (rows per tile) on
    int32_t* ent;                 // [m] neuron ids
    int* ent_n;                   // [wide_tiles(m)] their count per tile
    __nv_bfloat16* c_hi;          // [m][64] c = g u of the entries, hi part
    __nv_bfloat16* c_lo;          // [m][64] lo part (c - hi)
    float* partial;               // [ks][batch][d] down projection per slice of the listed rows
    int ks;                       // slices
    uint8_t* gbits;               // [batch][nbytes] gate-active bitmaps (per row-space position)
    uint8_t* bbits;               // [batch][nbytes] both-active bitmaps
    int nbytes;                   // bitmap bytes per token (multiple of 4)
    unsigned* status;
    float* y;                     // [batch][d] output, or
    float* h;                     // [batch][d] residual: h += y (residual_out)
    int residual_out;
};

// Whether a pass of `batch` tokens can take the wide kernels.
bool wide_supported(int wdtype, int d, int m, int batch);
// Slices of the listed rows for the down projection (one CTA per slice and 256 columns).
int wide_slices(int d, int num_sms);
// Most gate+up tiles of a pass over up to m rows.
int wide_tiles(int m, int num_sms);
cudaError_t prepare_wide();
// gate+up, down and the reduction of one pass (programmatic dependent launch
// between them; `pdl` for the first).
cudaError_t launch_wide(const WideLaunch& L, int num_sms, cudaStream_t stream, bool pdl);
// x = rmsnorm(h) with x[d-1] = 1, bf16, for the stacks.
cudaError_t launch_norm(int d, int batch, const float* h, __nv_bfloat16* xout, cudaStream_t stream, bool pdl);

}  // namespace tsffn
