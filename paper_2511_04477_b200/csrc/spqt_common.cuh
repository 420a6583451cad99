// Shared host-side helpers of the SpQt CUDA library (argument checks, geometry,
// device properties).  No kernel code lives here.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/spqt.h"

namespace spqt {

struct Format {
    int m, n, bits, group;
    int R;          // block-rows
    int B;          // bytes of codes per block
    size_t blocks;  // R * n
};

// Validates the format and fills the derived sizes.
inline spqt_status make_format(int m, int n, int bits, int group, Format* f)
{
    if (m <= 0 || n <= 0) return SPQT_ERR_INVALID_ARG;
    if (bits != 3 && bits != 4) return SPQT_ERR_UNSUPPORTED;
    if (group != 64 && group != 128) return SPQT_ERR_UNSUPPORTED;
    if (m % group != 0) return SPQT_ERR_UNSUPPORTED;
    f->m = m; f->n = n; f->bits = bits; f->group = group;
    f->R = m / group;
    f->B = group * bits / 8;
    f->blocks = (size_t)f->R * (size_t)n;
    return SPQT_OK;
}

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Workspace layout, the same for every shape, so that calls of different shapes may use one workspace: the status word, the last
// one of the first 256 bytes (the others are not used); then the slots in which CTAs that share a block-row leave their sums, 8
// bytes for each of its rows between every two neighbouring CTAs, zero between calls.  (The size is that of the first form, which
// had counters for the block-rows and at least one fp32 value per output row and block-row behind them.)
constexpr int kMaxPieceCtas = 160;
constexpr size_t kSlotsOffset = 256, kStatusOffset = kSlotsOffset - sizeof(int);
inline size_t slots_bytes(int group) { return (size_t)kMaxPieceCtas * (size_t)group * sizeof(unsigned long long); }

inline size_t workspace_bytes(const Format& f)
{
    const size_t header = (((size_t)(f.R + 1) * 4 + 255) / 256) * 256;   // (not less than kSlotsOffset)
    const size_t rows = ((size_t)f.m + (size_t)f.R) * sizeof(float), slots = slots_bytes(f.group);
    return header + (rows > slots ? rows : slots);
}

inline void* status_word(void* workspace) { return static_cast<unsigned char*>(workspace) + kStatusOffset; }

extern int g_no_pdl;          // 1 = launch strictly stream-ordered (spqt_set_tuning)
int sm_count();               // SMs of the current device (cached per device); <= 0 on error
void count_launch(int k = 1); // bump the process-wide launch counter

// Index collection over `batch` rows of X (columns active in at least one row, ascending; n < 2^16), one launch; the
// listed columns' values go to `gathered`, 4 (batch <= 4) or 8 fp16 values per list entry.
spqt_status launch_sparsify_rows(const __half* X, int ldx, int batch, int n, float t, int32_t* idx, int32_t* count,
                                 void* gathered, cudaStream_t stream);

}  // namespace spqt
