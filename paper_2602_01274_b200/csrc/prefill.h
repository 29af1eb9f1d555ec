// Prompt prefill of one model as tiled GEMMs and a flash attention kernel (host interface).
#pragma once
#include "fwd_phases.cuh"

namespace pf {

constexpr int ROWS = 2048;                 // prompt rows (all sequences together) of one chunk at most
constexpr int MIN_ROWS = 33;               // fewer rows in all go through the forward kernel

// Device buffers, in the workspace.
struct Bufs {
    float *x;                              // [rows][d] residual stream
    bf16 *xg, *att, *act;                  // operands of the projections, split bf16 in operand order (see operand_index)
    float *q;                              // [rows][H * hd] rotated and scaled queries (the bytes of act)
    float *ssq;                            // [parts][rows padded to 128] shares of sum(x^2)
};
struct Sizes {
    size_t x, xg, att, act, ssq;
};
Sizes sizes(int d_max, int hh_max, int f_max, int rows);

enum Input { EMBED = 0, HIDDEN = 1 };

// Rows j = 0 .. nj-1 (cache positions c0 + j) of `batch` sequences through model m: appends their keys and values.
// input: EMBED reads the prompt tokens, HIDDEN takes the rows that the run of the draft model before left in x, through
// its final norm `normf` (the pre-verification model's input).  need_x: the last layer's output is wanted in x; without it
// the last layer ends with its keys and values.  Returns the first CUDA error; *launches counts kernels.
cudaError_t run(const ModelDev &m, const DevPtrs &d, const Bufs &b, int32_t *abort_flag, int batch, int nj, int c0, Input input,
                const bf16 *normf, bool need_x, int n_sm, cudaStream_t st, int64_t *launches);

// End of the prefill: n rows in the caches of the given models.
cudaError_t set_lengths(const DevPtrs &d, int batch, int n, bool target, bool draft, bool mb, cudaStream_t st);

}  // namespace pf
