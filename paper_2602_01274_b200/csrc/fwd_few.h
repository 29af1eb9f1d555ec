// Host side of the few-row forward kernel.  The kernel is a translation unit of its own: compiled together with k_forward
// it made ptxas spill 660 bytes a thread there instead of 190 (verify forward of 25 rows, 14 layers of width 7168: 4.66
// against 4.21 ms).
#pragma once
#include "fwd_phases.cuh"

namespace fwd {

constexpr int FEW_ROWS = 16;                    // live token rows of such a forward at most
constexpr int FQ = 8;                           // query rows of an attention item
constexpr int FEW_XBYTES = 5120;                // shared memory for a block's columns of the residual stream
constexpr int FEW_ITEMS = 1024;                 // attention partials kept: items x FQ rows (or one per unsplit item)

// Whether a forward of these dimensions can take the kernel (when its live rows turn out to be few): the residual columns
// of a block fit its shared memory and one pass.
bool few_rows_ok(const ModelDev &m, const Geom &g, int kind, int ncta);
cudaError_t launch_few(const Args &a, int ncta, cudaStream_t st);

}  // namespace fwd
