// ESC accumulator of the light columns (Section 4): launcher.
#pragma once

#include "kernels.cuh"

namespace spg {

constexpr int kEscWarps = 8;  // warps per CTA, each working its own columns

// values = false: run counts into cnt_out[j + 1] (symbolic).  values = true:
// C's rows and values at base[j] + rank; the counts are written to cnt_out
// when given (single pass), else checked against base[j + 1] - base[j].
// t.bin is a lane-group bin; t.m rows are numbered.
cudaError_t launch_esc_bin(const BinTask &t, const Operands &o, const int64_t *base, int64_t *cnt_out,
                           int32_t *Crow, void *Cval, bool values, int dtype, int sms, cudaStream_t s);

}  // namespace spg
