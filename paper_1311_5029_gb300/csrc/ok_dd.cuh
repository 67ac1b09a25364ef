// FP64-accurate application of M on the FP32 pipes (double-float W and fields).
#pragma once
#include "ok_launch.cuh"

namespace okgb {

// The apply's input: a spinor field as double-float, in blocks of 32 sites (dd_field_bytes bytes).
size_t dd_field_bytes(const ok_W* W);
int launch_to_dd_field(const ok_W* W, const cx<double>* in, void* out, cudaStream_t st);
// out = M psi (EPI_NONE) or out = b - M psi with <out, out>, <b, b> reduced (EPI_RESID), in
// double-float arithmetic with the handle's OK_W_DF64 copy: psi from launch_to_dd_field, b and out FP64
// [V][12].  OK_EINVAL without the copy or for another epilogue.
int launch_apply_dd(const ok_W* W, const void* psi_dd, cx<double>* out, int epi, const EpiArgs<dd>& ep, cudaStream_t st);

}  // namespace okgb
