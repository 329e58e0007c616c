// Entry points of the data-consistency path that other translation units of the library use.
#pragma once
#include <cuda_runtime.h>
#include "../../include/gleam.h"

namespace gleam {

// RUN_PREPARE: only what depends on y and the mask alone (rank map, z table) is computed and left in
// the workspace; RUN_APPLY: the step with those tables taken from the workspace as they are; RUN_ADJOINT: A^H y
// (x and eta are ignored; the transforms of a zero image are left out).
enum { RUN_ALL = 0, RUN_PREPARE = 1, RUN_APPLY = 2, RUN_ADJOINT = 3 };

// How the one-pass 2-D kernel of a call leaves its inner products (dot_rows), and the shape of its launch.
struct DotForm {
    int sums;            // sums per example in each half of dot_rows
    int warps;           // warps of its blocks where it is one block per SM, 0 in its other forms
    bool shared;         // such a block: four warps share a line group
};

// out = x - eta A^H (A x - y)   (y == nullptr: out = x - eta A^H A x).  Validates its arguments,
// enqueues on d->stream, returns GLEAM_OK or a GLEAM_ERR_* code.  check_only: the argument checks
// alone (callers that must enqueue something of their own before the step run them first).
int run(const void* x, const void* y, const void* sens, const float* mask, float eta, void* out,
        const gleam_dims* d, int mode = RUN_ALL, double* dot_rows = nullptr, bool check_only = false,
        int layout = 0,      // layout: GLEAM_X_CHANNELS | GLEAM_OUT_CHANNELS (two-real-channel image arrays)
        const void* aty = nullptr,    // with y == nullptr: out = x - eta (A^H A x - aty), aty = A^H y as an image
        DotForm* dot_form = nullptr);    // set (also by check_only) to the form of the call's one-pass launch

// dot_rows (device, two arrays of one double per image row, B*T*n1): the one-pass 2-D kernel also stores
// Re<x_row, out_row> and <out_row, out_row> of every row it writes, so that a caller's inner products need no
// pass of their own.  Only where this returns true (2-D, readout-invariant mask, warp-resident row plan).
bool dot_rows_supported(const gleam_dims* d);

// GLEAM_OK for a device (or managed) pointer, GLEAM_ERR_NOT_DEVICE_POINTER otherwise
int check_device_ptr(const void* p);

// counts a launch of kernel class cls and, while per-kernel timing is on, records its event
cudaError_t prof_mark(int cls, cudaStream_t s);

}  // namespace gleam
