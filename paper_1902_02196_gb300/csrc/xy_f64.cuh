// FP64 xy transforms on square circulants of 8..128 (xy_f64.cu).
#pragma once

#include "fft.cuh"

// Forward (in: x [R][nc][nz][ny][nx] or on the support sp; out: the spectrum, planes of [L][L]) or inverse
// with the voxel-wise terms of e (in: the spectrum, out: y).  name, bytes: the launch's accounting.
int xy_f64(bool fwd, const char* name, double bytes, const vie_handle* h, const double2* in, double2* out,
           unsigned planes, int nx, int ny, const MatvecEpi& e, const Support& sp, cudaStream_t s);
