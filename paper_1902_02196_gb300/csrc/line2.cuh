// Line transforms of the matvec's line path with the two-pass register FFT (FP32: line2.cu; FP64: line_f64.cu).
#pragma once

#include "fft.cuh"

// FFT lengths the two-pass line kernels take (8..512, powers of two)
bool line2_ok(int L);

// Forward transform of the lines of `a` (natural order in, a.n_in <= L/2 elements, the rest
// zero): every frequency stored, at position q = colkx^-1 (colkx[q] = the frequency stored at q)
// or, with colkx NULL, in fft2's transposed order.
int line2_forward(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx, cudaStream_t s);
int line64_forward(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx, cudaStream_t s);

// Inverse (unnormalised) transform of the lines of `a`, spectrum in the order the forward transform
// stores, outputs l < a.n_out (<= L/2) written in natural order; with the voxel-wise terms of epi if given.
int line2_inverse(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx, cudaStream_t s);
int line64_inverse(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx,
                   const MatvecEpi* epi, cudaStream_t s);
