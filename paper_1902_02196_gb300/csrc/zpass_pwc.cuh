// z pass of the PWC system with its 3 x 3 block (zpass_pwc.cu).
#pragma once

#include "common.cuh"

struct ZPArgs {
    void* w;            // spectrum [R*3][Nz][Ly][Lx], in place
    const void* green;  // octant spectra [60][Oz][Oy][Ox] in the spectrum's precision
    const int* colkx;   // [Lx] kx of each stored column
    int R, nz, Lx, Ly, Ox, Oy, Oz;
    int ay, by;         // row py holds ky = py / by + ay * (py % by); by = 0: ky = py
};

// FFT lengths the PWC z pass takes
inline bool zpwc_ok(const vie_handle* h) { return h->L[2] >= 8 && h->L[2] <= 512 && h->L[0] >= 8; }
int zpass_pwc(const vie_handle* h, const ZPArgs& z, bool fp64, cudaStream_t s);
