// FP64 xy transforms of the matvec (Section IV-A) on square circulants of 8..128: per plane, zero-pad
// and transform along x and y; and back, with the crop and the voxel-wise terms.  The counterparts of
// xy_fwd_kernel and xy_inv_kernel (matvec.cu), with the same spectrum layout, on scaled 64-bit integers
// (fixed.cuh): sm_103a's two FP64 operations per clock and SM made these transforms take 11 to 13 ms each way
// for 16 right-hand sides on a 64^3 grid.
//
// Precision.  Every line has its own scale, a row along x and a column along y, from its largest element; with one scale for
// a plane, planes whose values or spectra have a peak came out up to five times further off.  Before each of
// the four passes a line is brought to the bits which that pass's worst case leaves room for (fx_room): 56 to
// 58 of them, so that a rounding is 2^-56 of the line's largest value or less, where FP64 rounds every
// operation to 2^-53 of its own result.  The lanes of a warp are on different lines, so a line's key is an atomic
// without conflicts.
//
// Measured, 16 right-hand sides on 64^3 voxels (12288 planes, 128 x 128 spectra): forward 3.09 ms and inverse
// 4.73 ms, the FP64 kernels 11.2 and 13.1 ms (3.18 and 4.67 ms with a scale for a plane).
//
// What bounds them: the forward transforms issue in 49% of the cycles with 16 warps to an SM and wait for the ALU (busy
// 51%) and for shared memory; the inverse ones in 34%, waiting for shared memory, at barriers and for the
// voxel-wise terms (FP64 pipe 37%).
//
// A CTA owns one plane.  The x spectra of its rows stay in shared memory; the y transforms run on
// chunks of CW stored columns, whose spectra go to or come from global memory in registers, 512
// contiguous bytes to a warp.
#include <climits>

#include "block.cuh"
#include "fft2.cuh"
#include "fixed.cuh"
#include "xy_f64.cuh"

namespace {

template <int L>
struct XYCfg64 {
    static constexpr int H = L / 2;                // rows that are non-zero before / needed after the y transform
    static constexpr int RS = L + 1;               // odd row stride
    static constexpr int CW = L < 32 ? L : 32;     // stored columns per y-transform chunk
    static constexpr int NT = L >= 128 ? 512 : (L >= 32 ? 256 : 64);
    static constexpr int MINB = L >= 128 ? 1 : (L >= 64 ? 2 : 4);
    static constexpr size_t smem = sizeof(fx2) * (size_t)(L * CW + H * RS + L) + sizeof(int4) * H + L + sizeof(int) * (4 * L);
};

// Forward: plane (r, alpha, z) of x -> W2 plane [Ly][Lx] (transposed ky, stored kx).  x is
// [R][nc][Nz][Ny][Nx], or [R][nc][ns] on a support (rows != NULL; zeros outside it).
template <int L>
__global__ void __launch_bounds__(XYCfg64<L>::NT, XYCfg64<L>::MINB)
    xy64_fwd_kernel(const double2* x, double2* w, int nx, int ny, int nz,
                    const int4* __restrict__ rows, long long ns, const unsigned char* __restrict__ cpos,
                    const int4* __restrict__ twg, const int* rmap, MatvecEpi dc) {
    using Cfg = XYCfg64<L>;
    constexpr int A = fft2::Split<L>::A, B = fft2::Split<L>::B, NT = Cfg::NT, RS = Cfg::RS, CW = Cfg::CW, H = Cfg::H;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* ck = reinterpret_cast<fx2*>(smem_raw);  // [L][CW] chunk of stored columns
    fx2* xr = ck + L * CW;                       // [H][RS] rows: the input, then its x spectra
    int4* tw = reinterpret_cast<int4*>(xr + H * RS);
    int4* rw = tw + L;  // [H] support rows of this plane
    unsigned char* pos = reinterpret_cast<unsigned char*>(rw + H);
    unsigned* krow = reinterpret_cast<unsigned*>(pos + L);  // [H] keys of the rows
    unsigned* kmid = krow + H;                              // [H] after the first x pass
    unsigned* kspec = kmid + H;                             // [H] of their x spectra
    int* rsh = reinterpret_cast<int*>(kspec + H);           // [H] shift of a row to the plane's scale
    unsigned* kcol = reinterpret_cast<unsigned*>(rsh + H);  // [L] of the stored columns after the first y pass
    const int tid = threadIdx.x;
    const long long p = blockIdx.x;  // spectrum plane; the input plane is pin (rmap: active right-hand sides)
    const long long rplanes = (long long)dc.nc * nz;  // planes per right-hand side
    grid_release();
    grid_wait();
    if (dc.nact) {  // planes of right-hand sides beyond the device count are skipped
        const int cnt = *dc.nact;
        dev_bytes_add(dc.bctr, dc.bfix + dc.bper * cnt, cnt > 0);
        if (p / rplanes >= cnt) return;
    }
    for (int m = tid; m < L; m += NT) {
        tw[m] = twg[m];
        pos[m] = cpos[m];
    }
    for (int m = tid; m < 4 * H + L; m += NT) krow[m] = 0;
    const long long pin = rmap ? (long long)rmap[p / rplanes] * rplanes + p % rplanes : p;
    const double2* src = x + pin * (long long)ny * nx;
    if (rows) {
        const int z = (int)(p % nz);
        for (int yy = tid; yy < ny; yy += NT) rw[yy] = rows[(long long)z * ny + yy];
        src = x + (pin / nz) * ns;
    }
    __syncthreads();
    for (int i0 = tid; i0 < ny * nx; i0 += 4 * NT) {  // four loads in flight
        double2 v[4];
        int dst[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int idx = i0 + q * NT, yy = idx / nx, xx = idx - yy * nx;
            v[q] = make_double2(0.0, 0.0);
            dst[q] = idx < ny * nx ? yy * RS + xx : -1;
            if (idx < ny * nx) {
                if (rows) {
                    const int4 s = rw[yy];
                    if (xx >= s.x && xx < s.y) v[q] = src[s.z + (xx - s.x)];
                } else {
                    v[q] = src[idx];
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (dst[q] >= 0) *reinterpret_cast<double2*>(xr + dst[q]) = v[q];
    }
    __syncthreads();
    // x transform; lanes are on different rows
    for (int t = tid; t < H * B; t += NT) {
        const int n = t % H, b = t / H;
        if (n >= ny) continue;
        const double2* ln = reinterpret_cast<const double2*>(xr + n * RS);
        unsigned key = 0;
#pragma unroll
        for (int a = 0; a < A / 2; ++a) {
            const int l = b + B * a;
            if (l < nx) key = max(key, fx_key(ln[l]));
        }
        atomicMax(krow + n, key);
    }
    __syncthreads();
    for (int t = tid; t < H * B; t += NT) {
        const int n = t % H, b = t / H;
        if (n >= ny) continue;
        const FxScale sc(krow[n], fx_room(A / 2));
        fx2* ln = xr + n * RS;
        fx2 v[A];
#pragma unroll
        for (int a = 0; a < A / 2; ++a) {
            const int l = b + B * a;
            v[a] = l < nx ? sc(*reinterpret_cast<const double2*>(ln + l)) : fx2{0, 0};
        }
        fft2::dft_half_in<A>(v, -1);
        unsigned key = 0;
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            if (k1 && b) v[k1] = cmul(v[k1], tw[b * k1]);
            ln[b + B * k1] = v[k1];
            key |= fx_key(v[k1]);
        }
        atomicOr(kmid + n, key);
    }
    __syncthreads();
    for (int t = tid; t < H * A; t += NT) {
        const int n = t % H, k1 = t / H;
        if (n >= ny) continue;
        const int k = excess(kmid[n], B);
        fx2* ln = xr + n * RS + B * k1;
        fx2 v[B];
#pragma unroll
        for (int b = 0; b < B; ++b) v[b] = fx_shift(ln[b], k);
        fft2::DFT<B, fx2>::run(v, -1);
        unsigned key = 0;
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            ln[k2] = v[k2];
            key |= fx_key(v[k2]);
        }
        atomicOr(kspec + n, key);
    }
    __syncthreads();
    // The rows' spectra go to one scale, with room for the y transform.  (No row is shifted up: a spectrum is as
    // large as its row, so its exponent is below the common one as it is.)
    auto row_ex = [&](int n) { return FxScale(krow[n], fx_room(A / 2)).ex + excess(kmid[n], B); };
    int ex = INT_MIN;
    unsigned kall = 0;
    for (int n = tid & 31; n < ny; n += 32) {
        const int e = row_ex(n);
        ex = max(ex, max(fx_bits(kspec[n]) - fx_room(A / 2), 0) + e);
        kall = max(kall, krow[n]);
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    for (int n = tid; n < ny; n += NT) rsh[n] = min(ex - row_ex(n), 62);
    const bool bad = __reduce_max_sync(0xffffffffu, kall) >= 0x7ff00000u;  // an Inf or NaN reaches the whole spectrum
    __syncthreads();
    double2* dst = w + p * (long long)L * L;
#pragma unroll 1
    for (int c0 = 0; c0 < L; c0 += CW) {
        // y transform, pass 1: stored column c0 + c from the x spectra.  An A-point DFT of A/2 values
        // is two A/2-point ones, of the even and (twisted) of the odd frequencies: a task each
        for (int t = tid; t < 2 * CW * B; t += NT) {
            const int c = t % CW, b = (t / CW) % B, odd = t / (CW * B);
            const fx2* col = xr + pos[c0 + c];
            fx2 v[A / 2];
#pragma unroll
            for (int a = 0; a < A / 2; ++a) {  // ny <= L/2: the upper half is zero
                const int yy = b + B * a;
                v[a] = yy < ny ? fx_shift(col[yy * RS], rsh[yy]) : fx2{0, 0};
            }
            if (odd) {
#pragma unroll
                for (int a = 0; a < A / 2; ++a) v[a] = fft2::twist<A>(v[a], a, -1);
            }
            fft2::DFT<A / 2, fx2>::run(v, -1);
            unsigned key = 0;
#pragma unroll
            for (int q = 0; q < A / 2; ++q) {
                const int k1 = 2 * q + odd;
                if (b && k1) v[q] = cmul(v[q], tw[b * k1]);
                ck[(b + B * k1) * CW + c] = v[q];
                key |= fx_key(v[q]);
            }
            atomicOr(kcol + c0 + c, key);
        }
        __syncthreads();
        for (int t = tid; t < CW * A; t += NT) {
            const int c = t % CW, k1 = t / CW;
            const int k = excess(kcol[c0 + c], B);
            const fx2* ln = ck + B * k1 * CW + c;
            fx2 v[B];
#pragma unroll
            for (int b = 0; b < B; ++b) v[b] = fx_shift(ln[b * CW], k);
            fft2::DFT<B, fx2>::run(v, -1);
            // the range is looked at once for a line's values, not for each: 3.22 to 3.09 ms at the size above
            auto store = [&](auto to_double) {
#pragma unroll
                for (int k2 = 0; k2 < B; ++k2) {
                    double2 o = to_double(v[k2], ex + k);
                    if (bad) o.x = o.y = __longlong_as_double(0x7ff8000000000000ll);
                    dst[(long long)(B * k1 + k2) * L + c0 + c] = o;
                }
            };
            if (fx_in_range(ex + k))
                store([](fx2 u, int e) { return fx_double<true>(u, e); });
            else
                store([](fx2 u, int e) { return fx_double(u, e); });
        }
        __syncthreads();
    }
}

// Inverse: W2 plane -> y plane [Ny][Nx] with the material / Gram / preconditioner epilogue;
// CONV: also the plane's (N - G) x at every voxel to epi.conv (full grid).
template <int L, bool CONV>
__global__ void __launch_bounds__(XYCfg64<L>::NT, XYCfg64<L>::MINB)
    xy64_inv_kernel(const double2* w, double2* y, MatvecEpi epi,
                    const unsigned char* __restrict__ cpos, const int4* __restrict__ twg) {
    using Cfg = XYCfg64<L>;
    constexpr int A = fft2::Split<L>::A, B = fft2::Split<L>::B, NT = Cfg::NT, RS = Cfg::RS, CW = Cfg::CW, H = Cfg::H;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* ck = reinterpret_cast<fx2*>(smem_raw);
    fx2* xr = ck + L * CW;
    int4* tw = reinterpret_cast<int4*>(xr + H * RS);
    int4* rw = tw + L;
    unsigned char* pos = reinterpret_cast<unsigned char*>(rw + H);
    unsigned* kcol = reinterpret_cast<unsigned*>(pos + L);   // [L] keys of the stored columns
    unsigned* kmid = kcol + L;                               // [L] after the first y pass
    int* cex = reinterpret_cast<int*>(kmid + L);             // [L] by x position: the exponent after the y transform
    int* rtop = cex + L;                                     // [H] bits and exponent of the largest value of a row
    unsigned* krow = reinterpret_cast<unsigned*>(rtop + H);  // [H] keys of the rows after the first x pass
    const int tid = threadIdx.x;
    const int nx = epi.nx, ny = epi.ny, nz = epi.nz;
    const long long p = blockIdx.x;  // spectrum plane (r * nc + alpha) * nz + z; output plane po
    const int nc = epi.nc;
    const long long rplanes = (long long)nc * nz;  // planes per right-hand side
    grid_release();
    grid_wait();
    if (epi.nact) {
        const int cnt = *epi.nact;
        dev_bytes_add(epi.bctr, epi.bfix + epi.bper * cnt, cnt > 0);
        if (p / rplanes >= cnt) return;
    }
    for (int m = tid; m < L; m += NT) {
        tw[m] = twg[m];
        pos[m] = cpos[m];
        kcol[m] = kmid[m] = 0;
    }
    for (int n = tid; n < H; n += NT) {
        rtop[n] = INT_MIN;
        krow[n] = 0;
    }
    const long long po = epi.rmap ? (long long)epi.rmap[p / rplanes] * rplanes + p % rplanes : p;
    if (epi.rows)
        for (int yy = tid; yy < ny; yy += NT) rw[yy] = epi.rows[(p % nz) * ny + yy];
    __syncthreads();
    const double2* src = w + p * (long long)L * L;
#pragma unroll 1
    for (int c0 = 0; c0 < L; c0 += CW) {
        // inverse y transform, pass 1.  One task per thread (CW A <= NT), so its inputs wait in registers
        // for the column's scale
        static_assert(CW * A <= NT || L < 32, "one pass-1 task per thread");
        constexpr int NTASK = (CW * A + NT - 1) / NT;
        double2 d[NTASK][B];
#pragma unroll
        for (int q = 0; q < NTASK; ++q) {
            const int t = tid + q * NT, c = t % CW, k1 = t / CW;
            unsigned key = 0;
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) {
                d[q][k2] = t < CW * A ? src[(long long)(B * k1 + k2) * L + c0 + c] : make_double2(0.0, 0.0);
                key = max(key, fx_key(d[q][k2]));
            }
            if (t < CW * A) atomicMax(kcol + c0 + c, key);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NTASK; ++q) {
            const int t = tid + q * NT, c = t % CW, k1 = t / CW;
            if (t >= CW * A) continue;
            const FxScale sc(kcol[c0 + c], fx_room(B));
            unsigned key = 0;
            fx2 v[B];
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k2] = sc(d[q][k2]);
            fft2::DFT<B, fx2>::run(v, +1);
#pragma unroll
            for (int b = 0; b < B; ++b) {
                if (b && k1) v[b] = cmul(v[b], fx_conj(tw[b * k1]));
                ck[(b + B * k1) * CW + c] = v[b];
                key |= fx_key(v[b]);
            }
            atomicOr(kmid + c0 + c, key);
        }
        __syncthreads();
        // pass 2: rows y < Ny scattered to the x-transform buffer at the column's x position
        for (int t = tid; t < CW * B; t += NT) {
            const int c = t % CW, b = t / CW, px = pos[c0 + c];
            const int k = excess(kmid[c0 + c], A);
            fx2 v[A];
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) v[k1] = fx_shift(ck[(b + B * k1) * CW + c], k);
            fft2::dft_half_out<A>(v, +1);
            const int ex = FxScale(kcol[c0 + c], fx_room(B)).ex + k;
            fx2* col = xr + px;
#pragma unroll
            for (int a = 0; a < A / 2; ++a) {  // ny <= L/2
                const int yy = b + B * a, top = fx_bits(fx_key(v[a])) + ex;
                if (yy >= ny) continue;
                col[yy * RS] = v[a];
                if constexpr (CW == 32) {  // a warp is on one row
                    const int m = __reduce_max_sync(0xffffffffu, top);
                    if (c == 0) atomicMax(rtop + yy, m);
                } else {
                    atomicMax(rtop + yy, top);
                }
            }
            if (b == 0) cex[px] = ex;
        }
        __syncthreads();
    }
    unsigned kall = 0;
    for (int m = tid & 31; m < L; m += 32) kall = max(kall, kcol[m]);
    const bool bad = __reduce_max_sync(0xffffffffu, kall) >= 0x7ff00000u;  // an Inf or NaN reaches the whole plane
    const long long base = po * (long long)ny * nx;
    const long long cbase = (po / nz) * epi.ns;  // component block on the support
    const double2* xin = reinterpret_cast<const double2*>(epi.x);
    // the epilogue's x values of this plane arrive in the free chunk buffer during the x transform
    static_assert(CW >= L / 4, "a plane of L/2 x L/2 values fits the chunk buffer");
    const bool pre = epi.op != VIE_OP_NSCAT;
    if (pre) {
        for (int idx = tid; idx < ny * nx; idx += NT) {
            const int yy = idx / nx, xx = idx % nx;
            long long o = base + idx;
            bool in = true;
            if (epi.rows) {
                const int4 q = rw[yy];
                in = xx >= q.x && xx < q.y;
                o = in ? cbase + q.z + (xx - q.x) : cbase;
            }
            cp_async_elem(reinterpret_cast<double2*>(ck) + idx, xin + o, in);
        }
        cp_async_commit();
    }
    // inverse x transform: a row's values, one of each column, on the scale of its largest
    for (int t = tid; t < H * A; t += NT) {
        const int n = t % H, k1 = t / H;
        if (n >= ny) continue;
        const int ex = rtop[n] - fx_room(B);
        fx2* ln = xr + n * RS + B * k1;
        fx2 v[B];
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            const int s = ex - cex[B * k1 + k2], up = max(-s, 0);  // up <= 25: the bits count 32 at least
            const fx2 u = fx_shift(ln[k2], min(max(s, 0), 62));
            v[k2] = fx2{u.x << up, u.y << up};
        }
        fft2::DFT<B, fx2>::run(v, +1);
        unsigned key = 0;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if (b && k1) v[b] = cmul(v[b], fx_conj(tw[b * k1]));
            ln[b] = v[b];
            key |= fx_key(v[b]);
        }
        atomicOr(krow + n, key);
    }
    __syncthreads();
    for (int t = tid; t < H * B; t += NT) {
        const int n = t % H, b = t / H;
        if (n >= ny) continue;
        const int k = excess(krow[n], A);
        fx2* ln = xr + n * RS;
        fx2 v[A];
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[k1] = fx_shift(ln[b + B * k1], k);
        fft2::dft_half_out<A>(v, +1);
#pragma unroll
        for (int a = 0; a < A / 2; ++a) {
            const int l = b + B * a;
            if (l < nx) ln[l] = v[a];
        }
        if (b == 0) rtop[n] += k - fx_room(B);  // now the exponent of the row's results
    }
    if (pre) cp_async_wait<0>();
    __syncthreads();
    const int alpha = (int)((p / nz) % nc);
    const long long zoff = (p % nz) * (long long)ny * nx;
    const double gl = comp_is_constant(alpha, nc) ? epi.g1 : epi.g234;
    const double ig = 1.0 / gl;
    const double2* c1 = reinterpret_cast<const double2*>(epi.c1);
    const double2* c2 = reinterpret_cast<const double2*>(epi.c2);
    const double2 sh = epi.shift ? epi.shift[po / rplanes] : make_double2(0.0, 0.0);  // op PA
    double2* conv = CONV ? reinterpret_cast<double2*>(epi.conv) : nullptr;
#pragma unroll 4
    for (int idx = tid; idx < ny * nx; idx += NT) {
        const int yy = idx / nx, xx = idx % nx;
        long long o = base + idx;
        bool in = true;
        if (epi.rows) {
            const int4 q = rw[yy];
            in = xx >= q.x && xx < q.y;
            o = cbase + q.z + (xx - q.x);
        }
        if (!CONV && !in) continue;
        double2 v = fx_double(xr[yy * RS + xx], rtop[yy]);
        if (bad) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
        if (CONV) conv[base + idx] = v;  // every voxel of the plane, full-grid layout
        if (!in) continue;
        if (epi.op == VIE_OP_A) {
            const double2 xv = reinterpret_cast<const double2*>(ck)[idx];
            v = csub(mk(gl * xv.x, gl * xv.y), cmul(c2[zoff + idx], v));
        } else if (epi.op == VIE_OP_PA) {
            const double2 xv = reinterpret_cast<const double2*>(ck)[idx];
            const double2 t = cmul(c2[zoff + idx], v);
            v = csub(cmul(csub(c1[zoff + idx], sh), xv), mk(ig * t.x, ig * t.y));
        }
        y[o] = v;
    }
}

template <int L>
int launch_L(bool fwd, const char* name, double bytes, const vie_handle* h, const double2* in, double2* out,
             unsigned planes, int nx, int ny, const MatvecEpi& e, const Support& sp, cudaStream_t s) {
    using Cfg = XYCfg64<L>;
    // set on every call: the attribute is per device and launches may come from several threads
    auto attr = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem);
    };
    const unsigned char* cpos = h->colmap + L;
    const int4* tw = h->twfx + L;
    if (fwd) {
        VIE_CUDA(attr(xy64_fwd_kernel<L>));
        VIE_LAUNCH(name, s, bytes, (xy64_fwd_kernel<L>), planes, Cfg::NT, Cfg::smem, in, out, nx, ny, h->nz, sp.rows,
                   sp.ns, cpos, tw, e.rmap, e);
    } else if (e.conv) {
        VIE_CUDA(attr(xy64_inv_kernel<L, true>));
        VIE_LAUNCH(name, s, bytes, (xy64_inv_kernel<L, true>), planes, Cfg::NT, Cfg::smem, in, out, e, cpos, tw);
    } else {
        VIE_CUDA(attr(xy64_inv_kernel<L, false>));
        VIE_LAUNCH(name, s, bytes, (xy64_inv_kernel<L, false>), planes, Cfg::NT, Cfg::smem, in, out, e, cpos, tw);
    }
    VIE_CHECK_LAUNCH();
    return VIE_OK;
}

}  // namespace

int xy_f64(bool fwd, const char* name, double bytes, const vie_handle* h, const double2* in, double2* out,
           unsigned planes, int nx, int ny, const MatvecEpi& e, const Support& sp, cudaStream_t s) {
    switch (h->L[0]) {
        case 8: return launch_L<8>(fwd, name, bytes, h, in, out, planes, nx, ny, e, sp, s);
        case 16: return launch_L<16>(fwd, name, bytes, h, in, out, planes, nx, ny, e, sp, s);
        case 32: return launch_L<32>(fwd, name, bytes, h, in, out, planes, nx, ny, e, sp, s);
        case 64: return launch_L<64>(fwd, name, bytes, h, in, out, planes, nx, ny, e, sp, s);
        case 128: return launch_L<128>(fwd, name, bytes, h, in, out, planes, nx, ny, e, sp, s);
    }
    set_error("xy transform: unsupported length");
    return VIE_EINVAL;
}
