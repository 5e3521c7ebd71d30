// z pass of the PWC system's matvec (Section IV-A with the l = 1 functions of Section V-A alone): z
// transform, 3 x 3 Green block and inverse z transform of TB stored columns per CTA, one right-hand
// side after another, with the two-pass transforms of fft2.cuh and, in FP64, on scaled integers
// (fixed.cuh).  It replaces the generic z pass (matvec.cu: radix-4 transforms, log4 L trips through
// shared memory) for FFT lengths along z of 8..512 and Lx >= 8: one right-hand side on 61^3 voxels (128^3 points)
// took 0.95 ms there in FP64, which the FP64 unit's two operations per clock bound.  The product itself,
// nine complex multiply-adds a point, stays on that unit.  Every line has its own scale, renewed before each pass.
// What bounds it is still that unit, busy for 71%.
//
// The six Green values of a point come from the octant spectra [60][Oz][Oy][Ox] (every tenth tensor), served by
// L2: a reordered copy would save less than it costs to set up for a system that is solved once or twice.
#include "block.cuh"
#include "fft2.cuh"
#include "fixed.cuh"
#include "zpass_pwc.cuh"

namespace {

template <typename T, int LZ>
struct ZPCfg {
    static constexpr int TB = LZ <= 256 ? 8 : 4;
    static constexpr int NL = 3 * TB;  // lines
    static constexpr int NT = LZ <= 16 ? 96 : (LZ == 256 ? 384 : 192);
    static constexpr int MINB = LZ <= 128 ? 3 : (LZ == 256 ? 1 : 2);
    static constexpr int GS = LZ * TB + 8;  // component stride: 8 elements of padding keep half-warps apart
    static constexpr size_t smem = (sizeof(T) == 8 ? 16 : 8) * (size_t)(3 * GS + LZ) + (sizeof(T) == 8 ? 4 * sizeof(int) * NL : 0);
};

// y = B x at one point: entry (p, q) is tensor 10 pq(p, q); m: components whose sign flips at this reflected point
template <typename C>
__device__ __forceinline__ void point3(const C* __restrict__ g, long long tstride, unsigned m, C* x) {
    C u[6];
#pragma unroll
    for (int t = 0; t < 6; ++t) u[t] = __ldg(g + 10 * t * tstride);  // xx, xy, xz, yy, yz, zz
#pragma unroll
    for (int b = 0; b < 3; ++b)
        if ((m >> b) & 1u) x[b] = cneg(x[b]);
    C y0 = C{}, y1 = C{}, y2 = C{};
    cfma(y0, u[0], x[0]);
    cfma(y1, u[1], x[0]);
    cfma(y2, u[2], x[0]);
    cfma(y0, u[1], x[1]);
    cfma(y1, u[3], x[1]);
    cfma(y2, u[4], x[1]);
    cfma(y0, u[2], x[2]);
    cfma(y1, u[4], x[2]);
    cfma(y2, u[5], x[2]);
    x[0] = (m & 1u) ? cneg(y0) : y0;
    x[1] = (m & 2u) ? cneg(y1) : y1;
    x[2] = (m & 4u) ? cneg(y2) : y2;
}

template <typename T, int LZ>
__global__ void __launch_bounds__(ZPCfg<T, LZ>::NT, ZPCfg<T, LZ>::MINB)
    zpwc_kernel(ZPArgs z, const float2* __restrict__ tw32, const int4* __restrict__ twfx) {
    using Cfg = ZPCfg<T, LZ>;
    using C = typename CT<T>::C;
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int A = fft2::Split<LZ>::A, B = fft2::Split<LZ>::B, NT = Cfg::NT, TB = Cfg::TB, GS = Cfg::GS, NL = Cfg::NL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* s = reinterpret_cast<C*>(smem_raw);
    fx2* f = reinterpret_cast<fx2*>(smem_raw);  // FP64: the same places, between the conversions
    float2* twf = reinterpret_cast<float2*>(s + 3 * GS);
    int4* twi = reinterpret_cast<int4*>(s + 3 * GS);
    // FP64: per line the keys of the inputs, after the first forward pass, of the product, after the first inverse pass
    unsigned* kin = reinterpret_cast<unsigned*>(s + 3 * GS + LZ);
    unsigned *kfwd = kin + NL, *kout = kfwd + NL, *kmid = kout + NL;
    const int tid = threadIdx.x, lane = tid & 31;
    grid_release();
    for (int m = tid; m < LZ; m += NT) {
        if constexpr (F64)
            twi[m] = twfx[m];
        else
            twf[m] = tw32[m];
    }
    if (F64)
        for (int i = tid; i < 4 * NL; i += NT) kin[i] = 0;
    grid_wait();
    __syncthreads();
    const int ntile = z.Lx / TB;
    const int py = blockIdx.x / ntile, sc0 = (blockIdx.x % ntile) * TB;
    const long long plane = (long long)z.Ly * z.Lx;
    const int ky = py / z.by + z.ay * (py % z.by);
    const int kyo = ky <= z.Ly / 2 ? ky : z.Ly - ky;
    const unsigned fy = ky > z.Ly / 2 ? 2u : 0u;  // reflection parity of component p under axis i: -1 iff p = i
    const int nz = z.nz;
    const unsigned nzq = 0xffffffffu / (unsigned)nz + 1u;  // e / nz = umulhi(e, nzq) for e < 2^11, 3 <= nz <= 512
    auto comp_of = [&](int e) { return (int)__umulhi((unsigned)e, nzq); };
    const C* green = reinterpret_cast<const C*>(z.green);
    const long long tstride = (long long)z.Ox * z.Oy * z.Oz;
    auto line = [](int n) { return (n / TB) * GS + n % TB; };
    // the largest key of the lanes on one column, TB apart, to the column's line of component a
    auto collect = [&](unsigned key, unsigned* dst, int a) {
#pragma unroll
        for (int d = TB; d < 32; d *= 2) key = max(key, __shfl_xor_sync(0xffffffffu, key, d));
        if (lane < TB) atomicMax(dst + a * TB + lane, key);
    };

#pragma unroll 1
    for (int r = 0; r < z.R; ++r) {
        C* base = reinterpret_cast<C*>(z.w) + (long long)r * 3 * nz * plane + (long long)py * z.Lx + sc0;
        for (int i0 = tid - lane; i0 < 3 * nz * TB; i0 += 4 * NT) {  // four loads in flight
            C v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int idx = i0 + q * NT + lane;
                v[q] = idx < 3 * nz * TB ? base[(idx / TB) * plane + idx % TB] : C{};
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int idx = i0 + q * NT + lane, e = min(idx / TB, 3 * nz - 1), a = comp_of(e);
                if (idx < 3 * nz * TB) s[a * GS + (e - a * nz) * TB + idx % TB] = v[q];
                if constexpr (F64) {
                    const unsigned key = fx_key(v[q]);
                    if (__all_sync(0xffffffffu, a == __shfl_sync(0xffffffffu, a, 0)))
                        collect(key, kin, a);
                    else
                        atomicMax(kin + a * TB + lane % TB, key);
                }
            }
        }
        __syncthreads();
        int top = 0;
        if constexpr (F64) {
            for (int w = tid; w < NL * B; w += NT) {
                const int ln = w % NL, b = w / NL;
                const FxScale sc(kin[ln], fx_room(A / 2));
                fx2* p = f + line(ln);
                fx2 v[A];
#pragma unroll
                for (int a = 0; a < A / 2; ++a) {
                    const int l = b + B * a;
                    v[a] = l < nz ? sc(*reinterpret_cast<const double2*>(p + l * TB)) : fx2{0, 0};
                }
                fft2::dft_half_in<A>(v, -1);
                unsigned key = 0;
#pragma unroll
                for (int k1 = 0; k1 < A; ++k1) {
                    if (k1 && b) v[k1] = cmul(v[k1], twi[b * k1]);
                    p[(b + B * k1) * TB] = v[k1];
                    key |= fx_key(v[k1]);
                }
                atomicOr(kfwd + ln, key);
            }
            __syncthreads();
            // the spectrum becomes FP64 numbers relative to its largest exponent: none of them, nor of the product, is subnormal
            // or out of range for the size of the inputs
            const int n = lane % NL;
            top = __reduce_max_sync(0xffffffffu, FxScale(kin[n], fx_room(A / 2)).ex + excess(kfwd[n], B));
            for (int w = tid; w < NL * A; w += NT) {
                const int ln = w % NL, k1 = w / NL;
                const int k = excess(kfwd[ln], B), ex = FxScale(kin[ln], fx_room(A / 2)).ex + k - top;
                fx2* p = f + line(ln) + B * k1 * TB;
                fx2 v[B];
#pragma unroll
                for (int b = 0; b < B; ++b) v[b] = fx_shift(p[b * TB], k);
                fft2::DFT<B, fx2>::run(v, -1);
#pragma unroll
                for (int k2 = 0; k2 < B; ++k2) *reinterpret_cast<double2*>(p + k2 * TB) = fx_double(v[k2], ex);
            }
            __syncthreads();
        } else {
            fft2::forward<LZ, NT>(s, NL, line, TB, twf, nz);
        }
        // block product
        static_assert(NT % TB == 0, "a thread stays on one column");
        unsigned key[3] = {0, 0, 0};
        for (int i = tid; i < LZ * TB; i += NT) {
            const int c = i % TB, p = i / TB;
            const int kz = fft2::freq_at(LZ, p), kx = z.colkx ? z.colkx[sc0 + c] : sc0 + c;
            const int kzo = kz <= LZ / 2 ? kz : LZ - kz, kxo = kx <= z.Lx / 2 ? kx : z.Lx - kx;
            const unsigned m = fy | (kx > z.Lx / 2 ? 1u : 0u) | (kz > LZ / 2 ? 4u : 0u);
            C x[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) x[a] = s[a * GS + i];
            point3<C>(green + ((long long)kzo * z.Oy + kyo) * z.Ox + kxo, tstride, m, x);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                s[a * GS + i] = x[a];
                if constexpr (F64) key[a] = max(key[a], fx_key(x[a]));
            }
        }
        if constexpr (F64) {
#pragma unroll
            for (int a = 0; a < 3; ++a) collect(key[a], kout, a);
        }
        __syncthreads();
        if constexpr (F64) {
            // an Inf or NaN reaches every component
            const bool bad = __any_sync(0xffffffffu, max(kin[lane % NL], kout[lane % NL]) >= 0x7ff00000u);
            for (int w = tid; w < NL * A; w += NT) {
                const int ln = w % NL, k1 = w / NL;
                const FxScale sc(kout[ln], fx_room(B));
                fx2* p = f + line(ln) + B * k1 * TB;
                fx2 v[B];
                unsigned key = 0;
#pragma unroll
                for (int k2 = 0; k2 < B; ++k2) v[k2] = sc(*reinterpret_cast<const double2*>(p + k2 * TB));
                fft2::DFT<B, fx2>::run(v, +1);
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    if (b && k1) v[b] = cmul(v[b], fx_conj(twi[b * k1]));
                    p[b * TB] = v[b];
                    key |= fx_key(v[b]);
                }
                atomicOr(kmid + ln, key);
            }
            __syncthreads();
            for (int w = tid; w < NL * B; w += NT) {
                const int ln = w % NL, b = w / NL;
                const int k = excess(kmid[ln], A), ex = FxScale(kout[ln], fx_room(B)).ex + k + top;
                const fx2* p = f + line(ln);
                fx2 v[A];
#pragma unroll
                for (int k1 = 0; k1 < A; ++k1) v[k1] = fx_shift(p[(b + B * k1) * TB], k);
                fft2::dft_half_out<A>(v, +1);
                double2* out = reinterpret_cast<double2*>(base) + (long long)(ln / TB) * nz * plane + ln % TB;
#pragma unroll
                for (int a = 0; a < A / 2; ++a) {
                    const int l = b + B * a;
                    if (l < nz) {
                        double2 o = fx_double(v[a], ex);
                        if (bad) o.x = o.y = __longlong_as_double(0x7ff8000000000000ll);
                        out[l * plane] = o;
                    }
                }
            }
            __syncthreads();
            for (int i = tid; i < 4 * NL; i += NT) kin[i] = 0;
        } else {
            fft2::inverse<LZ, NT>(s, NL, line, TB, twf, nz);
            for (int idx = tid; idx < 3 * nz * TB; idx += NT) {
                const int e = idx / TB, a = comp_of(e);
                base[e * plane + idx % TB] = s[a * GS + (e - a * nz) * TB + idx % TB];
            }
        }
        __syncthreads();
    }
}

template <typename T, int LZ>
int launch_L(const vie_handle* h, const ZPArgs& z, cudaStream_t s) {
    using Cfg = ZPCfg<T, LZ>;
    // set on every call: the attribute is per device and launches may come from several threads
    VIE_CUDA(cudaFuncSetAttribute(zpwc_kernel<T, LZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem));
    const double bytes = (sizeof(T) == 8 ? 16.0 : 8.0) * (2.0 * z.R * 3 * z.nz * z.Ly * z.Lx + 6.0 * z.Ox * z.Oy * z.Oz);
    VIE_LAUNCH(sizeof(T) == 8 ? "zpass_block_pwc_f64" : "zpass_block_pwc_f32", s, bytes, (zpwc_kernel<T, LZ>),
               (unsigned)(z.Ly * (z.Lx / Cfg::TB)), Cfg::NT, Cfg::smem, z, h->tw32 + LZ, h->twfx + LZ);
    VIE_CHECK_LAUNCH();
    return VIE_OK;
}

template <typename T>
int launch(const vie_handle* h, const ZPArgs& z, cudaStream_t s) {
    switch (h->L[2]) {
        case 8: return launch_L<T, 8>(h, z, s);
        case 16: return launch_L<T, 16>(h, z, s);
        case 32: return launch_L<T, 32>(h, z, s);
        case 64: return launch_L<T, 64>(h, z, s);
        case 128: return launch_L<T, 128>(h, z, s);
        case 256: return launch_L<T, 256>(h, z, s);
        case 512: return launch_L<T, 512>(h, z, s);
    }
    set_error("PWC z pass: unsupported length");
    return VIE_EINVAL;
}

}  // namespace

int zpass_pwc(const vie_handle* h, const ZPArgs& z, bool fp64, cudaStream_t s) {
    return fp64 ? launch<double>(h, z, s) : launch<float>(h, z, s);
}
