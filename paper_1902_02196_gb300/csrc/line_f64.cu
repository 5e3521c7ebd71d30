// FP64 line transforms of the matvec's line path (Section IV-A on grids whose xy circulant is not square or is
// longer than 128), for lengths 8..512: the forward FFTs along x and y, the inverse FFT along y and the inverse
// FFT along x with the voxel-wise terms, on scaled 64-bit integers (fixed.cuh).  The FP32 counterparts are line2.cu
// (same layouts and orders) and, for the inverse along x, line_fft_kernel.
//
// The FP64 pipe of two operations per clock and SM bounded these transforms.  Measured on a 78 x 26 x 81 grid with 10
// right-hand sides (256 x 64 x 256 circulant), FP64 line kernels and these: forward x 2.69 and 0.83 ms, forward y
// 4.49 and 1.60, inverse y 4.78 and 1.47, inverse x with the voxel-wise terms 4.27 and 1.09.  They now issue in 60% of the
// cycles with 15 warps to an SM and wait for the ALU (busy 60%); the inverse x transform waits for its
// voxel-wise terms, which keep the FP64 pipe busy for 60%.
//
// Every line has its own scale, from its largest element: neighbouring lines can belong to different components or
// right-hand sides.  Before the second pass a line drops as many bits as its values exceed the room that the pass's
// worst case leaves (fx_room), so that a rounding is 2^-56 of the line's largest value or less.
//
// A CTA owns TB lines in shared memory, which arrive as doubles by cp.async.  A transform task is one line's A or
// B points in registers; the tasks of a warp are on different lines, at an odd stride.
#include "block.cuh"
#include "fft2.cuh"
#include "fixed.cuh"
#include "line2.cuh"

namespace {

enum { FORWARD = 0, INVERSE = 1, INVERSE_EPI = 2 };

template <int L>
struct Line64Cfg {
    static constexpr int TB = 4096 / L > 32 ? 32 : 4096 / L;  // lines per CTA
    static constexpr int LS = L + 1;
    static constexpr int NT = TB * fft2::Split<L>::B;  // 64..256
    static constexpr int MINB = L >= 128 ? 2 : 3;
    static constexpr size_t smem = sizeof(fx2) * (size_t)(TB * LS + L) + 8 * TB;
};

// colkx: stored position q holds frequency colkx[q] (the x transforms), or NULL: position q holds transposed
// position q (the y transforms)
template <int L, int KIND>
__global__ void __launch_bounds__(Line64Cfg<L>::NT, Line64Cfg<L>::MINB)
    line64_kernel(LineArgs a, const int* __restrict__ colkx, const int4* __restrict__ twg, MatvecEpi epi) {
    using Cfg = Line64Cfg<L>;
    constexpr int A = fft2::Split<L>::A, B = fft2::Split<L>::B, TB = Cfg::TB, LS = Cfg::LS, NT = Cfg::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* s = reinterpret_cast<fx2*>(smem_raw);
    int4* tw = reinterpret_cast<int4*>(s + TB * LS);
    unsigned* kin = reinterpret_cast<unsigned*>(tw + L);  // a line's key
    unsigned* kmid = kin + TB;                            // its key after the first pass
    const int tid = threadIdx.x;
    const int ntile = (a.nb + TB - 1) / TB;
    const long long ai = blockIdx.x / ntile;
    const int b0 = (blockIdx.x % ntile) * TB;
    const double2* in = reinterpret_cast<const double2*>(a.in) + ai * a.ia;
    double2* out = reinterpret_cast<double2*>(a.out);
    for (int m = tid; m < L; m += NT) tw[m] = twg[m];
    if (tid < 2 * TB) kin[tid] = 0;
    // contiguous lines (il or ol == 1) put one line's elements on consecutive threads, strided lines put
    // the TB lines' element l on consecutive threads
    const int nl = KIND == FORWARD ? a.n_in : L;
    for (int idx = tid; idx < TB * nl; idx += NT) {
        const int n = a.il == 1 ? idx / nl : idx % TB, q = a.il == 1 ? idx % nl : idx / TB;
        const int p = KIND != FORWARD && colkx ? fft2::tpos(L, colkx[q]) : q;
        const bool ok = b0 + n < a.nb;
        cp_async_elem(reinterpret_cast<double2*>(s) + n * LS + p,
                      ok ? in + (long long)q * a.il + (long long)(b0 + n) * a.ib : in, ok);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    // first pass: N1-point transforms, NTASK1 of them per line
    constexpr int N1 = KIND == FORWARD ? A : B, NTASK1 = L / N1;
    auto elem1 = [](int n, int t, int i) { return n * LS + (KIND == FORWARD ? t + B * i : B * t + i); };
    constexpr int NLOAD = KIND == FORWARD ? A / 2 : B;
    for (int t = tid; t < TB * NTASK1; t += NT) {
        const int n = t % TB, j = t / TB;
        unsigned key = 0;
#pragma unroll
        for (int i = 0; i < NLOAD; ++i)
            if (KIND != FORWARD || j + B * i < nl) key = max(key, fx_key(reinterpret_cast<const double2*>(s)[elem1(n, j, i)]));
        atomicMax(kin + n, key);
    }
    __syncthreads();
    for (int t = tid; t < TB * NTASK1; t += NT) {
        const int n = t % TB, j = t / TB;
        const FxScale sc(kin[n], fx_room(NLOAD));
        fx2 v[N1];
#pragma unroll
        for (int i = 0; i < NLOAD; ++i)
            v[i] = KIND != FORWARD || j + B * i < nl ? sc(reinterpret_cast<const double2*>(s)[elem1(n, j, i)]) : fx2{0, 0};
        if constexpr (KIND == FORWARD)
            fft2::dft_half_in<A>(v, -1);
        else
            fft2::DFT<B, fx2>::run(v, +1);
        unsigned key = 0;
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            if (i && j) v[i] = cmul(v[i], KIND == FORWARD ? tw[j * i] : fx_conj(tw[i * j]));
            // forward: b = j, k1 = i, back to b + B k1; inverse: k1 = j, b = i
            s[elem1(n, j, i)] = v[i];
            key |= fx_key(v[i]);
        }
        atomicOr(kmid + n, key);
    }
    __syncthreads();
    // second pass, to doubles
    constexpr int N2 = L / N1;
    for (int t = tid; t < TB * N1; t += NT) {
        const int n = t % TB, j = t / TB;
        const int k = excess(kmid[n], N2);
        const int ex = FxScale(kin[n], fx_room(NLOAD)).ex + k;
        const bool bad = kin[n] >= 0x7ff00000u;  // an Inf or NaN reaches the whole line
        auto elem2 = [&](int i) { return n * LS + (KIND == FORWARD ? B * j + i : j + B * i); };
        fx2 v[N2];
#pragma unroll
        for (int i = 0; i < N2; ++i) v[i] = fx_shift(s[elem2(i)], k);
        if constexpr (KIND == FORWARD)
            fft2::DFT<B, fx2>::run(v, -1);
        else
            fft2::dft_half_out<A>(v, +1);
#pragma unroll
        for (int i = 0; i < (KIND == FORWARD ? B : A / 2); ++i) {
            double2 o = fx_double(v[i], ex);
            if (bad) o.x = o.y = __longlong_as_double(0x7ff8000000000000ll);
            if (KIND == FORWARD || j + B * i < a.n_out) reinterpret_cast<double2*>(s)[elem2(i)] = o;
        }
    }
    __syncthreads();
    const double2* res = reinterpret_cast<const double2*>(s);
    const bool outc = a.ol == 1;
    const int no = KIND == FORWARD ? L : a.n_out;
#pragma unroll 4
    for (int idx = tid; idx < TB * no; idx += NT) {
        const int n = outc ? idx / no : idx % TB, q = outc ? idx % no : idx / TB;
        const int b = b0 + n;
        if (b >= a.nb) continue;
        const int p = KIND == FORWARD && colkx ? fft2::tpos(L, colkx[q]) : q;
        const long long o = ai * a.oa + (long long)q * a.ol + (long long)b * a.ob;
        double2 v = res[n * LS + p];
        if constexpr (KIND == INVERSE_EPI) {
            // line b = ((r nc + alpha) nz + z) ny + y, element q = x
            if (epi.conv) reinterpret_cast<double2*>(epi.conv)[o] = v;  // full-grid output: o is the voxel index
            const int plane = epi.ny * epi.nz, c = b / plane;
            const long long vox = (long long)(b - c * plane) * epi.nx + q;
            const double gl = comp_is_constant(c % epi.nc, epi.nc) ? epi.g1 : epi.g234;
            if (epi.op == VIE_OP_A) {
                const double2 xv = reinterpret_cast<const double2*>(epi.x)[o];
                v = csub(mk(gl * xv.x, gl * xv.y), cmul(reinterpret_cast<const double2*>(epi.c2)[vox], v));
            } else if (epi.op == VIE_OP_PA) {
                const double2 xv = reinterpret_cast<const double2*>(epi.x)[o];
                double2 c1 = reinterpret_cast<const double2*>(epi.c1)[vox];
                const double2 t = cmul(reinterpret_cast<const double2*>(epi.c2)[vox], v);
                const double ig = 1.0 / gl;
                if (epi.shift) c1 = csub(c1, epi.shift[c / epi.nc]);
                v = csub(cmul(c1, xv), mk(ig * t.x, ig * t.y));
            }
        }
        out[o] = v;
    }
}

template <int L, int KIND>
int launch_L(const char* name, const vie_handle* h, const LineArgs& a, const int* colkx, const MatvecEpi& e,
             cudaStream_t s) {
    using Cfg = Line64Cfg<L>;
    // the two-pass transforms take at most L/2 non-zero inputs (forward) or outputs (inverse)
    if ((KIND == FORWARD ? a.n_in : a.n_out) > L / 2 || (KIND == FORWARD ? a.n_out : a.n_in) != L) {
        set_error("line transform: a line needs at most L/2 inputs and L outputs (forward), or the reverse");
        return VIE_EINVAL;
    }
    // set on every call: the attribute is per device and launches may come from several threads
    VIE_CUDA(cudaFuncSetAttribute(line64_kernel<L, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem));
    const long long blocks = (long long)a.na * ((a.nb + Cfg::TB - 1) / Cfg::TB);
    if (blocks <= 0) return VIE_OK;
    if (blocks > 0x7fffffffLL) {
        set_error("line FFT grid too large");
        return VIE_EINVAL;
    }
    // algorithmic bytes: inputs read once, outputs written once (+ x and the coefficient maps in the epilogue)
    double bytes = 16.0 * (double)a.na * a.nb * (a.n_in + a.n_out);
    if (KIND == INVERSE_EPI && e.op != VIE_OP_NSCAT)
        bytes += 16.0 * ((double)a.na * a.nb * a.n_out + (double)h->nv * (e.op == VIE_OP_PA ? 2 : 1));
    VIE_KLAUNCH_B(name, s, bytes,
                  line64_kernel<L, KIND><<<(unsigned)blocks, Cfg::NT, Cfg::smem, s>>>(a, colkx, h->twfx + L, e));
    VIE_CHECK_LAUNCH();
    return VIE_OK;
}

template <int KIND>
int launch(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx, const MatvecEpi& e,
           cudaStream_t s) {
    switch (L) {
        case 8: return launch_L<8, KIND>(name, h, a, colkx, e, s);
        case 16: return launch_L<16, KIND>(name, h, a, colkx, e, s);
        case 32: return launch_L<32, KIND>(name, h, a, colkx, e, s);
        case 64: return launch_L<64, KIND>(name, h, a, colkx, e, s);
        case 128: return launch_L<128, KIND>(name, h, a, colkx, e, s);
        case 256: return launch_L<256, KIND>(name, h, a, colkx, e, s);
        case 512: return launch_L<512, KIND>(name, h, a, colkx, e, s);
    }
    set_error("line transform: unsupported length " + std::to_string(L));
    return VIE_EINVAL;
}

}  // namespace

int line64_forward(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx, cudaStream_t s) {
    return launch<FORWARD>(name, h, L, a, colkx, MatvecEpi{}, s);
}

int line64_inverse(const char* name, const vie_handle* h, int L, const LineArgs& a, const int* colkx,
                   const MatvecEpi* epi, cudaStream_t s) {
    return epi ? launch<INVERSE_EPI>(name, h, L, a, colkx, *epi, s) : launch<INVERSE>(name, h, L, a, colkx, MatvecEpi{}, s);
}
