// FP64 z pass of the matvec (Section IV-A) with the 12 x 12 Green block product fused between the
// forward and inverse z transforms: the FP64 counterpart of zpass_f32.cu, for the refinement
// residuals, the post-processing and the plain FP64 solver; the N block from its 60 tensors, or
// (KOP) the K block (Eq. 8, 25) from its 30.
//
// sm_103a has two FP64 operations per clock and SM, which this pass would need 290 clocks of per
// frequency point for the product alone and 110 more for the transforms.  So it runs on
// scaled integers (fixed.cuh) and on the tensor cores:
//  - a CTA owns one ky row and one mirror pair of columns and loops over groups of RB right-hand
//    sides, 24 RB lines in shared memory.  The two lines of a component share one power-of-two
//    scale, taken from their largest element and again before the second pass, and the transforms are
//    those of fft2.cuh on 64-bit integers;
//  - the block product is exact up to its last digits: with X the spectrum and B the block in 62
//    bits below their largest values (the digit tables of green_digits), both are cut into seven
//    signed 9-bit digits, X = sum_i x_i 2^(9(6-i)), and the products of digits with i + j <= 6 are
//    summed by fp16 mma.sync into FP32, where every sum is an integer below 2^22 and so exact (the
//    splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).  The dropped digits
//    are 2^-59 of the product, where FP64 rounds its operands and every sum to 2^-53;
//  - B has an exponent per octant point, and X the one that goes with it, so that a unit of the product is 2^-58 of the
//    largest product of the two at any one point (not of X's largest value times B's, which a smooth
//    field has at different kz); a component of the product is then scaled by its own largest value.  With one exponent per
//    column and one for all twelve components the linear components of smooth fields came out up to twelve
//    times further off than from the FP64 kernel (8 x 7 x 200 voxels);
//  - the accumulators start at 1.5 2^23, so that their bit patterns are the integers and no
//    conversion instruction (16 per clock) is needed.
//
// Measured, 16 right-hand sides on 64^3 voxels (Lx = Ly = Lz = 128): 15.6 ms, the FP64 kernel of the same
// structure 70.8 ms; the K block of 8 right-hand sides 6.8 ms against 29.1 ms.
//
// What bounds it: 12 warps to an SM (168 registers, 115 KB of shared memory to a CTA), which issue in 49% of the cycles 268
// instructions per point and right-hand side, half of them the product's (digits, sums, recombination).  A warp's
// wait is on its own results (1.5 cycles per instruction), on the ALU (0.6), on shared memory (0.55) and at barriers
// (0.5); the tensor cores are busy for 13%.
//
// What the integers do not keep: FP64 holds 53 bits of every value, here a value has 58 bits below the largest of its
// line and of the twelve components at its point.  A component a million times weaker than the strongest
// of its right-hand side, in an output that the strong one does not reach, loses 20 of them.
//
// Roles in the mma: the 24 x 24 real form of B (rows re, im of the outputs; columns re, im of the
// inputs) is the 16-row operand, the points that share an octant point, +-kx, +-kz and RB = 2
// right-hand sides, are its 8 columns.  A lane's share of X is then three whole complex values and
// no digit is built twice.  Rows 0..15 take one instruction; rows 16..23 fill both halves of
// another with two successive digits of B, whose products belong to successive weights.
#include <cuda_fp16.h>

#include "block.cuh"
#include "fft2.cuh"
#include "fixed.cuh"
#include "zpass_f64.cuh"

namespace {

constexpr int kD = 7;  // digits of the spectrum and of the block
constexpr unsigned kMagicBits = 0x4B400000u;  // 1.5 2^23
// 256 in each digit: makes them 0..511 in a plain bit field
constexpr unsigned long long kBias =
    256ull * ((1ull << 54) + (1ull << 45) + (1ull << 36) + (1ull << 27) + (1ull << 18) + (1ull << 9) + 1);
constexpr int kLow = -100000;  // below every exponent
constexpr int kLowest = -2000;  // below the exponents of the spectra
constexpr int kBits = 62;   // |X|, |B| < 2^62
constexpr int kShift = 66;  // Y = X B 2^-66: |Y| < 24 2^(62 + 62 - 66) < 2^63

template <int LZ>
struct ZDCfg {
    static constexpr int RB = LZ <= 256 ? 2 : 1;  // right-hand sides per group
    static constexpr int NL = 24 * RB;            // lines: RB x 12 components x 2 columns
    static constexpr int NT = LZ <= 8 ? 96 : (LZ <= 128 ? 192 : 384);
    static constexpr int MINB = LZ <= 128 ? 2 : 1;
    static constexpr int GS = 2 * LZ + 2;  // component stride: four components and two columns on distinct banks
    static constexpr int KEYS = 68 * RB;  // words for the keys, a multiple of four
    static constexpr int NTW = (fft2::Split<LZ>::A - 1) * (fft2::Split<LZ>::B - 1) + 1;  // twiddles in use
    static constexpr size_t smem = sizeof(fx2) * (size_t)(RB * 12 * GS + NTW) + sizeof(int) * KEYS +
                                   (size_t)(NT / 32) * 60 * 32 + sizeof(short) * 2 * (LZ / 2 + 2);
};

__device__ __forceinline__ void mma16(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                      unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the first of a sum: starts at 1.5 2^23
__device__ __forceinline__ void mma16s(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                       unsigned b1) {
    const float m = __uint_as_float(kMagicBits);
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(m));
}
__device__ __forceinline__ void mma8(float* c, unsigned a0, unsigned a1, unsigned b0) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(b0));
}

// Sums of digit products of weight d: S_d = sum over i + j = d of (digit i of X) (digit j of B),
// for the lane's rows g, g + 8 (s[0..3]) and g + 16 (s[4], s[5]), columns 2t and 2t + 1.  A sum of 24
// products is below 2^20.6, so an accumulator takes two of them.  Rows g + 16: the lower half of the
// instruction's rows has the even digits j, the upper one j + 1, whose products have weight d + 1 and
// come back in next[2] (carry[2] of the call before).
template <int D>
__device__ __forceinline__ void digit_sums(const unsigned (&a)[3][3][kD], const unsigned (&b)[3][kD], int* s,
                                           const unsigned* carry, unsigned* next) {
    unsigned t[6] = {0, 0, 0, 0, carry[0], carry[1]};
#pragma unroll
    for (int j = 0; j <= D; j += 2) {
        const int i = D - j;
        float c[4];
        mma16s(c, a[0][0][j], a[1][0][j], a[0][1][j], a[1][1][j], b[0][i], b[1][i]);
        if (j + 1 <= D) {
            mma16(c, a[0][2][j], a[1][2][j], a[0][2][j + 1], a[1][2][j + 1], b[2][i], b[2][i - 1]);
            mma16(c, a[0][0][j + 1], a[1][0][j + 1], a[0][1][j + 1], a[1][1][j + 1], b[0][i - 1], b[1][i - 1]);
        } else {
            mma8(c, a[0][2][j], a[1][2][j], b[2][i]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) t[q] += __float_as_uint(c[q]) - kMagicBits;
    }
    next[0] = next[1] = 0;
#pragma unroll
    for (int j = 0; j <= D; j += 4) {  // even digits two at a time: j with D - j, j + 2 with D - j - 2
        const int i = D - j;
        // digit j + 1 of the upper half (past the last one: none)
        auto up = [&](int e, int d) { return d < kD ? a[2][e][d] : 0u; };
        float c[4];
        mma16s(c, a[2][0][j], up(0, j + 1), a[2][1][j], up(1, j + 1), b[0][i], b[1][i]);
        if (j + 2 <= D) {
            mma16(c, a[2][2][j], up(2, j + 1), a[2][2][j + 2], up(2, j + 3), b[2][i], b[2][i - 2]);
            mma16(c, a[2][0][j + 2], up(0, j + 3), a[2][1][j + 2], up(1, j + 3), b[0][i - 2], b[1][i - 2]);
        } else {
            mma8(c, a[2][2][j], up(2, j + 1), b[2][i]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            t[4 + q] += __float_as_uint(c[q]) - kMagicBits;
            next[q] += __float_as_uint(c[2 + q]) - kMagicBits;
        }
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) s[q] = (int)t[q];
}

// Y = sum_d S_d 2^(9 (12 - d) - kShift) for the lane's six values
__device__ __forceinline__ void block_digits(const unsigned (&a)[3][3][kD], const unsigned (&b)[3][kD], long long* y) {
    unsigned h[2] = {0, 0}, g[2];
    int s[6], low[6];
    digit_sums<0>(a, b, s, h, g);
#pragma unroll
    for (int q = 0; q < 6; ++q) y[q] = (long long)s[q] << 42;
    digit_sums<1>(a, b, s, g, h);
#pragma unroll
    for (int q = 0; q < 6; ++q) y[q] += (long long)s[q] << 33;
    digit_sums<2>(a, b, s, h, g);
#pragma unroll
    for (int q = 0; q < 6; ++q) y[q] = fx_mad(s[q], 1 << 24, y[q]);
    digit_sums<3>(a, b, s, g, h);
#pragma unroll
    for (int q = 0; q < 6; ++q) y[q] = fx_mad(s[q], 1 << 15, y[q]);
    digit_sums<4>(a, b, s, h, g);
#pragma unroll
    for (int q = 0; q < 6; ++q) low[q] = s[q] * 64;
    digit_sums<5>(a, b, s, g, h);
    int t5[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) t5[q] = s[q] + 4;
    digit_sums<6>(a, b, s, h, g);
#pragma unroll
    for (int q = 0; q < 6; ++q) y[q] += low[q] + ((t5[q] + ((s[q] + 256) >> 9)) >> 3);
}

// Digits of one complex value as fp16 pairs (re, im), most significant first: w = v 2^sh + bias,
// fields 0..511 (the top one to 1023); the fp16 1024 + u is 0x6400 | u.  sg (+-1, +-1) flips the sign.
__device__ __forceinline__ void split_digits(fx2 v, int sh, __half2 sg, unsigned* d) {
    const unsigned long long re = (unsigned long long)(sh >= 0 ? v.x << sh : v.x >> -sh) + kBias;
    const unsigned long long im = (unsigned long long)(sh >= 0 ? v.y << sh : v.y >> -sh) + kBias;
    const unsigned rl = (unsigned)re, rh = (unsigned)(re >> 32), il = (unsigned)im, ih = (unsigned)(im >> 32);
    const unsigned lo = 0x1ffu, hi = 0x1ff0000u, mg = 0x64006400u;
    unsigned u[kD];
    u[6] = (rl & lo) | mg | ((il << 16) & hi);
    u[5] = ((rl >> 9) & lo) | mg | ((il << 7) & hi);
    u[4] = ((rl >> 18) & lo) | mg | ((il >> 2) & hi);
    u[3] = (__funnelshift_r(rl, rh, 27) & lo) | mg | (__funnelshift_r(il, ih, 11) & hi);
    u[2] = ((rh >> 4) & lo) | mg | ((ih << 12) & hi);
    u[1] = ((rh >> 13) & lo) | mg | ((ih << 3) & hi);
    u[0] = ((rh >> 22) & 0x3ffu) | mg | ((ih >> 6) & 0x3ff0000u);
    const __half2 off = __hmul2(sg, __float2half2_rn(-1280.f));  // 1024 + 256
#pragma unroll
    for (int i = 0; i < kD; ++i) {
        const __half2 r = __hfma2(*reinterpret_cast<__half2*>(&u[i]), sg, off);
        d[i] = *reinterpret_cast<const unsigned*>(&r);
    }
}

__device__ __forceinline__ int pos_of(int L, int k) { return fft2::tpos(L, k); }

template <int LZ, bool KOP>
__global__ void __launch_bounds__(ZDCfg<LZ>::NT, ZDCfg<LZ>::MINB)
    zfused64_kernel(ZDArgs z, const int4* __restrict__ twg) {
    using Cfg = ZDCfg<LZ>;
    constexpr int NG = KOP ? 30 : 60;  // tensors per octant point
    constexpr int A = fft2::Split<LZ>::A, B = fft2::Split<LZ>::B, NT = Cfg::NT, RB = Cfg::RB, GS = Cfg::GS, NL = Cfg::NL;
    // bits of the inputs of the two passes of the forward transform, and of the inverse one
    constexpr int TF1 = fx_room(A / 2), TF2 = fx_room(B), TI1 = fx_room(B);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* s = reinterpret_cast<fx2*>(smem_raw);
    int4* tw = reinterpret_cast<int4*>(s + RB * 12 * GS);
    // per right-hand side and component: keys of the inputs, after the first forward pass, of the product and after the
    // first inverse pass; the spectrum's exponent; per right-hand side the product's exponent in both
    // columns, and the components that an Inf or NaN of the inputs reaches; those that one of the tensors reaches
    unsigned* kin = reinterpret_cast<unsigned*>(tw + Cfg::NTW);
    unsigned *kfwd = kin + 12 * RB, *kout = kfwd + 12 * RB, *kmid = kout + 12 * RB;
    int *sex = reinterpret_cast<int*>(kmid + 12 * RB), *pex = sex + 12 * RB, *bad = pex + 2 * RB,
        *gbad = bad + RB;  // [2 columns]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // the digits of the warp's next octant point, copied while the current one is multiplied
    uint4* gbuf = reinterpret_cast<uint4*>(kin + Cfg::KEYS) + wid * (NG * 2);
    // exponents of B at the octant points of the two columns
    short* bex = reinterpret_cast<short*>(reinterpret_cast<uint4*>(kin + Cfg::KEYS) + NT / 32 * 60 * 2);
    grid_release();
    if (z.nact) grid_wait();
    const int R = z.nact ? min(*z.nact, z.R) : z.R;
    dev_bytes_add(z.bctr, 16.0 * (2.0 * R * 12 * z.nz * z.Ly * z.Lx + (double)NG * z.Ox * z.Oy * z.Oz), R > 0);
    if (R <= 0) return;
    for (int m = tid; m < Cfg::NTW; m += NT) tw[m] = twg[m];
    auto reset = [&] {
        for (int i = tid; i < 48 * RB; i += NT) kin[i] = 0;
        if (tid < 2 * RB) pex[tid] = kLow;
    };
    reset();
    if (tid < 2) gbad[tid] = 0;
    __syncthreads();
    const int ntile = z.Lx / 2;
    const int py = blockIdx.x / ntile, ct = blockIdx.x % ntile, sc0 = 2 * ct;
    const long long plane = (long long)z.Ly * z.Lx;
    const int ky = py / z.by + z.ay * (py % z.by);
    const int kyo = ky <= z.Ly / 2 ? ky : z.Ly - ky;
    const unsigned fy = ky > z.Ly / 2 ? z.my : 0u;
    const bool ry = ky > z.Ly / 2;
    const int nz = z.nz;
    const unsigned nzq = 0xffffffffu / (unsigned)nz + 1u;  // idx / nz = umulhi(idx, nzq) for idx < 2^14, 3 <= nz <= 512
    const bool single = ct == ntile - 1;  // columns 0 and Lx/2: own octant columns
    const int kx0 = z.colkx[sc0], kx1 = z.colkx[sc0 + 1];
    const int kxo0 = kx0 <= z.Lx / 2 ? kx0 : z.Lx - kx0, kxo1 = kx1 <= z.Lx / 2 ? kx1 : z.Lx - kx1;
    const unsigned fx0 = kx0 > z.Lx / 2 ? z.mx : 0u, fx1 = kx1 > z.Lx / 2 ? z.mx : 0u;
    const int gc0 = kyo * z.Ox + kxo0, gc1 = kyo * z.Ox + kxo1;

    // block-product roles of this lane.  Points (mma columns) 0..7: bit 0 the column, bit 1 the sign of
    // kz, bit 2 the right-hand side; n is the point whose X this lane splits, components t, t + 4, t + 8.
    const int n = lane >> 2, t = lane & 3;
    const int ncol = n & 1, nneg = (n >> 1) & 1, nr_ = n >> 2;
    const int qcol = t & 1;  // of the outputs (points 2t, 2t + 1): the sign of kz; t >> 1 the right-hand side
    const int ra = (lane >> 2) >> 1, part = (lane >> 2) & 1;  // output rows: components ra, ra + 4, ra + 8, re or im
    // B: entry (row component 4 p + ra, input 4 q + t): scalar pair (ra, t), vector pair (p, q)
    const int l0 = min(ra, t), l1 = max(ra, t);
    const int ll = l0 == 0 ? l1 : (l0 == 1 ? 3 + l1 : (l0 == 2 ? 5 + l1 : 9));  // ll_index
    const bool swapneg = ra > t && (((ra > 0) + (t > 0)) & 1);  // l > l' with one of them constant: sign -1
    // re rows take (Br, -Bi), im rows (Bi, Br)
    const unsigned bsel = part ? 0x1032u : 0x3210u;
    const unsigned bneg = (part ? 0u : 0x80000000u) ^ (swapneg ? 0x80008000u : 0u);

    // exponents of the points and the raises of the two columns' linear functions (the last word of tensor 0), and the
    // outputs that a tensor with an Inf or NaN reaches (that of tensor 1)
    constexpr int NO = LZ / 2 + 1;
    auto point_word = [&](int c, int ko, int t) {
        return reinterpret_cast<const int*>(z.green_d)[(((long long)(c ? gc1 : gc0) * z.Oz + ko) * NG + t) * 8 + 7];
    };
    for (int i = tid; i < 2 * NO; i += NT) {
        const int c = i / NO, ko = i % NO, w = point_word(c, ko, 1);
        bex[i] = (short)(point_word(c, ko, 0) >> 8);
        if (w) atomicOr(gbad + c, w);
    }
    const int up0 = point_word(0, 0, 0) & 255, up1 = point_word(1, 0, 0) & 255;
    // octant points q of this CTA: 0..LZ/2, for each column when the columns are self-mirrored
    constexpr int NW = NT / 32;
    const int nq = single ? 2 * NO : NO;
    auto fetch = [&](int q) {
        const bool col = q >= NO;
        const uint4* src = z.green_d + ((long long)(col ? gc1 : gc0) * z.Oz + (q - (col ? NO : 0))) * (NG * 2);
        for (int i = lane; i < NG * 2; i += 32) cp_async16(gbuf + i, src + i);
        cp_async_commit();
    };
    if (wid < nq) fetch(wid);
    grid_wait();

#pragma unroll 1
    for (int r0 = 0; r0 < R; r0 += RB) {
        const int nr = min(RB, R - r0);
        // load, with the largest element of each component
#pragma unroll 1
        for (int rr = 0; rr < nr; ++rr) {
            const double2* base = z.w + (long long)(r0 + rr) * 12 * nz * plane + (long long)py * z.Lx + sc0;
#pragma unroll 1
            for (int i0 = tid - lane; i0 < 24 * nz; i0 += 8 * NT) {  // eight loads in flight
                double2 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int idx = i0 + q * NT + lane;
                    v[q] = idx < 24 * nz ? base[(long long)(idx >> 1) * plane + (idx & 1)] : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int idx = i0 + q * NT + lane, e = min(idx >> 1, 12 * nz - 1);
                    const int a = (int)__umulhi((unsigned)e, nzq);
                    if (idx < 24 * nz) *reinterpret_cast<double2*>(s + (rr * 12 + a) * GS + 2 * (e - a * nz) + (idx & 1)) = v[q];
                    const unsigned key = fx_key(v[q]);
                    if (__all_sync(0xffffffffu, a == __shfl_sync(0xffffffffu, a, 0))) {
                        const unsigned m = __reduce_max_sync(0xffffffffu, key);
                        if (lane == 0) atomicMax(kin + rr * 12 + a, m);
                    } else {
                        atomicMax(kin + rr * 12 + a, key);
                    }
                }
            }
        }
        __syncthreads();
        // forward z transform; pass 1 (A points, the upper half zero) converts to fixed point
        for (int w = tid; w < NL * B; w += NT) {
            const int ln = w % NL, b = w / NL, rr = ln / 24;
            if (RB > 1 && rr >= nr) continue;
            const FxScale sc(kin[ln >> 1], TF1);
            fx2* p = s + (ln >> 1) * GS + (ln & 1);
            fx2 v[A];
#pragma unroll
            for (int a = 0; a < A / 2; ++a) {
                const int l = b + B * a;
                v[a] = l < nz ? sc(*reinterpret_cast<const double2*>(p + 2 * l)) : fx2{0, 0};
            }
            fft2::dft_half_in<A>(v, -1);
#pragma unroll
            for (int k1 = 1; k1 < A; ++k1)
                if (b) v[k1] = cmul(v[k1], tw[b * k1]);
            unsigned m = 0;
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) {
                p[2 * (b + B * k1)] = v[k1];
                m |= fx_key(v[k1]);
            }
            atomicOr(kfwd + (ln >> 1), m);
        }
        __syncthreads();
        for (int w = tid; w < NL * A; w += NT) {
            const int ln = w % NL, k1 = w / NL;
            if (RB > 1 && ln / 24 >= nr) continue;
            const int k = excess(kfwd[ln >> 1], B);
            fx2* p = s + (ln >> 1) * GS + (ln & 1) + 2 * B * k1;
            fx2 v[B];
#pragma unroll
            for (int b = 0; b < B; ++b) v[b] = fx_shift(p[2 * b], k);
            fft2::DFT<B, fx2>::run(v, -1);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) p[2 * k2] = v[k2];
        }
        if (wid == 0) {  // a component with an Inf or NaN: so far down that the product has a unit of it at most
            const bool in = lane < 12 * RB, nan = in && kin[lane] >= 0x7ff00000u;
            if (in) sex[lane] = nan ? kLowest : FxScale(kin[lane], TF1).ex + excess(kfwd[lane], B);
            const unsigned m = __ballot_sync(0xffffffffu, nan) >> (12 * (lane % RB)) & 0xFFFu;
            // it reaches every output, through K those of the other two directions
            if (lane < RB)
                bad[lane] = KOP ? (m & 0xFF0 ? 0xF : 0) | (m & 0xF0F ? 0xF0 : 0) | (m & 0xFF ? 0xF00 : 0) : (m ? 0xFFF : 0);
        }
        __syncthreads();
        // The product's exponent: the largest, over the points, of the spectrum's exponent less that of B.  (In a pass of its
        // own: an exponent per point would be a reduction between the product's loads and its digits.)
        for (int w = tid; w < 2 * LZ * RB; w += NT) {  // whole warps
            const int c = w & 1, pos = (w >> 1) % LZ, rr = w / (2 * LZ), kz = fft2::freq_at(LZ, pos);
            const fx2* p = s + rr * 12 * GS + 2 * pos + c;
            int ec = kLow, el = kLow;
#pragma unroll
            for (int a = 0; a < 12; ++a) {
                const int e = fx_bits(fx_key(p[a * GS])) + sex[rr * 12 + a];
                if (a % 4)
                    el = max(el, e);
                else
                    ec = max(ec, e);
            }
            int g = max(ec, el - (c ? up1 : up0)) - bex[c * NO + (kz <= LZ / 2 ? kz : LZ - kz)];
            if (single || LZ < 16) {
                atomicMax(pex + 2 * rr + c, g);
                if (!single) atomicMax(pex + 2 * rr + (c ^ 1), g);
            } else {
                g = __reduce_max_sync(0xffffffffu, g);
                if (lane < 2) atomicMax(pex + 2 * rr + lane, g);
            }
        }
        __syncthreads();
        // block product, a warp per octant point
        {
            const int nrx = RB == 1 ? 0 : nr_;
            const bool nval = RB == 1 ? nr_ == 0 : nr_ < nr;
            const int rout = t >> 1;
            const bool oval = RB == 1 ? rout == 0 : rout < nr;
            // exponents of this lane's components t, t + 4, t + 8
            int xe[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) xe[e] = sex[nrx * 12 + t + 4 * e];
            const int xlift = kBits - pex[2 * nrx + ncol] - (t ? (ncol ? up1 : up0) : 0);
            unsigned key[3] = {0, 0, 0};  // of the lane's outputs, components ra, ra + 4, ra + 8
            for (int q = wid; q < nq; q += NW) {
                const int col = q >= NO, ko = q - (col ? NO : 0);
                const bool self = ko == 0 || ko == LZ / 2;
                // the point's exponent and digits of B: rows ra + 4 p, inputs t + 4 q
                unsigned a[3][3][kD];
                cp_async_wait<0>();
                __syncwarp();
                // of X, less B's exponent (its columns share an octant point unless they are self-mirrored)
                const int lift = xlift - ((int)gbuf[1].w >> 8);
#pragma unroll
                for (int p = 0; p < 3; ++p)
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        const bool zero = KOP && p == e;
                        const int tens = (KOP ? 10 * (3 - p - e) : 10 * pq_index(p, e)) + ll;
                        const unsigned neg = bneg ^ (KOP && kblock::levi_civita(p, 3 - p - e, e) > 0 ? 0x80008000u : 0u);
                        const uint4 g = zero ? make_uint4(0, 0, 0, 0) : gbuf[tens * 2];
                        const uint4 f = zero ? make_uint4(0, 0, 0, 0) : gbuf[tens * 2 + 1];
                        const unsigned v[kD] = {g.x, g.y, g.z, g.w, f.x, f.y, f.z};
#pragma unroll
                        for (int d = 0; d < kD; ++d) a[p][e][d] = zero ? 0u : __byte_perm(v[d], 0, bsel) ^ neg;
                    }
                __syncwarp();
                fetch(q + NW < nq ? q + NW : wid);  // after the last one, the next group's first
                // digits of X: components t + 4 e of point n, X = spectrum 2^lift: with that, every point's product has the exponent
                // pex, and X stays below 2^62; the linear components are lower by the raise of B's linear rows and columns
                unsigned b[3][kD];
                {
                    const bool v = nval && !(nneg && self) && !(single && ncol != col);
                    const int kz = nneg && ko ? LZ - ko : ko;
                    const unsigned m = fy ^ (ncol ? fx1 : fx0) ^ (nneg ? z.mz : 0u);
                    const fx2* p = s + (nrx * 12 + t) * GS + 2 * pos_of(LZ, kz) + ncol;
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        const fx2 x = v ? p[4 * e * GS] : fx2{0, 0};
                        const __half2 sg = __float2half2_rn(((m >> (t + 4 * e)) & 1u) ? -1.f : 1.f);
                        split_digits(x, max(lift + xe[e], -62), sg, b[e]);
                    }
                }
                long long y[6];
                block_digits(a, b, y);
                __syncwarp();
                // outputs: components ra + 4 p, re or im, points 2t (column 0) and 2t + 1 (column 1)
                {
                    const int kz = qcol && ko ? LZ - ko : ko;
                    const bool rz = qcol;
                    if (oval && !(qcol && self)) {
                        long long* p = reinterpret_cast<long long*>(s + ((RB == 1 ? 0 : rout) * 12 + ra) * GS + 2 * pos_of(LZ, kz)) + part;
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            if (single && c != col) continue;
                            unsigned m = fy ^ (c ? fx1 : fx0) ^ (rz ? z.mz : 0u);
                            if (KOP && (ry ^ rz ^ ((c ? fx1 : fx0) != 0))) m ^= 0xFFFu;
#pragma unroll
                            for (int e = 0; e < 3; ++e) {
                                long long v = y[2 * e + c];
                                if ((m >> (ra + 4 * e)) & 1u) v = -v;
                                key[e] |= fx_key(v);
                                p[8 * e * GS + 2 * c] = v;
                            }
                        }
                    }
                }
                __syncwarp();
            }
            if (oval) {  // a lane's outputs belong to one right-hand side
#pragma unroll
                for (int e = 0; e < 3; ++e) atomicOr(kout + (RB == 1 ? 0 : rout) * 12 + ra + 4 * e, key[e]);
            }
        }
        __syncthreads();
        // inverse z transform, a component rescaled before each pass
        for (int w = tid; w < NL * A; w += NT) {
            const int ln = w % NL, k1 = w / NL;
            if (RB > 1 && ln / 24 >= nr) continue;
            const int k = excess(kout[ln >> 1], B);
            fx2* p = s + (ln >> 1) * GS + (ln & 1) + 2 * B * k1;
            fx2 v[B];
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k2] = fx_shift(p[2 * k2], k);
            fft2::DFT<B, fx2>::run(v, +1);
#pragma unroll
            for (int b = 1; b < B; ++b)
                if (k1) v[b] = cmul(v[b], fx_conj(tw[b * k1]));
            unsigned m = 0;
#pragma unroll
            for (int b = 0; b < B; ++b) {
                p[2 * b] = v[b];
                m |= fx_key(v[b]);
            }
            atomicOr(kmid + (ln >> 1), m);
        }
        __syncthreads();
        for (int w = tid; w < NL * B; w += NT) {
            const int ln = w % NL, b = w / NL, rr = ln / 24;
            if (RB > 1 && rr >= nr) continue;
            const fx2* p = s + (ln >> 1) * GS + (ln & 1);
            const int k = excess(kmid[ln >> 1], A);
            fx2 v[A];
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) v[k1] = fx_shift(p[2 * (b + B * k1)], k);
            fft2::dft_half_out<A>(v, +1);
            const int comp = (ln % 24) >> 1, c = ln & 1;
            const bool nan = ((bad[rr] | gbad[c]) >> comp) & 1;
            // exponent of the result: that of the product and the bits dropped since
            const int ex = pex[2 * rr + c] - (comp % 4 ? (c ? up1 : up0) : 0) - kBits + kShift + excess(kout[ln >> 1], B) + k;
            double2* out = z.w + (long long)(r0 + rr) * 12 * nz * plane + (long long)py * z.Lx + sc0 + c;
            auto store = [&](auto to_double) {
#pragma unroll
                for (int a = 0; a < A / 2; ++a) {
                    const int l = b + B * a;
                    if (l < nz) {
                        double2 o = to_double(v[a], ex);
                        if (nan) o.x = o.y = __longlong_as_double(0x7ff8000000000000ll);
                        out[((long long)comp * nz + l) * plane] = o;
                    }
                }
            };
            if (fx_in_range(ex))
                store([](fx2 u, int e) { return fx_double<true>(u, e); });
            else
                store([](fx2 u, int e) { return fx_double(u, e); });
        }
        __syncthreads();
        reset();
        __syncthreads();
    }
    cp_async_wait<0>();
}

// Digit tables from the octant spectra g [NG][Oz][Oy][Ox].  Every octant point has an exponent be and every column a raise
// up: an entry B is stored as seven signed 9-bit digits of B 2^(be + c up), c the number of linear functions in its pair,
// below 2^62; be << 8 | up is in the unused last word of tensor 0, and
// in that of tensor 1 a mask of the outputs whose rows have an Inf or a NaN at that point (stored as zero).  The raise brings the linear rows and columns
// up to the constant ones (their Gram entries are 1/12, and where the spectrum is large they couple through
// differences); it is the largest that leaves the pairs of constant functions the largest values, give or
// take a bit or two.
// A block takes kDigitCols neighbouring columns, whose values of one (tensor, kz) are 128 contiguous bytes, and reads
// them twice; the digits of a value are 32 contiguous bytes.
constexpr int kDigitCols = 8, kMaxOz = 257;
__global__ void __launch_bounds__(256) digits_kernel(const double2* __restrict__ g, int Ox, int Oy, int Oz, int NG,
                                                     uint4* __restrict__ d) {
    __shared__ int top[3][kMaxOz][kDigitCols];  // per class of pairs: |B| < 2^(top - 1022); then [0]: be
    __shared__ int ctop[3][kDigitCols];         // the same over a column
    __shared__ unsigned reach[kMaxOz][kDigitCols];
    const int c = threadIdx.x % kDigitCols, kx = blockIdx.x * kDigitCols + c, ky = blockIdx.y;
    for (int i = threadIdx.x; i < 3 * kMaxOz * kDigitCols; i += 256) (&top[0][0][0])[i] = kLow;
    for (int i = threadIdx.x; i < kMaxOz * kDigitCols; i += 256) (&reach[0][0])[i] = 0;
    if (threadIdx.x < 3 * kDigitCols) (&ctop[0][0])[threadIdx.x] = kLow;
    __syncthreads();
    const int n = NG * Oz;
    auto linear = [](int t) {  // linear functions in the pair
        const int ll = t % 10;
        return ll == 0 ? 0 : (ll < 4 ? 1 : 2);
    };
    auto outputs_of = [&](int t) {
        unsigned m = 0;
        if (NG == 60)
            for (int i = kBlock.start[t]; i < kBlock.start[t + 1]; ++i) m |= 1u << kBlock.e[i].a;
        else
            for (int i = kKBlock.start[t]; i < kKBlock.start[t + 1]; ++i) m |= 1u << kKBlock.e[i].a;
        return m;
    };
    if (kx < Ox)
        for (int i = threadIdx.x / kDigitCols; i < n; i += 256 / kDigitCols) {
            const int t = i / Oz, kz = i - t * Oz;
            double2 v = g[((long long)i * Oy + ky) * Ox + kx];
            int e = (int)(fx_key(v) >> 20);
            if (e >= 2047) {
                atomicOr(&reach[kz][c], outputs_of(t));
                continue;
            }
            if (e == 0) {  // subnormal numbers
                v = make_double2(0x1p64 * v.x, 0x1p64 * v.y);
                e = v.x == 0.0 && v.y == 0.0 ? kLow : (int)(fx_key(v) >> 20) - 64;
            }
            atomicMax(&top[linear(t)][kz][c], e);
        }
    __syncthreads();
    for (int q = 0; q < 3; ++q)
        for (int kz = threadIdx.x / kDigitCols; kz < Oz; kz += 256 / kDigitCols) atomicMax(&ctop[q][c], top[q][kz][c]);
    __syncthreads();
    const int up = min(max(min((ctop[0][c] - ctop[2][c] + 1) >> 1, ctop[0][c] - ctop[1][c] + 2), 0), 60);
    for (int kz = threadIdx.x / kDigitCols; kz < Oz; kz += 256 / kDigitCols) {
        const int e = max(top[0][kz][c], max(top[1][kz][c] + up, top[2][kz][c] + 2 * up));
        top[0][kz][c] = e > kLow / 2 ? kBits + 1022 - e : 0;
    }
    __syncthreads();
    if (kx >= Ox) return;
    const long long col = (long long)ky * Ox + kx;
    for (int i = threadIdx.x / kDigitCols; i < n; i += 256 / kDigitCols) {
        const int t = i / Oz, kz = i - t * Oz;
        const int be = top[0][kz][c], sc = be + linear(t) * up;
        double2 v = g[((long long)i * Oy + ky) * Ox + kx];
        if (fx_key(v) >= 0x7ff00000u) v = make_double2(0.0, 0.0);
        if (sc > 1000 || sc < -1000) {
            v = make_double2(scalbn(v.x, sc), scalbn(v.y, sc));
        } else {
            const double f = __hiloint2double((1023 + sc) << 20, 0);
            v = make_double2(f * v.x, f * v.y);
        }
        unsigned long long re = (unsigned long long)__double2ll_rn(v.x) + kBias;
        unsigned long long im = (unsigned long long)__double2ll_rn(v.y) + kBias;
        unsigned u[8] = {};
#pragma unroll
        for (int q = kD - 1; q >= 0; --q) {
            const int mask = q ? 511 : 1023;
            const __half2 h = __halves2half2(__int2half_rn((int)(re & mask) - 256), __int2half_rn((int)(im & mask) - 256));
            u[q] = *reinterpret_cast<const unsigned*>(&h);
            re >>= 9;
            im >>= 9;
        }
        uint4* out = d + 2 * ((col * Oz + kz) * NG + t);
        out[0] = make_uint4(u[0], u[1], u[2], u[3]);
        out[1] = make_uint4(u[4], u[5], u[6], t == 0 ? (unsigned)(be << 8 | up) : (t == 1 ? reach[kz][c] : 0u));
    }
}

template <int LZ, bool KOP>
int launch_zd_L(const vie_handle* h, const ZDArgs& z, cudaStream_t s) {
    constexpr size_t smem = ZDCfg<LZ>::smem;
    constexpr double NG = KOP ? 30.0 : 60.0;
    // set on every call: the attribute is per device and launches may come from several threads
    VIE_CUDA(cudaFuncSetAttribute(zfused64_kernel<LZ, KOP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const long long blocks = (long long)z.Ly * (z.Lx / 2);
    const double bytes = z.nact ? kDevCounted : 16.0 * (2.0 * z.R * 12 * z.nz * z.Ly * z.Lx + NG * z.Ox * z.Oy * z.Oz);
    VIE_LAUNCH(KOP ? "zpass_block_k_f64" : "zpass_block_f64", s, bytes, (zfused64_kernel<LZ, KOP>), (unsigned)blocks,
               ZDCfg<LZ>::NT, smem, z, h->twfx + LZ);
    VIE_CHECK_LAUNCH();
    return VIE_OK;
}

template <bool KOP>
int launch_zd(const vie_handle* h, const ZDArgs& z, cudaStream_t s) {
    switch (h->L[2]) {
        case 8: return launch_zd_L<8, KOP>(h, z, s);
        case 16: return launch_zd_L<16, KOP>(h, z, s);
        case 32: return launch_zd_L<32, KOP>(h, z, s);
        case 64: return launch_zd_L<64, KOP>(h, z, s);
        case 128: return launch_zd_L<128, KOP>(h, z, s);
        case 256: return launch_zd_L<256, KOP>(h, z, s);
        case 512: return launch_zd_L<512, KOP>(h, z, s);
    }
    set_error("FP64 z pass: unsupported length");
    return VIE_EINVAL;
}

}  // namespace

int green_digits(const vie_handle* h, const double2* g, int ng, uint4* d, cudaStream_t s) {
    const dim3 grid((unsigned)((h->O[0] + kDigitCols - 1) / kDigitCols), (unsigned)h->O[1]);
    VIE_KLAUNCH("green_digits", s,
                digits_kernel<<<grid, 256, 0, s>>>(g, h->O[0], h->O[1], h->O[2], ng, d));
    VIE_CHECK_LAUNCH();
    return VIE_OK;
}

int zpass_f64_fused(const vie_handle* h, const ZDArgs& z, cudaStream_t s) { return launch_zd<false>(h, z, s); }

int zpass_f64_fused_k(const vie_handle* h, const ZDArgs& z, cudaStream_t s) { return launch_zd<true>(h, z, s); }
