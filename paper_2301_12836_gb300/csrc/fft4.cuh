// fft4.cuh - compile-time two-step ("four-step") FFT.
//
// A line of length L = A * B is transformed as
//   Y[t][k1] = W_L^(t k1) * sum_a x[t + B a] W_A^(a k1)      (B DFTs of length A, then twiddles)
//   X[k1 + A k2] = sum_t Y[t][k1] W_B^(t k2)                  (A DFTs of length B)
// with every short DFT held in registers and one exchange through shared memory between the steps.  A
// tile of NL lines is transformed by NL * min(A, B) threads: thread tid works on line tid % NL.
#pragma once
#include "fft.cuh"
#include <type_traits>

namespace lsm {

template <int S, typename C>
__device__ __forceinline__ C cmul_const(C a, double re, double im_s) {
    // multiply by (re + S * i * im_s)
    typedef typename real_of<C>::type T;
    const T cr = (T)re, ci = (T)(S * im_s);
    return mkc<C>(a.x * cr - a.y * ci, a.x * ci + a.y * cr);
}

// 16-point DFT in registers, natural order in and out: n = 4 n1 + n2, k = k1 + 4 k2.
// HALF: inputs 8..15 are zero, i.e. n1 = 2, 3 vanish in every first-layer 4-point DFT.
template <int S, bool HALF = false, typename C> __device__ __forceinline__ void bfly16(C* v) {
    const double c1 = 0.92387953251128675613;  // cos(pi/8)
    const double s1 = 0.38268343236508977173;  // sin(pi/8)
    const double r2 = 0.70710678118654752440;  // 1/sqrt(2)
    C y[16];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
        C a[4] = {v[n2], v[4 + n2], v[8 + n2], v[12 + n2]};
        if (HALF) bfly4_half<S>(a);
        else bfly4<S>(a);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) y[n2 * 4 + k1] = a[k1];
    }
    // twiddles W16^(n2 k1), W16^m = cos(2 pi m/16) + S i sin(2 pi m/16)
    y[5] = cmul_const<S>(y[5], c1, s1);      // m = 1
    y[6] = cmul_const<S>(y[6], r2, r2);      // m = 2
    y[7] = cmul_const<S>(y[7], s1, c1);      // m = 3
    y[9] = cmul_const<S>(y[9], r2, r2);      // m = 2
    y[10] = cmul_si<S>(y[10]);               // m = 4
    y[11] = cmul_const<S>(y[11], -r2, r2);   // m = 6
    y[13] = cmul_const<S>(y[13], s1, c1);    // m = 3
    y[14] = cmul_const<S>(y[14], -r2, r2);   // m = 6
    y[15] = cmul_const<S>(y[15], -c1, -s1);  // m = 9
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        C b[4] = {y[k1], y[4 + k1], y[8 + k1], y[12 + k1]};
        bfly4<S>(b);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = b[k2];
    }
}

// 16-point DFT whose inputs NZ..15 are zero, computing only its first NO outputs: the zero
// inputs drop out of the first-layer 4-point DFTs, the unneeded outputs out of the last-layer
// ones.  NZ = NO = 16 is bfly16 operation for operation.
template <int S, int NZ, int N2, typename C> __device__ __forceinline__ void b16_first(const C* v, C* y) {
    constexpr int nz = (NZ - N2 + 3) / 4 < 1 ? 0 : ((NZ - N2 + 3) / 4 > 4 ? 4 : (NZ - N2 + 3) / 4);
    C a[4];
    if constexpr (nz == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = czero<C>();
    } else {
#pragma unroll
        for (int k = 0; k < nz; ++k) a[k] = v[N2 + 4 * k];
        bfly4p<S, nz, 4>(a);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) y[N2 * 4 + k1] = a[k1];
}
template <int S, int NO, int K1, typename C> __device__ __forceinline__ void b16_last(const C* y, C* v) {
    constexpr int no = (NO - K1 + 3) / 4 < 1 ? 0 : ((NO - K1 + 3) / 4 > 4 ? 4 : (NO - K1 + 3) / 4);
    if constexpr (no > 0) {
        C b[4] = {y[K1], y[4 + K1], y[8 + K1], y[12 + K1]};
        bfly4p<S, 4, no>(b);
#pragma unroll
        for (int k2 = 0; k2 < no; ++k2) v[K1 + 4 * k2] = b[k2];
    }
}
template <int S, int NZ, int NO, typename C> __device__ __forceinline__ void bfly16p(C* v) {
    const double c1 = 0.92387953251128675613;  // cos(pi/8)
    const double s1 = 0.38268343236508977173;  // sin(pi/8)
    const double r2 = 0.70710678118654752440;  // 1/sqrt(2)
    C y[16];
    b16_first<S, NZ, 0>(v, y);
    b16_first<S, NZ, 1>(v, y);
    b16_first<S, NZ, 2>(v, y);
    b16_first<S, NZ, 3>(v, y);
    // twiddles W16^(n2 k1), as in bfly16
    y[5] = cmul_const<S>(y[5], c1, s1);
    y[6] = cmul_const<S>(y[6], r2, r2);
    y[7] = cmul_const<S>(y[7], s1, c1);
    y[9] = cmul_const<S>(y[9], r2, r2);
    y[10] = cmul_si<S>(y[10]);
    y[11] = cmul_const<S>(y[11], -r2, r2);
    y[13] = cmul_const<S>(y[13], s1, c1);
    y[14] = cmul_const<S>(y[14], -r2, r2);
    y[15] = cmul_const<S>(y[15], -c1, -s1);
    b16_last<S, NO, 0>(y, v);
    b16_last<S, NO, 1>(y, v);
    b16_last<S, NO, 2>(y, v);
    b16_last<S, NO, 3>(y, v);
}

// W32^k a, W32^k = cos(2 pi k/32) + S i sin(2 pi k/32), k < 16 a compile-time constant after
// unrolling
template <int S, typename C> __device__ __forceinline__ C tw32(C a, int k) {
    const double c1 = 0.98078528040323044913, s1 = 0.19509032201612826785;  // cos, sin(pi/16)
    const double c2 = 0.92387953251128675613, s2 = 0.38268343236508977173;  // cos, sin(pi/8)
    const double c3 = 0.83146961230254523708, s3 = 0.55557023301960222474;  // cos, sin(3 pi/16)
    const double r2 = 0.70710678118654752440;
    switch (k) {
        case 0: return a;
        case 1: return cmul_const<S>(a, c1, s1);
        case 2: return cmul_const<S>(a, c2, s2);
        case 3: return cmul_const<S>(a, c3, s3);
        case 4: return cmul_const<S>(a, r2, r2);
        case 5: return cmul_const<S>(a, s3, c3);
        case 6: return cmul_const<S>(a, s2, c2);
        case 7: return cmul_const<S>(a, s1, c1);
        case 8: return cmul_si<S>(a);
        case 9: return cmul_const<S>(a, -s1, c1);
        case 10: return cmul_const<S>(a, -s2, c2);
        case 11: return cmul_const<S>(a, -s3, c3);
        case 12: return cmul_const<S>(a, -r2, r2);
        case 13: return cmul_const<S>(a, -c3, s3);
        case 14: return cmul_const<S>(a, -c2, s2);
        default: return cmul_const<S>(a, -c1, s1);
    }
}

// 32-point DFT in registers, natural order in and out, inputs NZ..31 zero and only the first NO
// outputs wanted: radix 2 over the 16-point DFTs E of the even and O of the odd samples,
// X[k] = E[k] + W32^k O[k] and X[k + 16] = E[k] - W32^k O[k] (k < 16).  The even samples keep
// (NZ + 1) / 2 nonzero inputs, the odd ones NZ / 2, and both halves need outputs k < min(NO, 16).
template <int S, int NZ, int NO, typename C> __device__ __forceinline__ void bfly32p(C* v) {
    constexpr int NZE = (NZ + 1) / 2, NZO = NZ / 2, NH = NO < 16 ? NO : 16;
    C e[16], o[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        e[j] = v[2 * j];
        o[j] = v[2 * j + 1];
    }
    bfly16p<S, NZE, NH>(e);
    if constexpr (NZO >= 1) bfly16p<S, NZO, NH>(o);
#pragma unroll
    for (int k = 0; k < NH; ++k) {
        const C t = NZO >= 1 ? tw32<S>(o[k], k) : czero<C>();
        v[k] = cadd(e[k], t);
        if (k + 16 < NO) v[k + 16] = csub(e[k], t);
    }
}

// Fixed-point 32-point DFT times 1/4 (all inputs, first NO outputs), in two units.  Radix 8 over
// the samples t = 4 a + b in the inputs' unit, products with W32^(b k) / 4 into a unit four times
// coarser, and a last radix-4 layer of additions alone.  As 2 x 16 points in one unit (every inner
// product rounded in the outputs' unit, which had to leave one bit more of headroom), an inverse
// 512-point line of a Green-multiplied spectrum had 1.8 to 3.7 times the FP64 engine's error; it has
// 0.49 to 0.88 of it.  256^3 FP64 apply 20.03 -> 20.09 ms.
template <int S> __device__ __forceinline__ fxc fx_tw32_quarter(fxc a, int k) {
    const double c[8] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                         0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173, 0.19509032201612826785};
    const int q = k >> 3, j = k & 7;
    if (j == 0) {   // +-1, +-i
        const fxc r{fx_r((fx_ll(a.x) + 2) >> 2), fx_r((fx_ll(a.y) + 2) >> 2)};
        return q == 0 ? r : cmul_si<S>(r);   // k < 22: 0 or 8 here
    }
    const long long kc = fx_const(c[j]), ks = fx_const(c[8 - j]);   // cos, sin(2 pi j / 32)
    const long long re = q == 0 ? kc : (q == 1 ? -ks : -kc), im = q == 0 ? ks : (q == 1 ? kc : -ks);
    return fx_cmul_quarter(a, re, S * im);
}
template <int S> __device__ __forceinline__ void fx_bfly8_wide(fxc* v) {   // bfly8 for sums below 2^62.6
    const long long r2 = fx_const(0.70710678118654752440);
    fxc e[4] = {v[0], v[2], v[4], v[6]};
    fxc o[4] = {v[1], v[3], v[5], v[7]};
    bfly4<S>(e);
    bfly4<S>(o);
    // o[1] (1 + S i) / sqrt2 and o[3] (-1 + S i) / sqrt2 from sums and differences
    const fxr s1 = fx_scale_wide(fx_add(o[1].x, o[1].y), r2), d1 = fx_scale_wide(fx_sub(o[1].x, o[1].y), r2);
    const fxr s3 = fx_scale_wide(fx_add(o[3].x, o[3].y), r2), d3 = fx_scale_wide(fx_sub(o[3].x, o[3].y), r2);
    const fxc o1 = S > 0 ? fxc{d1, s1} : fxc{s1, fx_neg(d1)};
    const fxc o3 = S > 0 ? fxc{fx_neg(s3), d3} : fxc{fx_neg(d3), fx_neg(s3)};
    v[0] = cadd(e[0], o[0]);       v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], o1);         v[5] = csub(e[1], o1);
    v[2] = fx_addi<S>(e[2], o[2]); v[6] = fx_subi<S>(e[2], o[2]);
    v[3] = cadd(e[3], o3);         v[7] = csub(e[3], o3);
}
template <int S, int NZ, int NO> __device__ __forceinline__ void bfly32p(fxc* v) {
    static_assert(NZ == 32 && (NO == 17 || NO == 32), "whole lines in, a cropped or a whole line out");
    fxc y[4][8];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
#pragma unroll
        for (int a = 0; a < 8; ++a) y[b][a] = v[4 * a + b];
        fx_bfly8_wide<S>(y[b]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        fxc z[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) z[b] = fx_tw32_quarter<S>(y[b][k], b * k);
        if (NO == 32) bfly4p<S, 4, 4>(z);
        else if (k == 0) bfly4p<S, 4, 3>(z);
        else bfly4p<S, 4, 2>(z);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (k + 8 * j < NO) v[k + 8 * j] = z[j];
    }
}

// R-point DFT with inputs NZ..R-1 zero and only the first NO outputs needed.  Pruned forms exist
// for R = 32, 16 and 4 (and R = 8 with NZ <= 4, R = 2 with NZ = 1); otherwise the full DFT runs.
template <int R, int S, int NZ, int NO, typename C> __device__ __forceinline__ void dft_reg_p(C* v) {
    if constexpr (R == 32) {
        bfly32p<S, NZ, NO>(v);
    } else if constexpr (R == 16) {
        bfly16p<S, NZ, NO>(v);
    } else if constexpr (R == 4) {
        bfly4p<S, NZ, NO>(v);
    } else if constexpr (R == 8) {
        if constexpr (NZ <= 4) bfly8<S, true>(v);
        else bfly8<S>(v);
    } else {
        if constexpr (NZ == 1) v[1] = v[0];
        else bfly2<S>(v);
    }
}

// R-point DFT in registers; HALF: inputs R/2 .. R-1 are zero.
template <int R, int S, bool HALF = false, typename C> __device__ __forceinline__ void dft_reg(C* v) {
    if constexpr (R == 32) {
        bfly32p<S, HALF ? 16 : 32, 32>(v);
    } else if (R == 2) {
        if (HALF) v[1] = v[0];
        else bfly2<S>(v);
    } else if (R == 4) {
        if (HALF) bfly4_half<S>(v);
        else bfly4<S>(v);
    } else if (R == 8) {
        bfly8<S, HALF>(v);
    } else {
        bfly16<S, HALF>(v);
    }
}

template <int A, int B> struct FourStep {
    static constexpr int L = A * B;
    static constexpr int TPL = A < B ? A : B;   // threads per line
    static constexpr int I1 = B / TPL;          // step-1 DFTs per thread
    static constexpr int I2 = A / TPL;          // step-2 DFTs per thread
};

// Row stride (in elements) of the step-1 intermediate Y[t][k1] of fft4_io.  Threads of a warp
// write Y for consecutive t (groups of NL lanes) and read it back for consecutive k1; the skew
// PAD makes each group start on the banks where the previous one ended, so both accesses cost
// the minimum number of shared-memory wavefronts.  E = elements per 128-byte bank row.
template <int A, int E>
__host__ __device__ constexpr int fft4_pad(int NL) {
    return ((NL - A * NL) % E + E) % E;
}
template <int A, typename C>
__host__ __device__ constexpr int fft4_ystride(int NL) {
    return A * NL + fft4_pad<A, (int)(128 / sizeof(C))>(NL);
}

// fft4_io's transform of step-1 inputs already in registers: v[i][a] = element t + B a of line
// tid % NL, t = tid / NL + TPL i.
// Fixed point with an output of its own form (ODD: st takes a fourth argument whose call is a
// constant): a line whose outputs need the careful conversion (odd) stores in a second loop.
struct fft4_plain {};
template <bool V> struct fft4_flag {
    __device__ __forceinline__ constexpr bool operator()() const { return V; }
};
template <int A, int B, int S, bool IN_SMEM, bool OUT_SMEM, int NL, int NZ = A, int NO = B, typename C, typename Tw, class St, class Odd = fft4_plain>
__device__ __forceinline__ void fft4_run(C (&v)[FourStep<A, B>::I1][A], C* s, const Tw* __restrict__ tw, int tid, St st, Odd odd = Odd()) {
    typedef FourStep<A, B> F;
    const int l = tid % NL;
    const int q = tid / NL;
    constexpr int YS = fft4_ystride<A, C>(NL);
#pragma unroll
    for (int i = 0; i < F::I1; ++i) {
        const int t = q + F::TPL * i;
        dft_reg_p<A, S, NZ, A>(v[i]);
        tw_row<S, A * B, A>(v[i], tw, t);
    }
    if (IN_SMEM) __syncthreads();
#pragma unroll
    for (int i = 0; i < F::I1; ++i) {
        const int t = q + F::TPL * i;
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) s[t * YS + k1 * NL + l] = v[i][k1];
    }
    __syncthreads();
    C w2[F::I2][B];
#pragma unroll
    for (int i = 0; i < F::I2; ++i) {
        const int k1 = q + F::TPL * i;
#pragma unroll
        for (int t = 0; t < B; ++t) w2[i][t] = s[t * YS + k1 * NL + l];
        dft_reg_p<B, S, B, NO>(w2[i]);
    }
    if (OUT_SMEM) __syncthreads();
#pragma unroll
    for (int i = 0; i < F::I2; ++i) {
        const int k1 = q + F::TPL * i;
        if constexpr (std::is_same<Odd, fft4_plain>::value) {
#pragma unroll
            for (int k2 = 0; k2 < NO; ++k2) st(l, k1 + A * k2, w2[i][k2]);
        } else if (!odd) {
#pragma unroll
            for (int k2 = 0; k2 < NO; ++k2) st(l, k1 + A * k2, w2[i][k2], fft4_flag<false>());
        } else {
#pragma unroll
            for (int k2 = 0; k2 < NO; ++k2) st(l, k1 + A * k2, w2[i][k2], fft4_flag<true>());
        }
    }
    if (OUT_SMEM) __syncthreads();
}

// Four-step FFT with caller-supplied input and output.  ld(l, e) returns element e of line l
// (IN_SMEM: it reads the buffer s itself, so a barrier separates those reads from the first
// write into s); st(l, k, v) receives output k of line l (OUT_SMEM: it writes s, so a barrier
// separates the last reads of s from those writes).  Called by exactly NL * TPL threads.  The
// intermediate occupies B * fft4_ystride<A, C>(NL) elements of s.  Zero padding and cropping are
// pruned at compile time: inputs e >= NZ * B are known to be zero (ld is not called for them) and only
// outputs k < NO * A are produced (st is not called for the others).
template <int A, int B, int S, bool IN_SMEM, bool OUT_SMEM, int NL, int NZ = A, int NO = B, typename C, typename Tw, class Ld,
          class St>
__device__ __forceinline__ void fft4_io(C* s, const Tw* __restrict__ tw, int tid, Ld ld, St st) {
    typedef FourStep<A, B> F;
    const int l = tid % NL;
    const int q = tid / NL;
    C v[F::I1][A];
#pragma unroll
    for (int i = 0; i < F::I1; ++i) {
        const int t = q + F::TPL * i;
#pragma unroll
        for (int a = 0; a < A; ++a) v[i][a] = a < NZ ? ld(l, t + B * a) : czero<C>();
    }
    fft4_run<A, B, S, IN_SMEM, OUT_SMEM, NL, NZ, NO>(v, s, tw, tid, st);
}

}  // namespace lsm
