// fxg.cuh - runtime mixed-radix Stockham FFT (fft.cuh) of lines in shared memory, in 64-bit fixed point
// (fx.cuh): its plan and its stages.
//
// Every stage after the first takes its values to a unit 2^K coarser, with the twiddles' help.
// * Short lines: K = 1 .. 3 is the plan's, the smallest for which no line of that length can leave the
//   words; a line's error is that of its last stages (K = 2 or 3 by the radix alone lost up to 3 bits).
//   Against longdouble a line's rms error is 0.2 to 1.0 of that of the same plan in FP64.
// * Lines longer than 256, or longer than 128 in four stages or more: the headroom of the worst line
//   (all elements at the largest modulus, aligned) would cost more bits than FP64's roundings do
//   (errors up to 2.4 of FP64's, on lines whose spectra are peaked).  Here each stage sees how large the
//   values of the line really are and steps to the unit that they need (block floating point, stage by
//   stage): 0.2 to 0.55 of FP64's error.  One system, FP64 apply, against the plan's K: 144^3
//   5.69 -> 6.29 ms, 200^3 17.5 -> 18.9 ms, 250^3 41.4 -> 44.1 ms.
// tests/test_fixed_point_lines.py measures both.
#pragma once
#include "fft.cuh"

namespace lsm {

// Scaling of a plan's fixed-point stages: in log2 of the largest modulus, the first stage's outputs and
// every later stage's stay below 61.9 with the smallest K in 1 .. 3 that does it (K = 1 doubles the
// values before a product, which needs them below 60.9).  A dynamic plan uses fxbits alone.  Its rule:
// with the plan's K the worst of six kinds of fields had 0.97 of FP64's error at L = 200, 0.87 at 144
// (four stages), but 1.02 at 180 (four), 1.2 at 162 (five), 1.1 at 320 and 1.3 to 2.4 at the other
// lengths above 256.
inline void fixed_point_scaling(FxPlan& p) {
    const double top = 61.9;
    const double g0 = log2((double)p.radix[0]);
    p.fxbits = (int)floor(top - 0.5 - g0);
    double m = p.fxbits + 0.5 + g0;
    p.fxk[0] = 0;
    p.fxsum = 0;
    p.fxdyn = p.L > 256 || (p.L > 128 && p.nst > 3);
    for (int s = 1; s < p.nst; ++s) {
        const double g = log2((double)p.radix[s]);
        int k = (m <= top - 1.0 && m + g - 1.0 <= top) ? 1 : (m + g - 2.0 <= top ? 2 : 3);
        p.fxk[s] = k;
        p.fxsum += k;
        m += g - k;
    }
}

inline bool factor_plan(int L, FxPlan& p) {
    p.L = L;
    p.nst = 0;
    int m = L;
    const int rs[5] = {8, 4, 2, 3, 5};
    for (int k = 0; k < 5; ++k) {
        while (m % rs[k] == 0) {
            if (p.nst >= 12) return false;
            p.radix[p.nst++] = rs[k];
            m /= rs[k];
        }
    }
    if (m == 1) fixed_point_scaling(p);
    return m == 1;
}

// the two scaled twiddle tables of a line length: entries times 2^-2 and 2^-3
struct FxTables {
    const int4 *t2, *t3;
};

// Bits of the values before a dynamic stage's products: the quarter-scaled twiddles then keep every sum
// of the butterfly below 2^61.9 and every factor of its products in range.
template <int R> __device__ __forceinline__ constexpr int fxg_fill() { return R == 2 ? 62 : (R == 8 ? 60 : 61); }

// One stage.  K: the plan's step (0: the first stage); DYN: the left shift that fills the words of the
// line's values before the stage (the step is 2 - K).  bits: the high words of
// the results' moduli are or-ed into it (DYN).
template <int S, int R, int LD, bool DYN>
__device__ __forceinline__ void fxg_stage(const fxc* __restrict__ src, fxc* __restrict__ dst, int L, int Ns, int K,
                                          const FxTables& T, int l, int g, int m, unsigned& bits) {
    const int4* __restrict__ tw = !DYN && K == 3 ? T.t3 : T.t2;
    const int nb = L / R, tstep = L / (Ns * R);
    const unsigned magic = 0xffffffffu / (unsigned)Ns + 1;   // j / Ns = j magic 2^-32 for j < 2^16 (Ns > 1)
#pragma unroll 1
    for (int j = g; j < nb; j += m) {
        const int jq = Ns == 1 ? j : (int)__umulhi((unsigned)j, magic);
        const int k = j - jq * Ns;
        fxc v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src[(j + r * nb) * LD + l];
        if (DYN ? Ns > 1 : K != 0) {   // not the first stage
            if constexpr (DYN) {
                v[0] = fxc{fx_shift(v[0].x, 2 - K), fx_shift(v[0].y, 2 - K)};
#pragma unroll
                for (int r = 1; r < R; ++r)
                    v[r] = tw_mul32<S>(fxc{fx_shift(v[r].x, -K), fx_shift(v[r].y, -K)}, tw, r * k * tstep);
            } else {
                v[0].x = fx_r((fx_ll(v[0].x) + (1 << (K - 1))) >> K);
                v[0].y = fx_r((fx_ll(v[0].y) + (1 << (K - 1))) >> K);
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    if (K == 1) v[r] = cadd(v[r], v[r]);
                    v[r] = tw_mul32<S>(v[r], tw, r * k * tstep);
                }
            }
        }
        if constexpr (R == 2) bfly2<S>(v);
        else if constexpr (R == 3) bfly3<S>(v);
        else if constexpr (R == 4) bfly4<S>(v);
        else if constexpr (R == 5) bfly5<S>(v);
        else bfly8<S>(v);
        const int base = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            dst[(base + r * Ns) * LD + l] = v[r];
            if (DYN) bits |= fx_hibits(v[r]);
        }
    }
}

// Transform the tile in a (layout a[e * LD + l]); b is scratch of the same size.  Returns the buffer
// of the result.  The caller synchronises before; the result is visible to the block on return.
// esum: by how many powers of two the result's unit is coarser than the inputs'.
// DYN: lines with the same gi (< NG) share their units.  hi [3][NG] in shared memory, zeroed by the
// caller before its barrier: stage s reads the size of the values from row s % 3, collects that of its
// results in the next row and clears the third (read by the stage before, written by the next).
template <int S, int LD, bool DYN, int NG>
__device__ __forceinline__ fxc* fxg_fft(fxc* a, fxc* b, const FxPlan& p, const FxTables& T, int l, int g, int m,
                                        unsigned* hi, int gi, int& esum) {
    int Ns = 1;
    esum = DYN ? 0 : p.fxsum;
    for (int s = 0; s < p.nst; ++s) {
        const int R = p.radix[s];
        int K = DYN ? 0 : p.fxk[s];
        unsigned bits = 0;
        if (DYN && s > 0) {
            K = (R == 2 ? fxg_fill<2>() : (R == 8 ? fxg_fill<8>() : fxg_fill<3>())) - (64 - __clz((int)hi[s % 3 * NG + gi]));
            esum += 2 - K;
        }
        if (DYN && (int)threadIdx.x < NG) hi[(s + 2) % 3 * NG + threadIdx.x] = 0;
        switch (R) {
            case 8: fxg_stage<S, 8, LD, DYN>(a, b, p.L, Ns, K, T, l, g, m, bits); break;
            case 4: fxg_stage<S, 4, LD, DYN>(a, b, p.L, Ns, K, T, l, g, m, bits); break;
            case 2: fxg_stage<S, 2, LD, DYN>(a, b, p.L, Ns, K, T, l, g, m, bits); break;
            case 3: fxg_stage<S, 3, LD, DYN>(a, b, p.L, Ns, K, T, l, g, m, bits); break;
            default: fxg_stage<S, 5, LD, DYN>(a, b, p.L, Ns, K, T, l, g, m, bits); break;
        }
        if (DYN && bits) atomicOr(&hi[(s + 1) % 3 * NG + gi], bits);
        __syncthreads();
        fxc* t = a; a = b; b = t;
        Ns *= R;
    }
    return a;
}

// Groups per line, m <= most: the fewest butterfly rounds weighted by their size, then the most groups.
inline int fxg_groups(const FxPlan& p, int least, int most) {
    int best = least;
    double cost = 1e300;
    for (int m = least; m <= most; ++m) {
        double c = 0.0;
        for (int s = 0; s < p.nst; ++s) {
            const int nb = p.L / p.radix[s];
            c += (double)((nb + m - 1) / m) * (p.radix[s] + 2) * m;
        }
        c *= 1.0 + 4.0 / m;   // fewer threads hide less latency
        if (c <= cost) {
            cost = c;
            best = m;
        }
    }
    return best;
}

}  // namespace lsm
