// apply_fxg.cuh - the FP64 operator's transform passes in 64-bit fixed point for any line length with
// factors 2, 3 and 5 (and for the two-step lengths on request of the schedule), on the runtime stages
// of fxg.cuh.  Included by apply.cu after apply_fx.cuh.
//
// A thread keeps one line (l) and one of m groups of butterflies (g), so no stage divides by the tile's
// width; m is chosen on the host so that the groups fill every stage's butterflies as evenly as they
// can (fxg_groups).
//
// Bound by latency and the integer pipes (z pass at 96^3: issue 31% at 10 warps before the tile was
// halved).  One system, FP64 apply: 96^3 4.62 -> 1.44 ms (z pass 2.74 -> 0.65, y 0.51 -> 0.14 each, inverse x
// 0.30 -> 0.12), 60 x 45 x 50 0.92 -> 0.30 ms.
#pragma once
#include "fxg.cuh"

namespace lsm {

// Elements g, g + m, ... below n of a line, ld(e) -> raw[e * LD + l], four loads in flight; returns the
// largest magnitude word.
template <int LD, class Ld>
__device__ __forceinline__ unsigned fxg_load(double2* raw, int n, int l, int g, int m, Ld ld) {
    unsigned mag = 0;
    for (int e = g; e < n; e += 4 * m) {
        double2 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = e + k * m < n ? ld(e + k * m) : czero<double2>();
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (e + k * m < n) {
                raw[(e + k * m) * LD + l] = v[k];
                mag = max(mag, max(fx_mag(v[k].x), fx_mag(v[k].y)));
            }
    }
    return mag;
}

// ---- strided pass: NL consecutive lines along x per block
template <int DIR, int NL, bool DYN>
__global__ void __launch_bounds__(NL * 48) kg_strided_fx(FxPlan p, FxTables T, StridedArgs a, const ApplySys<double>* __restrict__ sys) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned s_mag[NL], s_hi[DYN ? 3 * NL : 1];
    const ApplySys<double>& S = sys[blockIdx.z / a.ncomp];
    if (S.run && !*S.run) return;
    const int c = blockIdx.z % a.ncomp;
    const int l = threadIdx.x % NL, g = threadIdx.x / NL, m = blockDim.x / NL;
    const int x = blockIdx.x * NL + l;
    const bool xin = x < a.nlines;
    const double2* __restrict__ src = pick<double2>(S, a.src_sel) + c * a.src_os2 + blockIdx.y * a.src_os1 + x;
    double2* __restrict__ dst = pick<double2>(S, a.dst_sel) + c * a.dst_os2 + blockIdx.y * a.dst_os1 + x;
    fxc* sa = reinterpret_cast<fxc*>(smem_raw);
    fxc* sb = sa + (size_t)p.L * NL;
    double2* raw = reinterpret_cast<double2*>(sb);
    if (threadIdx.x < NL) s_mag[threadIdx.x] = 0;
    if (DYN && threadIdx.x < 3 * NL) s_hi[threadIdx.x] = 0;
    __syncthreads();
    const unsigned mag = fxg_load<NL>(raw, a.in_count, l, g, m, [&](int e) { return xin ? src[(long long)e * a.src_es] : czero<double2>(); });
    atomicMax(&s_mag[l], mag);
    __syncthreads();
    const FxScale sc(s_mag[l]);
    for (int e = g; e < p.L; e += m) {
        const int es = e - a.in_off;
        sa[e * NL + l] = (es >= 0 && es < a.in_count) ? fx_from(raw[es * NL + l], sc, p.fxbits) : czero<fxc>();
    }
    __syncthreads();
    int esum;
    const fxc* r = fxg_fft<DIR, NL, DYN, NL>(sa, sb, p, T, l, g, m, s_hi, l, esum);
    const FxUnit un(sc.unit(p.fxbits) + esum, sc.bad, s_mag[l] == 0);
    if (xin)
        for (int eo = g; eo < a.out_count; eo += m) {
            const fxc v = r[(eo + a.out_off) * NL + l];
            dst[(long long)eo * a.dst_es] = un.odd ? fx_to_odd(v, un) : fx_to(v, un);
        }
}

// ---- contiguous rows: NL rows per block.  Row r of src holds in_count elements (placed at in_off),
// row r of dst out_count (from out_off).  OUT: the inverse x pass's epilogue, dst = S.out = u - result.
template <int DIR, int NL, bool OUT, bool DYN>
__global__ void __launch_bounds__(NL * 48) kg_rows_fx(FxPlan p, FxTables T, const ApplySys<double>* __restrict__ sys, int src_sel,
                                                      int dst_sel, long long nrows, int in_count, int in_off, int out_count,
                                                      int out_off) {
    constexpr int LD = NL + 1;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned s_mag[NL], s_hi[DYN ? 3 * NL : 1];
    __shared__ int s_sum[NL];
    const ApplySys<double>& S = sys[blockIdx.y];
    if (S.run && !*S.run) return;
    const int l = threadIdx.x % NL, g = threadIdx.x / NL, m = blockDim.x / NL;
    const long long r0 = (long long)blockIdx.x * NL;
    const int live = nrows - r0 < NL ? (int)(nrows - r0) : NL;
    const double2* __restrict__ src = pick<double2>(S, src_sel) + r0 * in_count;
    double2* __restrict__ dst = (OUT ? S.out : pick<double2>(S, dst_sel)) + r0 * out_count;
    const double2* __restrict__ uin = OUT ? S.u + r0 * out_count : nullptr;
    fxc* sa = reinterpret_cast<fxc*>(smem_raw);
    fxc* sb = sa + (size_t)p.L * LD;
    double2* raw = reinterpret_cast<double2*>(sb);
    if (threadIdx.x < NL) s_mag[threadIdx.x] = 0;
    if (DYN && threadIdx.x < 3 * NL) s_hi[threadIdx.x] = 0;
    __syncthreads();
    for (int k = 0; k < live; ++k) {
        unsigned mag = 0;
        for (int e = threadIdx.x; e < in_count; e += blockDim.x) {
            const double2 v = src[(long long)k * in_count + e];
            raw[e * LD + k] = v;
            mag = max(mag, max(fx_mag(v.x), fx_mag(v.y)));
        }
        if (mag) atomicMax(&s_mag[k], mag);
    }
    __syncthreads();
    const FxScale sc(s_mag[l]);
    for (int e = g; e < p.L; e += m) {
        const int es = e - in_off;
        sa[e * LD + l] = (l < live && es >= 0 && es < in_count) ? fx_from(raw[es * LD + l], sc, p.fxbits) : czero<fxc>();
    }
    __syncthreads();
    int esum;
    const fxc* r = fxg_fft<DIR, LD, DYN, NL>(sa, sb, p, T, l, g, m, s_hi, l, esum);
    if constexpr (DYN) {
        if (g == 0) s_sum[l] = esum;
        __syncthreads();
    }
    for (int k = 0; k < live; ++k) {
        const FxScale sk(s_mag[k]);
        const FxUnit un(sk.unit(p.fxbits) + (DYN ? s_sum[k] : esum), sk.bad, s_mag[k] == 0);
        for (int e = threadIdx.x; e < out_count; e += blockDim.x) {
            const fxc v = r[(e + out_off) * LD + k];
            const double2 w = un.odd ? fx_to_odd(v, un) : fx_to(v, un);
            const long long i = (long long)k * out_count + e;
            dst[i] = OUT ? csub(uin[i], w) : w;
        }
    }
    if (OUT && S.count && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(S.count, 1ull);
}

// ---- z pass with the Green multiply: TX columns of one ky, as k4_fftz_green_fx
template <bool CONJ, int TX, bool DYN>
__global__ void __launch_bounds__(3 * TX * 32) kg_fftz_green_fx(Dims d, FxPlan p, FxTables T, const ApplySys<double>* __restrict__ sys,
                                                                int nsys, int in_count, int in_off, int out_count, int out_off,
                                                                int src_sel, int dst_sel) {
    constexpr int NL = 3 * TX;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned s_mag[TX], s_hi[DYN ? 3 * TX : 1];
    __shared__ int s_key[TX];
    const ApplySys<double>& S = sys[blockIdx.x % nsys];
    if (S.run && !*S.run) return;
    const int L = p.L;
    const int x0 = (int)(blockIdx.x / nsys) * TX, ky = blockIdx.y;
    const int l = threadIdx.x % NL, g = threadIdx.x / NL, m = blockDim.x / NL;
    const int cl = l / TX, lx = l - cl * TX;
    const bool xin = x0 + lx < d.Lx;
    const unsigned plane = (unsigned)(d.Ly * d.Lx), col = (unsigned)(ky * d.Lx + x0 + lx);
    fxc* sa = reinterpret_cast<fxc*>(smem_raw);
    fxc* sb = sa + (size_t)L * NL;
    int* sE = reinterpret_cast<int*>(sb + (size_t)L * NL);   // [L][TX]
    double2* raw = reinterpret_cast<double2*>(sb);
    if (threadIdx.x < TX) {
        s_mag[threadIdx.x] = 0;
        s_key[threadIdx.x] = FX_NO_KEY;
    }
    if (DYN && threadIdx.x < 3 * TX) s_hi[threadIdx.x] = 0;
    __syncthreads();
    {
        const double2* __restrict__ src = pick<double2>(S, src_sel) + (size_t)cl * in_count * plane + col;
        const unsigned mag = fxg_load<NL>(raw, in_count, l, g, m, [&](int e) { return xin ? src[(size_t)e * plane] : czero<double2>(); });
        atomicMax(&s_mag[lx], mag);
    }
    __syncthreads();
    const FxScale sc(s_mag[lx]);
    for (int e = g; e < L; e += m) {
        const int es = e - in_off;
        sa[e * NL + l] = (es >= 0 && es < in_count) ? fx_from(raw[es * NL + l], sc, p.fxbits) : czero<fxc>();
    }
    __syncthreads();
    int esum, esum_inv;
    fxc* s = fxg_fft<-1, NL, DYN, TX>(sa, sb, p, T, l, g, m, s_hi, lx, esum);   // one unit per column: its components mix
    fxc* o = s == sa ? sb : sa;
    if (DYN && threadIdx.x < 3 * TX) s_hi[threadIdx.x] = 0;   // ordered before its use by the barrier after the multiply
    // ---- Green multiply
    {
        const int cx = threadIdx.x % TX, kx = x0 + cx;   // blockDim.x is a multiple of TX
        int key = FX_NO_KEY;
        if (kx < d.Lx) {
            const long long NO = (long long)(d.nx + 1) * (d.ny + 1) * (d.nz + 1);
            const int fy = ky <= d.ny ? ky : d.Ly - ky, fx = kx <= d.nx ? kx : d.Lx - kx;
            const int sgx = kx > d.nx ? -1 : 1, sgy = ky > d.ny ? -1 : 1;
            const unsigned o0 = (unsigned)(fy * (d.nx + 1) + fx), oz = (unsigned)((d.nx + 1) * (d.ny + 1));
            const int4* __restrict__ gx = S.gx;
            const int* __restrict__ gexp = S.ge;
            const int dk = blockDim.x / TX;
            int4 G[6];
            int ge = 0;
            auto fetch = [&](int k) {
                const unsigned w = (unsigned)(k <= d.nz ? k : L - k) * oz + o0;
#pragma unroll
                for (int c = 0; c < 6; ++c) G[c] = __ldg(gx + c * NO + w);
                ge = __ldg(gexp + w);
            };
            int kz = threadIdx.x / TX;
            if (kz < L) fetch(kz);
#pragma unroll 1
            for (; kz < L; kz += dk) {
                const int sgz = kz > d.nz ? -1 : 1;
                const int4 G0 = G[0], G1 = G[1], G2 = G[2];
                const int4 G3 = fx_flip(G[3], sgy * sgz), G4 = fx_flip(G[4], sgx * sgz), G5 = fx_flip(G[5], sgx * sgy);
                const int e = ge;
                if (kz + dk < L) fetch(kz + dk);   // in flight during this point's products
                fxc* row = s + kz * NL + cx;
                const FxQ qa(row[0]), qb(row[TX]), qc(row[2 * TX]);
                const fxc r0 = fx_gdot3<CONJ>(G0, qa, G5, qb, G4, qc);
                row[0] = r0;
                const fxc r1 = fx_gdot3<CONJ>(G5, qa, G1, qb, G3, qc);
                row[TX] = r1;
                const fxc r2 = fx_gdot3<CONJ>(G4, qa, G3, qb, G2, qc);
                row[2 * TX] = r2;
                sE[kz * TX + cx] = e;
                key = max(key, 64 - __clz((int)(fx_hibits(r0) | fx_hibits(r1) | fx_hibits(r2))) + e);
            }
            atomicMax(&s_key[cx], key);
        }
        __syncthreads();
    }
    // ---- inverse transform
    const int top = s_key[lx], ecom = top - p.fxbits;
    for (int e = g; e < L; e += m) {
        fxc v = s[e * NL + l];
        const int sh = ecom - (xin ? sE[e * TX + lx] : 0);
        s[e * NL + l] = fxc{fx_shift(v.x, sh), fx_shift(v.y, sh)};
    }
    __syncthreads();
    const fxc* r = fxg_fft<1, NL, DYN, TX>(s, o, p, T, l, g, m, s_hi, lx, esum_inv);
    const FxUnit un(sc.unit(p.fxbits) + esum + esum_inv + ecom, sc.bad || top > FxG::BAD_EXP / 2, s_mag[lx] == 0);
    if (xin) {
        double2* __restrict__ dst = pick<double2>(S, dst_sel) + (size_t)cl * out_count * plane + col;
        for (int eo = g; eo < out_count; eo += m) {
            const fxc v = r[(eo + out_off) * NL + l];
            dst[(size_t)eo * plane] = un.odd ? fx_to_odd(v, un) : fx_to(v, un);
        }
    }
}

// ---- Green spectrum setup: FFT of lines that are even or odd about element 0 (and zero at L / 2),
// stored as their first half 0 .. n, n = L / 2; outputs 0 .. n in place.  Component c of the six
// (blockIdx.z) is odd when bit c of `odd` is set.  Line i of outer group o starts at o os + i ls, its
// elements es apart; ROWS: es = 1, loads and stores run along the line.  Outputs that vanish by
// symmetry come out as zero or a few units: v and -v round to opposite values but for ties.
struct SymArgs {
    long long cs, os, ls, es;
    int nlines, odd;
};
template <int NL, bool ROWS, bool DYN>
__global__ void __launch_bounds__(NL * 48) kg_sym_fx(FxPlan p, FxTables T, SymArgs a, double2* __restrict__ buf) {
    constexpr int LD = ROWS ? NL + 1 : NL;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned s_mag[NL], s_hi[DYN ? 3 * NL : 1];
    __shared__ int s_sum[NL];
    const int n = p.L / 2, i0 = blockIdx.x * NL;
    const int l = threadIdx.x % NL, g = threadIdx.x / NL, m = blockDim.x / NL;
    const int live = a.nlines - i0 < NL ? a.nlines - i0 : NL;
    double2* tile = buf + blockIdx.z * a.cs + blockIdx.y * a.os + i0 * a.ls;
    fxc* sa = reinterpret_cast<fxc*>(smem_raw);
    fxc* sb = sa + (size_t)p.L * LD;
    double2* raw = reinterpret_cast<double2*>(sb);
    if (threadIdx.x < NL) s_mag[threadIdx.x] = 0;
    if (DYN && threadIdx.x < 3 * NL) s_hi[threadIdx.x] = 0;
    __syncthreads();
    if constexpr (ROWS) {
        for (int k = 0; k < live; ++k) {
            unsigned mag = 0;
            for (int e = threadIdx.x; e <= n; e += blockDim.x) {
                const double2 v = tile[k * a.ls + e];
                raw[e * LD + k] = v;
                mag = max(mag, max(fx_mag(v.x), fx_mag(v.y)));
            }
            if (mag) atomicMax(&s_mag[k], mag);
        }
    } else {
        const unsigned mag = fxg_load<LD>(raw, n + 1, l, g, m, [&](int e) { return l < live ? tile[l * a.ls + e * a.es] : czero<double2>(); });
        atomicMax(&s_mag[l], mag);
    }
    __syncthreads();
    const FxScale sc(s_mag[l]);
    const bool odd = (a.odd >> blockIdx.z & 1) != 0;
    if (l < live)
        for (int e = g; e < p.L; e += m) {
            fxc v = fx_from(raw[(e <= n ? e : p.L - e) * LD + l], sc, p.fxbits);
            if (odd && e > n) v = fxc{fx_neg(v.x), fx_neg(v.y)};
            sa[e * LD + l] = v;
        }
    __syncthreads();
    int esum;
    const fxc* r = fxg_fft<-1, LD, DYN, NL>(sa, sb, p, T, l, g, m, s_hi, l, esum);
    if constexpr (ROWS) {
        if constexpr (DYN) {
            if (g == 0) s_sum[l] = esum;
            __syncthreads();
        }
        for (int k = 0; k < live; ++k) {
            const FxScale sk(s_mag[k]);
            const FxUnit un(sk.unit(p.fxbits) + (DYN ? s_sum[k] : esum), sk.bad, s_mag[k] == 0);
            for (int e = threadIdx.x; e <= n; e += blockDim.x) {
                const fxc v = r[e * LD + k];
                tile[k * a.ls + e] = un.odd ? fx_to_odd(v, un) : fx_to(v, un);
            }
        }
    } else if (l < live) {
        const FxUnit un(sc.unit(p.fxbits) + esum, sc.bad, s_mag[l] == 0);
        for (int e = g; e <= n; e += m) {
            const fxc v = r[e * LD + l];
            tile[l * a.ls + e * a.es] = un.odd ? fx_to_odd(v, un) : fx_to(v, un);
        }
    }
}

}  // namespace lsm
