// apply_fx.cuh - the FP64 operator's transform passes in 64-bit fixed point (fx.cuh), for the line
// lengths of the compile-time two-step FFT.  Included by apply.cu.
//
// Each kernel reads FP64, finds the line's (z pass: the column's three lines') largest exponent,
// converts, transforms on the integer pipes and converts back.  The FP64 engine kept the FP64 pipe 87%
// busy; here the z pass keeps the wide multiplies' pipe 65% busy at 12 warps per SM (43% of issue
// slots), the y and x passes the integer-add pipe 64-66% at 15 warps.
#pragma once

namespace lsm {

template <int A, int B> struct FxStep {
    static constexpr int NZI = A / 2 + 1;   // nonzero inputs of a step-1 DFT of a padded line
    static constexpr int NOO = B / 2 + 1;   // wanted outputs of a step-2 DFT of a cropped line
};

// Strided pass: TX consecutive lines along x per block, as k4_strided.  bits: fx_bits of the line's
// nonzero inputs.  Bound by the integer-add pipe.  128^3, one system: 1.05 ms on the FP64 pipe, 0.175
// here (0.6 GB at 3.5 TB/s).
template <int DIR, int A, int B, int TX>
__global__ void __launch_bounds__(TX * FourStep<A LSM_COMMA B>::TPL, B == 32 ? 2 : 4) k4_strided_fx(
    const int4* __restrict__ tw, StridedArgs a, const ApplySys<double>* __restrict__ sys, int bits) {
    typedef FourStep<A, B> F;
    constexpr int NT = TX * F::TPL, NW = (NT + 31) / 32;
    constexpr int NZ = DIR < 0 ? FxStep<A, B>::NZI : A, NO = DIR > 0 ? FxStep<A, B>::NOO : B;
    static_assert(NT % 32 == 0 && 32 % TX == 0, "whole warps of whole groups of lines");
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned part[NW][TX];
    const int c = blockIdx.z % a.ncomp;
    const ApplySys<double> S = sys[blockIdx.z / a.ncomp];
    if (S.run && !*S.run) return;
    fxc* s = reinterpret_cast<fxc*>(smem_raw);
    const int l = threadIdx.x % TX, q = threadIdx.x / TX;
    const int x = blockIdx.x * TX + l;   // this thread's line
    const bool xin = x < a.nlines;
    const double2* __restrict__ src = pick<double2>(S, a.src_sel) + c * a.src_os2 + blockIdx.y * a.src_os1 + x;
    double2* __restrict__ dst = pick<double2>(S, a.dst_sel) + c * a.dst_os2 + blockIdx.y * a.dst_os1 + x;
    const int ses = (int)a.src_es, des = (int)a.dst_es;
    double2 in[F::I1][NZ];
    unsigned mag = 0;
#pragma unroll
    for (int i = 0; i < F::I1; ++i)
#pragma unroll
        for (int k = 0; k < NZ; ++k) {
            const int es = q + F::TPL * i + B * k - a.in_off;
            in[i][k] = (xin && es >= 0 && es < a.in_count) ? src[es * ses] : czero<double2>();
            mag = max(mag, max(fx_mag(in[i][k].x), fx_mag(in[i][k].y)));
        }
#pragma unroll
    for (int o = TX; o < 32; o <<= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    if constexpr (NW > 1) {
        if ((threadIdx.x & 31) < TX) part[threadIdx.x >> 5][l] = mag;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NW; ++w) mag = max(mag, part[w][l]);
    }
    const FxScale sc(mag);
    fxc v[F::I1][A];
#pragma unroll
    for (int i = 0; i < F::I1; ++i)
#pragma unroll
        for (int k = 0; k < A; ++k) v[i][k] = k < NZ ? fx_from(in[i][k < NZ ? k : 0], sc, bits + fx_prescale(A * B)) : czero<fxc>();
    const FxUnit un(sc.unit(bits), sc.bad, mag == 0);
    auto st = [&](int, int k, fxc r, auto odd) {
        const int eo = k - a.out_off;
        if (xin && eo >= 0 && eo < a.out_count) dst[eo * des] = odd() ? fx_to_odd(r, un) : fx_to(r, un);
    };
    fft4_run<A, B, DIR, false, false, TX, NZ, NO>(v, s, tw, threadIdx.x, st, un.odd);
}

// Contiguous rows: each line on TPL consecutive lanes of one warp, as k4_rows_w, for every A and B.
// The line's exponent is a shuffle reduction over its lanes and the exchange between the steps a
// tile of its own ordered by __syncwarp, so a block has no barrier.  Bound by the integer-add pipe.
// 128^3, one system: inverse x pass 0.57 -> 0.124 ms, contrast source and forward x 0.76 -> 0.31 (of
// which the source, on the FP64 pipe, 0.23).
template <int DIR, int A, int B, int NZ, int NO, class Tw, class St>
__device__ __forceinline__ void fx_row(double2 (&in)[FourStep<A, B>::I1][NZ], fxc* tl, const Tw* __restrict__ tw, int q, int bits, St st) {
    typedef FourStep<A, B> F;
    unsigned mag = 0;
#pragma unroll
    for (int i = 0; i < F::I1; ++i)
#pragma unroll
        for (int k = 0; k < NZ; ++k) mag = max(mag, max(fx_mag(in[i][k].x), fx_mag(in[i][k].y)));
#pragma unroll
    for (int o = 1; o < F::TPL; o <<= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    const FxScale sc(mag);
#pragma unroll
    for (int i = 0; i < F::I1; ++i) {
        const int t = q + F::TPL * i;
        fxc v[A];
#pragma unroll
        for (int k = 0; k < A; ++k) v[k] = k < NZ ? fx_from(in[i][k < NZ ? k : 0], sc, bits + fx_prescale(A * B)) : czero<fxc>();
        dft_reg_p<A, DIR, NZ, A>(v);
        tw_row<DIR, A * B, A>(v, tw, t);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) tl[t * (A + 1) + k1] = v[k1];
    }
    __syncwarp();
    const FxUnit un(sc.unit(bits), sc.bad, mag == 0);
#pragma unroll
    for (int i = 0; i < F::I2; ++i) {
        const int k1 = q + F::TPL * i;
        fxc w[B];
#pragma unroll
        for (int t = 0; t < B; ++t) w[t] = tl[t * (A + 1) + k1];
        dft_reg_p<B, DIR, B, NO>(w);
        if (!un.odd) {
#pragma unroll
            for (int k2 = 0; k2 < NO; ++k2) st(k1 + A * k2, fx_to(w[k2], un));
        } else {
#pragma unroll
            for (int k2 = 0; k2 < NO; ++k2) st(k1 + A * k2, fx_to_odd(w[k2], un));
        }
    }
}

// x FFT of contiguous rows: row r of src holds in_count elements (placed at in_off; forward: the rest
// of the line is zero), row r of dst receives outputs out_off .. out_off + out_count - 1 (inverse: the
// first half and a little, as cropped lines have)
template <int DIR, int A, int B, int LPB>
__global__ void __launch_bounds__(LPB * FourStep<A LSM_COMMA B>::TPL, B == 32 ? 2 : 4) k4_rows_fx(const int4* __restrict__ tw,
                                                                            const ApplySys<double>* __restrict__ sys,
                                                                            int src_sel, int dst_sel, long long nrows,
                                                                            int in_count, int in_off, int out_count,
                                                                            int out_off, int bits) {
    typedef FourStep<A, B> F;
    constexpr int NZ = DIR < 0 ? FxStep<A, B>::NZI : A, NO = DIR > 0 ? FxStep<A, B>::NOO : B;
    static_assert(LPB * F::TPL % 32 == 0, "whole warps");
    extern __shared__ unsigned char smem_raw[];
    const ApplySys<double> S = sys[blockIdx.y];
    if (S.run && !*S.run) return;
    const int ln = threadIdx.x / F::TPL, q = threadIdx.x % F::TPL;
    const long long row = (long long)blockIdx.x * LPB + ln;
    const bool live = row < nrows;
    const double2* __restrict__ src = pick<double2>(S, src_sel) + row * in_count;
    double2* __restrict__ dst = pick<double2>(S, dst_sel) + row * out_count;
    double2 in[F::I1][NZ];
#pragma unroll
    for (int i = 0; i < F::I1; ++i)
#pragma unroll
        for (int k = 0; k < NZ; ++k) {
            const int e = q + F::TPL * i + B * k - in_off;
            in[i][k] = (live && e >= 0 && e < in_count) ? src[e] : czero<double2>();
        }
    fxc* tl = reinterpret_cast<fxc*>(smem_raw) + ln * B * (A + 1);
    fx_row<DIR, A, B, NZ, NO>(in, tl, tw, q, bits, [&](int k, double2 r) {
        const int e = k - out_off;
        if (live && e >= 0 && e < out_count) dst[e] = r;
    });
}

// inverse x FFT of the rows of w2 [3][nz][ny][L], crop to x = k - xoff in [0, nx), Au = u - u_s
template <int A, int B, int LPB>
__global__ void __launch_bounds__(LPB * FourStep<A LSM_COMMA B>::TPL, B == 32 ? 2 : 4) k4_xout_fx(Dims d, const ApplySys<double>* __restrict__ sys,
                                                                            const int4* __restrict__ tw, int xoff, int bits) {
    typedef FourStep<A, B> F;
    constexpr int L = A * B, NO = FxStep<A, B>::NOO;
    extern __shared__ unsigned char smem_raw[];
    const ApplySys<double> S = sys[blockIdx.y];
    if (S.run && !*S.run) return;
    const int ln = threadIdx.x / F::TPL, q = threadIdx.x % F::TPL;
    const long long row = (long long)blockIdx.x * LPB + ln;
    const bool live = row < 3LL * d.nz * d.ny;
    const double2* __restrict__ src = S.w2 + row * L;
    const double2* __restrict__ uin = S.u + row * d.nx;
    double2* __restrict__ out = S.out + row * d.nx;
    double2 in[F::I1][A];
#pragma unroll
    for (int i = 0; i < F::I1; ++i)
#pragma unroll
        for (int k = 0; k < A; ++k) in[i][k] = live ? src[q + F::TPL * i + B * k] : czero<double2>();
    fxc* tl = reinterpret_cast<fxc*>(smem_raw) + ln * B * (A + 1);
    fx_row<1, A, B, A, NO>(in, tl, tw, q, bits, [&](int k, double2 r) {
        const int x = k - xoff;
        if (live && x >= 0 && x < d.nx) out[x] = csub(uin[x], r);
    });
    if (S.count && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(S.count, 1ull);
}

// ---------------------------------------------------------------------------------------------
// z pass with the Green multiply
// ---------------------------------------------------------------------------------------------

// The forms of the octant spectra, from their FP64 values times scale (1/P): gx [6][NO] = (G1, G0) of the
// real part, then of the imaginary part, ge [NO] = the point's exponent (fx.cuh), g32 and gdf FP32 and
// double-float copies (either may be null).  g and gx may be the same memory.
static __global__ void __launch_bounds__(NTH) k_spectrum_forms(const double2* g, double scale, long long NO, int4* gx, int* __restrict__ ge,
                                                               float2* __restrict__ g32, dfcplx* __restrict__ gdf) {
    for (long long i = (long long)blockIdx.x * NTH + threadIdx.x; i < NO; i += (long long)gridDim.x * NTH) {
        double2 v[6];
        unsigned mag = 0;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            v[c] = cscale(g[c * NO + i], scale);
            mag = max(mag, max(fx_mag(v[c].x), fx_mag(v[c].y)));
        }
        const FxScale sc(mag);
        // components below 2^60 in units of 2^-61: below 1/2; the multiply returns g q / 2
        const bool zero = mag == 0;
        ge[i] = sc.bad ? FxG::BAD_EXP : (zero ? FxG::ZERO_EXP : sc.unit(60) + 62);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const fxc q = fx_from(v[c], sc, 60);
            int4 w;
            w.x = (int)((fx_ll(q.x) + (1LL << 29)) >> 30);
            w.y = (int)(fx_ll(q.x) - ((long long)w.x << 30));
            w.z = (int)((fx_ll(q.y) + (1LL << 29)) >> 30);
            w.w = (int)(fx_ll(q.y) - ((long long)w.z << 30));
            if (zero) w = make_int4(0, 0, 0, 0);
            gx[c * NO + i] = w;
            if (g32) g32[c * NO + i] = make_float2((float)v[c].x, (float)v[c].y);
            if (gdf) gdf[c * NO + i] = dfcplx{df_from(v[c].x), df_from(v[c].y)};
        }
    }
}

// sg = +-1: g or -g, by multiplications (the FMA pipe; the integer-add pipe is the busy one)
__device__ __forceinline__ int4 fx_flip(int4 g, int sg) { return make_int4(g.x * sg, g.y * sg, g.z * sg, g.w * sg); }
// A transform value split for the multiply: its two lowest bits rounded off, q = 4 (h 2^30 + l),
// |l| <= 2^29.
struct FxQ {
    int xh, xl, yh, yl;
    __device__ __forceinline__ explicit FxQ(fxc q) {
        split(q.x, xh, xl);
        split(q.y, yh, yl);
    }
    static __device__ __forceinline__ void split(fxr v, int& h, int& l) {
        v = fx_add(v, fxr{2u, 0});
        h = v.h + (int)(v.l >> 31);
        l = (int)v.l >> 2;
    }
};
// g q / 2 (conj(g) for CONJ) is h + t 2^-30: with |g| < 1/2 per component and |q| < 2^62.6, over the
// three products of a row |h| < 2^62.7 and |t| < 6 2^29 2^30 + 3 2^30.6 2^29.5 < 2^62.7
template <bool CONJ>
__device__ __forceinline__ void fx_gmac(const int4& g, const FxQ& q, long long& hr, long long& tr, long long& hi, long long& ti) {
    const int gi1 = CONJ ? -g.z : g.z, gi0 = CONJ ? -g.w : g.w;
    hr = fx_mad(q.yh, -gi1, fx_mad(q.xh, g.x, hr));
    hi = fx_mad(q.xh, gi1, fx_mad(q.yh, g.x, hi));
    tr = fx_mad(q.yh, -gi0, fx_mad(q.yl, -gi1, fx_mad(q.xh, g.y, fx_mad(q.xl, g.x, tr))));
    ti = fx_mad(q.xh, gi0, fx_mad(q.xl, gi1, fx_mad(q.yh, g.y, fx_mad(q.yl, g.x, ti))));
}
__device__ __forceinline__ fxr fx_sr30(long long t) {
    const fxr v = fx_words(t);
    return fxr{__funnelshift_l(v.l, (unsigned)v.h, 2), v.h >> 30};
}
template <bool CONJ>
__device__ __forceinline__ fxc fx_gdot3(const int4& g0, const FxQ& qa, const int4& g1, const FxQ& qb, const int4& g2, const FxQ& qc) {
    long long tr = 1LL << 29, ti = 1LL << 29, hr = 0, hi = 0;
    fx_gmac<CONJ>(g0, qa, hr, tr, hi, ti);
    fx_gmac<CONJ>(g1, qb, hr, tr, hi, ti);
    fx_gmac<CONJ>(g2, qc, hr, tr, hi, ti);
    return fxc{fx_add(fx_words(hr), fx_sr30(tr)), fx_add(fx_words(hi), fx_sr30(ti))};
}
constexpr int FX_NO_KEY = -(1 << 24);   // below any exponent

// Maximum over the lanes of each aligned group of 16 whose numbers agree modulo TX (the same column
// of the z pass): its first TX lanes then hold it.  NT threads per block, a multiple of 16.
template <int TX, int NT, typename V> __device__ __forceinline__ V column_max(V v) {
    static_assert(NT % 16 == 0 && 16 % TX == 0, "groups of 16 lanes");
    const unsigned mask = (NT % 32 && threadIdx.x >= NT / 32 * 32) ? 0xffffu : 0xffffffffu;
#pragma unroll
    for (int o = TX; o < 16; o <<= 1) v = max(v, __shfl_xor_sync(mask, v, o));
    return v;
}

// Block = TX columns (kx) of one ky of one system (blockIdx.x = system + nsys * tile: the systems of a
// batch meet the tile's spectrum entries in the caches one after the other): 3 TX lines, element k of
// line l = c TX + lx at s[k NL + l].  The column's three lines share one exponent.  The multiply
// leaves each point's products in their own exponent (the point's spectrum exponent, kept in sE);
// the column's largest sets the inverse transform's, and the shift happens as its first step loads
// them.  TX = 4: 192 threads at L = 256, two blocks per SM whose loads, barriers and arithmetic overlap
// (TX = 2 with four to six smaller blocks: the same at 128^3, slower at 64^3 and 256^3); the spectrum is
// read through the caches, where the other systems and the mirrored rows find it again.  (One block for
// all systems in turn, hoisting what they share, spilled 110 registers.)  Bound by the wide multiplies'
// pipe and its latencies.  128^3, one system: 5.21 ms on the FP64 pipe, 0.93 here.
template <bool CONJ, int A, int B, int TX>
__global__ void __launch_bounds__(3 * TX * FourStep<A LSM_COMMA B>::TPL, 2) k4_fftz_green_fx(
    Dims d, const int4* __restrict__ tw, const ApplySys<double>* __restrict__ sys, int nsys, int in_count, int in_off,
    int out_count, int out_off, int src_sel, int dst_sel, int fbits, int ibits) {
    typedef FourStep<A, B> F;
    constexpr int NL = 3 * TX, L = A * B, NT = NL * F::TPL;
    constexpr int NZ = FxStep<A, B>::NZI, NO_ = FxStep<A, B>::NOO;
    constexpr int YB = B * fft4_ystride<A, fxc>(NL), SB = YB > L * NL ? YB : L * NL;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned s_mag[TX];
    __shared__ int s_key[TX];
    fxc* s = reinterpret_cast<fxc*>(smem_raw);
    int* sE = reinterpret_cast<int*>(s + SB);        // [L][TX]
    const int ky = blockIdx.y;
    const int x0 = (int)(blockIdx.x / nsys) * TX;
    const int fy = ky <= d.ny ? ky : d.Ly - ky;
    const int my = ky > d.ny ? -1 : 0;
    const long long NO = (long long)(d.nx + 1) * (d.ny + 1) * (d.nz + 1);
    const unsigned plane = (unsigned)(d.Ly * d.Lx);
    const ApplySys<double>& S = sys[blockIdx.x % nsys];
    if (S.run && !*S.run) return;
    const int tid = threadIdx.x;
    const int lt = tid % NL, q = tid / NL;
    const int cl = lt / TX, lxl = lt - cl * TX;      // this thread's line: component, column
    const bool xin = x0 + lxl < d.Lx;
    const unsigned col = (unsigned)(ky * d.Lx + x0 + lxl);
    if (tid < TX) {
        s_mag[tid] = 0;
        s_key[tid] = FX_NO_KEY;
    }
    __syncthreads();
    FxScale sc(0u);
    {
        const double2* __restrict__ src = pick<double2>(S, src_sel) + (size_t)cl * in_count * plane;
        double2 in[F::I1][NZ];
        unsigned mag = 0;
#pragma unroll
        for (int i = 0; i < F::I1; ++i)
#pragma unroll
            for (int k = 0; k < NZ; ++k) {
                const int es = q + F::TPL * i + B * k - in_off;
                in[i][k] = (xin && es >= 0 && es < in_count) ? src[(unsigned)es * plane + col] : czero<double2>();
                mag = max(mag, max(fx_mag(in[i][k].x), fx_mag(in[i][k].y)));
            }
        mag = column_max<TX, NT>(mag);
        if ((tid & 15) < TX) atomicMax(&s_mag[lxl], mag);
        __syncthreads();
        sc = FxScale(s_mag[lxl]);
        fxc v[F::I1][A];
#pragma unroll
        for (int i = 0; i < F::I1; ++i)
#pragma unroll
            for (int k = 0; k < A; ++k) v[i][k] = k < NZ ? fx_from(in[i][k < NZ ? k : 0], sc, fbits + fx_prescale(L)) : czero<fxc>();
        auto st_s = [&](int l, int k, fxc r) { s[k * NL + l] = r; };
        fft4_run<A, B, -1, false, true, NL, NZ, B>(v, s, tw, tid, st_s);
    }
    // ---- Green multiply, points (kz, lx) of the three lines
    {
        const int lx = tid % TX;   // NT is a multiple of TX
        const int kx = x0 + lx;
        int key = FX_NO_KEY;
        if (kx < d.Lx) {
            const int sgx = kx > d.nx ? -1 : 1, sgy = my ? -1 : 1;
            const int fx = kx <= d.nx ? kx : d.Lx - kx;
            const unsigned o0 = (unsigned)(fy * (d.nx + 1) + fx), oz = (unsigned)((d.nx + 1) * (d.ny + 1));
            const int4* __restrict__ gx = S.gx;
            const int* __restrict__ gexp = S.ge;
            constexpr int DK = NT / TX;
            int kz = tid / TX;
            int4 G[6];
            int ge = 0;
            auto fetch = [&](int k) {
                const unsigned o = (unsigned)(k <= d.nz ? k : L - k) * oz + o0;
#pragma unroll
                for (int c = 0; c < 6; ++c) G[c] = __ldg(gx + c * NO + o);
                ge = __ldg(gexp + o);
            };
            fetch(kz);
#pragma unroll 1
            for (; kz < L; kz += DK) {
                // mirrored octant entries: the off-diagonal ij entry is odd in axes i and j
                const int sgz = kz > d.nz ? -1 : 1;
                const int4 G0 = G[0], G1 = G[1], G2 = G[2];
                const int4 G3 = fx_flip(G[3], sgy * sgz), G4 = fx_flip(G[4], sgx * sgz), G5 = fx_flip(G[5], sgx * sgy);
                const int e = ge;
                if (kz + DK < L) fetch(kz + DK);   // in flight during this point's products
                fxc* row = s + kz * NL + lx;
                const FxQ qa(row[0]), qb(row[TX]), qc(row[2 * TX]);
                const fxc r0 = fx_gdot3<CONJ>(G0, qa, G5, qb, G4, qc);
                row[0] = r0;
                const fxc r1 = fx_gdot3<CONJ>(G5, qa, G1, qb, G3, qc);
                row[TX] = r1;
                const fxc r2 = fx_gdot3<CONJ>(G4, qa, G3, qb, G2, qc);
                row[2 * TX] = r2;
                sE[kz * TX + lx] = e;
                const unsigned b = fx_hibits(r0) | fx_hibits(r1) | fx_hibits(r2);
                // |components| < 2^(64 - clz): an upper bound when the high words are all zero
                key = max(key, 64 - __clz((int)b) + e);
            }
        }
        key = column_max<TX, NT>(key);
        if ((tid & 15) < TX) atomicMax(&s_key[lx], key);
        __syncthreads();
    }
    // ---- inverse transform: components below 2^ibits in the unit of its outputs
    const int top = s_key[lxl];
    const int ecom = top - ibits - fx_prescale(L);   // unit of the first step's inputs
    const FxUnit un(sc.unit(fbits) + ecom + fx_prescale(L), sc.bad || top > FxG::BAD_EXP / 2, s_mag[lxl] == 0);
    fxc v[F::I1][A];
#pragma unroll
    for (int i = 0; i < F::I1; ++i)
#pragma unroll
        for (int k = 0; k < A; ++k) {
            const int kz = q + F::TPL * i + B * k;
            fxc r = s[kz * NL + lt];
            const int sh = ecom - (xin ? sE[kz * TX + lxl] : 0);
            if (sh >= 0) {       // the usual case
                r.x = fx_r(fx_ll(r.x) >> min(sh, 63));
                r.y = fx_r(fx_ll(r.y) >> min(sh, 63));
            } else {             // a point whose products are small beside its spectrum entry
                r.x = fx_r((long long)((unsigned long long)fx_ll(r.x) << min(-sh, 63)));
                r.y = fx_r((long long)((unsigned long long)fx_ll(r.y) << min(-sh, 63)));
            }
            v[i][k] = r;
        }
    double2* __restrict__ dst = pick<double2>(S, dst_sel) + (size_t)cl * out_count * plane;
    auto st_g = [&](int, int k, fxc r, auto odd) {
        // the shift above rounded L inputs down, half a unit of the first step each on average: a sum
        // that lands on output 0 alone (a component that is zero in the whole column stays zero)
        if (k == 0) {
            constexpr unsigned half = L >> (fx_prescale(L) + 1);
            r = fxc{fx_add(r.x, fxr{r.x.l | (unsigned)r.x.h ? half : 0u, 0}), fx_add(r.y, fxr{r.y.l | (unsigned)r.y.h ? half : 0u, 0})};
        }
        const int eo = k - out_off;
        if (xin && eo >= 0 && eo < out_count) dst[(unsigned)eo * plane + col] = odd() ? fx_to_odd(r, un) : fx_to(r, un);
    };
    fft4_run<A, B, 1, true, false, NL, A, NO_>(v, s, tw, tid, st_g, un.odd);
}

}  // namespace lsm
