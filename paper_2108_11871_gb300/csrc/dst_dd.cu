// Sine-transform passes that keep double-float arithmetic (pairs of FP32, 48
// significant bits): the transform of u1 and of the boundary layers in the
// tensor-core modes, and the direct sums of line lengths without an FFT (FP64 or
// double-float).  Algorithm, data layout and epilogue of the FFT form are those of
// the pass in dst.cu; it runs on the FP32 pipe.
#include <type_traits>

#include "fft.cuh"

namespace idp {

namespace {

constexpr int NT = 256;

template <int K, int LBO = 0, int NTB = NT>
struct DstCfg {
    static constexpr int M = 2 * K;
    static constexpr int N = M - 1;
    // lines per block: 2 buffers x LB x M reals (32 KB for M >= 128), at
    // least 8 lines so that the scan groups fit a warp; LBO = 8 gives the
    // minimum (more blocks for small launches)
    static constexpr int LBr = (2048 / M) > 32 ? 32 : (2048 / M);
    // a power of two (so that LB * G = 256)
    static constexpr int LB0 = LBr >= 32 ? 32 : LBr >= 16 ? 16 : LBr >= 8 ? 8 : 4;
    static constexpr int LB = LBO ? LBO : (LB0 < 8 ? 8 : LB0);
    static constexpr int T = NTB;                 // threads per block
    static constexpr int G = T / LB;              // threads per line in the scan
    static constexpr int C = (K + G - 1) / G;     // scan elements per thread (the last ones guarded)
};

// element access for the two storage forms of a real value: FP64, or a
// double-float pair (the DD kernels keep intermediates in that form)
template <class R>
struct Io;
template <>
struct Io<double> {
    static __device__ __forceinline__ double ld(const void *p, int64_t i, int) { return reinterpret_cast<const double *>(p)[i]; }
    static __device__ __forceinline__ void st(void *p, int64_t i, double v, int) { reinterpret_cast<double *>(p)[i] = v; }
};
template <>
struct Io<ddr> {
    static __device__ __forceinline__ ddr ld(const void *p, int64_t i, int dd)
    {
        if (dd) return reinterpret_cast<const ddr *>(p)[i];
        return dd_from_bits(reinterpret_cast<const double *>(p)[i]);
    }
    static __device__ __forceinline__ void st(void *p, int64_t i, ddr v, int dd)
    {
        if (dd) reinterpret_cast<ddr *>(p)[i] = v;
        else reinterpret_cast<double *>(p)[i] = dd_to_bits(v);
    }
};

__device__ __forceinline__ double times4_exact(double x) { return x * 4.0; }
__device__ __forceinline__ ddr times4_exact(ddr x) { return Ar<ddr>::times4(x); }

// strides of a view along the line (u, v) coordinates and the element index e
// of a pass along `axis` (u, v = the other two axes in order)
__device__ __forceinline__ void view_strides(const View3 &w, int axis, int64_t &su, int64_t &sv, int64_t &se)
{
    if (axis == 2) { su = w.s0; sv = w.s1; se = w.s2; }
    else if (axis == 1) { su = w.s0; sv = w.s2; se = w.s1; }
    else { su = w.s1; sv = w.s2; se = w.s0; }
}

template <int K, int LBO, int NTB>
__global__ void __launch_bounds__(NTB) dst_dd_kernel(const DstPass a)
{
    pdl_enter();
    using R = ddr;
    using Cfg = DstCfg<K, LBO, NTB>;
    constexpr int NT = NTB;
    using A = Ar<R>;
    using Cx = typename A::C;
    constexpr int M = Cfg::M, N = Cfg::N, LB = Cfg::LB;
    extern __shared__ double2 smem_raw[];
    Cx *bufA = reinterpret_cast<Cx *>(smem_raw);   // LB * K complex
    Cx *bufB = bufA + LB * K;                      // LB * K complex
    // the FFT's K / 2 twiddles, copied into shared memory once (read in every pass; from
    // the global table they are long-scoreboard loads); visible after the first barrier
    using TwT = typename Ar<R>::T;
    static_assert(sizeof(TwT) <= 32, "the shared-memory size counts 32 bytes per twiddle");
    TwT *twsm = reinterpret_cast<TwT *>(bufB + LB * K);
    // in the bank-spread planes of tw_stage
    constexpr bool TWS = TwSwz<K>::ok;
    if constexpr (TWS) {
        tw_stage<K>(twsm, a.twd, threadIdx.x, NT);
    } else {
        const TwT *tg = a.twd;
        for (int i = threadIdx.x; i < K / 2; i += NT) twsm[i] = tg[i];
    }

    // line (u, v) coordinates: the two non-transform axes, v fastest.  The
    // strides are taken from the parameters where they are used, so that none
    // of them stays live across the FFT.
    const int nv = a.axis == 2 ? a.n1 : a.n2;
    const int u = blockIdx.y;
    const int v0 = blockIdx.x * LB;
    const int nl = min(LB, nv - v0);
    const bool contig = (a.axis == 2);

    // 1. load and pre-process in one step: the thread that forms y'_j and
    //    y'_{M-j} loads x_j and x_{M-j} itself (consecutive threads take
    //    consecutive j of a contiguous line, or consecutive lines), into bufA
    //    viewed as R[LB][M] (zf[j] = y'_j); lines past the end give zeros
    R *zf = reinterpret_cast<R *>(bufA);
    int64_t isu, isv, ise;
    view_strides(a.in, a.axis, isu, isv, ise);
    const int64_t inb = (int64_t)u * isu + (int64_t)v0 * isv;
    // all loads of the thread first (their latencies overlap), then the pre-pass
    // arithmetic and the shared-memory stores
    constexpr int IT = (LB * K + NT - 1) / NT;
    R xa[IT], xb[IT], sv[IT];
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int f = threadIdx.x + i * NT;
        xa[i] = A::zero();
        xb[i] = A::zero();
        sv[i] = A::zero();
        if (f < LB * K) {
            int l, j;
            if (contig) { l = f / K; j = f - l * K; }
            else { j = f / LB; l = f - j * LB; }
            const int64_t lb = inb + (int64_t)l * isv;   // x_i at element i-1 of the line
            if (j == 0) {
                if (l < nl) xa[i] = Io<R>::ld(a.in.p, lb + (int64_t)(K - 1) * ise, a.in_dd);
            } else {
                if (l < nl) {
                    xa[i] = Io<R>::ld(a.in.p, lb + (int64_t)(j - 1) * ise, a.in_dd);
                    xb[i] = Io<R>::ld(a.in.p, lb + (int64_t)(M - j - 1) * ise, a.in_dd);
                }
                sv[i] = a.sin2d[j];
            }
        }
    }
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int f = threadIdx.x + i * NT;
        if (f >= LB * K) break;
        int l, j;
        if (contig) { l = f / K; j = f - l * K; }
        else { j = f / LB; l = f - j * LB; }
        R *zl = zf + l * M;
        if (j == 0) {
            zl[0] = A::zero();
            zl[K] = l < nl ? times4_exact(xa[i]) : A::zero();
        } else {
            const R p = A::add(xa[i], xb[i]), m = A::sub(xa[i], xb[i]);
            zl[j] = A::fma(sv[i], p, m);
            zl[M - j] = A::fma(sv[i], p, A::neg(m));
        }
    }
    __syncthreads();

    // 3. complex FFT of length K, by the block
    Cx *Z = cta_fft_t<R, K, LB, NT, false, false, TWS>(bufA, bufB, twsm, false);
    R *o = reinterpret_cast<R *>(Z == bufA ? bufB : bufA);   // R[LB][M]

    // 4. post-processing: even outputs final, odd slots get Re T_k
    for (int f = threadIdx.x; f < LB * (K / 2); f += NT) {
        const int l = f / (K / 2);
        const int k = f - l * (K / 2) + 1;      // 1..K/2
        const Cx *zl = Z + l * K;
        R *ol = o + l * M;
        const Cx zk = zl[k], zc = zl[K - k];
        const R Er = A::add(A::re(zk), A::re(zc)), Ei = A::sub(A::im(zk), A::im(zc));
        const R Or = A::sub(A::re(zk), A::re(zc)), Oi = A::add(A::im(zk), A::im(zc));
        {
            const Cx w = a.halfd[k];
            const R Pr = A::mul_sub(A::re(w), Or, A::im(w), Oi);
            const R Pi = A::mul_add(A::re(w), Oi, A::im(w), Or);
            ol[2 * k - 1] = A::sub(Pr, Ei);
            ol[2 * (K - k) - 1] = A::add(Ei, Pr);
            ol[2 * k] = A::add(Er, Pi);
            ol[2 * (K - k)] = A::sub(Er, Pi);
        }
        if (k == 1) ol[0] = A::add(A::re(zl[0]), A::im(zl[0]));
    }
    __syncthreads();

    // 5. prefix sum over the odd slots o[2k], k = 0..K-1
    {
        constexpr int G = Cfg::G, C = Cfg::C;
        const int l = threadIdx.x / G;
        const int g = threadIdx.x - l * G;
        R vals[C];
        R run = A::zero();
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (g * C + c < K) run = A::add(run, o[l * M + 2 * (g * C + c)]);
            vals[c] = run;
        }
        // inclusive scan of the group totals (groups of G consecutive lanes)
        R incl = run;
#pragma unroll
        for (int dd = 1; dd < G; dd <<= 1) {
            const R nb = A::shfl_up(incl, dd, G);
            if (g >= dd) incl = A::add(incl, nb);
        }
        const R off = A::sub(incl, run);
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (g * C + c < K) o[l * M + 2 * (g * C + c)] = A::add(vals[c], off);
    }
    __syncthreads();

    // 6. epilogue and store
    int64_t osu, osv, ose, tsu, tsv, tse;
    view_strides(a.out, a.axis, osu, osv, ose);
    {
        // the tables are dense interior arrays n0 x n1 x n2
        const View3 tv{nullptr, (int64_t)a.n1 * a.n2, a.n2, 1};
        view_strides(tv, a.axis, tsu, tsv, tse);
    }
    const int64_t outb = (int64_t)u * osu + (int64_t)v0 * osv;
    const int64_t tabb = (int64_t)u * tsu + (int64_t)v0 * tsv;
    const bool has_tab = a.tab || a.tabd;
    if (!has_tab) {
        for (int f = threadIdx.x; f < LB * N; f += NT) {
            int l, e;
            if (contig) { l = f / N; e = f - l * N; }
            else { e = f / LB; l = f - e * LB; }
            if (l >= nl) continue;
            Io<R>::st(a.out.p, outb + (int64_t)l * osv + (int64_t)e * ose, o[l * M + e], a.out_dd);
        }
        return;
    }
    // groups of EG outputs: the table loads of a group go out before its stores
    // (which, as far as the compiler knows, could alias them)
    constexpr int EG = 4;
    for (int f0 = threadIdx.x; f0 < LB * N; f0 += EG * NT) {
        R tv[EG];
#pragma unroll
        for (int g = 0; g < EG; ++g) {
            const int f = f0 + g * NT;
            tv[g] = A::zero();
            if (f >= LB * N) continue;
            int l, e;
            if (contig) { l = f / N; e = f - l * N; }
            else { e = f / LB; l = f - e * LB; }
            if (l >= nl) continue;
            const int64_t ti = tabb + (int64_t)l * tsv + (int64_t)e * tse;
            tv[g] = Io<R>::ld(a.tabd ? (const void *)a.tabd : (const void *)a.tab, ti, a.tabd != nullptr);
        }
#pragma unroll
        for (int g = 0; g < EG; ++g) {
            const int f = f0 + g * NT;
            if (f >= LB * N) break;
            int l, e;
            if (contig) { l = f / N; e = f - l * N; }
            else { e = f / LB; l = f - e * LB; }
            if (l >= nl) continue;
            Io<R>::st(a.out.p, outb + (int64_t)l * osv + (int64_t)e * ose, A::mul(tv[g], o[l * M + e]), a.out_dd);
        }
    }
}

// Direct sine sums for line lengths without an FFT here (any M <= 513): every
// output U_e = 4 sum_i S[i][e] x_i with S[i][e] = sin(pi (i+1)(e+1) / M) from the
// table a.sinm (FP64, or double-float pairs when R is ddr), stored with e fastest
// so that consecutive threads read consecutive entries.  LBD lines per block, held
// in shared memory; thread t computes modes t, t + 256 for all of them.  The same
// epilogue as the FFT pass.
constexpr int LBD = 16, DMAX = 2;   // lines per block, modes per thread (N <= 512)

template <class R>
__global__ void __launch_bounds__(NT) dst_direct_kernel(const DstPass a)
{
    pdl_enter();
    using A = Ar<R>;
    const int M = a.M, N = M - 1;
    extern __shared__ double2 smem_raw[];
    R *xs = reinterpret_cast<R *>(smem_raw);   // [LBD][N]
    const int nv = a.axis == 2 ? a.n1 : a.n2;
    const int u = blockIdx.y;
    const int v0 = blockIdx.x * LBD;
    const int nl = min(LBD, nv - v0);
    const bool contig = (a.axis == 2);
    int64_t isu, isv, ise;
    view_strides(a.in, a.axis, isu, isv, ise);
    const int64_t inb = (int64_t)u * isu + (int64_t)v0 * isv;
    for (int f = threadIdx.x; f < LBD * N; f += NT) {
        int l, i;
        if (contig) { l = f / N; i = f - l * N; }
        else { i = f / LBD; l = f - i * LBD; }
        xs[l * N + i] = l < nl ? Io<R>::ld(a.in.p, inb + (int64_t)l * isv + (int64_t)i * ise, a.in_dd) : A::zero();
    }
    __syncthreads();
    R acc[DMAX][LBD];
#pragma unroll
    for (int j = 0; j < DMAX; ++j)
#pragma unroll
        for (int l = 0; l < LBD; ++l) acc[j][l] = A::zero();
    const R *S = reinterpret_cast<const R *>(a.sinm);
    for (int i = 0; i < N; ++i) {
#pragma unroll
        for (int j = 0; j < DMAX; ++j) {
            const int e = threadIdx.x + j * NT;
            if (e >= N) break;
            const R sv = S[(int64_t)i * N + e];
#pragma unroll
            for (int l = 0; l < LBD; ++l) acc[j][l] = A::fma(sv, xs[l * N + i], acc[j][l]);
        }
    }
    int64_t osu, osv, ose, tsu, tsv, tse;
    view_strides(a.out, a.axis, osu, osv, ose);
    {
        const View3 tv{nullptr, (int64_t)a.n1 * a.n2, a.n2, 1};
        view_strides(tv, a.axis, tsu, tsv, tse);
    }
    const int64_t outb = (int64_t)u * osu + (int64_t)v0 * osv;
    const int64_t tabb = (int64_t)u * tsu + (int64_t)v0 * tsv;
    const bool has_tab = a.tab || a.tabd;
#pragma unroll
    for (int j = 0; j < DMAX; ++j) {
        const int e = threadIdx.x + j * NT;
        if (e >= N) break;
#pragma unroll
        for (int l = 0; l < LBD; ++l) {
            if (l >= nl) break;
            R y = times4_exact(acc[j][l]);
            const int64_t ti = tabb + (int64_t)l * tsv + (int64_t)e * tse;
            if (has_tab)
                y = A::mul(Io<R>::ld(a.tabd ? (const void *)a.tabd : (const void *)a.tab, ti, a.tabd != nullptr), y);
            Io<R>::st(a.out.p, outb + (int64_t)l * osv + (int64_t)e * ose, y, a.out_dd);
        }
    }
}

template <class R>
cudaError_t launch_direct(const DstPass &a, cudaStream_t st)
{
    if (a.M - 1 > DMAX * NT || !a.sinm) return cudaErrorInvalidValue;
    int nu, nv;
    if (a.axis == 2) { nu = a.n0; nv = a.n1; }
    else if (a.axis == 1) { nu = a.n0; nv = a.n2; }
    else { nu = a.n1; nv = a.n2; }
    const size_t sm = sizeof(R) * LBD * (a.M - 1);
    dim3 grid((nv + LBD - 1) / LBD, nu);
    return launch_pdl(dst_direct_kernel<R>, grid, dim3(NT), sm, st, a);
}

template <int K, int LBO, int NTB = NT>
cudaError_t launch_lb(const DstPass &a, int nu, int nv, cudaStream_t st)
{
    using Cfg = DstCfg<K, LBO, NTB>;
    static_assert(Cfg::G <= 32, "scan group must fit a warp");
    static_assert(Cfg::LB * Cfg::G == NTB, "every thread belongs to one scan group");
    const size_t sm = 2 * sizeof(double2) * Cfg::LB * K + 32 * (K / 2);   // + the twiddles
    dim3 grid((nv + Cfg::LB - 1) / Cfg::LB, nu);
    return launch_pdl(dst_dd_kernel<K, LBO, NTB>, grid, dim3(NTB), sm, st, a);
}

template <int K>
cudaError_t launch_k(const DstPass &a, cudaStream_t st)
{
    int nu, nv;
    if (a.axis == 2) { nu = a.n0; nv = a.n1; }
    else if (a.axis == 1) { nu = a.n0; nv = a.n2; }
    else { nu = a.n1; nv = a.n2; }
    // 32 lines (M = 128) or 16 lines (M = 256) per block: the per-line prefix sum
    // then runs on at least half a warp (an FP64 warp instruction costs the pipe the
    // same whatever its active lanes)
    if constexpr (K == 64) {
        if (a.lines == 32) return launch_lb<K, 32>(a, nu, nv, st);
    }
    if constexpr (K == 128) {
        if (a.lines == 16) return launch_lb<K, 16>(a, nu, nv, st);
    }
    // 4 lines on 128 threads (M = 256, 512): a warp per line, smaller blocks
    if constexpr (K == 128 || K == 256) {
        if (a.lines == 4) return launch_lb<K, 4, 128>(a, nu, nv, st);
    }
    if constexpr (DstCfg<K>::LB > 8) {
        // a launch of less than two blocks per SM (the layer transforms) runs faster
        // on more, smaller blocks
        const int64_t blocks = (int64_t)nu * ((nv + DstCfg<K>::LB - 1) / DstCfg<K>::LB);
        if (a.lines == 8 || blocks < 2 * 152) return launch_lb<K, 8>(a, nu, nv, st);
        // 8 lines on 128 threads: one radix-4 unit per thread per pass for K = 64
        if (a.lines == -8 && K == 64) return launch_lb<K, 8, 128>(a, nu, nv, st);
    }
    return launch_lb<K, 0>(a, nu, nv, st);
}

template <int K, int LBO, int NTB = NT>
cudaError_t attr_lb()
{
    using Cfg = DstCfg<K, LBO, NTB>;
    const int sm = (int)(2 * sizeof(double2) * Cfg::LB * K + 32 * (K / 2));
    return cudaFuncSetAttribute(dst_dd_kernel<K, LBO, NTB>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

template <int K>
cudaError_t attr_k()
{
    cudaError_t e = attr_lb<K, 0>();
    if (e != cudaSuccess) return e;
    if constexpr (DstCfg<K>::LB > 8) {
        e = attr_lb<K, 8>();
    }
    if constexpr (K == 64) {
        if (e == cudaSuccess) e = attr_lb<K, 8, 128>();
        if (e == cudaSuccess) e = attr_lb<K, 32>();
    }
    if constexpr (K == 128) {
        if (e == cudaSuccess) e = attr_lb<K, 16>();
    }
    if constexpr (K == 128 || K == 256) {
        if (e == cudaSuccess) e = attr_lb<K, 4, 128>();
    }
    return e;
}

#define IDP_DST_SWITCH(M, CALL, OTHER)  \
    switch (M) {                         \
    case 16: { constexpr int K = 8; return CALL; }    \
    case 32: { constexpr int K = 16; return CALL; }   \
    case 48: { constexpr int K = 24; return CALL; }   \
    case 64: { constexpr int K = 32; return CALL; }   \
    case 96: { constexpr int K = 48; return CALL; }   \
    case 128: { constexpr int K = 64; return CALL; }  \
    case 192: { constexpr int K = 96; return CALL; }  \
    case 256: { constexpr int K = 128; return CALL; } \
    case 384: { constexpr int K = 192; return CALL; } \
    case 512: { constexpr int K = 256; return CALL; } \
    default: return OTHER;               \
    }

cudaError_t attr_m(int M) { IDP_DST_SWITCH(M, attr_k<K>(), cudaErrorInvalidValue) }

}  // namespace

cudaError_t dst_dd_set_attributes()
{
    cudaError_t e;
    for (int M : {16, 32, 48, 64, 96, 128, 192, 256, 384, 512})
        if ((e = attr_m(M)) != cudaSuccess) return e;
    const int sm = (int)(sizeof(double) * LBD * DMAX * NT);
    if ((e = cudaFuncSetAttribute(dst_direct_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm)))
        return e;
    return cudaFuncSetAttribute(dst_direct_kernel<ddr>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

// double-float FFT passes (dd = 1), and direct sums in FP64 or double-float for the
// lengths without an FFT
cudaError_t launch_dst_dd(const DstPass &a, cudaStream_t st)
{
    if (!a.dd) return launch_direct<double>(a, st);
    IDP_DST_SWITCH(a.M, launch_k<K>(a, st), launch_direct<ddr>(a, st))
}

}  // namespace idp
