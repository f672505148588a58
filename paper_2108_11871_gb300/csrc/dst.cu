// Sine-transform pass (section 3, eqs. rhoSinSeries / phiStarSoln2D; section 5,
// the sine eigenvectors of the compact operator): for every line of an
// interior box along one axis, U = 4 S x with S_{k,i} = sin(pi k i / M),
// k, i = 1..M-1, followed by a pointwise epilogue.
//
// Algorithm per line (M = 2K):
//   y'_j = 2 sin(pi j/M)(x_j + x_{M-j}) + (x_j - x_{M-j}),  y'_K = 4 x_K, y'_0 = 0
//   Z    = FFT_K(y'_{2m} + i y'_{2m+1})                    (complex, length K)
//   T_k  = (Z_k + conj Z_{K-k}) - i e^{-2 pi i k/M} (Z_k - conj Z_{K-k})
//   U_{2k} = -Im T_k,   U_{2k+1} = U_{2k-1} + Re T_k,   U_1 = Re Z_0 + Im Z_0
// (the real-FFT form of the DST-I; T = 4 Y where Y is the real FFT of y), in the
// block fixed-point arithmetic of q64.cuh, FP64 in and out.
#include "arith.cuh"
#include "q64.cuh"

namespace idp {

namespace {

// strides of a view along the line (u, v) coordinates and the element index e
// of a pass along `axis` (u, v = the other two axes in order)
__device__ __forceinline__ void view_strides(const View3 &w, int axis, int64_t &su, int64_t &sv, int64_t &se)
{
    if (axis == 2) { su = w.s0; sv = w.s1; se = w.s2; }
    else if (axis == 1) { su = w.s0; sv = w.s2; se = w.s1; }
    else { su = w.s1; sv = w.s2; se = w.s0; }
}

// Largest radix of the FFT of length K: short lines come in small launches, whose time
// is the latency of one block and shorter with radix-4 units (K <= 48); long ones are bound
// by the integer pipes, where radix 8 saves products and shared-memory round trips.
__host__ __device__ constexpr int dst_radix(int K) { return K <= 48 ? 4 : 8; }

// G threads per line, each with C = K / G of the line's pairs (x_j, x_{M-j}) in the
// load and of its odd outputs in the prefix sum; LB lines per block; radices up to RM
// (by the length alone: every shape runs the same arithmetic on a line).
template <int K, int LBO, int GO>
struct DstCfg {
    static constexpr int M = 2 * K, N = M - 1;
    static constexpr int G = GO, C = K / G, RM = dst_radix(K);
    static constexpr int LB = LBO, T = LB * G;
    static constexpr int LS = K + 1;                      // line stride of the FFT buffers (16-byte elements)
    static constexpr int OS = (2 * K + G + 1) | 1;        // line stride of the outputs (8-byte words, odd: lanes
                                                          // on consecutive lines hit different banks)
    static constexpr int BUF = (LB * (OS > 2 * LS ? OS : 2 * LS) + 1) / 2;   // 16-byte elements of one buffer
    // tables: FFT factors, e^{-i pi k/K} (k = 0..K/2), sin(pi j/M) (j = 0..K-1, 8 bytes each)
    static constexpr int TW = q_tw_count(K, RM), HALF = TW, SIN = TW + K / 2 + 1, TAB = SIN + K / 2;
    static constexpr size_t SMEM = sizeof(qc) * (2 * BUF + TAB);
    static_assert(K % G == 0 && (G & (G - 1)) == 0 && G <= 32 && T % 32 == 0 && T <= 256,
                  "whole warps; a group fits a warp");
};

template <class Cfg, int K>
__global__ void __launch_bounds__(Cfg::T) dst_pass_kernel(const DstPass a)
{
    constexpr int M = Cfg::M, N = Cfg::N, LB = Cfg::LB, NT = Cfg::T, G = Cfg::G, C = Cfg::C, RM = Cfg::RM;
    constexpr int LS = Cfg::LS, OS = Cfg::OS;
    extern __shared__ qc smem_q[];
    qc *bufA = smem_q, *bufB = smem_q + Cfg::BUF;
    int4 *tabs = reinterpret_cast<int4 *>(bufB + Cfg::BUF);
    __shared__ int s_emax[LB], s_scale[LB];
    __shared__ unsigned s_sum[LB];
    // the tables, made with the plan, come in while the previous launch drains (they are
    // visible after the first barrier)
    pdl_launch();
    {
        for (int i = threadIdx.x; i < Cfg::TAB; i += NT) tabs[i] = __ldg(a.qtab + i);
    }
    if (threadIdx.x < LB) {
        s_emax[threadIdx.x] = 1;
        s_sum[threadIdx.x] = 0;
    }
    pdl_wait();

    const int nv = a.axis == 2 ? a.n1 : a.n2;
    const int u = blockIdx.y;
    const int v0 = blockIdx.x * LB;
    const int nl = min(LB, nv - v0);
    const bool contig = (a.axis == 2);

    // 1. load: thread (l, g) takes the pairs x_j, x_{M-j}, j = g + i G, of line l
    //    (consecutive threads on consecutive j of a contiguous line, or on
    //    consecutive lines); j = 0 stands for the middle element x_K
    const int l = contig ? threadIdx.x / G : threadIdx.x % LB;
    const int g = contig ? threadIdx.x % G : threadIdx.x / LB;
    double xa[C], xb[C];
    {
        int64_t isu, isv, ise;
        view_strides(a.in, a.axis, isu, isv, ise);
        const double *in = a.in.p + (int64_t)u * isu + (int64_t)(v0 + l) * isv;   // x_i at element i - 1
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int j = g + i * G;
            xa[i] = 0.0;
            xb[i] = 0.0;
            if (l < nl) {
                xa[i] = in[(int64_t)((j ? j : K) - 1) * ise];
                if (j) xb[i] = in[(int64_t)(M - j - 1) * ise];
            }
        }
        if (a.in_dd) {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                xa[i] = dd_to_bits(*reinterpret_cast<const ddr *>(&xa[i]));
                xb[i] = dd_to_bits(*reinterpret_cast<const ddr *>(&xb[i]));
            }
        }
    }

    // 2. the line's scale, from its largest exponent and its absolute sum
    int emax = 1;
#pragma unroll
    for (int i = 0; i < C; ++i) emax = max(emax, max(q_expo(xa[i]), q_expo(xb[i])));
    // lanes of one line: G consecutive ones, or those LB apart
    const int d0 = contig ? 1 : LB, d1 = contig ? G : 32;
    for (int d = d0; d < d1; d <<= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, d));
    __syncthreads();
    const bool lead = contig ? g == 0 : (threadIdx.x & 31) < LB;
    if (lead) atomicMax(&s_emax[l], emax);
    __syncthreads();
    emax = s_emax[l];
    unsigned sum = 0;
#pragma unroll
    for (int i = 0; i < C; ++i) sum += q_weight(xa[i], emax) + q_weight(xb[i], emax);
    for (int d = d0; d < d1; d <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lead) atomicAdd(&s_sum[l], sum);
    __syncthreads();
    const int bits = q_bits(s_sum[l]);
    if (threadIdx.x < LB) {
        const int e = s_emax[threadIdx.x];
        s_scale[threadIdx.x] = e == 0x7ff ? Q_NAN : 1101 - e - q_bits(s_sum[threadIdx.x]);
    }

    // 3. pre-processing into bufA viewed as y'[LB][M] (y'_j in component j mod 2 of
    //    element j / 2): y'_j = sin(pi j/M) (2 x_j + 2 x_{M-j}) + (x_j - x_{M-j})
    {
        long long *zl = reinterpret_cast<long long *>(bufA + l * LS);
        const int shift = emax + bits - 19;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int j = g + i * G;
            const long long va = q_from(xa[i], shift), vb = q_from(xb[i], shift);
            const int2 sn = reinterpret_cast<const int2 *>(tabs + Cfg::SIN)[j];
            const long long p = q_rmul((va + vb) << 1, sn.x, sn.y), m = va - vb;
            const int j1 = j ? M - j : K;
            zl[2 * q_slot(j >> 1) + (j & 1)] = j ? p + m : 0;
            zl[2 * q_slot(j1 >> 1) + (j1 & 1)] = j ? p - m : va << 2;
        }
    }
    __syncthreads();

    // 4. complex FFT of length K
    q_fft<K, RM, LB, NT, LS>(bufA, bufB, tabs);
    constexpr bool INA = q_passes(K, RM) % 2 == 0;
    const qc *Z = INA ? bufA : bufB;
    long long *o = reinterpret_cast<long long *>(INA ? bufB : bufA);
    // outputs of a line: U_{2k} at word k - 1; the odd slots (Re T_k, then U_{2k+1}) at
    // word K + k + k / C (one word of padding per thread of the prefix sum)

    // 5. post-processing: even outputs final, odd slots get Re T_k
    for (int f = threadIdx.x; f < LB * (K / 2); f += NT) {
        const int ll = f / (K / 2);
        const int k = f - ll * (K / 2) + 1;      // 1..K/2
        const qc *zl = Z + ll * LS;
        long long *ol = o + ll * OS;
        const qc zk = zl[q_slot(k)], zc = zl[q_slot(K - k)];
        const long long Er = zk.re + zc.re, Ei = zk.im - zc.im;
        const qc P = q_cmul(qc{zk.re - zc.re, zk.im + zc.im}, tabs[Cfg::HALF + k]);
        ol[k - 1] = P.re - Ei;
        ol[K - k - 1] = P.re + Ei;
        ol[K + k + k / C] = Er + P.im;
        ol[K + (K - k) + (K - k) / C] = Er - P.im;
        if (k == 1) ol[K] = zl[0].re + zl[0].im;
    }
    __syncthreads();

    // 6. prefix sum over the odd slots: G lanes per line, C consecutive slots each
    {
        const int ll = threadIdx.x / G, gg = threadIdx.x % G;
        long long *ol = o + ll * OS + K + gg * (C + 1);
        long long val[C], run = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            run += ol[c];
            val[c] = run;
        }
        long long incl = run;
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            const long long nb = __shfl_up_sync(0xffffffffu, incl, d, G);
            if (gg >= d) incl += nb;
        }
        const long long below = incl - run;
#pragma unroll
        for (int c = 0; c < C; ++c) ol[c] = val[c] + below;
    }
    __syncthreads();

    // 7. epilogue and store
    int64_t osu, osv, ose, asu, asv, ase, tsu, tsv, tse;
    view_strides(a.out, a.axis, osu, osv, ose);
    view_strides(a.add, a.axis, asu, asv, ase);
    {
        // the tables are dense interior arrays n0 x n1 x n2
        const View3 tv{nullptr, (int64_t)a.n1 * a.n2, a.n2, 1};
        view_strides(tv, a.axis, tsu, tsv, tse);
    }
    double *out = a.out.p + (int64_t)u * osu + (int64_t)v0 * osv;
    const double *tab = a.tab + ((int64_t)u * tsu + (int64_t)v0 * tsv);
    const double *add = a.add.p + ((int64_t)u * asu + (int64_t)v0 * asv);
    // groups of EG outputs: the table and addend loads of a group go out before
    // its stores (which, as far as the compiler knows, could alias them)
    constexpr int EG = 4;
    for (int f0 = threadIdx.x; f0 < LB * N; f0 += EG * NT) {
        double tv[EG], av[EG];
        if (a.tab || a.add.p) {
#pragma unroll
            for (int q = 0; q < EG; ++q) {
                const int f = f0 + q * NT;
                int ll, e;
                if (contig) { ll = f / N; e = f - ll * N; }
                else { e = f / LB; ll = f - e * LB; }
                tv[q] = 1.0;
                av[q] = 0.0;
                if (f >= LB * N || ll >= nl) continue;
                if (a.tab) tv[q] = tab[(int64_t)ll * tsv + (int64_t)e * tse];
                if (a.add.p) av[q] = add[(int64_t)ll * asv + (int64_t)e * ase];
            }
        }
#pragma unroll
        for (int q = 0; q < EG; ++q) {
            const int f = f0 + q * NT;
            if (f >= LB * N) break;
            int ll, e;
            if (contig) { ll = f / N; e = f - ll * N; }
            else { e = f / LB; ll = f - e * LB; }
            if (ll >= nl) continue;
            const int h = e >> 1, s = s_scale[ll];
            const long long w = o[ll * OS + ((e & 1) ? h : K + h + h / C)];
            double y = q_to(w, s, q_fast(s));
            if (a.tab) y = a.add.p ? fma(tv[q], y, av[q]) : tv[q] * y;
            else if (a.add.p) y += av[q];
            out[(int64_t)ll * osv + (int64_t)e * ose] = y;
        }
    }
}

template <class Cfg, int K>
cudaError_t launch_cfg(const DstPass &a, int nu, int nv, cudaStream_t st)
{
    return launch_pdl(dst_pass_kernel<Cfg, K>, dim3((nv + Cfg::LB - 1) / Cfg::LB, nu), dim3(Cfg::T), Cfg::SMEM, st, a);
}

// The shapes of a pass: Big (up to 256 threads, C = 8 or 12 pairs a thread), Mid with half
// its lines, and Thin with up to four times the threads per line, for launches that leave most of the chip idle and so are as long as one block.
template <int K>
struct DstShapes {
    static constexpr int G = K % 3 == 0 ? K / 12 : K / 8;
    static constexpr int BIG = 256 / G < 32 ? 256 / G : 32;
    static constexpr int MID = BIG / 2 * G >= 32 ? BIG / 2 : BIG;
    static constexpr int GT = 4 * G < 32 ? 4 * G : 32;
    static constexpr int THIN = GT >= 32 ? 2 : GT >= 16 ? 4 : 8;
    using Big = DstCfg<K, BIG, G>;
    using Mid = DstCfg<K, MID, G>;
    using Thin = DstCfg<K, THIN, GT>;
};

template <int K>
cudaError_t launch_k(const DstPass &a, cudaStream_t st)
{
    using S = DstShapes<K>;
    int nu, nv;
    if (a.axis == 2) { nu = a.n0; nv = a.n1; }
    else if (a.axis == 1) { nu = a.n0; nv = a.n2; }
    else { nu = a.n1; nv = a.n2; }
    int lines = a.lines > 0 ? a.lines : 0;
    if (!lines) {
        const int64_t all = (int64_t)nu * nv;
        // Big from twelve of its blocks per SM on (129^3, 508 Big blocks: 250 us per solve
        // with Big, 235 with Mid; 257^3 and 513^3: Big 3 % and 10 % ahead), Thin below four Mid
        // blocks per SM (33 x 65 x 97: 117 us per solve with Mid, 77 with Thin)
        lines = all >= (int64_t)152 * 12 * S::BIG ? 32 : all >= (int64_t)152 * 4 * S::MID ? 16 : 8;
    }
    if (lines == 32) return launch_cfg<typename S::Big, K>(a, nu, nv, st);
    if (lines == 16) return launch_cfg<typename S::Mid, K>(a, nu, nv, st);
    return launch_cfg<typename S::Thin, K>(a, nu, nv, st);
}

template <class Cfg, int K>
cudaError_t attr_cfg()
{
    return cudaFuncSetAttribute(dst_pass_kernel<Cfg, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
}

template <int K>
cudaError_t attr_k()
{
    using S = DstShapes<K>;
    cudaError_t e = attr_cfg<typename S::Big, K>();
    if (e == cudaSuccess) e = attr_cfg<typename S::Mid, K>();
    if (e == cudaSuccess) e = attr_cfg<typename S::Thin, K>();
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

cudaError_t dst_set_attributes()
{
    cudaError_t e;
    for (int M : {16, 32, 48, 64, 96, 128, 192, 256, 384, 512})
        if ((e = attr_m(M)) != cudaSuccess) return e;
    return dst_dd_set_attributes();
}

cudaError_t launch_dst_pass(const DstPass &a, cudaStream_t st)
{
    if (a.dd) return launch_dst_dd(a, st);
    IDP_DST_SWITCH(a.M, launch_k<K>(a, st), launch_dst_dd(a, st))
}

int q_table_radix(int L, int Ns, int RM) { return q_radix(L, Ns, RM); }
int q_table_count(int L, int RM) { return q_tw_count(L, RM); }
int dst_table_radix(int K) { return dst_radix(K); }

}  // namespace idp
