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
//
// What bounds it (257^3, 115 us a pass, of which its bytes need 40): no single unit.  The two
// integer pipes are busy 36-47 % of the time, the FP64 pipe, which converts, 47-60 %, and
// shared memory 34-47 %, in turns, because the blocks of an SM are in different phases; half
// of the warps fit (64 registers).  In FP64 the pass was bound by the FP64 pipe: 250 us at
// 257^3, 3.9 ms at 513^3 (now 0.98).
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
    static constexpr int LS = q_line(K);                  // line stride of the FFT buffers (16-byte elements)
    // outputs of a line (8-byte words): U_{2k} at q_slot(k - 1), the odd slots (Re T_k, then
    // U_{2k+1}) at OD + q_slot(k); line stride OS, odd (lanes on consecutive lines hit
    // different banks)
    static constexpr int OD = q_slot(K), OS = 2 * OD - 1;
    static constexpr int BUF = LB * LS;                   // 16-byte elements of one buffer
    static_assert(OS <= 2 * LS, "the outputs fit a buffer");
    // tables: FFT factors, e^{-i pi k/K} (k = 0..K/2), sin(pi j/M) (j = 0..K-1, 8 bytes each)
    static constexpr int TW = q_tw_count(K, RM), HALF = TW, SIN = TW + K / 2 + 1, TAB = SIN + K / 2;
    static constexpr size_t SMEM = sizeof(qc) * (BUF + TAB);
    static constexpr int BPS = 1024 / T;   // blocks per SM that the registers allow
    // contiguous outputs: whole warps on one line at a time (LW lines of a warp)
    static constexpr bool WIDE = G < 32 && (2 * K) % 32 == 0;
    static constexpr int LW = 32 / G;
    static_assert(K % G == 0 && (G & (G - 1)) == 0 && G <= 32 && T % 32 == 0 && T <= 256,
                  "whole warps; a group fits a warp");
};

template <class Cfg, int K>
__global__ void __launch_bounds__(Cfg::T, Cfg::BPS) dst_pass_kernel(const DstPass a)
{
    constexpr int M = Cfg::M, N = Cfg::N, LB = Cfg::LB, NT = Cfg::T, G = Cfg::G, C = Cfg::C, RM = Cfg::RM;
    constexpr int LS = Cfg::LS, OS = Cfg::OS, LW = Cfg::LW;
    constexpr bool WIDE = Cfg::WIDE;
    extern __shared__ qc smem_q[];
    qc *buf = smem_q;
    int4 *tabs = reinterpret_cast<int4 *>(buf + Cfg::BUF);
    __shared__ int s_high[LB], s_scale[LB], s_gmax;
    __shared__ unsigned s_sum[LB];
    // the tables, made with the plan, come in while the previous launch drains (they are
    // visible after the first barrier)
    pdl_launch();
    {
        for (int i = threadIdx.x; i < Cfg::TAB; i += NT) tabs[i] = __ldg(a.qtab + i);
    }
    if (threadIdx.x == 0) s_gmax = 0;
    if (threadIdx.x < LB) {
        s_high[threadIdx.x] = 0;
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
        const double *pa = in + (int64_t)(g - 1) * ise, *pb = in + (int64_t)(M - 1 - g) * ise;
        const int64_t step = G * ise;
        const bool on = l < nl;
#pragma unroll
        for (int i = 0; i < C; ++i, pa += step, pb -= step) {
            const bool mid = i == 0 && g == 0;
            xa[i] = on ? *(mid ? in + (int64_t)(K - 1) * ise : pa) : 0.0;
            xb[i] = on && !mid ? *pb : 0.0;
        }
    }

    // 2. the line's scale, from its largest exponent and its absolute sum (q64.cuh)
    int high = 0;
#pragma unroll
    for (int i = 0; i < C; ++i) high = max(high, max(q_high(xa[i]), q_high(xb[i])));
    // values that are not finite stay out of the conversions: the line's marker stands for them.
    // (With many values a thread the compiler mixes the loads and the reductions without a branch
    // here, 112 -> 123 us a pass at 257^3; short launches are faster without it, 33 x 65 x 97
    // 142 -> 137 us per solve.)
    if (C > 4 && high >= 0x7ff00000) {
#pragma unroll
        for (int i = 0; i < C; ++i) xa[i] = xb[i] = 0.0;
    }
    // lanes of one line: G consecutive ones, or those LB apart
    const int d0 = contig ? 1 : LB, d1 = contig ? G : 32;
    for (int d = d0; d < d1; d <<= 1) high = max(high, __shfl_xor_sync(0xffffffffu, high, d));
    __syncthreads();
    const bool lead = contig ? g == 0 : (threadIdx.x & 31) < LB;
    if (lead) atomicMax(&s_high[l], high);
    __syncthreads();
    const int emax = q_emax(s_high[l]);
    unsigned sum = 2 * C;
#pragma unroll
    for (int i = 0; i < C; ++i) sum += q_weight(xa[i], emax) + q_weight(xb[i], emax);
    for (int d = d0; d < d1; d <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lead) atomicAdd(&s_sum[l], sum);
    __syncthreads();
    const int eb = emax + q_bits(s_sum[l]), scale = 1101 - eb;   // absolute sum below 2^58 units
    if (g == 0) {
        s_scale[l] = emax == 0x7ff ? Q_NAN : scale;
        if (a.gmax && l < nl) atomicMax(&s_gmax, emax == 0x7ff ? Q_GNAN : eb);
    }

    // 3. pre-processing into buf viewed as y'[LB][M] (y'_j in component j mod 2 of
    //    element j / 2): y'_j = sin(pi j/M) (2 x_j + 2 x_{M-j}) + (x_j - x_{M-j})
    {
        long long *zl = reinterpret_cast<long long *>(buf + l * LS);
        const int2 *sn = reinterpret_cast<const int2 *>(tabs + Cfg::SIN) + g;
        const QFrom from(scale, emax);
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int j = g + i * G;
            const bool mid = i == 0 && g == 0;
            const long long va = from(xa[i]), vb = from(xb[i]);
            const int2 w = sn[i * G];
            const long long p = q_rmul((va + vb) << 1, w.x, w.y), m = va - vb;
            const int j1 = mid ? K : M - j;
            zl[2 * q_slot(j >> 1) + (j & 1)] = mid ? 0 : p + m;
            zl[2 * q_slot(j1 >> 1) + (j1 & 1)] = mid ? va << 2 : p - m;
        }
    }
    __syncthreads();

    if (a.gmax && threadIdx.x == 0 && *a.gmax < s_gmax) atomicMax(a.gmax, s_gmax);

    // 4. complex FFT of length K
    q_fft<K, RM, LB, NT, LS>(buf, tabs);

    // 5. post-processing, in place like the passes: even outputs final, odd slots get
    //    Re T_k.  From here to the prefix sum: G consecutive threads per line
    const int ll = threadIdx.x / G, gg = threadIdx.x % G;
    long long *o = reinterpret_cast<long long *>(buf), *ol = o + ll * OS;
    {
        constexpr int H = (K / 2 + G - 1) / G;
        const qc *zl = buf + ll * LS;
        const int4 *half = tabs + Cfg::HALF;
        qc zk[H], zc[H], z0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const int k = min(1 + gg + i * G, K / 2);   // 1..K/2
            zk[i] = zl[q_slot(k)];
            zc[i] = zl[q_slot(K - k)];
        }
        if (gg == 0) z0 = zl[0];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const int k = min(1 + gg + i * G, K / 2);
            const long long Er = zk[i].re + zc[i].re, Ei = zk[i].im - zc[i].im;
            const qc P = q_cmul(qc{zk[i].re - zc[i].re, zk[i].im + zc[i].im}, half[k]);
            ol[q_slot(k - 1)] = P.re - Ei;
            ol[q_slot(K - k - 1)] = P.re + Ei;
            ol[Cfg::OD + q_slot(k)] = Er + P.im;
            ol[Cfg::OD + q_slot(K - k)] = Er - P.im;
        }
        if (gg == 0) ol[Cfg::OD] = z0.re + z0.im;
    }
    __syncthreads();

    // 6. prefix sum over the odd slots: C consecutive ones per lane
    {
        long long val[C], run = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            run += ol[Cfg::OD + q_slot(gg * C + c)];
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
        for (int c = 0; c < C; ++c) ol[Cfg::OD + q_slot(gg * C + c)] = val[c] + below;
    }
    __syncthreads();

    // 7. epilogue and store: thread (l, g) of the load takes the outputs e = g + i G of line l
    //    (U_{e+1}); consecutive threads again on consecutive e or on consecutive lines
    int64_t osu, osv, ose;
    view_strides(a.out, a.axis, osu, osv, ose);
    if (WIDE && contig && !a.tab) {
        // lines along axis 2: a warp writes its lines one after the other, 32 outputs at a time,
        // in half as many pieces of 128-byte lines as the mapping below has: nothing to gain in
        // device memory (257^3: 114.5 us a pass either way), but phi in host memory goes out over
        // the link (host-buffer solve at 129^3: 662 -> 624 us)
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int b = 0; b < LW; ++b) {
            const int ln = threadIdx.x / 32 * LW + b;
            if (ln >= nl) return;
            double *out = a.out.p + (int64_t)u * osu + (int64_t)(v0 + ln) * osv + lane;
            const QTo to(s_scale[ln]);
            const long long *w0 = o + ln * OS + ((lane & 1) ? 0 : Cfg::OD);
#pragma unroll
            for (int i = 0; i < 2 * K / 32; ++i)
                if (i < 2 * K / 32 - 1 || lane < 31) out[i * 32] = to(w0[q_slot(i * 16 + (lane >> 1))]);
        }
        return;
    }
    if (l >= nl) return;
    double *out = a.out.p + (int64_t)u * osu + (int64_t)(v0 + l) * osv + (int64_t)g * ose;
    const int64_t step = G * ose;
    const QTo to(s_scale[l]);
    const long long *w0 = o + l * OS;
    auto word = [&](int i) -> long long {
        const int e = g + i * G, h = e >> 1;
        return w0[((e & 1) ? 0 : Cfg::OD) + q_slot(h)];
    };
    if (!a.tab) {
#pragma unroll
        for (int i = 0; i < 2 * C; ++i, out += step)
            if (i < 2 * C - 1 || g + i * G < N) *out = to(word(i));
        return;
    }
    int64_t tsu, tsv, tse;
    // the table is a dense interior array n0 x n1 x n2
    view_strides(View3{nullptr, (int64_t)a.n1 * a.n2, a.n2, 1}, a.axis, tsu, tsv, tse);
    const double *tab = a.tab + ((int64_t)u * tsu + (int64_t)(v0 + l) * tsv + (int64_t)g * tse);
    // groups of EG outputs: the table loads of a group go out before its stores (which, as
    // far as the compiler knows, could alias them)
    constexpr int EG = (2 * C) % 4 == 0 ? 4 : 2;
#pragma unroll
    for (int i0 = 0; i0 < 2 * C; i0 += EG) {
        double tv[EG];
#pragma unroll
        for (int q = 0; q < EG; ++q) {
            const int i = i0 + q;
            tv[q] = i < 2 * C - 1 || g + i * G < N ? tab[(int64_t)(i * G) * tse] : 1.0;
        }
#pragma unroll
        for (int q = 0; q < EG; ++q, out += step) {
            const int i = i0 + q;
            if (i == 2 * C - 1 && g + i * G >= N) break;
            *out = tv[q] * to(word(i));
        }
    }
}

template <class Cfg, int K>
cudaError_t launch_cfg(const DstPass &a, int nu, int nv, cudaStream_t st)
{
    return launch_pdl(dst_pass_kernel<Cfg, K>, dim3((nv + Cfg::LB - 1) / Cfg::LB, nu), dim3(Cfg::T), Cfg::SMEM, st, a);
}

// The shapes of a pass: Big (up to 256 threads, C = 8 or 6 pairs a thread), Mid with half
// its lines, and Thin with up to four times the threads per line, for launches that leave most
// of the chip idle and so are as long as one block.
template <int K>
struct DstShapes {
    static constexpr int G = K % 3 == 0 ? K / 6 : K / 8;
    static constexpr int BIG = 256 / G < 32 ? 256 / G : 32;
    static constexpr int MID = BIG / 2 * G >= 32 ? BIG / 2 : BIG;
    static constexpr int GT = (K % 3 == 0 ? 2 : 4) * G < 32 ? (K % 3 == 0 ? 2 : 4) * G : 32;
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
        // Big from twelve of its blocks per SM on (passes of a solve, Big and Mid: 129^3,
        // 508 Big blocks, 197 and 179 us; 257^3 1001 and 1035 us; 513^3 7.8 and 10.8 ms), Thin
        // below four Mid blocks per SM (33 x 65 x 97: 117 us per solve with Mid, 77 with Thin)
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
