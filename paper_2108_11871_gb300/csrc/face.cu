// Boundary stage 2 (section 4) in block fixed point: for the two faces of axis a, the FFT
// of length L = 2 P_b along b of every slice p, times the kernel spectra, summed over
// the slices (and the sum of the partial results, stage 3a's input).
//
// The two faces are mirror images: with p' = np - 1 - p, face 0 weighs slice p by k_p
// and face 1 by k_p'.  So the kernel works on the pair sums X_p + X_p' with
// (k_p + k_p') / 2 and on the differences X_p - X_p' with (k_p - k_p') / 2; their
// sums over the pairs, S and D, give face 0 = S + D and face 1 = S - D.  Against weighing
// every slice twice this halves the products and reads every spectrum once.
//
// Arithmetic (q64.cuh): one scale for all columns and slices of a pass, from bounds on the
// lines of stage 1 summed over each slice (slices x the largest line's bound left a single charged
// line eight bits short at 257^3: g off by 1.9e-13, with the sums by 2.4e-15, FP64 2.2e-15); the
// spectra of each frequency pair (b, c) are fractions of a power of two, up to 1 each and up to 4
// in sum over the slices: a low frequency weighs every slice alike, by a few hundredths at most,
// and what a product is rounded to counts against that.  So neither a transform nor a sum can
// overflow: columns are below 2^61 units, S and D below 2^62 and S +- D below 2^63.  (One power
// for all frequencies leaves the products' rounding as white noise over them: measured 1e-12
// of g on mixed-sign densities.)  White noise, g off by, with the first bounds and now (FP64): 129^3 5.5e-15 and 1.6e-15
// (1.5e-15), 257^3 2.5e-14 and 4.5e-15 (2.5e-15), 513^3 8.7e-14 and 5.1e-15 (2.4e-15).
#include "fft.cuh"
#include "q64.cuh"

namespace idp {

namespace {

// TC columns (consecutive frequencies c) per block and E = 8 elements (3 * 2^m: 6) of a
// column per thread: one or two units of the last pass, whose sums it keeps in registers.
// The line stride makes the first pass's writes conflict-free (8 / TC units of TC columns
// at a time).
template <int L_>
struct FaceQCfg {
    static constexpr int L = L_, RM = 8, E = L % 3 == 0 ? 6 : 8;
    static constexpr int last(int Ns)
    {
        return Ns * q_radix(L_, Ns, 8) == L_ ? q_radix(L_, Ns, 8) : last(Ns * q_radix(L_, Ns, 8));
    }
    static constexpr int RL = last(1), UL = L / RL, IL = E / RL;   // the last pass: radix, units, units per thread
    static constexpr int TC = 256 * E / L < 32 ? 256 * E / L : 32, NT = TC * L / E;
    // the registers allow 768 threads of 80 (with two blocks of 256 of them at 124 registers
    // the passes ran 15 % slower at 257^3)
    static constexpr int BPS = 768 / NT;
    static constexpr int LSM = TC <= 4 ? 2 : 1, LS = q_slot(L) + (LSM + 8 - q_slot(L) % 8) % 8;
    static constexpr int Ph = L / 2, KS = Ph + 1;
    static constexpr int R0 = q_radix(L, 1, RM), TW = q_tw_count(L, RM);
    static constexpr size_t SMEM = sizeof(qc) * (TC * LS + TW) + sizeof(int2) * TC * KS;
};

__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Signs in turn (q64.cuh) over the pairs and the column blocks, by the pair's number, so that
// the sums are the same integers for every chunk count.  ALT: an odd number of chunks, where
// the pairs of a chunk alternate and the sum so far is turned with each of them (r - sum in place
// of sum + r); with an even number all pairs of a chunk have one sign.
template <int L, bool ALT>
__global__ void __launch_bounds__(FaceQCfg<L>::NT, FaceQCfg<L>::BPS) face_q_kernel(const FaceQPass a)
{
    using Cfg = FaceQCfg<L>;
    constexpr int TC = Cfg::TC, NT = Cfg::NT, LS = Cfg::LS, KS = Cfg::KS, Ph = Cfg::Ph, R0 = Cfg::R0;
    constexpr int RL = Cfg::RL, UL = Cfg::UL, IL = Cfg::IL;
    extern __shared__ qc smem_q[];
    qc *buf = smem_q;
    int4 *tws = reinterpret_cast<int4 *>(buf + TC * LS);
    int2 *ks = reinterpret_cast<int2 *>(tws + Cfg::TW);
    const int c0 = blockIdx.x * TC, ncl = min(TC, a.nc - c0);
    const int chunk = blockIdx.y, diff = blockIdx.z;
    const int npair = (a.np + 1) / 2;
    // (the factors come in while the unit is found)
    for (int f = threadIdx.x; f < Cfg::TW; f += NT)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(tws + f)),
                     "l"(a.q + f)
                     : "memory");
    const int g = min(*a.gmax, 2100);
    // The unit: every column's absolute sum, at most twice that of the slices' line bounds, below 2^61
    // units.  b: the largest sum over a pair of slices in units of 2^(32 win - 1064); lines two
    // windows below the largest one's add up to less than the 1
    __shared__ int s_bound[NT / 32];
    const int win = g >> 5;
    {
        float b = 0.0f;
        for (int pr = threadIdx.x; pr < npair; pr += NT) {
            const int p2 = a.np - 1 - pr;
            const unsigned long long *s1 = a.sums + (int64_t)win * a.nsum, *s0 = s1 - a.nsum;
            const unsigned long long hi = s1[pr] + (p2 > pr ? s1[p2] : 0);
            const unsigned long long lo = win > 0 ? s0[pr] + (p2 > pr ? s0[p2] : 0) : 0;
            b = fmaxf(b, __fadd_ru(__ull2float_ru(hi), __fmul_ru(__ull2float_ru(lo), 0x1p-32f)));
        }
        const int m = __reduce_max_sync(0xffffffffu, __float_as_int(__fadd_ru(b, 1.0f)));
        if ((threadIdx.x & 31) == 0) s_bound[threadIdx.x >> 5] = m;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    int bound = 0;
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) bound = max(bound, s_bound[i]);
    const int unit = 1124 - ((bound >> 23) - 126) - 32 * win;
    if (threadIdx.x == 0 && blockIdx.x + blockIdx.y + blockIdx.z == 0) *a.unit = unit;
    int turns = blockIdx.x + chunk;
    QFrom from(unit, g - 31, q_turn(turns));
    const int2 *kq = a.kq + ((int64_t)diff * npair * a.nc + c0) * KS;

    // a unit of the last pass: column, frequencies j + q UL
    auto column = [](int it) { return (int)(threadIdx.x + it * NT) / UL; };
    auto freq = [](int it) { return (int)(threadIdx.x + it * NT) % UL; };
    qc acc[IL][RL];
#pragma unroll
    for (int it = 0; it < IL; ++it)
#pragma unroll
        for (int q = 0; q < RL; ++q) acc[it][q] = qc{0, 0};

    for (int pr = chunk; pr < npair; pr += a.nchunk) {
        const int p2 = a.np - 1 - pr;
        const bool two = pr != p2;
        // slices of zeros contribute nothing; the middle slice has no difference
        if (!(a.sliceflag[pr] | a.sliceflag[p2]) || (!two && diff)) {
            if constexpr (ALT) {
                from.flip();
                ++turns;
#pragma unroll
                for (int it = 0; it < IL; ++it)
#pragma unroll
                    for (int q = 0; q < RL; ++q) acc[it][q] = qc{-acc[it][q].re, -acc[it][q].im};
            }
            continue;
        }
        {
            const int2 *src = kq + (int64_t)pr * a.nc * KS;
            for (int f = threadIdx.x; f < ncl * KS; f += NT) cp_async8(ks + f, src + f);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        }
        // the first pass (radix R0, no factors) on the load: data at positions 1..Mb-1 of
        // a column, zeros elsewhere, in particular from L / 2 on
        {
            constexpr int U0 = L / R0, NZ = R0 / 2;   // units, inputs that can be non-zero
            const double2 *x1 = a.D + (int64_t)pr * a.sp + (int64_t)c0 * a.sc;
            const double2 *x2 = a.D + (int64_t)p2 * a.sp + (int64_t)c0 * a.sc;
#pragma unroll 2
            for (int f = threadIdx.x; f < TC * U0; f += NT) {
                const int jj = f / TC, t = f - jj * TC;   // consecutive threads: consecutive columns
                double2 y1[NZ], y2[NZ];
#pragma unroll
                for (int q = 0; q < NZ; ++q) {
                    const int pos = jj + q * U0;
                    const bool on = t < ncl && pos >= 1 && pos < a.Mb;
                    const int64_t at = (int64_t)(pos - 1) * a.sb + (int64_t)t * a.sc;
                    y1[q] = on ? x1[at] : make_double2(0.0, 0.0);
                    y2[q] = on && two ? x2[at] : make_double2(0.0, 0.0);
                }
                qc v[R0];
#pragma unroll
                for (int q = 0; q < R0; ++q) {
                    v[q] = qc{0, 0};
                    if (q < NZ) {
                        const double sr = diff ? y1[q].x - y2[q].x : y1[q].x + y2[q].x;
                        const double si = diff ? y1[q].y - y2[q].y : y1[q].y + y2[q].y;
                        v[q] = qc{from(sr), from(si)};
                    }
                }
                q_dft<R0>(v);
                qc *y = buf + t * LS;
#pragma unroll
                for (int q = 0; q < R0; ++q) y[q_slot(jj * R0 + q)] = v[q];
            }
        }
        __syncthreads();
        q_fft<L, Cfg::RM, TC, NT, LS, R0, false, UL>(buf, tws);
        // the last pass, its outputs times the spectra
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int it = 0; it < IL; ++it) {
            const int ct = column(it), j = freq(it);
            const qc *x = buf + ct * LS + q_slot(j);
            const int4 *tw = tws + (Cfg::TW - (RL - 1) * UL) + j;
            qc v[RL];
#pragma unroll
            for (int q = 0; q < RL; ++q) v[q] = x[UL % 8 == 0 ? q_slot(q * UL) : q_slot(j + q * UL) - q_slot(j)];
            if (j != 0) {   // (see q_pass)
#pragma unroll
                for (int q = 1; q < RL; ++q) v[q] = q_cmul(v[q], tw[(q - 1) * UL]);
            }
            q_dft<RL>(v);
            const int2 *k = ks + ct * KS;
#pragma unroll
            for (int q = 0; q < RL; ++q) {
                const int m = j + q * UL;
                const int2 w = k[m <= Ph ? m : L - m];
                if constexpr (ALT) {
                    acc[it][q].re = q_rmul(v[q].re, w.x, w.y) - acc[it][q].re;
                    acc[it][q].im = q_rmul(v[q].im, w.x, w.y) - acc[it][q].im;
                } else {
                    acc[it][q].re += q_rmul(v[q].re, w.x, w.y);
                    acc[it][q].im += q_rmul(v[q].im, w.x, w.y);
                }
            }
        }
        if constexpr (ALT) {
            from.flip();
            ++turns;
        }
        __syncthreads();   // the buffer is free
    }
#pragma unroll
    for (int it = 0; it < IL; ++it) {
        const int ct = column(it);
        if (ct >= ncl) continue;
        qc *part = a.part + (((int64_t)chunk * 2 + diff) * a.nc + c0 + ct) * L + freq(it);
        const bool back = ((turns ^ (ALT ? 0 : 1)) & 1) != 0;   // the last pair was not turned
#pragma unroll
        for (int q = 0; q < RL; ++q) part[q * UL] = back ? acc[it][q] : qc{-acc[it][q].re, -acc[it][q].im};
    }
}

// spectra of the pair sums and differences as fractions of 2^ek, and ek (see FaceQPass::kq)
__global__ void face_kq_kernel(const double *__restrict__ khat, int np, int64_t per, int2 *__restrict__ kq,
                               int *__restrict__ ek)
{
    const int npair = (np + 1) / 2;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < per; x += (int64_t)gridDim.x * blockDim.x) {
        double sum = 0.0, big = 0.0;
        for (int p = 0; p < np; ++p) {
            sum += fabs(khat[p * per + x]);
            big = fmax(big, fabs(khat[p * per + x]));
        }
        int e = 0;
        if (sum > 0.0) frexp(fmax(0.25 * sum, big) * (1.0 + 1e-9), &e);
        ek[x] = e;
        const double scale = ldexp(0.5, 62 - e);
        for (int p = 0; p < npair; ++p) {
            const double k1 = khat[p * per + x], k2 = khat[(np - 1 - p) * per + x];
            const long long s = __double2ll_rn((k1 + k2) * scale), d = __double2ll_rn((k1 - k2) * scale);
            // low words of either sign: what a product drops is then no bias over the slices
            // (|s| < 2^62 (1 - 1e-9) keeps the high word in range)
            const int sh = (int)((s + (1LL << 30)) >> 31), dh = (int)((d + (1LL << 30)) >> 31);
            kq[p * per + x] = make_int2(sh, (int)(s - ((long long)sh << 31)));
            kq[(npair + p) * per + x] = make_int2(dh, (int)(d - ((long long)dh << 31)));
        }
    }
}

#define IDP_FACE_SWITCH(LEN, ...)              \
    switch (LEN) {                             \
    case 32: { constexpr int L = 32; __VA_ARGS__; }   \
    case 64: { constexpr int L = 64; __VA_ARGS__; }   \
    case 96: { constexpr int L = 96; __VA_ARGS__; }   \
    case 128: { constexpr int L = 128; __VA_ARGS__; } \
    case 192: { constexpr int L = 192; __VA_ARGS__; } \
    case 256: { constexpr int L = 256; __VA_ARGS__; } \
    case 384: { constexpr int L = 384; __VA_ARGS__; } \
    case 512: { constexpr int L = 512; __VA_ARGS__; } \
    case 768: { constexpr int L = 768; __VA_ARGS__; } \
    case 1024: { constexpr int L = 1024; __VA_ARGS__; } \
    default: return cudaErrorInvalidValue;     \
    }

template <int L>
cudaError_t face_attr()
{
    const cudaError_t e = cudaFuncSetAttribute(face_q_kernel<L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)FaceQCfg<L>::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(face_q_kernel<L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)FaceQCfg<L>::SMEM);
}

}  // namespace

cudaError_t face_q_set_attributes()
{
    for (int len : {32, 64, 96, 128, 192, 256, 384, 512, 768, 1024}) {
        const cudaError_t e = [&]() -> cudaError_t { IDP_FACE_SWITCH(len, return face_attr<L>()) }();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_face_q(const FaceQPass &a, cudaStream_t st)
{
    IDP_FACE_SWITCH(2 * a.Pb, {
        using Cfg = FaceQCfg<L>;
        const dim3 grid((a.nc + Cfg::TC - 1) / Cfg::TC, a.nchunk, 2);
        if (a.nchunk & 1) face_q_kernel<L, true><<<grid, Cfg::NT, Cfg::SMEM, st>>>(a);
        else face_q_kernel<L, false><<<grid, Cfg::NT, Cfg::SMEM, st>>>(a);
        return cudaGetLastError();
    })
}

cudaError_t launch_face_kq(const double *khat, int np, int64_t per, int2 *kq, int *ek, cudaStream_t st)
{
    face_kq_kernel<<<1024, 256, 0, st>>>(khat, np, per, kq, ek);
    return cudaGetLastError();
}

int face_q_columns(int L)
{
    IDP_FACE_SWITCH(L, return FaceQCfg<L>::TC;)
}

int face_q_blocks_per_sm(int L)
{
    IDP_FACE_SWITCH(L, return FaceQCfg<L>::BPS;)
}

}  // namespace idp
