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
// Arithmetic (q64.cuh): one scale for all columns and slices of a pass, from a bound on
// the absolute sum of every line of stage 1; the spectra of each frequency pair (b, c)
// are fractions of a power of two that bounds their sum over the slices, so that
// neither a transform nor a sum can overflow.  (One power for all frequencies leaves the
// products' rounding as white noise over them: measured 1e-12 of g on mixed-sign
// densities, against 1e-15 with the spectra's decay in the scale.)
#include "fft.cuh"
#include "q64.cuh"

namespace idp {

namespace {

// TC columns (consecutive frequencies c) per block, a thread for each radix-8 unit of the
// last pass, which keeps the unit's 8 sums in registers
template <int L_>
struct FaceQCfg {
    static constexpr int L = L_, RM = 8, U = L / 8;
    static constexpr int TC = (L % 3 == 0 ? 1536 : 2048) / L < 32 ? (L % 3 == 0 ? 1536 : 2048) / L : 32;
    static constexpr int NT = TC * U, LS = q_line(L), Ph = L / 2, KS = Ph + 1;
    static constexpr int R0 = q_radix(L, 1, RM), TW = q_tw_count(L, RM);
    static constexpr size_t SMEM = sizeof(qc) * (TC * LS + TW) + sizeof(int2) * TC * KS;
};

__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int L>
__global__ void __launch_bounds__(FaceQCfg<L>::NT, 2) face_q_kernel(const FaceQPass a)
{
    using Cfg = FaceQCfg<L>;
    constexpr int TC = Cfg::TC, NT = Cfg::NT, LS = Cfg::LS, KS = Cfg::KS, U = Cfg::U, Ph = Cfg::Ph, R0 = Cfg::R0;
    extern __shared__ qc smem_q[];
    qc *buf = smem_q;
    int4 *tws = reinterpret_cast<int4 *>(buf + TC * LS);
    int2 *ks = reinterpret_cast<int2 *>(tws + Cfg::TW);
    const int c0 = blockIdx.x * TC, ncl = min(TC, a.nc - c0);
    const int chunk = blockIdx.y, diff = blockIdx.z;
    const int npair = (a.np + 1) / 2;
    const int g = *a.gmax;
    const QFrom from(1102 - min(g, 2100) - a.lgn, g - 31);   // every column's absolute sum below 2^61 units
    for (int f = threadIdx.x; f < Cfg::TW; f += NT) tws[f] = __ldg(a.q + f);
    const int2 *kq = a.kq + ((int64_t)diff * npair * a.nc + c0) * KS;

    // the unit of the last pass: column ct, frequencies j + q U
    const int ct = threadIdx.x / U, j = threadIdx.x - ct * U;
    qc acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = qc{0, 0};

    for (int pr = chunk; pr < npair; pr += a.nchunk) {
        const int p2 = a.np - 1 - pr;
        const bool two = pr != p2;
        // slices of zeros contribute nothing; the middle slice has no difference
        if (!(a.sliceflag[pr] | a.sliceflag[p2]) || (!two && diff)) continue;
        {
            const int2 *src = kq + (int64_t)pr * a.nc * KS;
            for (int f = threadIdx.x; f < ncl * KS; f += NT) cp_async8(ks + f, src + f);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        }
        // the first pass (radix R0, no factors) on the load: data at positions 1..Mb-1 of
        // a column, zeros elsewhere, in particular from L / 2 on
        {
            constexpr int U0 = L / R0, NZ = R0 == 3 ? 2 : R0 / 2;   // units, inputs that can be non-zero
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
        q_fft<L, Cfg::RM, TC, NT, LS, R0, false, U>(buf, tws);
        // the last pass, its outputs times the spectra
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
        {
            const qc *x = buf + ct * LS;
            const int4 *tw = tws + (Cfg::TW - 7 * U);
            qc v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = x[q_slot(j + q * U)];
#pragma unroll
            for (int q = 1; q < 8; ++q) v[q] = q_cmul(v[q], tw[(q - 1) * U + j]);
            q_dft8(v);
            const int2 *k = ks + ct * KS;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int m = j + q * U;
                const int2 w = k[m <= Ph ? m : L - m];
                acc[q].re += q_rmul(v[q].re, w.x, w.y);
                acc[q].im += q_rmul(v[q].im, w.x, w.y);
            }
        }
        __syncthreads();   // the buffer is free
    }
    if (ct < ncl) {
        qc *part = a.part + (((int64_t)chunk * 2 + diff) * a.nc + c0 + ct) * L;
#pragma unroll
        for (int q = 0; q < 8; ++q) part[j + q * U] = acc[q];
    }
}

// spectra of the pair sums and differences as fractions of 2^ek, and ek (see FaceQPass::kq)
__global__ void face_kq_kernel(const double *__restrict__ khat, int np, int64_t per, int2 *__restrict__ kq,
                               int *__restrict__ ek)
{
    const int npair = (np + 1) / 2;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < per; x += (int64_t)gridDim.x * blockDim.x) {
        double sum = 0.0;
        for (int p = 0; p < np; ++p) sum += fabs(khat[p * per + x]);
        int e = 0;
        if (sum > 0.0) frexp(0.5 * sum * (1.0 + 1e-9), &e);
        ek[x] = e;
        const double scale = ldexp(0.5, 62 - e);
        for (int p = 0; p < npair; ++p) {
            const double k1 = khat[p * per + x], k2 = khat[(np - 1 - p) * per + x];
            const long long s = __double2ll_rn((k1 + k2) * scale), d = __double2ll_rn((k1 - k2) * scale);
            kq[p * per + x] = make_int2((int)(s >> 31), (int)(s & 0x7fffffff));
            kq[(npair + p) * per + x] = make_int2((int)(d >> 31), (int)(d & 0x7fffffff));
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
    return cudaFuncSetAttribute(face_q_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FaceQCfg<L>::SMEM);
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
        face_q_kernel<L><<<dim3((a.nc + Cfg::TC - 1) / Cfg::TC, a.nchunk, 2), Cfg::NT, Cfg::SMEM, st>>>(a);
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

}  // namespace idp
