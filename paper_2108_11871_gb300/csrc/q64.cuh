// Block fixed-point ("q64") arithmetic for the FP64-class transforms, and the
// block-cooperative complex FFT built on it.
//
// GB300 issues FP64 at 2 lanes per clock and SM (measured: 64 cycles per warp
// instruction and scheduler), but a 32 x 32 -> 64-bit integer multiply-add at 60 lanes
// (2.1 cycles).  A radix-4 unit with its three twiddle products takes about 200
// cycles in 64-bit integers against 1540 in FP64, so the transforms run in
// integers: the values of one line share a power-of-two scale, chosen from a bound on
// the line's absolute sum so that no intermediate can overflow, and every value is
// a signed 64-bit integer in units of that scale.  Additions are exact; a
// product with a twiddle (62 fractional bits) is off by about one unit at most.  A unit
// is 2^-58 to 2^-59 of the line's absolute sum, and every output is bounded by that sum.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "idp_internal.cuh"

namespace idp {

struct __align__(16) qc {
    long long re, im;
};

__device__ __forceinline__ long long q_mulw(int a, int b)
{
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ long long q_madw(int a, int b, long long c)
{
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

__device__ __forceinline__ qc q_add(qc a, qc b) { return qc{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ qc q_sub(qc a, qc b) { return qc{a.re - b.re, a.im - b.im}; }

// A factor c in [-1, 1] is ch 2^-31 + cl 2^-62 (|cl| <= 2^30, except c = 1: ch = cl =
// 2^31 - 1, 2^-62 below 1); a value x is xh 2^31 + xl with 0 <= xl < 2^31:
//   x c = xh ch + (xh cl + xl ch) 2^-31 + xl cl 2^-62,
// the last term (below one unit) dropped and the bracket rounded to nearest (a rounding
// down is a bias, which the lowest modes add up over the line: measured ten times the
// error of FP64 on noise at M = 512, against the same).  |x| <= 2^61 keeps the bracket
// (for a complex product, the sum of two of them with c^2 + s^2 = 1) within 63 bits.
constexpr long long Q_HALF = 1LL << 30;
__device__ __forceinline__ long long q_rmul(long long x, int ch, int cl)
{
    const int xh = (int)(x >> 31), xl = (int)((unsigned)x & 0x7fffffffu);
    const long long m = q_madw(xl, ch, q_madw(xh, cl, Q_HALF));
    return q_madw(xh, ch, m >> 31);
}

__device__ __forceinline__ qc q_cmul(qc a, int4 w)   // w = (ch, cl, sh, sl): a (c + i s)
{
    const int xh = (int)(a.re >> 31), xl = (int)((unsigned)a.re & 0x7fffffffu);
    const int yh = (int)(a.im >> 31), yl = (int)((unsigned)a.im & 0x7fffffffu);
    // the two halves of the real part are formed apart and subtracted (measured 6 %
    // faster than negating the factor words)
    const long long m = q_madw(xl, w.x, q_madw(xh, w.y, Q_HALF)) - q_madw(yl, w.z, q_mulw(yh, w.w));
    const long long n = q_madw(yl, w.x, q_madw(yh, w.y, q_madw(xl, w.z, q_madw(xh, w.w, Q_HALF))));
    qc r;
    r.re = q_madw(xh, w.x, m >> 31) - q_mulw(yh, w.z);
    r.im = q_madw(yh, w.x, q_madw(xh, w.z, n >> 31));
    return r;
}

constexpr int Q_R2H = 1518500250, Q_R2L = -25716447;    // sqrt(1/2)
constexpr int Q_S3H = 1859775393, Q_S3L = 815355111;    // sqrt(3)/2

// forward DFTs (e^{-2 pi i/R}) in registers, natural order in and out
__device__ __forceinline__ void q_dft2(qc *v)
{
    const qc a = v[0];
    v[0] = q_add(a, v[1]);
    v[1] = q_sub(a, v[1]);
}
__device__ __forceinline__ void q_dft3(qc &a0, qc &a1, qc &a2)
{
    const qc t = q_add(a1, a2), d = q_sub(a1, a2);
    // t / 2, an odd t rounded up or down by the last bit of another value (no bias)
    const qc m = qc{a0.re - ((t.re + (a0.re & 1)) >> 1), a0.im - ((t.im + (a0.im & 1)) >> 1)};
    const long long pr = q_rmul(d.im, Q_S3H, Q_S3L), pi = q_rmul(d.re, Q_S3H, Q_S3L);
    a0 = q_add(a0, t);
    a1 = qc{m.re + pr, m.im - pi};
    a2 = qc{m.re - pr, m.im + pi};
}
// 6 = 2 * 3 by the residues (x_{3a+2b} -> X_{3c+4d}): two 3-point transforms, no factors
__device__ __forceinline__ void q_dft6(qc *v)
{
    qc s0 = q_add(v[0], v[3]), s1 = q_add(v[2], v[5]), s2 = q_add(v[4], v[1]);
    qc d0 = q_sub(v[0], v[3]), d1 = q_sub(v[2], v[5]), d2 = q_sub(v[4], v[1]);
    q_dft3(s0, s1, s2);
    q_dft3(d0, d1, d2);
    v[0] = s0; v[4] = s1; v[2] = s2;
    v[3] = d0; v[1] = d1; v[5] = d2;
}
__device__ __forceinline__ void q_dft4(qc &a0, qc &a1, qc &a2, qc &a3)
{
    const qc c0 = q_add(a0, a2), c1 = q_sub(a0, a2), e0 = q_add(a1, a3), e1 = q_sub(a1, a3);
    a0 = q_add(c0, e0);
    a2 = q_sub(c0, e0);
    a1 = qc{c1.re + e1.im, c1.im - e1.re};
    a3 = qc{c1.re - e1.im, c1.im + e1.re};
}
__device__ __forceinline__ void q_dft8(qc *v)
{
    q_dft4(v[0], v[2], v[4], v[6]);   // E_0..3
    q_dft4(v[1], v[3], v[5], v[7]);   // O_0..3
    const qc t0 = v[1];
    const qc t1 = qc{q_rmul(v[3].re + v[3].im, Q_R2H, Q_R2L), q_rmul(v[3].im - v[3].re, Q_R2H, Q_R2L)};
    const qc t2 = qc{v[5].im, -v[5].re};
    const qc t3 = qc{q_rmul(v[7].im - v[7].re, Q_R2H, Q_R2L), -q_rmul(v[7].re + v[7].im, Q_R2H, Q_R2L)};
    const qc e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    v[0] = q_add(e0, t0);
    v[4] = q_sub(e0, t0);
    v[1] = q_add(e1, t1);
    v[5] = q_sub(e1, t1);
    v[2] = q_add(e2, t2);
    v[6] = q_sub(e2, t2);
    v[3] = q_add(e3, t3);
    v[7] = q_sub(e3, t3);
}
template <int R>
__device__ __forceinline__ void q_dft(qc *v)
{
    if constexpr (R == 2) q_dft2(v);
    else if constexpr (R == 3) q_dft3(v[0], v[1], v[2]);
    else if constexpr (R == 6) q_dft6(v);
    else if constexpr (R == 4) q_dft4(v[0], v[1], v[2], v[3]);
    else q_dft8(v);
}

// Shared-memory place of element e of a line (16-byte elements): one element of padding
// after every eight, so that the eight lanes of a quarter-warp hit eight bank groups in a
// pass's reads (consecutive e) and in its writes (stride R), at offsets that are constants
// of the pass (an XOR of the low bits does the same, but costs integer instructions on
// every access).  q_line: padded length of a line, odd.
__host__ __device__ constexpr int q_slot(int e) { return e + (e >> 3); }
__host__ __device__ constexpr int q_line(int L) { return q_slot(L) | 1; }

// The radix of the pass of length L after a span of Ns, RM = 4 or 8.
//   2^m:     a radix-4 pass (RM = 4: radix-2) first where 2^m is no power of RM, then radix
//            RM, and for 2^m = 2 * 8^i a last radix-4 pass (two radix-4 passes in a row
//            would write two elements to one bank group)
//   3 * 2^m: the same with a last pass of radix 3, or 6 for 2^m = 2 * RM^i (radix 3 first
//            has no factors, but costs a radix-8 pass that has none and leaves spans that are
//            no powers of two: 193^3 with radix 3 first, face passes 640 us per solve, sine passes 442;
//            with it last 503 and 354)
__host__ __device__ constexpr int q_radix(int L, int Ns, int RM)
{
    const int rest = L / Ns, three = L % 3 == 0 ? 3 : 1, two = rest / three;   // 2^m left
    int p = 1;
    while (p * RM <= two) p *= RM;
    const int head = two / p;   // 1, 2 or 4
    if (three == 3) {
        if (two <= 2) return three * two;
        return head == 4 && Ns == 1 ? 4 : RM;
    }
    if (rest <= RM) return rest;
    if (Ns > 1 && RM == 8) return 8;
    if (head == 1) return RM;
    return RM == 8 ? 4 : 2;
}
// entries of the factor table of length L, from span Ns on
__host__ __device__ constexpr int q_tw_count(int L, int RM, int Ns = 1)
{
    return Ns == L ? 0 : (Ns > 1 ? (q_radix(L, Ns, RM) - 1) * Ns : 0) + q_tw_count(L, RM, Ns * q_radix(L, Ns, RM));
}

// One Stockham pass of radix R at span Ns over LB lines (line stride LS elements) by
// NT threads, in place: every thread takes its units into registers, and after a block
// barrier writes their results.  tw: the pass's factors w_{R Ns}^{k q}, [q - 1][k].  HZ: the
// elements from L / 2 on are zero and not read.  Ends with a block barrier.
// (One buffer and a second barrier per pass against two buffers: at M = 256 the sine
// pass then keeps four blocks per SM where two buffers with their padding allowed two.)
template <int L, int Ns, int RM, int LB, int NT, int LS, bool HZ = false>
__device__ __forceinline__ void q_pass(qc *X, const int4 *__restrict__ tw)
{
    constexpr int R = q_radix(L, Ns, RM), U = L / R, UNITS = LB * U, IT = (UNITS + NT - 1) / NT;
    // j + q U and (j - k) R + k + q Ns: place of the first plus a constant where nothing
    // carries into the padding count
    constexpr bool RLIN = U % 8 == 0, WLIN = Ns % 8 == 0 || (R != 3 && (Ns & (Ns - 1)) == 0);
    qc v[IT][R];
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int b = threadIdx.x + it * NT, line = b / U, j = b - line * U;
        if (UNITS % NT != 0 && b >= UNITS) break;
        const qc *x = X + line * LS + (RLIN ? q_slot(j) : 0);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int at = RLIN ? q_slot(q * U) : q_slot(j + q * U);
            if (HZ && q * U >= L / 2) v[it][q] = qc{0, 0};
            else if (HZ && (q + 1) * U > L / 2) v[it][q] = j + q * U < L / 2 ? x[at] : qc{0, 0};
            else v[it][q] = x[at];
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int b = threadIdx.x + it * NT, line = b / U, j = b - line * U, k = j % Ns;
        if (UNITS % NT != 0 && b >= UNITS) break;
        // no factors at k = 0: the word pairs end 2^-62 below 1, and with it half of such
        // products would come out one unit low, a bias that DC adds up over the line (noise at
        // 257^3: boundary values off by 2.6e-13 with these products, 2.1e-14 without, before the
        // signs in turn and the slice sums of face.cu)
        if (Ns > 1 && k != 0) {
            const int4 *w = tw + k;
#pragma unroll
            for (int q = 1; q < R; ++q) v[it][q] = q_cmul(v[it][q], w[(q - 1) * Ns]);
        }
        q_dft<R>(v[it]);
        const int base = (j - k) * R + k;
        qc *y = X + line * LS + (WLIN ? q_slot(base) : 0);
#pragma unroll
        for (int q = 0; q < R; ++q) y[WLIN ? q_slot(q * Ns) : q_slot(base + q * Ns)] = v[it][q];
    }
    __syncthreads();
}

// Forward FFT of LB lines of length L (a multiple of 8) in place, from span Ns on up to
// span NE.  tw: the factors of the passes after span Ns, one after the other (none for
// the first pass at Ns = 1).  HZ (first pass): see q_pass.
template <int L, int RM, int LB, int NT, int LS, int Ns = 1, bool HZ = false, int NE = L>
__device__ __forceinline__ void q_fft(qc *X, const int4 *__restrict__ tw)
{
    if constexpr (Ns < NE) {
        constexpr int R = q_radix(L, Ns, RM);
        q_pass<L, Ns, RM, LB, NT, LS, HZ>(X, tw);
        q_fft<L, RM, LB, NT, LS, Ns * R, false, NE>(X, tw + (Ns > 1 ? (R - 1) * Ns : 0));
    }
}

// ---- scales --------------------------------------------------------------------
// A line's scale from two reductions over its FP64 values: the largest high word (sign off),
// whose exponent field is emax, and the sum S of the magnitudes in units of
// 2^(emax - 1043), each rounded up.  With bits = bit length of S, the absolute sum is below
// 2^(emax - 1043 + bits).  (A subnormal value counts as the smallest normal one here.)
__device__ __forceinline__ int q_high(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int q_emax(int high) { return max(high >> 20, 1); }
__device__ __forceinline__ unsigned q_shr(unsigned x, int n)   // 0 for n >= 32
{
    unsigned r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
// one unit less than the value's part of S
__device__ __forceinline__ unsigned q_weight(double x, int emax)
{
    const int h = q_high(x);
    return q_shr(((unsigned)h & 0xfffffu) | 0x100000u, max(emax - (h >> 20), 0));
}
__device__ __forceinline__ int q_bits(unsigned S) { return max(32 - __clz((int)S), 21); }

// Signs in turn.  The parts of a product that are dropped or rounded have a mean that
// depends on the factor, so that an output of an FFT is off by a few units on average (5 at
// frequency 1 of length 512), the same ones in every line on the same scale: sums over lines and
// slices add them up (noise, boundary values: 513^2 off by 4.1e-15, 513 x 33^2 by 3.5e-15, in turns 1.8e-15
// and 1.5e-15, FP64 1.8e-15 and 1.0e-15).  So every second block of lines goes through its
// transform with its sign turned, in the exponent word that the conversions change anyway, and its mean
// errors come out turned as well.  (Not in the sine passes, whose errors are below FP64's without.)
constexpr unsigned Q_TURN = 0x80000000u;
__device__ __forceinline__ unsigned q_turn(int k) { return (unsigned)k << 31; }   // odd k

// x 2^s (turn: -x 2^s) rounded to nearest, |x| 2^s < 2^60
struct QFrom {
    int add, low, s;
    unsigned turn;
    __device__ __forceinline__ QFrom(int s_, int emax, unsigned turn_ = 0)
        : add((int)(((unsigned)s_ << 20) ^ turn_)), s(s_), turn(turn_)
    {
        // values whose exponent field plus s is below 1 give 0 (their half unit is far
        // above them); next to the smallest numbers the general form below runs instead
        low = emax < 128 ? -1 : max(1 - s_, 1) << 20;
    }
    __device__ __forceinline__ long long operator()(double x) const
    {
        const int h = __double2hiint(x);
        if (low >= 0) {
            // the power of two goes into the exponent field, the conversion runs on the
            // otherwise idle FP64 pipe (18 integer instructions if done by shifts)
            const int g = (h & 0x7fffffff) < low ? 0 : h + add;
            return __double2ll_rn(__hiloint2double(g, __double2loint(x)));
        }
        return shifted(x, (h & 0x7ff00000) ? 0x100000u : 0u);
    }
    // the same by integer shifts, for a kernel whose outputs keep the FP64 pipe busy (the real
    // FFTs, two outputs to an input: 257^3 325 -> 303 us per solve; no gain in the sine pass)
    __device__ __forceinline__ long long by_int(double x) const
    {
        return shifted(x, low >= 0 || (__double2hiint(x) & 0x7ff00000) ? 0x100000u : 0u);
    }
    __device__ __forceinline__ void flip()
    {
        add ^= Q_TURN;
        turn ^= Q_TURN;
    }

private:
    __device__ __forceinline__ long long shifted(double x, unsigned lead) const
    {
        const int h = __double2hiint(x);
        const unsigned long long f =
            (((unsigned long long)(((unsigned)h & 0xfffffu) | lead) << 32) | (unsigned)__double2loint(x)) << 10;
        const int r = max(min(1085 - s - q_emax(h & 0x7fffffff), 64), 1);
        const long long v = (long long)(((f >> (r - 1)) + 1) >> 1), t = (int)(h ^ turn) >> 31;
        return (v ^ t) - t;
    }
};
constexpr int Q_NAN = 1 << 30;   // scale of a line with a NaN or an infinity
constexpr int Q_GNAN = 1 << 20;  // emax + bits of such a line in a maximum over lines
// v 2^-s (turn: -v 2^-s) as FP64
struct QTo {
    int sub, s;
    bool fast;   // 2^-s and every |v| keep the result normal
    __device__ __forceinline__ explicit QTo(int s_, unsigned turn = 0)
        : sub((int)(((unsigned)s_ << 20) ^ turn)), s(s_), fast(s_ <= 1022 && s_ >= -960)
    {
    }
    __device__ __forceinline__ double operator()(long long v) const
    {
        const double d = __ll2double_rn(v);
        const int h = __double2hiint(d);
        if (fast) return __hiloint2double(h ? h - sub : 0, __double2loint(d));
        if (s == Q_NAN) return __longlong_as_double(0x7ff8000000000000LL);
        return scalbn(sub != s << 20 ? -d : d, -s);
    }
};

}  // namespace idp
