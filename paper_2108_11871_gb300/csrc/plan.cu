// C ABI of the infinite-domain Poisson solver: plans, workspace, tables and
// the order of the stages of one solve (section 2: phi = phi* + phi_H).
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <atomic>
#include <mutex>
#include <new>
#include <tuple>
#include <algorithm>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "dd.cuh"
#include "idp_internal.cuh"
#include "../../include/idp.h"

using namespace idp;

namespace {

thread_local char g_cuda_err[256] = "";

int cuda_fail(cudaError_t e, const char *what)
{
    snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s", what, cudaGetErrorString(e));
    return IDP_ECUDA;
}

#define IDP_CK(call)                                       \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

bool is_pow2(int64_t x) { return x > 0 && (x & (x - 1)) == 0; }
// panel counts with a transform kernel: 2^a in [16, 512] or 3 * 2^a in [48, 384]
bool supported_panels(int64_t M)
{
    return M >= 16 && M <= 512 && (is_pow2(M) || (M >= 48 && M % 3 == 0 && is_pow2(M / 3)));
}

// panel counts whose sine transform runs as an FFT here
bool has_fft_dst(int64_t M) { return supported_panels(M); }

// half the length of the zero-padded boundary convolutions for M panels: the
// smallest complex FFT length here that is >= M (M itself where it has one)
int conv_half(int64_t M)
{
    const int lens[12] = {16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024};
    for (int L : lens)
        if (L >= M) return L;
    return 0;
}

// the smallest supported panel count >= M (0 if there is none)
int64_t padded_panels(int64_t M)
{
    for (int64_t m = M < 16 ? 16 : M; m <= 512; ++m)
        if (supported_panels(m)) return m;
    return 0;
}

// host tables ----------------------------------------------------------------
// sin(pi m / L) and cos(pi m / L) with the integer argument reduced to [0, 2L).
double sinpi_frac(int64_t m, int64_t L)
{
    m %= 2 * L;
    if (m < 0) m += 2 * L;
    return std::sin(M_PI * (double)m / (double)L);
}
double cospi_frac(int64_t m, int64_t L)
{
    m %= 2 * L;
    if (m < 0) m += 2 * L;
    return std::cos(M_PI * (double)m / (double)L);
}

Tw make_tw(double c, double s)
{
    Tw t;
    if (std::fabs(c) >= std::fabs(s)) {
        t.r = s / c; t.mre = c; t.mim = c; t.swap = 0;
    } else {
        t.r = c / s; t.mre = -s; t.mim = s; t.swap = 1;
    }
    t.pad = 0;
    return t;
}

struct DevFft {
    Tw *fwd = nullptr, *inv = nullptr;
    double2 *half = nullptr;
    Tw *halfr = nullptr;
    TwD *fwdd = nullptr, *invd = nullptr;   // double-float forms
    ddc *halfd = nullptr;
    FftTables view(int L) const { return FftTables{L, fwd, inv, half, halfr, fwdd, invd, halfd}; }
};

// double-float pair of a double (host): hi = nearest float, lo = nearest float of the rest
ddr host_dd(double x)
{
    ddr r;
    r.hi = (float)x;
    r.lo = (float)(x - (double)r.hi);
    return r;
}
TwD make_twd(const Tw &t)
{
    TwD d;
    d.r = host_dd(t.r);
    d.mre = host_dd(t.mre);
    d.mim = host_dd(t.mim);
    d.swap = t.swap;
    d.pad = 0;
    return d;
}

// a factor in [-1, 1] in the two-word fixed-point form of q64.cuh: ch 2^-31 + cl 2^-62
int2 fixed_factor(long double c)
{
    const long double top = 2147483647.0L, a = c * 2147483648.0L;
    const long double h = std::min(top, std::nearbyint(a));
    return make_int2((int)h, (int)std::min(top, std::nearbyint((a - h) * 2147483648.0L)));
}
// cos and sin of pi m / L to the precision of that form (argument reduced to the first octant)
void cossinpi(int64_t m, int64_t L, long double &c, long double &s)
{
    const long double pi = 3.14159265358979323846264338327950288L;
    m %= 2 * L;
    if (m < 0) m += 2 * L;
    int64_t r = m % L;                     // angle pi r / L in [0, pi)
    const bool neg = m >= L, obtuse = 2 * r > L;
    if (obtuse) r = L - r;
    const bool swap = 4 * r > L;
    const long double t = swap ? pi * (long double)(L - 2 * r) / (long double)(2 * L) : pi * (long double)r / (long double)L;
    c = swap ? std::sin(t) : std::cos(t);
    s = swap ? std::cos(t) : std::sin(t);
    if (obtuse) c = -c;
    if (neg) { c = -c; s = -s; }
}
int4 fixed_unit(int64_t m, int64_t L)      // e^{-i pi m / L}
{
    long double c, s;
    cossinpi(m, L, c, s);
    const int2 x = fixed_factor(c), y = fixed_factor(-s);
    return make_int4(x.x, x.y, y.x, y.y);
}

// Host copies of the tables, which depend on the kind and the length alone: made once per
// process (the long-double sines cost milliseconds on Arm), at most one per supported length
std::mutex g_table_mu;
std::map<std::pair<int, int>, std::vector<char>> g_tables;
template <class Fill>
const std::vector<char> &host_table(int kind, int key, Fill fill)
{
    std::lock_guard<std::mutex> lk(g_table_mu);
    auto it = g_tables.find({kind, key});
    if (it == g_tables.end()) {
        std::vector<char> v;
        fill(v);
        it = g_tables.emplace(std::make_pair(kind, key), std::move(v)).first;
    }
    return it->second;   // entries are never changed or removed
}

std::mutex g_attr_mu;
std::atomic<uint64_t> g_serial{1};
std::vector<int> g_attr_done;

int ensure_attributes(int dev)
{
    std::lock_guard<std::mutex> lk(g_attr_mu);
    for (int d : g_attr_done)
        if (d == dev) return IDP_OK;
    IDP_CK(dst_set_attributes());
    IDP_CK(boundary_set_attributes());
    IDP_CK(mp_set_attributes());
    g_attr_done.push_back(dev);
    return IDP_OK;
}

}  // namespace

struct BatchCache {
    std::vector<uint64_t> serials;
    std::vector<const double *> rho;
    std::vector<double *> phi;
    cudaGraphExec_t exec = nullptr;
    std::vector<cudaEvent_t> joins;
    cudaEvent_t fork = nullptr;
};

struct idp_plan_s {
    int d = 0, order = 0, dev = 0;
    uint64_t serial = 0;                 // unique per plan (keys the batch graph cache)
    uint64_t version = 0;                // bumped when an option changes the queued work
    cudaStream_t bst = nullptr;          // this plan's branch stream in a batched graph
    BatchCache *batch = nullptr;         // batched graph owned by this plan (first of its batch)
    int n[3] = {1, 1, 1};      // internal node counts (2-D: n[0] = 1)
    int M[3] = {0, 0, 0};
    int P[3] = {0, 0, 0};      // half the length of the boundary convolutions along each axis (P >= M)
    int ni[3] = {1, 1, 1};     // interior extents
    int act[3] = {0, 0, 0};
    double h[3] = {1, 1, 1};
    int64_t nodes = 0, nint = 0;
    // automatic padding (section 2: the domain is extended by a few panels so that
    // every panel count suits the transforms): the caller's node counts, the offset
    // of the caller's node 0 in the grid solved on, the caller's node count, and
    // the padded copies of rho and phi
    int padded = 0;
    int un[3] = {1, 1, 1}, uoff[3] = {0, 0, 0};
    int64_t unodes = 0;
    double *rho_pad = nullptr, *phi_pad = nullptr;
    int64_t ns[3] = {0, 0, 0};  // node strides
    int64_t is[3] = {0, 0, 0};  // interior strides
    Grid3 grid{};
    StencilCoef coef{};

    std::map<int, DevFft> fft;        // by complex length
    std::map<int, ddr *> sin2d;       // by M: 2 sin(pi j / M), j = 0..M/2, double-float pairs
    std::map<std::pair<int, int>, int4 *> qtab;   // fixed-point tables by kind (FFTs, sine passes) and length
    std::map<int, double *> sinm;     // by M (lengths without an FFT): sine matrices for direct sums
    std::map<int, ddr *> sinmd;       // double-float form
    int exact = 0;                    // created by idp_create_plan_exact
    std::vector<void *> allocs;
    static constexpr size_t GUARD = 256;              // keeps the buffers 256-byte aligned
    static constexpr unsigned char GUARD_BYTE = 0xA5;
    std::vector<std::pair<char *, size_t>> guarded;   // allocation base, payload bytes
    int64_t bytes = 0;
    bool released_dirty = false;                      // a guard of a released buffer was overwritten

    double *A = nullptr, *B = nullptr, *C = nullptr, *U = nullptr, *W = nullptr;
    double *tabc = nullptr, *tab4 = nullptr;
    double *tabc2 = nullptr;   // -2 * tabc (forward transform of rho continued from T0)
    double *Q0 = nullptr, *Q1 = nullptr, *Q2 = nullptr, *sin4 = nullptr;   // gtilde parts
    double *tabR = nullptr;    // tab4 * Lambda_R / Lambda4 + tab4 (R_spec's smoothing solve plus u1)
    double *E0 = nullptr, *E1 = nullptr, *E2 = nullptr, *sin4b = nullptr;   // layers of E = R - R_spec
    double *ld = nullptr;      // per-axis eigenvalues of D2_s (axis s at ldoff[s])
    int64_t ldoff[3] = {0, 0, 0};
    // zeroed at the start of every solve, one allocation: the slice sums of the face passes
    // (FaceQPass::sums, slices of axes 0, 1, 2), then the flags
    unsigned long long *sums = nullptr;
    int nsum = 0;
    int *flags = nullptr;        // support flags of rho: rows along axes 2 and 1, slices of axes 0, 1, 2
    int64_t nflags = 0;
    int *row2 = nullptr, *row1 = nullptr, *sl[3] = {nullptr, nullptr, nullptr};
    double2 *T0 = nullptr, *T1 = nullptr, *part = nullptr, *F = nullptr;
    double *khat[3] = {nullptr, nullptr, nullptr};
    ddr *khatd[3] = {nullptr, nullptr, nullptr};   // double-float copies (IDP_KEY_MIXED_BOUNDARY_DF32)
    int64_t khat_n[3] = {0, 0, 0};
    int2 *kq[3] = {nullptr, nullptr, nullptr};   // fixed-point spectra (FaceQPass) and their exponents
    int *kq_ek[3] = {nullptr, nullptr, nullptr};
    int qchunk[3] = {1, 1, 1};        // chunks of pairs of slices of the fixed-point face passes
    int *gmax[4] = {};                // bounds of the lines along axes 2 and 1 (FaceQPass::gmax), of the layers
                                      // of gtilde and of E; zeroed with the flags
    int *unit[3] = {};                // units of the parts of the face passes (FaceQPass::unit)
    int2 *sinq = nullptr, *sinq2 = nullptr;   // fixed-point forms of sin4 / 4 and sin4b / 4
    int nchunk[3] = {1, 1, 1}, pchunk[3] = {1, 1, 1};
    int dst_lines = 0;                // lines per block of the full-volume sine passes (0 = default)

    // mixed precision (IDP_KEY_PRECISION = 1): sine passes on the tensor cores
    int mixed = 0;
    int stall_test = 0;               // IDP_KEY_STALL_TEST: next tensor-core pass waits in vain
    int mixed_path = 0;               // mixed precision: 0 = tensor-core matrix pass, 1 = df32 FFT pass
    int mixed_bdd = 0;                // IDP_KEY_MIXED_BOUNDARY_DF32: tensor-core modes, 3-D boundary in double-float
    int64_t part_cap = 0;             // capacity (complex) of the partial face sums of one axis
    int64_t f_cap = 0;                // capacity (complex) of the face spectra of one axis
    int tuned = 0;
    std::map<int, void *> mp_img;     // by M: BF16 pieces of the sine matrix
    float *t32[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};   // [stream][ping/pong]
    int *d_err = nullptr;
    int validate = 0;                 // IDP_KEY_VALIDATE: margin k (0: off)
    int *d_val = nullptr;             // validation word (bit 1: NaN/inf, bit 2: support too close)

    // per-launch timing (idp_profile_solve)
    int profiling = 0;
    std::vector<cudaEvent_t> ev;
    std::vector<int> ev_kind;
    int ev_used = 0;
    int64_t launches = 0;      // kernel launches queued by the last enqueue

    // staging for idp_solve_host
    double *h_rho = nullptr, *h_phi = nullptr;

    // CUDA graph of one solve for a fixed (rho, phi)
    int use_graph = 1;
    int nvtx = 0;                     // IDP_KEY_NVTX: NVTX ranges around launches and stages
    cudaStream_t cap = nullptr;
    cudaStream_t side = nullptr;          // second stream of a solve (forward transform of rho)
    cudaEvent_t fork = nullptr, join = nullptr;
    // 3-D faces: axes 0 and 1 run on their own streams beside axis 2 (each axis
    // with its own partial sums and face spectra)
    cudaStream_t fst[2] = {nullptr, nullptr};
    cudaEvent_t fev[3] = {nullptr, nullptr, nullptr};   // T0 ready; axis 0 done; axis 1 done
    // host-buffer solves (page-locked buffers, captured into their own graph): the
    // first row transform reads rho from the host buffer (through its device view)
    // and the kernels that write phi write the host buffer directly, so that the
    // upload and the download overlap their work
    const double *hio_rho = nullptr;   // host rho of the solve being queued (null: none)
    const double *hio_view = nullptr;  // its device view
    cudaGraphExec_t hexec = nullptr;
    const double *hg_rho = nullptr;
    double *hg_phi = nullptr;
    uint64_t hg_version = ~0ull;
    cudaGraphExec_t gexec = nullptr;
    const double *g_rho = nullptr;
    double *g_phi = nullptr;
    cudaStream_t last = nullptr;
    int last_valid = 0;

    template <class T>
    int alloc(T **p, int64_t count)
    {
        // every buffer sits between two guard regions of GUARD bytes filled with
        // GUARD_BYTE; idp_plan_check_guards reports one that was overwritten (an
        // out-of-bounds write), in place of a memory checker
        void *q = nullptr;
        const size_t b = (size_t)count * sizeof(T);
        const size_t payload = b > 0 ? b : 16;
        cudaError_t e = cudaMalloc(&q, payload + 2 * GUARD);
        if (e != cudaSuccess) {
            cuda_fail(e, "cudaMalloc");
            return IDP_ENOMEM;
        }
        char *c = static_cast<char *>(q);
        e = cudaMemset(c, GUARD_BYTE, GUARD);
        if (e == cudaSuccess) e = cudaMemset(c + GUARD + payload, GUARD_BYTE, GUARD);
        allocs.push_back(q);
        guarded.emplace_back(c, payload);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemset (guards)");
        bytes += (int64_t)payload;
        *p = (T *)(c + GUARD);
        return IDP_OK;
    }

    // frees a buffer of alloc() (synchronises the device); its guards are looked at first
    int release(void *q)
    {
        char *c = static_cast<char *>(q) - GUARD;
        for (size_t i = 0; i < guarded.size(); ++i)
            if (guarded[i].first == c) {
                int rc = IDP_OK;
                bool intact = true;
                if ((rc = guards_intact(guarded[i], &intact))) return rc;
                released_dirty = released_dirty || !intact;
                bytes -= (int64_t)guarded[i].second;
                guarded.erase(guarded.begin() + i);
                allocs.erase(std::find(allocs.begin(), allocs.end(), (void *)c));
                const cudaError_t e = cudaFree(c);
                return e == cudaSuccess ? IDP_OK : cuda_fail(e, "cudaFree");
            }
        return IDP_EINVAL;
    }

    static int guards_intact(const std::pair<char *, size_t> &g, bool *intact)
    {
        unsigned char h[GUARD];
        for (int side = 0; side < 2; ++side) {
            const cudaError_t e = cudaMemcpy(h, side ? g.first + GUARD + g.second : g.first, GUARD, cudaMemcpyDeviceToHost);
            if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy (guards)");
            for (unsigned char v : h) *intact = *intact && v == GUARD_BYTE;
        }
        return IDP_OK;
    }
};

namespace {

// NVTX range names of the IDP_KERNEL_* families
const char *kernel_range(int kind)
{
    switch (kind) {
    case IDP_KERNEL_DST: return "idp:dst";
    case IDP_KERNEL_RFFT: return "idp:rfft";
    case IDP_KERNEL_FACE: return "idp:face";
    case IDP_KERNEL_FACE_INVB: return "idp:face_invb";
    case IDP_KERNEL_FACE_C2R: return "idp:face_c2r";
    case IDP_KERNEL_GTILDE: return "idp:gtilde";
    case IDP_KERNEL_RHS6_W: return "idp:rhs6_w";
    case IDP_KERNEL_RHS6_CORE: return "idp:rhs6_core";
    case IDP_KERNEL_RHS6_EXTRAP: return "idp:rhs6_extrap";
    case IDP_KERNEL_GTILDE_EXPAND: return "idp:gtilde_expand";
    case IDP_KERNEL_DST_PARTS: return "idp:dst_layers";
    case IDP_KERNEL_MIXED: return "idp:mixed";
    case IDP_KERNEL_RHS6_EXPAND: return "idp:rhs6_expand";
    case IDP_KERNEL_LINE1D: return "idp:line1d";
    case IDP_KERNEL_PAD: return "idp:pad";
    case IDP_KERNEL_VALIDATE: return "idp:validate";
    default: return "idp:kernel";
    }
}

// An NVTX range over a stage of a solve (IDP_KEY_NVTX), closed at the end of scope.
struct Range {
    bool on;
    Range(idp_plan p, const char *name) : on(p->nvtx != 0)
    {
        if (on) nvtxRangePushA(name);
    }
    ~Range()
    {
        if (on) nvtxRangePop();
    }
};

// Marks one kernel launch: counts it, with IDP_KEY_NVTX encloses it in an NVTX
// range named after its family and, while profiling, brackets it with CUDA events
// recorded on the launch stream.
struct Mark {
    idp_plan p;
    cudaStream_t st;
    int idx = -1;
    Range r;
    Mark(idp_plan p_, int kind, cudaStream_t st_) : p(p_), st(st_), r(p_, kernel_range(kind))
    {
        ++p->launches;
        if (p->profiling && p->ev_used + 2 <= (int)p->ev.size()) {
            idx = p->ev_used;
            p->ev_used += 2;
            p->ev_kind.push_back(kind);
            cudaEventRecord(p->ev[idx], st);
        }
    }
    ~Mark()
    {
        if (idx >= 0) cudaEventRecord(p->ev[idx + 1], st);
    }
};

int get_fft(idp_plan p, int L, FftTables *out)
{
    auto it = p->fft.find(L);
    if (it != p->fft.end()) {
        *out = it->second.view(L);
        return IDP_OK;
    }
    // one upload of all tables, made once per process
    const size_t h = L / 2, f = L + 1;
    const size_t size[7] = {h * sizeof(Tw), h * sizeof(Tw), f * sizeof(double2), f * sizeof(Tw),
                            h * sizeof(TwD), h * sizeof(TwD), f * sizeof(ddc)};
    size_t off[8] = {0};
    for (int i = 0; i < 7; ++i) off[i + 1] = (off[i] + size[i] + 31) / 32 * 32;
    const std::vector<char> &blob = host_table(0, L, [&](std::vector<char> &v) {
        v.resize(off[7]);
        Tw *fw = reinterpret_cast<Tw *>(v.data() + off[0]), *iv = reinterpret_cast<Tw *>(v.data() + off[1]);
        double2 *hf = reinterpret_cast<double2 *>(v.data() + off[2]);
        Tw *hr = reinterpret_cast<Tw *>(v.data() + off[3]);
        TwD *fwd2 = reinterpret_cast<TwD *>(v.data() + off[4]), *ivd2 = reinterpret_cast<TwD *>(v.data() + off[5]);
        ddc *hfd = reinterpret_cast<ddc *>(v.data() + off[6]);
        for (int j = 0; j < L / 2; ++j) {
            const double c = cospi_frac(2 * j, L), s = sinpi_frac(2 * j, L);
            fw[j] = make_tw(c, -s);
            iv[j] = make_tw(c, s);
            fwd2[j] = make_twd(fw[j]);
            ivd2[j] = make_twd(iv[j]);
        }
        for (int k = 0; k <= L; ++k) {
            hf[k] = make_double2(cospi_frac(k, L), -sinpi_frac(k, L));
            hr[k] = make_tw(hf[k].x, hf[k].y);
            hfd[k].re = host_dd(hf[k].x);
            hfd[k].im = host_dd(hf[k].y);
        }
    });
    char *d = nullptr;
    int rc;
    if ((rc = p->alloc(&d, (int64_t)blob.size()))) return rc;
    IDP_CK(cudaMemcpy(d, blob.data(), blob.size(), cudaMemcpyHostToDevice));
    DevFft t;
    t.fwd = reinterpret_cast<Tw *>(d + off[0]);
    t.inv = reinterpret_cast<Tw *>(d + off[1]);
    t.half = reinterpret_cast<double2 *>(d + off[2]);
    t.halfr = reinterpret_cast<Tw *>(d + off[3]);
    t.fwdd = reinterpret_cast<TwD *>(d + off[4]);
    t.invd = reinterpret_cast<TwD *>(d + off[5]);
    t.halfd = reinterpret_cast<ddc *>(d + off[6]);
    p->fft[L] = t;
    *out = t.view(L);
    return IDP_OK;
}

// 2 sin(pi j / M), j <= M/2, as double-float pairs
int get_sin2d(idp_plan p, int M, const ddr **out)
{
    auto it = p->sin2d.find(M);
    if (it == p->sin2d.end()) {
        std::vector<ddr> s(M / 2 + 1);
        for (int j = 0; j <= M / 2; ++j) s[j] = host_dd(2.0 * sinpi_frac(j, M));
        ddr *d = nullptr;
        int rc;
        if ((rc = p->alloc(&d, M / 2 + 1))) return rc;
        IDP_CK(cudaMemcpy(d, s.data(), sizeof(ddr) * s.size(), cudaMemcpyHostToDevice));
        it = p->sin2d.emplace(M, d).first;
    }
    *out = it->second;
    return IDP_OK;
}

// factors of the fixed-point FFT of length L, pass by pass (q64.cuh), radices up to RM
std::vector<int4> q_factors(int L, int RM)
{
    std::vector<int4> q;
    for (int Ns = 1; Ns < L;) {
        const int R = q_table_radix(L, Ns, RM);
        if (Ns > 1)
            for (int r = 1; r < R; ++r)
                for (int k = 0; k < Ns; ++k) q.push_back(fixed_unit(2 * (int64_t)r * k, (int64_t)R * Ns));
        Ns *= R;
    }
    return q;
}

// uploads a table once per plan
template <class Fill>
int cached_table(idp_plan p, int kind, int key, Fill fill, const int4 **out)
{
    auto it = p->qtab.find({kind, key});
    if (it == p->qtab.end()) {
        const std::vector<char> &t = host_table(kind, key, [&](std::vector<char> &v) {
            std::vector<int4> q;
            fill(q);
            v.resize(sizeof(int4) * q.size());
            std::memcpy(v.data(), q.data(), v.size());
        });
        char *d = nullptr;
        int rc;
        if ((rc = p->alloc(&d, (int64_t)t.size()))) return rc;
        IDP_CK(cudaMemcpy(d, t.data(), t.size(), cudaMemcpyHostToDevice));
        it = p->qtab.emplace(std::make_pair(kind, key), reinterpret_cast<int4 *>(d)).first;
    }
    *out = it->second;
    return IDP_OK;
}

// fixed-point tables of a complex FFT of length L (radices up to 8) and, for the real
// transforms, e^{-i pi m/L}, m = 0..L/2
int get_fft_tables(idp_plan p, int L, const int4 **q, const int4 **qhalf)
{
    const int rc = cached_table(p, 1, L, [&](std::vector<int4> &v) {
        v = q_factors(L, 8);
        for (int m = 0; m <= L / 2; ++m) v.push_back(fixed_unit(m, L));
    }, q);
    *qhalf = *q + q_table_count(L, 8);
    return rc;
}

// the tables of the sine passes of M panels: see DstPass
int get_dst_tables(idp_plan p, int M, const int4 **out)
{
    return cached_table(p, 2, M, [&](std::vector<int4> &q) {
        const int K = M / 2;
        q = q_factors(K, dst_table_radix(K));
        for (int k = 0; k <= K / 2; ++k) q.push_back(fixed_unit(k, K));
        int2 sn[2];
        for (int j = 0; j < K; ++j) {
            long double c, s;
            cossinpi(j, M, c, s);
            sn[j & 1] = fixed_factor(s);
            if (j & 1) q.push_back(make_int4(sn[0].x, sn[0].y, sn[1].x, sn[1].y));
        }
    }, out);
}

// sine matrix S[i][e] = sin(pi (i+1)(e+1) / M), i, e < M - 1, e fastest, for the
// direct sums of the lengths without an FFT; FP64 and double-float forms
int get_sinm(idp_plan p, int M, const void **out, int dd)
{
    auto it = p->sinm.find(M);
    if (it == p->sinm.end()) {
        const int N = M - 1;
        std::vector<double> s((size_t)N * N);
        std::vector<ddr> sd((size_t)N * N);
        for (int i = 0; i < N; ++i)
            for (int e = 0; e < N; ++e) {
                s[(size_t)i * N + e] = sinpi_frac((int64_t)(i + 1) * (e + 1), M);
                sd[(size_t)i * N + e] = host_dd(s[(size_t)i * N + e]);
            }
        double *d = nullptr;
        ddr *d2 = nullptr;
        int rc;
        if ((rc = p->alloc(&d, (int64_t)N * N)) || (rc = p->alloc(&d2, (int64_t)N * N))) return rc;
        IDP_CK(cudaMemcpy(d, s.data(), sizeof(double) * s.size(), cudaMemcpyHostToDevice));
        IDP_CK(cudaMemcpy(d2, sd.data(), sizeof(ddr) * sd.size(), cudaMemcpyHostToDevice));
        p->sinm[M] = d;
        p->sinmd[M] = d2;
    }
    *out = dd ? (const void *)p->sinmd[M] : (const void *)p->sinm[M];
    return IDP_OK;
}

View3 node_interior(idp_plan p, const double *base)
{
    int64_t off = 0;
    for (int s = 0; s < 3; ++s)
        if (p->act[s]) off += p->ns[s];
    return View3{const_cast<double *>(base) + off, p->ns[0], p->ns[1], p->ns[2]};
}
View3 dense(idp_plan p, const double *base) { return View3{const_cast<double *>(base), p->is[0], p->is[1], p->is[2]}; }

uint16_t bf16_bits(float f)
{
    uint32_t u;
    std::memcpy(&u, &f, 4);
    u += 0x7FFFu + ((u >> 16) & 1u);   // round to nearest even (finite values)
    return (uint16_t)(u >> 16);
}
double bf16_value(uint16_t b)
{
    const uint32_t u = (uint32_t)b << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return (double)f;
}

// FP32 bits rounded to TF32 (11 significant bits, to nearest, ties to even)
uint32_t tf32_bits(float x)
{
    uint32_t u;
    std::memcpy(&u, &x, 4);
    return (u + 0xFFFu + ((u >> 13) & 1u)) & 0xFFFFE000u;
}
double tf32_value(uint32_t u)
{
    float f;
    std::memcpy(&f, &u, 4);
    return (double)f;
}

// TF32 pieces of S (variant 1): [mode tile][k stage][2][W rows m x KB k] FP32
// containers (W = mp_tile_modes(n), KB = mp_stage_k(1)), element (r, c) at byte
// (c/4)*(16 W) + (r/8)*128 + (r%8)*16 + (c%4)*4
int get_mp_image_tf32(idp_plan p, int M, const void **out)
{
    const int KB = mp_stage_k(1);
    const int n = M - 1, W = mp_tile_modes(n), nt = (n + W - 1) / W, nkb = (n + KB - 1) / KB;
    const size_t tile = (size_t)W * KB;
    std::vector<uint32_t> img((size_t)nt * nkb * 2 * tile, 0);
    for (int t = 0; t < nt; ++t)
        for (int kb = 0; kb < nkb; ++kb)
            for (int r = 0; r < W; ++r)
                for (int c = 0; c < KB; ++c) {
                    const int m = t * W + r, k = kb * KB + c;
                    const double s = (m < n && k < n) ? sinpi_frac((int64_t)(m + 1) * (k + 1), M) : 0.0;
                    const uint32_t a = tf32_bits((float)s);
                    const uint32_t b = tf32_bits((float)(s - tf32_value(a)));
                    const size_t off = ((size_t)(c / 4) * (16 * W) + (r / 8) * 128 + (r % 8) * 16 + (c % 4) * 4) / 4;
                    const size_t base = (((size_t)t * nkb + kb) * 2) * tile;
                    img[base + off] = a;
                    img[base + tile + off] = b;
                }
    uint32_t *d;
    int rc = p->alloc(&d, (int64_t)img.size());
    if (rc) return rc;
    IDP_CK(cudaMemcpy(d, img.data(), img.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
    *out = d;
    return IDP_OK;
}

int64_t pad4(int64_t x) { return (x + 3) & ~(int64_t)3; }
// floats of one FP32 intermediate of the tensor-core transforms (the larger of the
// two padded layouts)
int64_t t32_count(idp_plan p)
{
    const int64_t n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
    if (p->d == 3) return std::max(n2 * n0 * pad4(n1), n1 * n2 * pad4(n0));
    return n2 * pad4(n1);
}

// the tensor-core pass variant of the plan's precision (0: BF16X3, 1: TF32X3)
int mp_variant(idp_plan p) { return p->mixed == IDP_PRECISION_MIXED_TF32X3 ? 1 : 0; }
bool tensor_mode(idp_plan p)
{
    return p->mixed == IDP_PRECISION_MIXED_BF16X3 || p->mixed == IDP_PRECISION_MIXED_TF32X3;
}
// the 3-D boundary convolutions (and so T0) in double-float arithmetic: a tensor-core
// mode with IDP_KEY_MIXED_BOUNDARY_DF32
int boundary_dd(idp_plan p)
{
    return p->d == 3 && tensor_mode(p) && p->mixed_bdd ? 1 : 0;
}

// the boundary in fixed point (else FP64 or double-float).  Not in the tensor-core modes: a
// last-bit change of their FP64 intermediates flips FP32 roundings of the tensor-core
// inputs, which moves single values of phi by up to 1e-7, within the modes' error of 1e-5
// but not the same result
int boundary_fx(idp_plan p) { return !tensor_mode(p) && !boundary_dd(p) ? 1 : 0; }

// Pieces of S_{m,k} = sin(pi (m+1)(k+1)/M) for a tensor-core variant, laid out
// as the kernel's shared-memory tiles, one contiguous block per (mode tile,
// K stage).  BF16 (variant 0): [mode tile][k stage][3][W rows m x KB k] with
// W = mp_tile_modes(n), KB = mp_stage_k(0), element (r, c) at byte
// (c/8)*(16 W) + (r/8)*128 + (r%8)*16 + (c%8)*2.  Cached per (M, variant).
int get_mp_image(idp_plan p, int M, int variant, const void **out)
{
    const int key = M + (variant << 24);
    auto it = p->mp_img.find(key);
    if (it != p->mp_img.end()) {
        *out = it->second;
        return IDP_OK;
    }
    if (variant) {
        int rc = get_mp_image_tf32(p, M, out);
        if (!rc) p->mp_img[key] = const_cast<void *>(*out);
        return rc;
    }
    const int KB = mp_stage_k(0);
    const int n = M - 1, W = mp_tile_modes(n), nt = (n + W - 1) / W, nkb = (n + KB - 1) / KB;
    const size_t tile = (size_t)W * KB;
    std::vector<uint16_t> img((size_t)nt * nkb * 3 * tile, 0);
    for (int t = 0; t < nt; ++t)
        for (int kb = 0; kb < nkb; ++kb)
            for (int r = 0; r < W; ++r)
                for (int c = 0; c < KB; ++c) {
                    const int m = t * W + r, k = kb * KB + c;
                    const double s = (m < n && k < n) ? sinpi_frac((int64_t)(m + 1) * (k + 1), M) : 0.0;
                    const uint16_t a = bf16_bits((float)s);
                    const double r1 = s - bf16_value(a);
                    const uint16_t b = bf16_bits((float)r1);
                    const double r2 = r1 - bf16_value(b);
                    const uint16_t cc = bf16_bits((float)r2);
                    const size_t off = ((size_t)(c / 8) * (16 * W) + (r / 8) * 128 + (r % 8) * 16 + (c % 8) * 2) / 2;
                    const size_t base = (((size_t)t * nkb + kb) * 3) * tile;
                    img[base + off] = a;
                    img[base + tile + off] = b;
                    img[base + 2 * tile + off] = cc;
                }
    uint16_t *d;
    int rc = p->alloc(&d, (int64_t)img.size());
    if (rc) return rc;
    IDP_CK(cudaMemcpy(d, img.data(), img.size() * sizeof(uint16_t), cudaMemcpyHostToDevice));
    p->mp_img[key] = d;
    *out = d;
    return IDP_OK;
}

// Sine transform of all active axes with the tensor-core pass (mixed.cu).
// The passes rotate the axes: (a,b,c) -> (c',a,b) -> (b',c',a) -> (a',b',c').
int transform_mixed(idp_plan p, View3 in, View3 out, const double *tab, int sidx, cudaStream_t st)
{
    const int n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
    float *ta = p->t32[sidx][0], *tb = p->t32[sidx][1];
    std::vector<MpPass> ps;
    MpPass a{};
    a.err = p->d_err;
    a.variant = mp_variant(p);
    // the FP32 intermediates keep their contiguous (next pass's k) axis padded to
    // whole 16-byte vectors, so that the next pass loads its lines as vectors
    const int64_t n0p = pad4(n0), n1p = pad4(n1);
    if (p->d == 3) {
        a.in = in.p; a.in_f64 = 1; a.is_p = in.s0; a.is_q = in.s1; a.is_k = in.s2;
        a.out = ta; a.out_f64 = 0; a.os_m = (int64_t)n0 * n1p; a.os_p = n1p; a.os_q = 1;
        a.P = n0; a.Q = n1; a.n = n2;
        ps.push_back(a);
        a.in = ta; a.in_f64 = 0; a.in_vec4 = 1; a.is_p = (int64_t)n0 * n1p; a.is_q = n1p; a.is_k = 1;
        a.out = tb; a.os_m = (int64_t)n2 * n0p; a.os_p = n0p; a.os_q = 1;
        a.P = n2; a.Q = n0; a.n = n1;
        ps.push_back(a);
        a.in = tb; a.is_p = (int64_t)n2 * n0p; a.is_q = n0p; a.is_k = 1;
        a.P = n1; a.Q = n2; a.n = n0;
    } else {
        a.in = in.p; a.in_f64 = 1; a.is_p = 0; a.is_q = in.s1; a.is_k = in.s2;
        a.out = ta; a.out_f64 = 0; a.os_m = n1p; a.os_p = 0; a.os_q = 1;
        a.P = 1; a.Q = n1; a.n = n2;
        ps.push_back(a);
        a.in = ta; a.in_f64 = 0; a.in_vec4 = 1; a.is_p = 0; a.is_q = n1p; a.is_k = 1;
        a.P = 1; a.Q = n2; a.n = n1;
    }
    // last pass: FP64 output in the original layout with the epilogue
    const int s0 = p->d == 3 ? 0 : 1;   // output axis of the modes
    const int64_t os[3] = {out.s0, out.s1, out.s2};
    const int64_t ts[3] = {p->is[0], p->is[1], p->is[2]};
    a.out = out.p; a.out_f64 = 1;
    a.os_m = os[s0]; a.os_p = p->d == 3 ? os[1] : 0; a.os_q = os[2];
    a.tab = tab; a.ts_m = ts[s0]; a.ts_p = p->d == 3 ? ts[1] : 0; a.ts_q = ts[2];
    ps.push_back(a);
    // pass i transforms axis 2, 1, 0 (3-D) / 2, 1 (2-D) of the original array
    const int axes3[3] = {2, 1, 0}, axes2[2] = {2, 1};
    if (p->stall_test) {
        ps[0].stall_test = 1;
        p->stall_test = 0;
    }
    for (size_t i = 0; i < ps.size(); ++i) {
        const int ax = p->d == 3 ? axes3[i] : axes2[i];
        int rc = get_mp_image(p, p->M[ax], ps[i].variant, &ps[i].bimg);
        if (rc) return rc;
        Mark mk(p, IDP_KERNEL_MIXED, st);
        IDP_CK(launch_mp_pass(ps[i], st));
    }
    return IDP_OK;
}

// one full sine transform (all active axes); `first` pass reads `in`, the
// last pass applies the epilogue (tab) and writes `out`; intermediate
// passes run in place on `work`.
// allow_reduced = false: FP64 passes in every precision mode except that
// fp64_only = false lets the tensor-core modes run them as double-float passes
// (the transform producing u1: FP64-class there, never the tensor cores)
int transform(idp_plan p, View3 in, double *work, View3 out, const double *tab, bool forward, cudaStream_t st,
              bool allow_reduced = true, bool skip_axis2 = false, int in_dd0 = 0,
              bool fp64_only = true)
{
    Range rg(p, forward ? "idp:sine transform (forward)" : "idp:sine transform (inverse)");
    if (tensor_mode(p) && allow_reduced && p->mixed_path == 0)
        return transform_mixed(p, in, out, tab, st == p->side ? 1 : 0, st);
    // df32 passes: precision DF32, or precision MIXED when the autotuner found the
    // double-float FFT faster than the matrix pass (it is also more accurate), or the
    // double-float transform of u1 in the tensor-core modes
    const bool dd = ((p->mixed == IDP_PRECISION_DF32 || (tensor_mode(p) && p->mixed_path == 1)) && allow_reduced) ||
                    (tensor_mode(p) && !allow_reduced && !fp64_only);
    int axes[3], na = 0;
    if (forward) {
        for (int s = skip_axis2 ? 1 : 2; s >= 0; --s)
            if (p->act[s]) axes[na++] = s;
    } else {
        for (int s = 0; s < 3; ++s)
            if (p->act[s]) axes[na++] = s;
    }
    for (int q = 0; q < na; ++q) {
        const int s = axes[q];
        DstPass a{};
        a.lines = p->dst_lines;
        a.in = (q == 0) ? in : dense(p, work);
        a.out = (q == na - 1) ? out : dense(p, work);
        a.tab = (q == na - 1) ? tab : nullptr;
        a.n0 = p->ni[0]; a.n1 = p->ni[1]; a.n2 = p->ni[2];
        a.axis = s;
        a.M = p->M[s];
        FftTables t{};
        int rc;
        if (has_fft_dst(p->M[s])) {
            if ((rc = get_fft(p, p->M[s] / 2, &t))) return rc;
            if ((rc = get_dst_tables(p, p->M[s], &a.qtab))) return rc;
        } else if ((rc = get_sinm(p, p->M[s], &a.sinm, dd ? 1 : 0))) {   // direct sums
            return rc;
        }
        // the tensor-core modes keep double-float passes (boundary_fx says why); precision
        // DF32 runs the fixed-point FFT, and double-float only in the direct sums
        a.in_dd = (q == 0) ? in_dd0 : 0;
        if (dd && (tensor_mode(p) || !has_fft_dst(p->M[s]))) {
            a.dd = 1;
            if (tensor_mode(p)) {   // intermediate passes keep double-float pairs
                if (q > 0) a.in_dd = 1;
                a.out_dd = q < na - 1;
            }
            a.twd = t.fwdd;
            a.halfd = t.halfd;
            if (has_fft_dst(p->M[s]) && (rc = get_sin2d(p, p->M[s], &a.sin2d))) return rc;
        }
        Mark mk(p, IDP_KERNEL_DST, st);
        IDP_CK(launch_dst_pass(a, st));
    }
    return IDP_OK;
}

// The transformed layers as fixed-point numbers and their expansions in integers: where every
// sine pass of the layers is a fixed-point one (its bound sets the scale)
bool layers_fx(idp_plan p)
{
    bool fx = !tensor_mode(p);
    for (int s = 0; s < 3; ++s) fx = fx && (!p->act[s] || has_fft_dst(p->M[s]));
    return fx;
}

// in-place sine passes over a dense box b0 x b1 x b2 along axis 2, then axis 1
// (if M1 > 0), with panel counts M2 / M1
int dst_box(idp_plan p, double *x, int b0, int b1, int b2, int M2, int M1, cudaStream_t st, int *gmax)
{
    const int axes[2] = {2, 1};
    const int Ms[2] = {M2, M1};
    for (int q = 0; q < 2; ++q) {
        if (Ms[q] <= 0) continue;
        DstPass a{};
        const View3 v{x, (int64_t)b1 * b2, b2, 1};
        a.in = v; a.out = v; a.tab = nullptr;
        a.n0 = b0; a.n1 = b1; a.n2 = b2;
        a.axis = axes[q];
        a.M = Ms[q];
        a.gmax = q == 1 || Ms[1] <= 0 ? gmax : nullptr;   // the last pass
        FftTables t{};
        int rc;
        const bool ddm = p->mixed == IDP_PRECISION_DF32 || tensor_mode(p);
        if (has_fft_dst(Ms[q])) {
            if ((rc = get_fft(p, Ms[q] / 2, &t))) return rc;
            if ((rc = get_dst_tables(p, Ms[q], &a.qtab))) return rc;
        } else if ((rc = get_sinm(p, Ms[q], &a.sinm, ddm ? 1 : 0))) {   // direct sums
            return rc;
        }
        if (ddm && (tensor_mode(p) || !has_fft_dst(Ms[q]))) {
            a.dd = 1;
            a.twd = t.fwdd;
            a.halfd = t.halfd;
            if (has_fft_dst(Ms[q]) && (rc = get_sin2d(p, Ms[q], &a.sin2d))) return rc;
        }
        Mark mk(p, IDP_KERNEL_DST_PARTS, st);
        IDP_CK(launch_dst_pass(a, st));
    }
    return IDP_OK;
}

// (d-1)-dimensional sine transforms of `nl` layers per axis.  Equal shapes form one box; else
// each axis has its own box, and with conc they run beside each other on the plan's face
// streams (each is one or two launches of a few microseconds that fill a part of the chip:
// 33 x 65 x 97 has twelve of them per solve)
int layer_transforms(idp_plan p, double *P0, double *P1, double *P2, int nl, cudaStream_t st, int *gm, bool conc)
{
    const int n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
    if (p->d == 3 && n0 == n1 && n1 == n2) return dst_box(p, P0, 3 * nl, n1, n2, p->M[2], p->M[1], st, gm);
    const int nside = p->d == 3 ? 2 : 1;   // boxes on other streams
    cudaStream_t s1 = st, s2 = st;
    if (conc) {
        s1 = p->fst[0];
        if (nside == 2) s2 = p->fst[1];
        IDP_CK(cudaEventRecord(p->fev[0], st));
        for (int i = 0; i < nside; ++i) IDP_CK(cudaStreamWaitEvent(p->fst[i], p->fev[0], 0));
    }
    int rc;
    if (p->d == 3) {
        if ((rc = dst_box(p, P0, nl, n1, n2, p->M[2], p->M[1], st, gm))) return rc;
        if ((rc = dst_box(p, P1, nl, n0, n2, p->M[2], p->M[0], s1, gm))) return rc;
        if ((rc = dst_box(p, P2, nl, n0, n1, p->M[1], p->M[0], s2, gm))) return rc;
    } else {
        if ((rc = dst_box(p, P1, nl, 1, n2, p->M[2], 0, st, gm))) return rc;
        if ((rc = dst_box(p, P2, nl, 1, n1, p->M[1], 0, s1, gm))) return rc;
    }
    if (conc)
        for (int i = 0; i < nside; ++i) {
            IDP_CK(cudaEventRecord(p->fev[1 + i], p->fst[i]));
            IDP_CK(cudaStreamWaitEvent(st, p->fev[1 + i], 0));
        }
    return IDP_OK;
}

// gtilde parts Q0, Q1, Q2 and their (d-1)-dimensional sine transforms
int gtilde_parts(idp_plan p, bool transform_parts, cudaStream_t st, bool conc)
{
    {
        Mark mk(p, IDP_KERNEL_GTILDE, st);
        IDP_CK(launch_gtilde_planes(p->grid, p->coef, p->U, p->Q0, p->Q1, p->Q2, st));
    }
    if (!transform_parts) return IDP_OK;
    int *gm = layers_fx(p) ? p->gmax[2] : nullptr;
    const int n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
    const int rc = layer_transforms(p, p->Q0, p->Q1, p->Q2, 2, st, gm, conc);
    if (rc) return rc;
    Mark mk(p, IDP_KERNEL_GTILDE, st);
    IDP_CK(launch_layers_combine(p->Q0, p->d == 3 ? (int64_t)n1 * n2 : 0, p->Q1, (int64_t)n0 * n2, p->Q2,
                                 (int64_t)n0 * n1, 1, st, gm));
    return IDP_OK;
}

// (d-1)-dimensional sine transforms of the layers of E (two per face)
int e_layers(idp_plan p, cudaStream_t st, bool conc)
{
    int *gm = layers_fx(p) ? p->gmax[3] : nullptr;
    const int n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
    const int rc = layer_transforms(p, p->E0, p->E1, p->E2, 4, st, gm, conc);
    if (rc) return rc;
    Mark mk(p, IDP_KERNEL_RHS6_EXPAND, st);
    IDP_CK(launch_layers_combine(p->E0, p->d == 3 ? (int64_t)n1 * n2 : 0, p->E1, (int64_t)n0 * n2, p->E2,
                                 (int64_t)n0 * n1, 2, st, gm));
    return IDP_OK;
}

// Forward transform of rho scaled by 1/lambda_c into A, starting from the
// boundary stage 1a output: T0 = 2 * (real FFT of the zero-padded rows along
// axis 2), whose imaginary part at m = 1..M2-1 is -2 times the sine sums of
// the rows, i.e. -1/2 of the first sine pass (4 S).  The remaining passes run
// on that data and the factor -2 is in tabc2.
int transform_rho_from_T0(idp_plan p, cudaStream_t st)
{
    const int64_t row = 2 * (int64_t)(p->P[2] + 1);   // doubles per T0 row
    const View3 im{reinterpret_cast<double *>(p->T0) + 3, (int64_t)p->ni[1] * row, row, 2};
    const int dd = boundary_dd(p);   // T0 holds pairs
    return transform(p, im, p->A, dense(p, p->A), p->tabc2, true, st, true, true, dd);
}

// about n chunks of the np slices of a face pass, no more than pairs: ceil(np / slices per chunk)
int face_q_chunks(int np, int n)
{
    n = std::max(1, std::min(n, (np + 1) / 2));
    const int per = (np + n - 1) / n;
    return (np + per - 1) / per;
}

// the fixed-point face pass of axis a_ into `part`, and what the inverse transform of
// its parts needs
int face_q_pass(idp_plan p, int a_, int nchunk, double2 *part, FaceQPass *q, FaceInvB *ib)
{
    const int b = a_ == 0 ? 1 : 0, c = a_ == 2 ? 1 : 2;
    const int64_t r2 = p->P[2] + 1, r1 = p->P[1] + 1;
    q->D = a_ == 2 ? p->T1 : p->T0;
    q->sp = a_ == 0 ? p->ni[1] * r2 : a_ == 1 ? r2 : r1;
    q->sb = a_ == 0 ? r2 : a_ == 1 ? p->ni[1] * r2 : p->ni[2] * r1;
    q->sc = 1;
    q->np = p->ni[a_]; q->Mb = p->M[b]; q->Pb = p->P[b]; q->nc = p->P[c] + 1;
    q->kq = p->kq[a_];
    q->part = reinterpret_cast<qc *>(part);
    q->nchunk = nchunk;
    q->sliceflag = p->sl[a_];
    q->gmax = p->gmax[a_ == 2 ? 1 : 0];
    q->sums = p->sums + (a_ == 0 ? 0 : a_ == 1 ? p->ni[0] : p->ni[0] + p->ni[1]);
    q->nsum = p->nsum;
    q->unit = p->unit[a_];
    ib->fx = 1; ib->nchunk = nchunk; ib->ek = p->kq_ek[a_]; ib->gmax = q->gmax; ib->unit = q->unit;
    const int4 *half;
    const int rc = get_fft_tables(p, 2 * p->P[b], &q->q, &half);
    ib->q = q->q;
    return rc;
}

// boundary values g into the boundary nodes of dst0 (and dst1 if not null).
// rho_src (optional): the node array that the first row transform reads instead
// of rho, copying its interior into rho for the later stages (a page-locked host
// buffer, through its device view: the upload then runs inside that pass).
// stage: g is the output itself: a tensor-core mode with FP64 boundary then gives the
// values of an FP64 plan
int boundary(idp_plan p, const double *rho, double *dst0, double *dst1, cudaStream_t st,
             bool fork_rho = false, const double *rho_src = nullptr, bool stage = false)
{
    Range rg(p, "idp:boundary values g");
    const View3 r = node_interior(p, rho);
    int rc;
    FftTables t;
    // double-float arithmetic for the 3-D convolutions, on request, in the tensor-core modes
    const int dd = boundary_dd(p);
    const int fx = stage ? !dd : boundary_fx(p);
    // support flags of rho: set by the first row transform
    IDP_CK(cudaMemsetAsync(p->sums, 0, (size_t)((char *)(p->flags + p->nflags) - (char *)p->sums), st));
    // stage 1a: along axis 2 -> T0[i0][i1][m2]; stage 1b: along axis 1 -> T1[i0][i2][m1]
    RfftPass a2{}, a1{};
    a2.in = rho_src ? node_interior(p, rho_src).p : r.p;
    a2.copy = rho_src ? r.p : nullptr;
    a2.is0 = r.s0; a2.is1 = r.s1; a2.is2 = r.s2;
    a2.out = p->T0;
    a2.os2 = 1; a2.os1 = p->P[2] + 1; a2.os0 = (int64_t)p->ni[1] * (p->P[2] + 1);
    a2.n0 = p->ni[0]; a2.n1 = p->ni[1]; a2.n2 = p->ni[2];
    a2.axis = 2; a2.M = p->M[2]; a2.P = p->P[2];
    if ((rc = get_fft(p, p->P[2], &t))) return rc;
    a2.t = t;
    a2.fx = a1.fx = fx;
    a2.gmax = p->gmax[0];
    a1.gmax = p->gmax[1];
    if (fx && p->d == 3) {
        a2.sums = a1.sums = p->sums;
        a2.nsum = a1.nsum = p->nsum;
        a2.sumu = 0;
        a2.sumv = p->ni[0];
        a1.sumu = -1;
        a1.sumv = p->ni[0] + p->ni[1];
    }
    if ((rc = get_fft_tables(p, p->P[2], &a2.q, &a2.qhalf))) return rc;
    a2.dd = dd;
    // the pass along axis 2 reads every value of rho once: it also marks which
    // rows and slices are non-zero (zero ones are skipped below; their
    // contributions are exactly zero)
    a2.fl_row2 = p->row2; a2.fl_row1 = p->row1;
    a2.fl_sl0 = p->sl[0]; a2.fl_sl1 = p->sl[1]; a2.fl_sl2 = p->sl[2];
    a1.in = r.p; a1.is0 = r.s0; a1.is1 = r.s1; a1.is2 = r.s2;
    a1.out = p->T1;
    a1.os1 = 1; a1.os2 = p->P[1] + 1; a1.os0 = (int64_t)p->ni[2] * (p->P[1] + 1);
    a1.n0 = p->ni[0]; a1.n1 = p->ni[1]; a1.n2 = p->ni[2];
    a1.axis = 1; a1.M = p->M[1]; a1.P = p->P[1];
    if ((rc = get_fft(p, p->P[1], &t))) return rc;
    a1.t = t;
    if ((rc = get_fft_tables(p, p->P[1], &a1.q, &a1.qhalf))) return rc;
    a1.dd = dd;
    a1.lineflag = p->row1;
    {
        Mark mk(p, IDP_KERNEL_RFFT, st);
        IDP_CK(launch_rfft_pass(a2, st));
    }
    if (fork_rho) {
        // the rest of the forward transform of rho runs beside the boundary stages
        IDP_CK(cudaEventRecord(p->fork, st));
        IDP_CK(cudaStreamWaitEvent(p->side, p->fork, 0));
        if ((rc = transform_rho_from_T0(p, p->side))) return rc;
        IDP_CK(cudaEventRecord(p->join, p->side));
    }
    // the faces of axes 0 and 1 read only T0: with fork_rho they start on their
    // own streams while the rest runs on st
    // (2-D: the faces of axis 1)
    const bool conc = fork_rho;
    const int nbr = p->d == 3 ? 2 : 1;   // branches
    if (conc) {
        IDP_CK(cudaEventRecord(p->fev[0], st));
        for (int i = 0; i < nbr; ++i) IDP_CK(cudaStreamWaitEvent(p->fst[i], p->fev[0], 0));
    }
    {
        Mark mk(p, IDP_KERNEL_RFFT, st);
        IDP_CK(launch_rfft_pass(a1, st));
    }
    if (p->d == 2) {
        // faces of axis 1 (rows i1 = 0, M1; data along axis 2) and of axis 2
        for (int face = 1; face <= 2; ++face) {
            FacePass2D a{};
            const int other = face == 1 ? 2 : 1;
            cudaStream_t sa = conc && face == 1 ? p->fst[0] : st;
            double2 *F = p->F + (face - 1) * p->f_cap;
            if (face == 1) { a.T = p->T0; a.sp = p->P[2] + 1; a.sm = 1; }
            else { a.T = p->T1; a.sp = p->P[1] + 1; a.sm = 1; }
            a.np = p->ni[face];
            a.nm = p->P[other] + 1;
            a.khat = p->khat[face];
            a.acc = F;
            a.split = fx;   // (the tensor-core modes keep the order of the sum)
            {
                Mark mk(p, IDP_KERNEL_FACE, sa);
                IDP_CK(launch_face_pass_2d(a, sa));
            }
            FaceC2R c{};
            c.in = F; c.nrows = 1; c.Mc = p->M[other]; c.Pc = p->P[other];
            c.dst0 = dst0; c.dst1 = dst1;
            c.base[0] = 0; c.base[1] = (int64_t)p->M[face] * p->ns[face];
            c.row_stride = 0; c.col_stride = p->ns[other];
            c.skip_row_edges = 0; c.skip_col_edges = (face == 2);
            if ((rc = get_fft(p, p->P[other], &t))) return rc;
            c.t = t;
            c.fx = fx;
            if ((rc = get_fft_tables(p, p->P[other], &c.q, &c.qhalf))) return rc;
            Mark mk(p, IDP_KERNEL_FACE_C2R, sa);
            IDP_CK(launch_face_c2r(c, sa));
        }
        if (conc) {
            IDP_CK(cudaEventRecord(p->fev[1], p->fst[0]));
            IDP_CK(cudaStreamWaitEvent(st, p->fev[1], 0));
        }
        return IDP_OK;
    }
    // 3-D: faces of axis a; b < c the other axes; data and strides per face
    for (int a_ = 0; a_ < 3; ++a_) {
        const int b = a_ == 0 ? 1 : 0;
        const int c = a_ == 2 ? 1 : 2;
        cudaStream_t sa = (conc && a_ < 2) ? p->fst[a_] : st;
        double2 *part = p->part + a_ * p->part_cap, *F = p->F + a_ * p->f_cap;
        FacePass f{};
        if (a_ == 0) { f.D = p->T0; f.sp = (int64_t)p->ni[1] * (p->P[2] + 1); f.sb = p->P[2] + 1; f.sc = 1; }
        else if (a_ == 1) { f.D = p->T0; f.sp = p->P[2] + 1; f.sb = (int64_t)p->ni[1] * (p->P[2] + 1); f.sc = 1; }
        else { f.D = p->T1; f.sp = p->P[1] + 1; f.sb = (int64_t)p->ni[2] * (p->P[1] + 1); f.sc = 1; }
        f.np = p->ni[a_];
        f.Mb = p->M[b];
        f.Pb = p->P[b];
        f.nc = p->P[c] + 1;
        f.khat = p->khat[a_];
        f.part = part;
        f.pchunk = p->pchunk[a_];
        if ((rc = get_fft(p, 2 * p->P[b], &t))) return rc;
        f.t = t;
        f.dd = dd;
        f.khatd = p->khatd[a_];
        f.sliceflag = p->sl[a_];
        FaceInvB ib{};
        ib.part = part; ib.nchunk = p->nchunk[a_];
        {
            Mark mk(p, IDP_KERNEL_FACE, sa);
            if (fx) {
                FaceQPass q{};
                if ((rc = face_q_pass(p, a_, p->qchunk[a_], part, &q, &ib))) return rc;
                IDP_CK(launch_face_q(q, sa));
            } else {
                IDP_CK(launch_face_pass(f, p->nchunk[a_], sa));
            }
        }
        ib.Mb = p->M[b]; ib.Pb = p->P[b]; ib.nc = f.nc; ib.out = F; ib.t = t;
        ib.dd = dd;
        {
            Mark mk(p, IDP_KERNEL_FACE_INVB, sa);
            IDP_CK(launch_face_inv_b(ib, sa));
        }
        FaceC2R cr{};
        cr.in = F; cr.nrows = p->M[b] + 1; cr.Mc = p->M[c]; cr.Pc = p->P[c];
        cr.dst0 = dst0; cr.dst1 = dst1;
        cr.base[0] = 0; cr.base[1] = (int64_t)p->M[a_] * p->ns[a_];
        cr.row_stride = p->ns[b]; cr.col_stride = p->ns[c];
        cr.skip_row_edges = (a_ >= 1);
        cr.skip_col_edges = (a_ == 2);
        if ((rc = get_fft(p, p->P[c], &t))) return rc;
        cr.t = t;
        cr.dd = dd;
        cr.fx = fx;
        if ((rc = get_fft_tables(p, p->P[c], &cr.q, &cr.qhalf))) return rc;
        Mark mk(p, IDP_KERNEL_FACE_C2R, sa);
        IDP_CK(launch_face_c2r(cr, sa));
    }
    if (conc)
        for (int i = 0; i < 2; ++i) {
            IDP_CK(cudaEventRecord(p->fev[1 + i], p->fst[i]));
            IDP_CK(cudaStreamWaitEvent(st, p->fev[1 + i], 0));
        }
    return IDP_OK;
}

enum { RUN_PHI = 0 };

// Queue the stages of one solve.  stop: 0 = full solve into phi; otherwise an
// IDP_STAGE_* value whose result is written to `out`.
// d = 1 (section 5): phi* by one forward and one inverse sine pass, then g at
// the two ends and the straight line through them added inside
int enqueue_1d(idp_plan p, const double *rho, double *phi, int stop, cudaStream_t st)
{
    const size_t node_bytes = sizeof(double) * p->nodes;
    const int M = p->M[2];
    if (stop == 0 && p->hio_rho)
        IDP_CK(cudaMemcpyAsync(p->h_rho, p->hio_rho, node_bytes, cudaMemcpyHostToDevice, st));
    if (stop == IDP_STAGE_BOUNDARY || stop == IDP_STAGE_U1) {
        Mark mk(p, IDP_KERNEL_LINE1D, st);
        IDP_CK(launch_line1d(rho, phi, M, p->h[2], stop == IDP_STAGE_BOUNDARY ? LINE1D_ENDS : LINE1D_LINE, st));
        return IDP_OK;
    }
    if (stop != 0 && stop != IDP_STAGE_PHISTAR) return IDP_ESUPPORT;
    int rc;
    if (stop == IDP_STAGE_PHISTAR) IDP_CK(cudaMemsetAsync(phi, 0, node_bytes, st));
    if ((rc = transform(p, node_interior(p, rho), p->A, dense(p, p->A), p->tabc, true, st))) return rc;
    if ((rc = transform(p, dense(p, p->A), p->A, node_interior(p, phi), nullptr, false, st))) return rc;
    if (stop == IDP_STAGE_PHISTAR) return IDP_OK;
    Mark mk(p, IDP_KERNEL_LINE1D, st);
    IDP_CK(launch_line1d(rho, phi, M, p->h[2], LINE1D_ADD, st));
    return IDP_OK;
}

int enqueue_grid(idp_plan p, const double *rho, double *phi, int stop, cudaStream_t st);

// A padded plan: the interior nodes of the caller's rho go into the padded array
// (the rest of it stays zero: the caller's boundary entries of rho are not used,
// as in an unpadded solve), the solve runs on the padded grid, and phi is read
// back at the caller's nodes.  Full solves only.
int enqueue_padded(idp_plan p, const double *rho, double *phi, int stop, cudaStream_t st)
{
    if (stop != 0) return IDP_ESUPPORT;
    if (p->hio_rho)
        IDP_CK(cudaMemcpyAsync(p->h_rho, p->hio_rho, sizeof(double) * p->unodes, cudaMemcpyHostToDevice, st));
    int lo[3], ext[3];
    for (int s = 0; s < 3; ++s) {
        lo[s] = p->act[s] ? 1 : 0;
        ext[s] = p->act[s] ? p->un[s] - 2 : 1;
    }
    const int64_t u1 = p->un[2], u0 = (int64_t)p->un[1] * p->un[2];
    const int64_t n1 = p->n[2], n0 = (int64_t)p->n[1] * p->n[2];
    const int64_t uo = (int64_t)p->uoff[0] * n0 + (int64_t)p->uoff[1] * n1 + p->uoff[2];
    {
        Mark mk(p, IDP_KERNEL_PAD, st);
        IDP_CK(launch_box_copy(rho + lo[0] * u0 + lo[1] * u1 + lo[2], u0, u1,
                               p->rho_pad + uo + lo[0] * n0 + lo[1] * n1 + lo[2], n0, n1, ext[0], ext[1], ext[2],
                               st));
    }
    const double *hio = p->hio_rho;
    p->hio_rho = nullptr;
    const int rc = enqueue_grid(p, p->rho_pad, p->phi_pad, 0, st);
    p->hio_rho = hio;
    if (rc) return rc;
    Mark mk(p, IDP_KERNEL_PAD, st);
    IDP_CK(launch_box_copy(p->phi_pad + uo, n0, n1, phi, u0, u1, p->un[0], p->un[1], p->un[2], st));
    return IDP_OK;
}

int enqueue(idp_plan p, const double *rho, double *phi, int stop, cudaStream_t st)
{
    Range rg(p, stop ? "idp:stage" : "idp:solve");
    if (p->validate) {
        // validation mode: the caller's rho is checked first (in a host-buffer
        // solve it goes up in one copy, and the check reads the copy)
        const double *hio = p->hio_rho;
        if (hio) {
            IDP_CK(cudaMemcpyAsync(p->h_rho, hio, sizeof(double) * p->unodes, cudaMemcpyHostToDevice, st));
            p->hio_rho = nullptr;
        }
        {
            Mark mk(p, IDP_KERNEL_VALIDATE, st);
            IDP_CK(launch_validate_rho(rho, p->un[0], p->un[1], p->un[2], p->act[0], p->act[1], p->act[2],
                                       p->validate, p->d_val, st));
        }
        const int rc = p->padded ? enqueue_padded(p, rho, phi, stop, st) : enqueue_grid(p, rho, phi, stop, st);
        p->hio_rho = hio;
        return rc;
    }
    if (p->padded) return enqueue_padded(p, rho, phi, stop, st);
    return enqueue_grid(p, rho, phi, stop, st);
}

// one solve (or stage) on the plan's own grid
int enqueue_grid(idp_plan p, const double *rho, double *phi, int stop, cudaStream_t st)
{
    if (p->d == 1) return enqueue_1d(p, rho, phi, stop, st);
    int rc;
    const size_t node_bytes = sizeof(double) * p->nodes;
    if (stop == IDP_STAGE_BOUNDARY) {
        IDP_CK(cudaMemsetAsync(phi, 0, node_bytes, st));
        return boundary(p, rho, phi, nullptr, st, false, nullptr, true);
    }
    if (stop == IDP_STAGE_PHISTAR) {
        IDP_CK(cudaMemsetAsync(phi, 0, node_bytes, st));
        if ((rc = transform(p, node_interior(p, rho), p->A, dense(p, p->A), p->tabc, true, st))) return rc;
        return transform(p, dense(p, p->A), p->A, node_interior(p, phi), nullptr, false, st);
    }
    // 0. the forward transform of rho does not depend on the boundary values:
    //    queue it on the side stream so it overlaps the boundary convolutions
    // (profiling keeps one stream so that every launch is timed on its own)
    const bool overlap_rho = (stop == 0) && !p->profiling;
    // FP64 / df32 transforms: the first pass of the forward transform of rho is
    // the imaginary part of the boundary's first real FFT (see transform_rho_from_T0)
    const bool rho_from_T0 = (stop == 0) && !(tensor_mode(p) && p->mixed_path == 0) &&
                             has_fft_dst(p->M[2]) && p->P[2] == p->M[2];
    // host-buffer solve: the first row transform reads rho from the host buffer
    // and leaves the device copy for the later stages; where rho is needed before
    // it (the tensor-core transform of rho starts at once), rho goes up first
    const double *rho_src = (stop == 0 && p->hio_rho && rho_from_T0) ? p->hio_view : nullptr;
    if (stop == 0 && p->hio_rho && !rho_src)
        IDP_CK(cudaMemcpyAsync(p->h_rho, p->hio_rho, sizeof(double) * p->nodes, cudaMemcpyHostToDevice, st));
    // the tensor-core transform of rho leaves out the eigenvalue factor tabc: the
    // expansion kernels below apply it (an FP64 table read in the epilogue of a
    // tensor-core pass is latency-bound there)
    const bool rho_unscaled = (stop == 0) && !rho_from_T0;
    const double *ascale = rho_unscaled ? p->tabc : nullptr;
    if (overlap_rho && !rho_from_T0) {
        IDP_CK(cudaEventRecord(p->fork, st));
        IDP_CK(cudaStreamWaitEvent(p->side, p->fork, 0));
        if ((rc = transform(p, node_interior(p, rho), p->A, dense(p, p->A), nullptr, true, p->side)))
            return rc;
        IDP_CK(cudaEventRecord(p->join, p->side));
    }
    // 1. boundary values: phi boundary and U boundary
    if ((rc = boundary(p, rho, stop == 0 ? phi : p->U, stop == 0 ? p->U : nullptr, st,
                       overlap_rho && rho_from_T0, rho_src)))
        return rc;
    // 2. gtilde on the boundary-adjacent layers, and the transforms of its parts
    if ((rc = gtilde_parts(p, stop != IDP_STAGE_GTILDE, st, overlap_rho))) return rc;
    if (stop == IDP_STAGE_GTILDE) {
        IDP_CK(launch_gtilde_scatter(p->grid, p->Q0, p->Q1, p->Q2, phi, st));
        return IDP_OK;
    }
    // 3. the forward transform of rho, scaled by 1/lambda_c (on the side stream
    //    in a full solve, joined before A is first used)
    if (stop == 0 && !overlap_rho) {
        if (rho_from_T0) {
            if ((rc = transform_rho_from_T0(p, st))) return rc;
        } else if ((rc = transform(p, node_interior(p, rho), p->A, dense(p, p->A), nullptr, true, st))) {
            return rc;
        }
    }
    if (p->order == 4 && stop == 0) {
        if (overlap_rho) IDP_CK(cudaStreamWaitEvent(st, p->join, 0));
        // A += tab4 * S gtilde; phi = S A inside
        {
            Mark mk(p, IDP_KERNEL_GTILDE_EXPAND, st);
            IDP_CK(layers_fx(p) ? launch_gtilde_expand_q(p->grid, p->Q0, p->Q1, p->Q2, p->sinq, p->gmax[2], p->tab4,
                                                         p->A, p->A, nullptr, nullptr, nullptr, st)
                                : launch_gtilde_expand(p->grid, p->Q0, p->Q1, p->Q2, p->sin4, p->tab4, p->A, p->A,
                                                       st, nullptr, nullptr, nullptr, 0, ascale));
        }
        return transform(p, dense(p, p->A), p->A, node_interior(p, phi), nullptr, false, st);
    }
    // 4. u1 = S B, B = tab4 * S gtilde; in a full solve also C = A + tabR * S gtilde,
    //    the solution coefficients less the layer correction (R_spec's share)
    if (stop == 0 && overlap_rho) IDP_CK(cudaStreamWaitEvent(st, p->join, 0));
    // the final transform takes u1 in C (S C + S B = S (C + B)), in every mode
    {
        Mark mk(p, IDP_KERNEL_GTILDE_EXPAND, st);
        double *C = stop == 0 ? p->C : nullptr;
        IDP_CK(layers_fx(p) ? launch_gtilde_expand_q(p->grid, p->Q0, p->Q1, p->Q2, p->sinq, p->gmax[2], p->tab4,
                                                     nullptr, p->B, p->tabR, p->A, C, st)
                            : launch_gtilde_expand(p->grid, p->Q0, p->Q1, p->Q2, p->sin4, p->tab4, nullptr, p->B,
                                                   st, p->tabR, p->A, C, 1, ascale));
    }
    // u1 feeds the sixth differences of R, which amplify its rounding by ~1e4-1e7:
    // this inverse transform stays FP64 in the FP64 and DF32 modes, and is a
    // double-float one (48 bits, never the tensor cores) in the tensor-core modes
    if ((rc = transform(p, dense(p, p->B), p->B, node_interior(p, p->U), nullptr, false, st, false, false, 0,
                        false)))
        return rc;
    if (stop == IDP_STAGE_U1) {
        IDP_CK(cudaMemcpyAsync(phi, p->U, node_bytes, cudaMemcpyDeviceToDevice, st));
        return IDP_OK;
    }
    // 5. E = R - R_spec on the layers next to the faces: W of the odd continuation
    //    near the faces, R at the extrapolation taps (into A, free now), E
    {
        Mark mk(p, IDP_KERNEL_RHS6_W, st);
        IDP_CK(launch_rhs6_spectral(p->grid, p->coef, p->U, p->W, p->A, p->E0, p->E1, p->E2, 0, st));
    }
    {
        Mark mk(p, IDP_KERNEL_RHS6_CORE, st);
        IDP_CK(launch_rhs6_spectral(p->grid, p->coef, p->U, p->W, p->A, p->E0, p->E1, p->E2, 1, st));
    }
    {
        Mark mk(p, IDP_KERNEL_RHS6_EXTRAP, st);
        IDP_CK(launch_rhs6_spectral(p->grid, p->coef, p->U, p->W, p->A, p->E0, p->E1, p->E2, 2, st));
    }
    if (stop == IDP_STAGE_R) {
        // R = S (Lambda_R b) + E with b the coefficients of u1 (recomputed), as a
        // dense interior array
        {
            Mark mk(p, IDP_KERNEL_GTILDE_EXPAND, st);
            IDP_CK(layers_fx(p) ? launch_gtilde_expand_q(p->grid, p->Q0, p->Q1, p->Q2, p->sinq, p->gmax[2], p->tab4,
                                                         nullptr, p->C, nullptr, nullptr, nullptr, st)
                                : launch_gtilde_expand(p->grid, p->Q0, p->Q1, p->Q2, p->sin4, p->tab4, nullptr,
                                                       p->C, st));
        }
        IDP_CK(launch_rhs6_symbol(p->grid, p->ld, p->ldoff[1], p->ldoff[2], p->C, st));
        if ((rc = transform(p, dense(p, p->C), p->C, dense(p, phi), nullptr, false, st, false))) return rc;
        IDP_CK(launch_rhs6_e_scatter(p->grid, p->E0, p->E1, p->E2, phi, st));
        return IDP_OK;
    }
    // 6. the layer transforms of E; C += tab4 * S E;  phi = S C + u1 inside
    if ((rc = e_layers(p, st, overlap_rho))) return rc;
    {
        Mark mk(p, IDP_KERNEL_RHS6_EXPAND, st);
        IDP_CK(layers_fx(p) ? launch_rhs6_e_expand_q(p->grid, p->E0, p->E1, p->E2, p->sinq, p->sinq2, p->gmax[3],
                                                     p->tab4, p->C, st)
                            : launch_rhs6_e_expand(p->grid, p->E0, p->E1, p->E2, p->sin4, p->sin4b, p->tab4, p->C,
                                                   st));
    }
    return transform(p, dense(p, p->C), p->C, node_interior(p, phi), nullptr, false, st);
}

// the plan's streams and events (graph capture forks and joins through them)
int plan_streams(idp_plan p)
{
    IDP_CK(cudaStreamCreateWithFlags(&p->side, cudaStreamNonBlocking));
    IDP_CK(cudaStreamCreateWithFlags(&p->bst, cudaStreamNonBlocking));
    if (!p->cap) IDP_CK(cudaStreamCreateWithFlags(&p->cap, cudaStreamNonBlocking));
    IDP_CK(cudaEventCreateWithFlags(&p->fork, cudaEventDisableTiming));
    IDP_CK(cudaEventCreateWithFlags(&p->join, cudaEventDisableTiming));
    for (int i = 0; i < 2; ++i) IDP_CK(cudaStreamCreateWithFlags(&p->fst[i], cudaStreamNonBlocking));
    for (int i = 0; i < 3; ++i) IDP_CK(cudaEventCreateWithFlags(&p->fev[i], cudaEventDisableTiming));
    return IDP_OK;
}

// d = 1: the sine-pass tables (made by plan_setup), the coefficient array and
// tabc = (2/M) / lambda_c(k) / 16 with lambda_c(k) = -(pi k / L)^2, L = M h: the
// forward sums scaled by 2/M and divided by the continuum eigenvalue (section 3);
// each sine pass returns 4 S x, hence the 1/16
int plan_setup_1d(idp_plan p)
{
    int rc;
    const int M = p->M[2], N = p->ni[2];
    if ((rc = p->alloc(&p->A, p->nint)) || (rc = p->alloc(&p->tabc, p->nint))) return rc;
    std::vector<double> tc(N);
    const double L = (double)M * p->h[2];
    for (int k = 1; k <= N; ++k) {
        const double w = 3.14159265358979323846 * k / L;
        tc[k - 1] = (2.0 / M) / (-(w * w)) / 16.0;
    }
    IDP_CK(cudaMemcpy(p->tabc, tc.data(), sizeof(double) * N, cudaMemcpyHostToDevice));
    return plan_streams(p);
}

// the first face axis whose kernel spectra are those of axis a_
int spectra_like(idp_plan p, int a_)
{
    auto key = [&](int s) {
        const int b = s == 0 ? 1 : 0, c = s == 2 ? 1 : 2;
        return std::make_tuple(p->ni[s], p->P[b], p->P[c], p->h[s], p->h[b], p->h[c]);
    };
    int s = 0;
    while (key(s) != key(a_)) ++s;
    return s;
}

int plan_setup(idp_plan p)
{
    int rc;
    // every table a solve uses is created here, so that solves (and their
    // graph capture) never allocate
    for (int s = 0; s < 3; ++s) {
        if (!p->act[s]) continue;
        FftTables t;
        const int4 *qt, *qh;
        const ddr *sd;
        const void *sm_;
        if ((has_fft_dst(p->M[s]) && ((rc = get_fft(p, p->M[s] / 2, &t)) || (rc = get_dst_tables(p, p->M[s], &qt)) || (rc = get_sin2d(p, p->M[s], &sd)))) ||
            (!has_fft_dst(p->M[s]) && (rc = get_sinm(p, p->M[s], &sm_, 0))) ||
            (rc = get_fft(p, p->P[s], &t)) || (rc = get_fft(p, 2 * p->P[s], &t)) ||
            (rc = get_fft_tables(p, p->P[s], &qt, &qh)) || (rc = get_fft_tables(p, 2 * p->P[s], &qt, &qh)))
            return rc;
    }
    if (p->padded) {
        if ((rc = p->alloc(&p->rho_pad, p->nodes)) || (rc = p->alloc(&p->phi_pad, p->nodes))) return rc;
        IDP_CK(cudaMemset(p->rho_pad, 0, sizeof(double) * p->nodes));
    }
    if (p->d == 1) return plan_setup_1d(p);
    // workspace
    if ((rc = p->alloc(&p->A, p->nint)) || (rc = p->alloc(&p->B, p->nint)) || (rc = p->alloc(&p->C, p->nint)) ||
        (rc = p->alloc(&p->U, p->nodes)) || (rc = p->alloc(&p->W, 3 * p->nodes)) ||
        (rc = p->alloc(&p->tabc, p->nint)) || (rc = p->alloc(&p->tab4, p->nint)) ||
        (rc = p->alloc(&p->tabc2, p->nint)))
        return rc;
    if ((rc = p->alloc(&p->T0, (int64_t)p->ni[0] * p->ni[1] * (p->P[2] + 1))) ||
        (rc = p->alloc(&p->T1, (int64_t)p->ni[0] * p->ni[2] * (p->P[1] + 1))))
        return rc;
    {
        const int64_t q0 = 2 * (int64_t)p->ni[1] * p->ni[2], q1 = 2 * (int64_t)p->ni[0] * p->ni[2],
                      q2 = 2 * (int64_t)p->ni[0] * p->ni[1];
        if ((rc = p->alloc(&p->Q0, q0 + q1 + q2))) return rc;
        p->Q1 = p->Q0 + q0;
        p->Q2 = p->Q1 + q1;
    }
    {
        const int64_t n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
        p->nflags = n0 * n1 + n0 * n2 + n0 + n1 + n2 + 7;
        p->nsum = (int)(n0 + n1 + n2);
        const int64_t ns = p->d == 3 ? (int64_t)FACE_WINDOWS * p->nsum : 0;
        if ((rc = p->alloc(&p->sums, ns + (p->nflags + 1) / 2))) return rc;
        p->flags = reinterpret_cast<int *>(p->sums + ns);
        p->row2 = p->flags;
        p->row1 = p->row2 + n0 * n1;
        p->sl[0] = p->row1 + n0 * n2;
        p->sl[1] = p->sl[0] + n0;
        p->sl[2] = p->sl[1] + n1;
        p->gmax[0] = p->sl[2] + n2;
        for (int i = 1; i < 4; ++i) p->gmax[i] = p->gmax[0] + i;
        for (int i = 0; i < 3; ++i) p->unit[i] = p->gmax[3] + 1 + i;
    }
    if ((rc = plan_streams(p))) return rc;
    {
        std::vector<double> s4;
        for (int s = 0; s < 3; ++s) {
            if (!p->act[s]) continue;
            for (int k = 0; k < p->ni[s]; ++k) s4.push_back(4.0 * sinpi_frac(k + 1, p->M[s]));
        }
        if ((rc = p->alloc(&p->sin4, (int64_t)s4.size()))) return rc;
        IDP_CK(cudaMemcpy(p->sin4, s4.data(), sizeof(double) * s4.size(), cudaMemcpyHostToDevice));
        std::vector<double> s4b;
        for (int s = 0; s < 3; ++s) {
            if (!p->act[s]) continue;
            for (int k = 0; k < p->ni[s]; ++k) s4b.push_back(4.0 * sinpi_frac(2 * (k + 1), p->M[s]));
        }
        if ((rc = p->alloc(&p->sin4b, (int64_t)s4b.size()))) return rc;
        IDP_CK(cudaMemcpy(p->sin4b, s4b.data(), sizeof(double) * s4b.size(), cudaMemcpyHostToDevice));
        std::vector<int2> sq;
        for (int m = 1; m <= 2; ++m)
            for (int s = 0; s < 3; ++s) {
                if (!p->act[s]) continue;
                for (int k = 0; k < p->ni[s]; ++k) {
                    long double c, sn;
                    cossinpi((int64_t)m * (k + 1), p->M[s], c, sn);
                    sq.push_back(fixed_factor(sn));
                }
            }
        if ((rc = p->alloc(&p->sinq, (int64_t)sq.size()))) return rc;
        IDP_CK(cudaMemcpy(p->sinq, sq.data(), sizeof(int2) * sq.size(), cudaMemcpyHostToDevice));
        p->sinq2 = p->sinq + s4.size();
    }
    {
        // layers of E (two per face): E0 [2][2][n1][n2] (3-D), E1 [2][2][n0][n2], E2 [2][2][n0][n1]
        const int64_t n0 = p->ni[0], n1 = p->ni[1], n2 = p->ni[2];
        const int64_t e0 = p->d == 3 ? 4 * n1 * n2 : 0, e1 = 4 * n0 * n2, e2 = 4 * n0 * n1;
        if ((rc = p->alloc(&p->E0, e0 + e1 + e2))) return rc;
        p->E1 = p->E0 + e0;
        p->E2 = p->E1 + e1;
        if ((rc = p->alloc(&p->tabR, p->nint))) return rc;
    }
    IDP_CK(cudaMemset(p->U, 0, sizeof(double) * p->nodes));
    IDP_CK(cudaMemset(p->W, 0, sizeof(double) * 3 * p->nodes));

    // eigenvalue tables (sections 3 and 5)
    {
        std::vector<double> lc, ld;
        int64_t off[3] = {0, 0, 0};
        for (int s = 0; s < 3; ++s) {
            off[s] = (int64_t)lc.size();
            if (!p->act[s]) { lc.push_back(0.0); ld.push_back(0.0); continue; }
            const double L = p->M[s] * p->h[s];
            for (int k = 1; k < p->M[s]; ++k) {
                lc.push_back(-(M_PI * M_PI) * (double)k * k / (L * L));
                const double sn = sinpi_frac(k, 2 * p->M[s]);
                ld.push_back(-(4.0 / (p->h[s] * p->h[s])) * sn * sn);
            }
        }
        double *dlc, *dld;
        if ((rc = p->alloc(&dlc, (int64_t)lc.size())) || (rc = p->alloc(&dld, (int64_t)ld.size()))) return rc;
        IDP_CK(cudaMemcpy(dlc, lc.data(), sizeof(double) * lc.size(), cudaMemcpyHostToDevice));
        IDP_CK(cudaMemcpy(dld, ld.data(), sizeof(double) * ld.size(), cudaMemcpyHostToDevice));
        double sc = 1.0;
        int da = 0;
        for (int s = 0; s < 3; ++s)
            if (p->act[s]) { sc *= 2.0 / p->M[s]; ++da; }
        for (int q = 0; q < 2 * da; ++q) sc *= 0.25;   // each sine pass returns 4 S x
        IDP_CK(launch_eigen_tables(p->grid, dlc, dld, off[1], off[2], sc, p->tabc, p->tab4, p->tabR, 0));
        IDP_CK(launch_eigen_tables(p->grid, dlc, dld, off[1], off[2], -2.0 * sc, p->tabc2, p->B, nullptr, 0));
        p->ld = dld;
        for (int s = 0; s < 3; ++s) p->ldoff[s] = off[s];
    }

    // kernel spectra of the boundary convolutions (section 4)
    if (p->d == 2) {
        int64_t fmax = 0;
        for (int face = 1; face <= 2; ++face) {
            const int other = face == 1 ? 2 : 1;
            const int Mb = p->P[other];   // spectra of the cyclic kernel of length 2P
            const int np = p->ni[face];
            if ((rc = p->alloc(&p->khat[face], (int64_t)np * (Mb + 1)))) return rc;
            double *kb, *tb;
            if ((rc = p->alloc(&kb, (int64_t)np * (Mb + 1))) || (rc = p->alloc(&tb, (int64_t)(Mb + 1) * (Mb + 1))))
                return rc;
            KernelFill kf{kb, 2, np, Mb, 0, p->h[face], p->h[other], 0.0, 0, 0};
            IDP_CK(launch_kernel_fill(kf, 0));
            // DCT-I table Cb[t][m] = w_t cos(pi m t / Mb) * h_a h_b / (4 Mb)
            std::vector<double> cb((size_t)(Mb + 1) * (Mb + 1));
            const double sc = p->h[face] * p->h[other] / (4.0 * Mb);
            for (int tt = 0; tt <= Mb; ++tt)
                for (int m = 0; m <= Mb; ++m)
                    cb[(size_t)tt * (Mb + 1) + m] = ((tt == 0 || tt == Mb) ? 1.0 : 2.0) *
                                                    cospi_frac((int64_t)m * tt, Mb) * sc;
            IDP_CK(cudaMemcpy(tb, cb.data(), sizeof(double) * cb.size(), cudaMemcpyHostToDevice));
            IDP_CK(launch_gemm_batched(np, Mb + 1, Mb + 1, kb, Mb + 1, 0, tb, Mb + 1, 0, p->khat[face], Mb + 1, 0,
                                       1, 0));
            // (kb and tb stay: a few MB, and giving them back takes a tenth of the set-up)
            fmax = std::max<int64_t>(fmax, 2 * (Mb + 1));
        }
        if ((rc = p->alloc(&p->F, 2 * fmax))) return rc;
        p->f_cap = fmax;
    } else {
        int64_t pmax = 0, fmax = 0;
        // temporaries of the spectra, built in slabs of slices that bound them: the kernel's
        // values and their transform along c, the two cosine tables; one buffer for all axes
        auto slab_of = [](int np, int64_t per) { return (int)std::max<int64_t>(1, std::min<int64_t>(np, (64 << 20) / (per * 8))); };
        int64_t tslab = 0, ttab = 0;
        for (int a_ = 0; a_ < 3; ++a_) {
            const int b = a_ == 0 ? 1 : 0, c = a_ == 2 ? 1 : 2;
            const int64_t per = (int64_t)(p->P[b] + 1) * (p->P[c] + 1);
            tslab = std::max(tslab, (slab_of(p->ni[a_], per) * per + 31) / 32 * 32);
            ttab = std::max(ttab, ((int64_t)(p->P[a_] + 1) * (p->P[a_] + 1) + 31) / 32 * 32);
        }
        double *kb;
        if ((rc = p->alloc(&kb, 2 * (tslab + ttab)))) return rc;
        double *yb = kb + tslab, *tcb = yb + tslab, *tbb = tcb + ttab;
        for (int a_ = 0; a_ < 3; ++a_) {
            const int b = a_ == 0 ? 1 : 0;
            const int c = a_ == 2 ? 1 : 2;
            // spectra of the cyclic kernel of length 2P along b and c
            const int Mb = p->P[b], Mc = p->P[c], np = p->ni[a_];
            const int L = 2 * Mb;
            const int TC = face_columns_per_block(L);
            const int tiles = (Mc + 1 + TC - 1) / TC;
            // one wave of resident blocks; fewer chunks = fewer partial sums
            int nsm = 152;
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->dev);
            const int slots = nsm * face_blocks_per_sm(L);
            int nch = std::max(1, std::min(np, slots / tiles));
            int pch = (np + nch - 1) / nch;
            nch = (np + pch - 1) / pch;
            p->nchunk[a_] = nch;
            p->pchunk[a_] = pch;
            pmax = std::max<int64_t>(pmax, (int64_t)nch * 2 * L * (Mc + 1));
            const int npair = (np + 1) / 2;
            // three waves of resident blocks with at least 8 pairs a block; one wave with at least
            // 2 on small grids
            const int qtiles = 2 * ((Mc + face_q_columns(L)) / face_q_columns(L));
            const int qslots = face_q_blocks_per_sm(L) * nsm;
            p->qchunk[a_] = face_q_chunks(np, std::max(std::min(3 * qslots / qtiles, npair / 8), std::min(qslots / qtiles, npair / 2)));
            pmax = std::max<int64_t>(pmax, (int64_t)p->qchunk[a_] * 2 * L * (Mc + 1));
            fmax = std::max<int64_t>(fmax, (int64_t)2 * (Mb + 1) * (Mc + 1));
            const int64_t per = (int64_t)(Mb + 1) * (Mc + 1);
            p->khat_n[a_] = (int64_t)np * per;
            // axes with the same lengths and mesh sizes have the same spectra (all three of a
            // cube): kept once
            const int like = spectra_like(p, a_);
            if (like < a_) {
                p->khat[a_] = p->khat[like];
                p->kq[a_] = p->kq[like];
                p->kq_ek[a_] = p->kq_ek[like];
                continue;
            }
            if ((rc = p->alloc(&p->khat[a_], (int64_t)np * per))) return rc;
            const int slab = slab_of(np, per);
            // the spectra are stored transposed, [slice][frequency c][frequency b]:
            //   khat^T = Cc^T K^T Cb^T  with  K^T[t_c][t_b] = G(d_p, t_b h_b, t_c h_c)
            std::vector<double> cct((size_t)(Mc + 1) * (Mc + 1)), cbt((size_t)(Mb + 1) * (Mb + 1));
            const double sc = p->h[0] * p->h[1] * p->h[2] / (8.0 * Mb * Mc);
            for (int m = 0; m <= Mc; ++m)        // Cc^T[m][t] = w_t cos(pi m t / Mc) * sc
                for (int tt = 0; tt <= Mc; ++tt)
                    cct[(size_t)m * (Mc + 1) + tt] = ((tt == 0 || tt == Mc) ? 1.0 : 2.0) *
                                                     cospi_frac((int64_t)m * tt, Mc) * sc;
            for (int tt = 0; tt <= Mb; ++tt)     // Cb^T[t][m] = w_t cos(pi m t / Mb)
                for (int m = 0; m <= Mb; ++m)
                    cbt[(size_t)tt * (Mb + 1) + m] = ((tt == 0 || tt == Mb) ? 1.0 : 2.0) *
                                                     cospi_frac((int64_t)m * tt, Mb);
            IDP_CK(cudaMemcpy(tcb, cct.data(), sizeof(double) * cct.size(), cudaMemcpyHostToDevice));
            IDP_CK(cudaMemcpy(tbb, cbt.data(), sizeof(double) * cbt.size(), cudaMemcpyHostToDevice));
            for (int p0 = 0; p0 < np; p0 += slab) {
                const int cnt = std::min(slab, np - p0);
                KernelFill kf{kb, 3, cnt, Mb, Mc, p->h[a_], p->h[b], p->h[c], p0, 1};
                IDP_CK(launch_kernel_fill(kf, 0));
                // Y^T = Cc^T K^T: rows (frequency c) x cols (t_b)
                IDP_CK(launch_gemm_batched(Mc + 1, Mb + 1, Mc + 1, tcb, Mc + 1, 0, kb, Mb + 1, per, yb, Mb + 1, per,
                                           cnt, 0));
                // khat^T = Y^T Cb^T: rows (frequency c) x cols (frequency b)
                IDP_CK(launch_gemm_batched(Mc + 1, Mb + 1, Mb + 1, yb, Mb + 1, per, tbb, Mb + 1, 0,
                                           p->khat[a_] + (int64_t)p0 * per, Mb + 1, per, cnt, 0));
            }
            // fixed-point spectra
            if ((rc = p->alloc(&p->kq[a_], 2 * (int64_t)npair * per)) || (rc = p->alloc(&p->kq_ek[a_], per))) return rc;
            IDP_CK(launch_face_kq(p->khat[a_], np, per, p->kq[a_], p->kq_ek[a_], 0));
        }
        if ((rc = p->release(kb))) return rc;
        if ((rc = p->alloc(&p->part, 3 * pmax)) || (rc = p->alloc(&p->F, 3 * fmax))) return rc;
        p->part_cap = pmax;
        p->f_cap = fmax;
    }
    IDP_CK(cudaDeviceSynchronize());
    return IDP_OK;
}

// Times candidate settings on the plan's own buffers and keeps the fastest:
// the slice chunking of each 3-D face pass, and (precision MIXED) the
// tensor-core matrix pass versus the df32 FFT pass for the reduced-precision
// transforms.  Results depend only on timing, not on the data.
int autotune(idp_plan p)
{
    if (p->d == 1) {   // one line per pass: nothing to choose
        p->tuned = 1;
        return IDP_OK;
    }
    cudaStream_t st = p->cap;
    cudaEvent_t e0, e1;
    IDP_CK(cudaEventCreate(&e0));
    IDP_CK(cudaEventCreate(&e1));
    int rc = IDP_OK;
    auto timed = [&](auto &&fn) -> float {
        float best = 1e30f;
        for (int r = 0; r < 4 && !rc; ++r) {
            cudaEventRecord(e0, st);
            rc = fn();
            cudaEventRecord(e1, st);
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (r > 0 && ms < best) best = ms;   // first run warms up
        }
        return best;
    };
    if (boundary_fx(p) && p->d == 3) {
        // chunk counts of the fixed-point face passes: around the set-up's choice and the
        // counts that fill whole waves of resident blocks; timed with every slice, and with the
        // sum of the parts that follows
        IDP_CK(cudaMemsetAsync(p->flags, 1, sizeof(int) * p->nflags, st));
        for (int a_ = 0; a_ < 3 && !rc; ++a_) {
            const int b = a_ == 0 ? 1 : 0, c = a_ == 2 ? 1 : 2;
            const int L = 2 * p->P[b], nc = p->P[c] + 1, n0 = p->qchunk[a_];
            int nsm = 152;
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->dev);
            const int tiles = 2 * ((nc + face_q_columns(L) - 1) / face_q_columns(L));
            std::vector<int> cands = {n0, face_q_chunks(p->ni[a_], n0 / 2), face_q_chunks(p->ni[a_], 2 * n0)};
            for (int w = 1; w <= 4; ++w)
                cands.push_back(face_q_chunks(p->ni[a_], w * face_q_blocks_per_sm(L) * nsm / tiles));
            float best_t = 1e30f;
            for (size_t i = 0; i < cands.size() && !rc; ++i) {
                if (std::find(cands.begin(), cands.begin() + i, cands[i]) != cands.begin() + i) continue;
                const int64_t need = (int64_t)cands[i] * 2 * L * nc;
                if (need > p->part_cap) {
                    double2 *np_part;
                    if ((rc = p->alloc(&np_part, 3 * need))) break;
                    p->part = np_part;
                    p->part_cap = need;
                }
                FaceQPass f{};
                FaceInvB ib{};
                if ((rc = face_q_pass(p, a_, cands[i], p->part, &f, &ib))) break;
                FftTables t;
                if ((rc = get_fft(p, L, &t))) break;
                ib.part = p->part; ib.Mb = p->M[b]; ib.Pb = p->P[b]; ib.nc = nc; ib.out = p->F; ib.t = t;
                const float ms = timed([&]() -> int {
                    cudaError_t e = launch_face_q(f, st);
                    if (e == cudaSuccess) e = launch_face_inv_b(ib, st);
                    return e == cudaSuccess ? IDP_OK : cuda_fail(e, "face pass (autotune)");
                });
                if (ms < best_t) { best_t = ms; p->qchunk[a_] = cands[i]; }
            }
        }
    }
    if (!boundary_fx(p) && p->d == 3) {
        for (int a_ = 0; a_ < 3 && !rc; ++a_) {
            const int b = a_ == 0 ? 1 : 0, c = a_ == 2 ? 1 : 2;
            const int np = p->ni[a_], L = 2 * p->P[b], nc = p->P[c] + 1;
            const int n0 = p->nchunk[a_];
            // around the set-up's choice, and the chunk counts that fill whole waves
            // of resident blocks (one column block per chunk: the block count is
            // chunks x column blocks, and a part-filled last wave leaves SMs idle)
            std::vector<int> cands = {std::max(1, n0 / 2), n0, std::min(np, 2 * n0), std::min(np, 4 * n0)};
            {
                int nsm = 152;
                cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->dev);
                const int slots = nsm * face_blocks_per_sm(L);
                const int tiles = (nc + face_columns_per_block(L) - 1) / face_columns_per_block(L);
                for (int w = 1; w <= 8; ++w) {
                    const int c = std::min(np, std::max(1, (int)(((int64_t)w * slots + tiles - 1) / tiles)));
                    if (std::find(cands.begin(), cands.end(), c) == cands.end()) cands.push_back(c);
                }
            }
            int best_n = n0, best_p = p->pchunk[a_];
            float best_t = 1e30f;
            for (size_t ci = 0; ci < cands.size() && !rc; ++ci) {
                const int pch = (np + cands[ci] - 1) / cands[ci];
                const int nch = (np + pch - 1) / pch;
                if ((int64_t)nch * 2 * L * nc > p->part_cap) {
                    double2 *np_part;
                    if ((rc = p->alloc(&np_part, 3 * (int64_t)nch * 2 * L * nc))) break;
                    p->part = np_part;
                    p->part_cap = (int64_t)nch * 2 * L * nc;
                }
                FacePass f{};
                if (a_ == 0) { f.D = p->T0; f.sp = (int64_t)p->ni[1] * (p->P[2] + 1); f.sb = p->P[2] + 1; f.sc = 1; }
                else if (a_ == 1) { f.D = p->T0; f.sp = p->P[2] + 1; f.sb = (int64_t)p->ni[1] * (p->P[2] + 1); f.sc = 1; }
                else { f.D = p->T1; f.sp = p->P[1] + 1; f.sb = (int64_t)p->ni[2] * (p->P[1] + 1); f.sc = 1; }
                f.np = np; f.Mb = p->M[b]; f.Pb = p->P[b]; f.nc = nc; f.khat = p->khat[a_]; f.part = p->part;
                f.pchunk = pch;
                FftTables t;
                if ((rc = get_fft(p, L, &t))) break;
                f.t = t;
                // the chunk count sets the work of the face pass and of the
                // partial-sum reduction that follows it: time both
                FaceInvB ib{};
                ib.part = p->part; ib.nchunk = nch; ib.Mb = p->M[b]; ib.Pb = p->P[b]; ib.nc = nc; ib.out = p->F;
                ib.t = t;
                const float ms = timed([&]() -> int {
                    cudaError_t e = launch_face_pass(f, nch, st);
                    if (e == cudaSuccess) e = launch_face_inv_b(ib, st);
                    return e == cudaSuccess ? IDP_OK : cuda_fail(e, "face pass (autotune)");
                });
                if (ms < best_t) { best_t = ms; best_n = nch; best_p = pch; }
            }
            p->nchunk[a_] = best_n;
            p->pchunk[a_] = best_p;
        }
    }
    if (!rc) {
        // block shape of the full-volume sine passes: the default, most lines per block (32),
        // half of them (16) or few (8); in the tensor-core modes, whose double-float passes
        // have shapes of their own, also 8 and 4 lines on 128 threads (-8: M = 128, 4: M = 256,
        // 512).  Shapes that do not apply to a length fall back to the default.  Timed in
        // whole solves: the transform of rho runs beside the boundary stages, so what a shape
        // costs depends on what runs next to it (a shape can win alone and lose in the
        // solve).  The density is a smooth bump over the middle of the box, zero near the boundary.
        std::vector<double> hr((size_t)p->nodes, 0.0);
        for (int i0 = 0; i0 < p->n[0]; ++i0)
            for (int i1 = 0; i1 < p->n[1]; ++i1)
                for (int i2 = 0; i2 < p->n[2]; ++i2) {
                    const int ii[3] = {i0, i1, i2};
                    double r2 = 0.0;
                    for (int s = 0; s < 3; ++s)
                        if (p->act[s]) {
                            const double t = 2.0 * ii[s] / p->M[s] - 1.0;
                            r2 += t * t;
                        }
                    const double q = 1.0 - r2 / 0.36;
                    hr[((size_t)i0 * p->n[1] + i1) * p->n[2] + i2] = q > 0.0 ? q * q * q * q : 0.0;
                }
        double *trho = nullptr, *tphi = nullptr;
        cudaError_t e = cudaMalloc(&trho, sizeof(double) * p->nodes);
        if (e == cudaSuccess) e = cudaMalloc(&tphi, sizeof(double) * p->nodes);
        if (e == cudaSuccess) e = cudaMemcpy(trho, hr.data(), sizeof(double) * p->nodes, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) rc = cuda_fail(e, "autotune buffers");
        const int opts[6] = {0, 8, 32, 16, -8, 4};
        const int nopt = tensor_mode(p) ? 6 : 4;   // (-8 and 4 are 0 and 8 to the fixed-point pass)
        int best = 0;
        float bt = 1e30f;
        for (int i = 0; i < nopt && !rc; ++i) {
            p->dst_lines = opts[i];
            const float t = timed([&]() -> int { return enqueue_grid(p, trho, tphi, 0, st); });
            if (t < bt) { bt = t; best = opts[i]; }
        }
        cudaStreamSynchronize(st);
        if (trho) cudaFree(trho);
        if (tphi) cudaFree(tphi);
        p->dst_lines = best;
    }
    if (!rc && tensor_mode(p)) {
        float tm[2];
        for (int path = 0; path < 2 && !rc; ++path) {
            p->mixed_path = path;
            tm[path] = timed([&]() -> int {
                return transform(p, dense(p, p->C), p->C, dense(p, p->C), nullptr, false, st);
            });
        }
        p->mixed_path = (tm[1] < tm[0]) ? 1 : 0;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    IDP_CK(cudaStreamSynchronize(st));
    p->tuned = 1;
    ++p->version;
    if (p->gexec) {
        cudaGraphExecDestroy(p->gexec);
        p->gexec = nullptr;
    }
    return rc;
}

bool overlap(const void *a, size_t na, const void *b, size_t nb)
{
    const char *x = (const char *)a, *y = (const char *)b;
    return x < y + nb && y < x + na;
}

int run_solve(idp_plan p, const double *rho, double *phi, cudaStream_t st)
{
    p->last = st;
    p->last_valid = 1;
    // a stall test is never baked into a graph, and NVTX ranges recorded while one is
    // captured would not recur on its replays
    if (!p->use_graph || p->stall_test || p->nvtx) {
        p->launches = 0;
        return enqueue(p, rho, phi, 0, st);
    }
    if (!p->gexec || p->g_rho != rho || p->g_phi != phi) {
        if (!p->cap) IDP_CK(cudaStreamCreateWithFlags(&p->cap, cudaStreamNonBlocking));
        IDP_CK(cudaStreamBeginCapture(p->cap, cudaStreamCaptureModeThreadLocal));
        p->launches = 0;
        int rc = enqueue(p, rho, phi, 0, p->cap);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(p->cap, &g);
        if (rc) {
            if (g) cudaGraphDestroy(g);
            return rc;
        }
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
        if (p->gexec) {
            cudaGraphExecDestroy(p->gexec);
            p->gexec = nullptr;
        }
        e = cudaGraphInstantiate(&p->gexec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
        p->g_rho = rho;
        p->g_phi = phi;
    }
    IDP_CK(cudaGraphLaunch(p->gexec, st));
    return IDP_OK;
}

// device view of page-locked (or registered, mapped) host memory: the address at
// which kernels read and write it directly; null for other memory
double *device_view(const void *ptr)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? static_cast<double *>(at.devicePointer) : nullptr;
}

// a solve from page-locked host buffers: the first row transform reads rho through
// the buffer's device view (leaving a device copy for the later stages), and the
// kernels that produce phi (the boundary values and the last sine pass) write the
// host buffer directly, so that the upload and the download run inside those
// kernels instead of before and after them.  Its own cached graph, keyed by the
// host pointers and the plan's settings.
int run_solve_host(idp_plan p, const double *rho_h, double *phi_h, double *phi_view, cudaStream_t st)
{
    p->last = st;
    p->last_valid = 1;
    if (!p->hexec || p->hg_rho != rho_h || p->hg_phi != phi_h || p->hg_version != p->version) {
        IDP_CK(cudaStreamBeginCapture(p->cap, cudaStreamCaptureModeThreadLocal));
        p->hio_rho = rho_h;
        p->hio_view = device_view(rho_h);
        int rc = enqueue(p, p->h_rho, phi_view, 0, p->cap);
        p->hio_rho = nullptr;
        p->hio_view = nullptr;
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(p->cap, &g);
        if (rc) {
            if (g) cudaGraphDestroy(g);
            return rc;
        }
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
        if (p->hexec) {
            cudaGraphExecDestroy(p->hexec);
            p->hexec = nullptr;
        }
        e = cudaGraphInstantiate(&p->hexec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
        p->hg_rho = rho_h;
        p->hg_phi = phi_h;
        p->hg_version = p->version;
    }
    IDP_CK(cudaGraphLaunch(p->hexec, st));
    return IDP_OK;
}

int create_plan(idp_plan *out, int d, const int64_t n[], const double h[], int order, int exact)
{
    if (!out || !n || !h) return IDP_EINVAL;
    *out = nullptr;
    if (d < 1 || d > 3) return IDP_EINVAL;
    if (order != 4 && order != 6) return IDP_EINVAL;
    for (int s = 0; s < d; ++s) {
        if (!(h[s] > 0.0) || !std::isfinite(h[s])) return IDP_EINVAL;
        if (n[s] < (exact ? 8 : 3)) return IDP_EINVAL;
        if (exact ? n[s] - 1 > 512 : !padded_panels(n[s] - 1)) return IDP_ESUPPORT;
    }
    idp_plan p = new (std::nothrow) idp_plan_s();
    if (!p) return IDP_ENOMEM;
    p->d = d;
    p->order = order;
    p->exact = exact;
    p->serial = g_serial.fetch_add(1);
    const int o = 3 - d;
    for (int s = 0; s < d; ++s) {
        // an unsupported panel count is padded to the next supported one, the
        // extra panels split between the two ends (h unchanged); an exact plan
        // solves on the given grid
        const int64_t Mp = exact ? n[s] - 1 : padded_panels(n[s] - 1);
        p->n[s + o] = (int)Mp + 1;
        p->un[s + o] = (int)n[s];
        p->uoff[s + o] = (int)((Mp - (n[s] - 1)) / 2);
        if (Mp != n[s] - 1) p->padded = 1;
        p->h[s + o] = h[s];
        p->act[s + o] = 1;
    }
    p->unodes = (int64_t)p->un[0] * p->un[1] * p->un[2];
    for (int s = 0; s < 3; ++s) {
        p->M[s] = p->n[s] - 1;
        p->P[s] = p->act[s] ? conv_half(p->M[s]) : p->M[s];
        p->ni[s] = p->act[s] ? p->n[s] - 2 : 1;
    }
    p->ns[2] = 1; p->ns[1] = p->n[2]; p->ns[0] = (int64_t)p->n[1] * p->n[2];
    p->is[2] = 1; p->is[1] = p->ni[2]; p->is[0] = (int64_t)p->ni[1] * p->ni[2];
    p->nodes = (int64_t)p->n[0] * p->n[1] * p->n[2];
    p->nint = (int64_t)p->ni[0] * p->ni[1] * p->ni[2];
    p->grid = Grid3{d, p->n[0], p->n[1], p->n[2], p->h[0], p->h[1], p->h[2]};
    p->coef = make_stencil_coef(p->grid);
    int rc;
    cudaError_t e = cudaGetDevice(&p->dev);
    if (e != cudaSuccess) rc = cuda_fail(e, "cudaGetDevice");
    else if (!(rc = ensure_attributes(p->dev))) rc = plan_setup(p);
    if (rc) {
        idp_destroy_plan(p);
        return rc;
    }
    *out = p;
    return IDP_OK;
}

}  // namespace

extern "C" {

int idp_create_plan(idp_plan *out, int d, const int64_t n[], const double h[], int order)
{
    return create_plan(out, d, n, h, order, 0);
}

int idp_create_plan_exact(idp_plan *out, int d, const int64_t n[], const double h[], int order)
{
    return create_plan(out, d, n, h, order, 1);
}

int idp_plan_set(idp_plan p, int key, int64_t value)
{
    if (!p) return IDP_EINVAL;
    if (key == IDP_KEY_USE_GRAPH) {
        p->use_graph = value ? 1 : 0;
        return IDP_OK;
    }
    if (key == IDP_KEY_NVTX) {
        p->nvtx = value ? 1 : 0;
        return IDP_OK;
    }
    if (key == IDP_KEY_AUTOTUNE) {
        if (!value) return IDP_OK;
        return autotune(p);
    }
    if (key == IDP_KEY_DST_SHAPE) {
        if (value != 0 && value != 8 && value != -8 && value != 32 && value != 16 && value != 4) return IDP_EINVAL;
        p->dst_lines = (int)value;
        ++p->version;
        if (p->gexec) {
            cudaGraphExecDestroy(p->gexec);
            p->gexec = nullptr;
        }
        return IDP_OK;
    }
    if (key == IDP_KEY_VALIDATE) {
        if (value < 0 || value > 1 << 20) return IDP_EINVAL;
        if (value && !p->d_val) {
            int rc;
            if ((rc = p->alloc(&p->d_val, 1))) return rc;
            IDP_CK(cudaMemset(p->d_val, 0, sizeof(int)));
        }
        p->validate = (int)value;
        ++p->version;
        if (p->gexec) {
            cudaGraphExecDestroy(p->gexec);
            p->gexec = nullptr;
        }
        return IDP_OK;
    }
    if (key == IDP_KEY_MIXED_BOUNDARY_DF32) {
        if (value != 0 && value != 1) return IDP_EINVAL;
        if (value && p->d == 3 && !p->khatd[0]) {
            int rc;
            ddr *d[3];
            for (int a_ = 0; a_ < 3; ++a_) {
                const int like = spectra_like(p, a_);
                if (like < a_) {
                    d[a_] = d[like];
                    continue;
                }
                if ((rc = p->alloc(&d[a_], p->khat_n[a_]))) return rc;
                IDP_CK(launch_to_dd(p->khat[a_], d[a_], p->khat_n[a_], 0));
            }
            IDP_CK(cudaDeviceSynchronize());
            for (int a_ = 0; a_ < 3; ++a_) p->khatd[a_] = d[a_];
        }
        if (p->mixed_bdd != (int)value) {
            p->mixed_bdd = (int)value;
            ++p->version;
            if (p->gexec) {
                cudaGraphExecDestroy(p->gexec);
                p->gexec = nullptr;
            }
        }
        return IDP_OK;
    }
    if (key == IDP_KEY_GUARD_TEST) {
        // test hook: overwrite (1) or restore (0) the first byte of the guard
        // region in front of the plan's first buffer; the write stays inside
        // that allocation
        if (value != 0 && value != 1) return IDP_EINVAL;
        if (p->guarded.empty()) return IDP_ESUPPORT;
        IDP_CK(cudaDeviceSynchronize());
        IDP_CK(cudaMemset(p->guarded.front().first, value ? 0x5A : idp_plan_s::GUARD_BYTE, 1));
        IDP_CK(cudaDeviceSynchronize());
        return IDP_OK;
    }
    if (key == IDP_KEY_STALL_TEST) {
        if (!tensor_mode(p)) return IDP_EINVAL;
        p->stall_test = value ? 1 : 0;
        ++p->version;
        if (p->gexec) {
            cudaGraphExecDestroy(p->gexec);
            p->gexec = nullptr;
        }
        return IDP_OK;
    }
    if (key == IDP_KEY_PRECISION) {
        if (value != IDP_PRECISION_FP64 && value != IDP_PRECISION_MIXED_BF16X3 && value != IDP_PRECISION_DF32 &&
            value != IDP_PRECISION_MIXED_TF32X3)
            return IDP_EINVAL;
        if (p->d == 1 && value != IDP_PRECISION_FP64) return IDP_ESUPPORT;
        if (value == IDP_PRECISION_MIXED_BF16X3 || value == IDP_PRECISION_MIXED_TF32X3) {
            int rc;
            if (!p->d_err) {
                if ((rc = p->alloc(&p->d_err, 1))) return rc;
                IDP_CK(cudaMemset(p->d_err, 0, sizeof(int)));
            }
            for (int s = 0; s < 2; ++s)
                for (int q = 0; q < 2; ++q)
                    if (!p->t32[s][q] && (rc = p->alloc(&p->t32[s][q], t32_count(p)))) return rc;
            for (int s = 0; s < 3; ++s) {
                const void *img;
                if (p->act[s] &&
                    (rc = get_mp_image(p, p->M[s], value == IDP_PRECISION_MIXED_TF32X3 ? 1 : 0, &img)))
                    return rc;
            }
        }
        if (p->mixed != (int)value) {
            p->mixed = (int)value;
            p->mixed_path = 0;
            ++p->version;
            if (p->gexec) {
                cudaGraphExecDestroy(p->gexec);
                p->gexec = nullptr;
            }
        }
        return IDP_OK;
    }
    return IDP_EINVAL;
}

int idp_solve(idp_plan p, const double *rho, double *phi, void *stream)
{
    if (!p || !rho || !phi) return IDP_EINVAL;
    const size_t b = sizeof(double) * p->unodes;
    if (overlap(rho, b, phi, b)) return IDP_EALIAS;
    return run_solve(p, rho, phi, (cudaStream_t)stream);
}

int idp_solve_host(idp_plan p, const double *rho_host, double *phi_host, void *stream)
{
    if (!p || !rho_host || !phi_host) return IDP_EINVAL;
    const size_t b = sizeof(double) * p->unodes;
    if (overlap(rho_host, b, phi_host, b)) return IDP_EALIAS;
    int rc;
    if (!p->h_rho && ((rc = p->alloc(&p->h_rho, p->unodes)) || (rc = p->alloc(&p->h_phi, p->unodes)))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    double *phi_view = nullptr;
    if (p->use_graph && !p->stall_test && !p->nvtx && device_view(rho_host) && (phi_view = device_view(phi_host))) {
        // page-locked buffers: phi is written in place by the kernels
        if ((rc = run_solve_host(p, rho_host, phi_host, phi_view, st))) return rc;
    } else {
        IDP_CK(cudaMemcpyAsync(p->h_rho, rho_host, b, cudaMemcpyHostToDevice, st));
        if ((rc = run_solve(p, p->h_rho, p->h_phi, st))) return rc;
        IDP_CK(cudaMemcpyAsync(phi_host, p->h_phi, b, cudaMemcpyDeviceToHost, st));
    }
    IDP_CK(cudaStreamSynchronize(st));
    return IDP_OK;
}

int idp_solve_batched(int count, const idp_plan plans[], const double *const rho[], double *const phi[],
                      void *stream)
{
    if (count < 0 || (count > 0 && (!plans || !rho || !phi))) return IDP_EINVAL;
    for (int i = 0; i < count; ++i) {
        if (!plans[i] || !rho[i] || !phi[i]) return IDP_EINVAL;
        for (int j = 0; j < i; ++j)
            if (plans[j] == plans[i]) return IDP_EINVAL;
    }
    // the problems run concurrently (branches of one graph): an output may
    // overlap no input and no other output, of its own problem or another
    for (int i = 0; i < count; ++i) {
        const size_t bi = sizeof(double) * plans[i]->unodes;
        for (int j = 0; j < count; ++j) {
            const size_t bj = sizeof(double) * plans[j]->unodes;
            if (overlap(phi[i], bi, rho[j], bj)) return IDP_EALIAS;
            if (j != i && overlap(phi[i], bi, phi[j], bj)) return IDP_EALIAS;
        }
    }
    if (count == 0) return IDP_OK;
    cudaStream_t st = (cudaStream_t)stream;
    idp_plan p0 = plans[0];
    bool graphs = true;
    for (int i = 0; i < count; ++i)
        graphs = graphs && plans[i]->use_graph && !plans[i]->nvtx && plans[i]->dev == p0->dev;
    if (!graphs) {
        for (int i = 0; i < count; ++i) {
            int rc = run_solve(plans[i], rho[i], phi[i], st);
            if (rc) return rc;
        }
        return IDP_OK;
    }
    // one CUDA graph: a branch per problem (each with its own two streams), all
    // forked from and joined into the launch stream, so that independent
    // problems of different sizes run concurrently
    BatchCache *bc = p0->batch;
    bool hit = bc && (int)bc->serials.size() == count;
    for (int i = 0; hit && i < count; ++i)
        hit = bc->serials[i] == (plans[i]->serial << 16 ^ plans[i]->version) && bc->rho[i] == rho[i] &&
              bc->phi[i] == phi[i];
    if (!hit) {
        if (!bc) bc = p0->batch = new BatchCache();
        if (bc->exec) {
            cudaGraphExecDestroy(bc->exec);
            bc->exec = nullptr;
        }
        if (!bc->fork) IDP_CK(cudaEventCreateWithFlags(&bc->fork, cudaEventDisableTiming));
        while ((int)bc->joins.size() < count) {
            cudaEvent_t e;
            IDP_CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
            bc->joins.push_back(e);
        }
        cudaStream_t origin = p0->cap;
        IDP_CK(cudaStreamBeginCapture(origin, cudaStreamCaptureModeThreadLocal));
        int rc = IDP_OK;
        cudaError_t e = cudaEventRecord(bc->fork, origin);
        for (int i = 0; i < count && !rc && e == cudaSuccess; ++i) {
            idp_plan q = plans[i];
            e = cudaStreamWaitEvent(q->bst, bc->fork, 0);
            if (e != cudaSuccess) break;
            q->launches = 0;
            rc = enqueue(q, rho[i], phi[i], 0, q->bst);
            if (!rc) e = cudaEventRecord(bc->joins[i], q->bst);
            if (!rc && e == cudaSuccess) e = cudaStreamWaitEvent(origin, bc->joins[i], 0);
        }
        cudaGraph_t g = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(origin, &g);
        if (rc || e != cudaSuccess || e2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            if (rc) return rc;
            return cuda_fail(e != cudaSuccess ? e : e2, "batched capture");
        }
        e = cudaGraphInstantiate(&bc->exec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
        bc->serials.assign(count, 0);
        bc->rho.assign(rho, rho + count);
        bc->phi.assign(phi, phi + count);
        for (int i = 0; i < count; ++i) bc->serials[i] = plans[i]->serial << 16 ^ plans[i]->version;
    }
    for (int i = 0; i < count; ++i) {
        plans[i]->last = st;
        plans[i]->last_valid = 1;
    }
    IDP_CK(cudaGraphLaunch(bc->exec, st));
    return IDP_OK;
}

int idp_solve_stage(idp_plan p, int stage, const double *rho, double *out, void *stream)
{
    if (!p || !rho || !out) return IDP_EINVAL;
    if (stage < IDP_STAGE_BOUNDARY || stage > IDP_STAGE_PHI) return IDP_EINVAL;
    if (stage == IDP_STAGE_R && p->order != 6) return IDP_EINVAL;
    const size_t b = sizeof(double) * p->unodes;
    if (overlap(rho, b, out, b)) return IDP_EALIAS;
    p->last = (cudaStream_t)stream;
    p->last_valid = 1;
    return enqueue(p, rho, out, stage == IDP_STAGE_PHI ? 0 : stage, (cudaStream_t)stream);
}

int idp_plan_status(idp_plan p)
{
    if (!p) return IDP_EINVAL;
    if (p->last_valid) IDP_CK(cudaStreamSynchronize(p->last));
    IDP_CK(cudaGetLastError());
    if (p->d_val) {
        int v = 0;
        IDP_CK(cudaMemcpy(&v, p->d_val, sizeof(int), cudaMemcpyDeviceToHost));
        if (v) {
            IDP_CK(cudaMemset(p->d_val, 0, sizeof(int)));   // reported once
            return (v & 1) ? IDP_EINVAL : IDP_ESUPPORT;
        }
    }
    if (p->d_err) {
        int e = 0;
        IDP_CK(cudaMemcpy(&e, p->d_err, sizeof(int), cudaMemcpyDeviceToHost));
        if (e) {
            IDP_CK(cudaMemset(p->d_err, 0, sizeof(int)));   // reported once
            return IDP_ETIMEOUT;
        }
    }
    return IDP_OK;
}

int idp_profile_solve(idp_plan p, const double *rho, double *phi, void *stream, int capacity, int *kinds,
                      float *ms)
{
    if (!p || !rho || !phi || capacity < 0 || (capacity > 0 && (!kinds || !ms))) return IDP_EINVAL;
    const size_t b = sizeof(double) * p->unodes;
    if (overlap(rho, b, phi, b)) return IDP_EALIAS;
    cudaStream_t st = (cudaStream_t)stream;
    while ((int)p->ev.size() < 2 * capacity) {
        cudaEvent_t e;
        IDP_CK(cudaEventCreate(&e));
        p->ev.push_back(e);
    }
    p->profiling = 1;
    p->ev_used = 0;
    p->ev_kind.clear();
    p->launches = 0;
    p->last = st;
    p->last_valid = 1;
    const int rc = enqueue(p, rho, phi, 0, st);
    p->profiling = 0;
    if (rc) return rc;
    IDP_CK(cudaStreamSynchronize(st));
    const int n = (int)p->ev_kind.size();
    for (int i = 0; i < n; ++i) {
        kinds[i] = p->ev_kind[i];
        IDP_CK(cudaEventElapsedTime(&ms[i], p->ev[2 * i], p->ev[2 * i + 1]));
    }
    return n;
}

int idp_plan_check_guards(idp_plan p)
{
    if (!p) return IDP_EINVAL;
    IDP_CK(cudaDeviceSynchronize());
    bool intact = !p->released_dirty;
    int rc;
    for (const auto &g : p->guarded)
        if ((rc = idp_plan_s::guards_intact(g, &intact))) return rc;
    return intact ? IDP_OK : IDP_EGUARD;
}

int idp_plan_grid(idp_plan p, int64_t n_solved[], int64_t offset[])
{
    if (!p || !n_solved || !offset) return IDP_EINVAL;
    const int o = 3 - p->d;
    for (int s = 0; s < p->d; ++s) {
        n_solved[s] = p->n[s + o];
        offset[s] = p->uoff[s + o];
    }
    return IDP_OK;
}

int idp_plan_info(idp_plan p, int64_t *nodes, int64_t *interior, int64_t *workspace_bytes)
{
    if (!p) return IDP_EINVAL;
    if (nodes) *nodes = p->unodes;
    if (interior) *interior = p->nint;
    if (workspace_bytes) *workspace_bytes = p->bytes;
    return IDP_OK;
}

int idp_destroy_plan(idp_plan p)
{
    if (!p) return IDP_EINVAL;
    cudaDeviceSynchronize();
    if (p->gexec) cudaGraphExecDestroy(p->gexec);
    if (p->hexec) cudaGraphExecDestroy(p->hexec);
    if (p->cap) cudaStreamDestroy(p->cap);
    if (p->side) cudaStreamDestroy(p->side);
    if (p->bst) cudaStreamDestroy(p->bst);
    if (p->batch) {
        if (p->batch->exec) cudaGraphExecDestroy(p->batch->exec);
        for (cudaEvent_t e : p->batch->joins) cudaEventDestroy(e);
        if (p->batch->fork) cudaEventDestroy(p->batch->fork);
        delete p->batch;
    }
    if (p->fork) cudaEventDestroy(p->fork);
    if (p->join) cudaEventDestroy(p->join);
    for (int i = 0; i < 2; ++i)
        if (p->fst[i]) cudaStreamDestroy(p->fst[i]);
    for (int i = 0; i < 3; ++i)
        if (p->fev[i]) cudaEventDestroy(p->fev[i]);
    for (cudaEvent_t e : p->ev) cudaEventDestroy(e);
    for (void *q : p->allocs) cudaFree(q);
    delete p;
    return IDP_OK;
}

const char *idp_strerror(int code)
{
    switch (code) {
    case IDP_OK: return "ok";
    case IDP_EINVAL: return "invalid argument";
    case IDP_ENOMEM: return "out of memory";
    case IDP_ECUDA: return "CUDA error";
    case IDP_EALIAS: return "input and output overlap";
    case IDP_ESUPPORT: return "size or option not supported (panel counts must be 2^a in [16, 512] or 3*2^a in [48, 384])";
    case IDP_ETIMEOUT: return "a device-side wait exceeded its iteration limit";
    case IDP_EGUARD: return "a guard region around a workspace buffer was overwritten";
    case IDP_ESCRATCH: return "problem larger than the fixed scratch of idp_rhs6_noalloc (524288 nodes)";
    default: return "unknown error";
    }
}

const char *idp_last_cuda_error(void) { return g_cuda_err; }

int idp_plan_tuning(idp_plan p, int64_t out[9])
{
    if (!p || !out) return IDP_EINVAL;
    out[0] = p->tuned;
    out[1] = p->mixed_path;
    for (int a = 0; a < 3; ++a) {
        const bool fx = boundary_fx(p) && p->d == 3;
        out[2 + a] = fx ? p->qchunk[a] : p->nchunk[a];
        out[5 + a] = fx ? (p->ni[a] + p->qchunk[a] - 1) / p->qchunk[a] : p->pchunk[a];
    }
    out[8] = p->dst_lines;
    return IDP_OK;
}

int idp_plan_launches(idp_plan p, int64_t *launches)
{
    if (!p || !launches) return IDP_EINVAL;
    *launches = p->launches;
    return IDP_OK;
}

}  // extern "C"
