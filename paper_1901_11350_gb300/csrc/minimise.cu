// minimise.cu -- velocity projection (Appendix D) and GNEB (Sec. GNEB,
// Appendix F) on the GPU.
//
// Work is cut into blocks of kBlock spins of one image ("image" = one system
// of one chain; a plain minimisation is one image).  Per-image scalars
// (energy, geodesic distance, tangent norm, projections, max force) are
// reduced deterministically: every block writes its partial, and the last
// block of the image to finish (atomic ticket) sums the image's partials in
// a fixed order and re-arms the ticket.  Kernels of one iteration:
//   move    v = c F, c = v.F / F.F or 0 from the previous force pass,
//           x <- normalise(x + dt v + dt^2/(2m) F)          (interior images)
//   field   B(x), E_v, Pg = -(B - (B.x)x), theta^2 to image v+1, and the
//           products of the differences d+ and d- to the neighbouring images
//           with each other and with Pg
//   coefs   per chain, from its images' sums: tangent weights, |tau|^2,
//           Pg.tau, the climbing image, force coefficients a
//   force   tau = P(w+ d+ + w- d-), F' = -Pg + a tau, v.F', F'.F', max |F'| with v = c F + dt/(2m)(F + F')
// What bounds them: memory.  The projected velocity is a multiple of F, so no
// pass stores it (the call's last one does), and tau is formed again in the
// force pass rather than stored: 144 B per spin and iteration.  |tau|^2 and
// Pg.tau follow from the field pass's products (tau is linear in the weights).
// 3.6 M spins in 12 chains: 335 -> 240 us an iteration (with tau and v stored,
// 288 B, and a neighbour loop with indices).  The field pass is 55% of it and
// bound by the instructions it issues (865 a spin, 65% of the issue slots).
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "minimise.h"

namespace spgb {

namespace {

struct ImgInfo {
    long long spin0;  // record offset of image 0 of the chain
    int N, chain, nu, M, g0, blk0, bpi;
    int kind;  // SP_IMAGE_* or -1: climbing decided by the climbing flag
    int spt;   // spins per thread (GNEB passes; 1 elsewhere)
    int unused;
};
// layouts are compared byte by byte: a padding byte, which holds whatever the stack
// did, would make an equal one look changed, and its upload cannot be captured
static_assert(sizeof(ImgInfo) == sizeof(long long) + 10 * sizeof(int), "no padding");
struct alignas(16) BlkInfo {
    int g, t, chain, ne;  // image, block of the image, the image's chain, its stencil's entries
};

// per-image scalar slots (kS doubles per image): energy, squared geodesic
// distance to the next image, products d+.d+, d+.d-, d-.d-, Pg.d+, Pg.d- of
// the projected differences to the next and the previous image, v.F, F.F,
// max_i |F_i|^2, energy-weighted segment length, tangent weights of the
// forward and backward differences, |tau|^2, Pg.tau, force coefficient a
// (F = -Pg + a tau), velocity projection coefficient v.F / F.F, max |F|
// (minimiser)
enum { kE = 0, kL2, kPP, kPM, kMM, kGP, kGM, kVF, kFF, kFMAX, kLW, kWP, kWM, kTT, kGT, kA, kC, kFN, kS = 18 };

struct Buf {
    void *p = nullptr;
    size_t bytes = 0;
};

int grow(Buf &b, size_t bytes)
{
    if (b.p && b.bytes >= bytes) return 0;
    if (b.p) cudaFree(b.p);
    b.p = nullptr;
    b.bytes = 0;
    if (cudaMalloc(&b.p, bytes) != cudaSuccess) return SP_ERR_CUDA;
    b.bytes = bytes;
    return 0;
}

}  // namespace

struct MinScratch {
    Buf F, G, scal, part, cnt, blk, img, sten, state, aux, sync;
    int *host_state = nullptr;  // pinned: iters, active
    double *host_fmax = nullptr;
    // batch layout last uploaded (block/image tables and stencils)
    std::vector<char> layout;
    int n_img = 0, n_blk = 0, n_chains = 0;
    // CUDA graph of kGraphIters steady-state GNEB iterations
    cudaStream_t gstream = nullptr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    cudaGraphExec_t gexec = nullptr;
    std::vector<char> gkey;
};

constexpr int kGraphIters = 8;
constexpr int kPartRow = 8;  // doubles of a block's partials, at most
// blocks per SM the register allocation is held to (FP32): GNEB field pass 4
// (240 us an iteration; 3: 246, 2: 274)
#ifndef SPGB_VP_MINB
#define SPGB_VP_MINB 6
#endif
#ifndef SPGB_GF_MINB
#define SPGB_GF_MINB 4
#endif

void min_scratch_destroy(MinScratch *s)
{
    if (!s) return;
    Buf *bufs[] = {&s->F, &s->G, &s->scal, &s->part, &s->cnt, &s->blk, &s->img, &s->sten, &s->state, &s->aux,
                   &s->sync};
    for (Buf *b : bufs)
        if (b->p) cudaFree(b->p);
    if (s->host_state) cudaFreeHost(s->host_state);
    if (s->host_fmax) cudaFreeHost(s->host_fmax);
    if (s->gexec) cudaGraphExecDestroy(s->gexec);
    if (s->gstream) cudaStreamDestroy(s->gstream);
    if (s->ev0) cudaEventDestroy(s->ev0);
    if (s->ev1) cudaEventDestroy(s->ev1);
    delete s;
}

namespace {

int scratch(MinScratch **s)
{
    if (!*s) {
        *s = new (std::nothrow) MinScratch();
        if (!*s) return SP_ERR_STATE;
        if (cudaMallocHost(&(*s)->host_state, 4 * sizeof(int)) != cudaSuccess) return SP_ERR_CUDA;
        if (cudaMallocHost(&(*s)->host_fmax, sizeof(double)) != cudaSuccess) return SP_ERR_CUDA;
    }
    return 0;
}

// Counters must start at zero; the reduction leaves them at zero.
int grow_counters(Buf &b, size_t n, cudaStream_t st)
{
    size_t bytes = n * sizeof(unsigned);
    if (b.p && b.bytes >= bytes) return 0;
    if (grow(b, bytes)) return SP_ERR_CUDA;
    return cudaMemsetAsync(b.p, 0, b.bytes, st) == cudaSuccess ? 0 : SP_ERR_CUDA;
}

// Per-image dot-product accumulators: float-float for FP32 (the FP64 sum of
// the same exact products to ~1e-14), plain FP64 for FP64.
template <typename T> struct Acc {
    using type = double;
};
template <> struct Acc<float> {
    using type = f2sum;
};
// exact_dot with products that no addition is fused with
__device__ __forceinline__ f2sum acc_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ f2sum acc_dot(v3<float> a, v3<float> b)
{
    return acc_prod(a.x, b.x) + acc_prod(a.y, b.y) + acc_prod(a.z, b.z);
}
// r += a.b for a sum of a few spins: the products and the errors of the
// additions to r.hi go to r.lo one after another
__device__ __forceinline__ void acc_add(f2sum &r, float a, float b)
{
    const float p = __fmul_rn(a, b);
    const f2sum s = two_sum(r.hi, p);
    r.hi = s.hi;
    r.lo += s.lo + fmaf(a, b, -p);
}
__device__ __forceinline__ void acc_add(f2sum &r, v3<float> a, v3<float> b)
{
    acc_add(r, a.x, b.x);
    acc_add(r, a.y, b.y);
    acc_add(r, a.z, b.z);
}
__device__ __forceinline__ void acc_add(double &r, double a, double b) { r = fma(a, b, r); }
__device__ __forceinline__ double acc_dot(v3<double> a, v3<double> b) { return xdot(a, b); }
__device__ __forceinline__ void acc_add(double &r, v3<double> a, v3<double> b) { r += xdot(a, b); }

__device__ __forceinline__ float xor_of(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double xor_of(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ f2sum xor_of(f2sum v, int o)
{
    return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// Sums over a warp of NS values per lane (a power of two); the 32 / NS lanes
// l with l NS / 32 = k receive the sum of value k.  Each step halves the
// values a lane carries: NS - 1 additions and one more per step that is left,
// not five per value.
template <int NS, typename V> __device__ __forceinline__ V warp_sums(V (&v)[NS])
{
    const int l = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = NS / 2; n > 0; n >>= 1, o >>= 1) {
        const bool up = (l & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const V send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = keep + xor_of(send, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) v[0] = v[0] + xor_of(v[0], o);
    return v[0];
}

// The type a block's sums are combined in: float-float for float.
template <typename V> struct Wide {
    using type = V;
};
template <> struct Wide<float> {
    using type = f2sum;
};
__device__ __forceinline__ f2sum widen(float v) { return {v, 0.f}; }
__device__ __forceinline__ f2sum widen(f2sum v) { return v; }
__device__ __forceinline__ double widen(double v) { return v; }

// Deterministic per-image reduction of NS sums (2 or 8) and, with MAX, one
// maximum (of non-negative values).  Every thread of every block of the image
// must call it.  The block's sums run in the values' own type V (float, double
// or f2sum), the image's in FP64.  After one
// barrier warps 1.. leave; warp 0 combines the warp results by a fixed shuffle
// tree into the block's partials and takes a ticket; warp 0 of the image's
// last block sums the partials in a fixed order, writes the totals to
// out[0..NS) (and out[NS]) and calls post(lane).
template <int NS, bool MAX, typename V, typename Post>
__device__ __forceinline__ void image_sums(V (&v)[NS], V m, double *__restrict__ part, int blk, int blk0, int bpi,
                                           unsigned *counter, double *out, Post post)
{
    constexpr int NW = kBlock / 32, LPV = 32 / NS, ROW = MAX ? 4 : 8, NV = NS + (MAX ? 1 : 0);
    static_assert(NV <= ROW && ROW <= kPartRow, "a row holds the values");
    // (the block's own sums in V, float-float for float: a conversion to FP64 per
    // warp and value was a fifth of the time of a minimiser's force pass)
    using W = typename Wide<V>::type;
    __shared__ V sh[NW][NV];
    const V s = warp_sums(v);
    if (MAX)
        for (int o = 16; o > 0; o >>= 1) m = nan_max(m, shfl_down(m, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l % LPV == 0) sh[w][l / LPV] = s;
    if (MAX && l == 0) sh[w][NS] = m;
    __syncthreads();
    if (w != 0) return;
    W t{};
    for (int k = l % LPV; k < NW; k += LPV) t = t + widen(sh[k][l / LPV]);
    for (int o = LPV / 2; o > 0; o >>= 1) t = t + xor_of(t, o);
    const double a = to_double(t);
    double mx = 0.0;
    if (MAX) {
        V mv = l < NW ? sh[l][NS] : V{};
        for (int o = NW / 2; o > 0; o >>= 1) mv = nan_max(mv, shfl_down(mv, o));
        mx = to_double(mv);
    }
    if (l % LPV == 0) part[(size_t)blk * ROW + l / LPV] = a;
    if (MAX && l == 0) part[(size_t)blk * ROW + NS] = mx;
    // the fences are lane 0's, between the warp's barriers and the ticket: it is
    // lane 0 that publishes the other lanes' partials and sees the other blocks'
    __syncwarp();
    int last = 0;
    if (l == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == (unsigned)(bpi - 1);
        __threadfence();
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __syncwarp();
    // lane l adds the rows l, l + 32, ..., four rows' loads in flight; the
    // maximum as an integer (the bits of non-negative numbers are in their order,
    // NaN above all), which the FP64 pipe has no part in: an image of a million
    // spins has thousands of rows (1024 x 1024, an iteration of the minimiser: 55 us
    // in FP32 and 267 in FP64; with eight rows at a time and their maxima in FP64
    // 131 and 345)
    double acc[NS] = {};
    unsigned long long top = 0;
    const double2 *row = reinterpret_cast<const double2 *>(part + (size_t)blk0 * ROW);
#pragma unroll 4
    for (int p = l; p < bpi; p += 32) {
        double2 r[ROW / 2];
#pragma unroll
        for (int k = 0; k < (NV + 1) / 2; ++k) r[k] = __ldcg(row + (size_t)p * (ROW / 2) + k);
#pragma unroll
        for (int k = 0; k < NS / 2; ++k) {
            acc[2 * k] += r[k].x;
            acc[2 * k + 1] += r[k].y;
        }
        if (MAX) top = max(top, (unsigned long long)__double_as_longlong(r[NS / 2].x));
    }
    const double total = warp_sums(acc);
    if (MAX)
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (l % LPV == 0) out[l / LPV] = total;
    if (MAX && l == 0) out[NS] = __longlong_as_double((long long)top);
    __threadfence();
    __syncwarp();
    if (l == 0) atomicExch(counter, 0u);
    post(l);
}

// After a force pass (out = scal + kS g + kVF): the projection coefficient
// v.F / F.F (0 unless both are positive) of the next move, and max |F|.
struct ForcePost {
    double *out;
    __device__ void operator()(int l) const
    {
        if (l != 0) return;
        const double vf = out[0], ff = out[kFF - kVF];
        out[kC - kVF] = (vf > 0 && ff > 0) ? vf / ff : 0.0;
        out[kFN - kVF] = sqrt(out[kFMAX - kVF]);
    }
};

// ============================================================ VP minimiser
// state (ints): [0] iterations performed, [1] active flag
// scal (doubles): the image slots kVF.. and, at kVP, whether the last force
// pass had a velocity.
// (max |F|^2 rather than max |F|: one square root per image instead of one
// per spin; sqrt is monotonic and correctly rounded, so sqrt(max |F|^2) is
// exactly max |F| in FP64)
// Between two force passes the velocity is a multiple c F of the force, so
// neither pass stores it; the last move of a call does.
constexpr int kVP = 0;  // slot kE, which the minimiser does not use

// Force pass of spin p = i of a system; mode 0: F only; 1: v from memory (the
// call's first iteration); 2: v = c F, c the projection coefficient of the
// previous force pass (read before this block's ticket, so before the
// system's last block replaces it).
template <typename T>
__device__ __forceinline__ void vp_force(const Stencil<T> &S, const rec_t<T> *x, const rec_t<T> *v, rec_t<T> *F, int i,
                                         T dth_m, int mode, T c, T (&r)[2], T &mx)
{
    int b;
    const v3<T> ni = ld(x, i);
    const v3<T> B = local_field(S, x, i, ni, b);
    const v3<T> Fn = tangent(B, ni);
    if (mode) {
        const v3<T> Fo = ldc((const rec_t<T> *)F, i);
        const v3<T> vi = axpy(dth_m, Fo + Fn, mode == 1 ? ldc(v, i) : c * Fo);
        r[0] = xdot(vi, Fn);
    }
    st(F, i, Fn);
    r[1] = xdot(Fn, Fn);
    mx = r[1];
}

// Move of spin i (done: none); last: the projected velocity is stored.
template <typename T>
__device__ __forceinline__ void vp_move(rec_t<T> *x, rec_t<T> *v, const rec_t<T> *F, int i, T dt, T dt2_2m, bool proj,
                                        T c, bool done, bool last)
{
    if (done && !last) return;
    const v3<T> Fi = ldc(F, i), vi = proj ? c * Fi : ldc((const rec_t<T> *)v, i);
    if (last && proj) st(v, i, vi);
    if (!done) st(x, i, xunit(axpy(dt2_2m, Fi, axpy(dt, vi, ldc((const rec_t<T> *)x, i)))));
}

template <typename T>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? SPGB_VP_MINB : 1)
    k_vp_force(const __grid_constant__ Stencil<T> S, const rec_t<T> *__restrict__ x, const rec_t<T> *__restrict__ v,
               rec_t<T> *__restrict__ F, T dth_m, int mode, double *part, unsigned *cnt, double *scal, const int *state)
{
    allow_dependents();
    wait_prerequisite(x, v, F, scal, state);  // state, scalars and records come from the kernels before
    if (mode && state[1] == 0) return;
    const int i = blockIdx.x * kBlock + threadIdx.x;
    const T c = mode == 2 ? (T)scal[kC] : T(0);
    T r[2] = {0, 0}, mx = 0;
    if (i < S.N) vp_force(S, x, v, F, i, dth_m, mode, c, r, mx);
    image_sums<2, true>(r, mx, part, blockIdx.x, 0, gridDim.x, cnt, scal + kVF, ForcePost{scal + kVF});
    if (blockIdx.x == 0 && threadIdx.x == 0) scal[kVP] = mode;
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_vp_move(int N, rec_t<T> *__restrict__ x, rec_t<T> *__restrict__ v,
                                                    const rec_t<T> *__restrict__ F, T dt, T dt2_2m, double tol,
                                                    int k, int max_iter, const double *scal, int *state)
{
    allow_dependents();
    wait_prerequisite(x, v, F, scal, state);  // state, scalars and records come from the kernels before
    const bool done = scal[kFN] < tol || k >= max_iter;
    const int i = blockIdx.x * kBlock + threadIdx.x;
    if (i < N) vp_move(x, v, F, i, dt, dt2_2m, scal[kVP] != 0.0, (T)scal[kC], done, k >= max_iter);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state[1] = done ? 0 : 1;
        if (!done) state[0] = k + 1;
    }
}

// ============================================================ GNEB
// The GNEB passes are written as bodies for one work block `vb` (an entry of
// the block table), so that the per-pass kernels (vb = blockIdx.x) and the
// persistent kernel (a CTA takes several vb in turn) run the same code.
// R: the record type the mutable buffers are read through -- rec_t<T> (the
// per-pass kernels: spins by the read-only path) or the plain-load record
// type of ShRec<T> (the persistent kernel, which reads what other blocks
// wrote earlier in the same launch).

// Spins per thread of a chain's passes: the reductions at the end of a block
// cost as much as two spins, so long chains share them among four; a chain
// with fewer blocks than two per SM of 256 spins each is spread out instead.
// It depends on the chain alone: a chain gets the same sums in any batch.
inline int gneb_spt(long long spins)
{
    const long long two_per_sm = 2LL * 152 * kBlock;
    return spins >= 4 * two_per_sm ? 4 : (spins >= 2 * two_per_sm ? 2 : 1);
}

// Every product and sum of the per-image scalars is written with the
// non-contracting intrinsics: the same bits in every kernel they are inlined
// into.
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }

// Weights (w+, w-) of the forward and backward differences in the improved
// tangent (Henkelman and Jonsson 2000) of an interior image of energy E0, from
// its neighbours' energies.
__device__ __forceinline__ void tangent_weights(double Em, double E0, double Ep, double *wp_out, double *wm_out)
{
    double wp, wm;
    if (Ep > E0 && E0 > Em) {
        wp = 1;
        wm = 0;
    } else if (Ep < E0 && E0 < Em) {
        wp = 0;
        wm = 1;
    } else {
        double dmax = fmax(fabs(Ep - E0), fabs(Em - E0)), dmin = fmin(fabs(Ep - E0), fabs(Em - E0));
        if (Ep > Em) {
            wp = dmax;
            wm = dmin;
        } else {
            wp = dmin;
            wm = dmax;
        }
    }
    *wp_out = wp;
    *wm_out = wm;
}

// Energy-weighted length of the segment from image a to a+1 (reading of the
// paper's spring modulation: arc length of the curve ((1-w) r, w E(r)) over
// the geodesic distance h, E(r) the cubic Hermite interpolant of the two
// images' energies and slopes), by adaptive Simpson with Lyness' criterion
// and Richardson correction to 1e-13 h, subdivision depth at most 40 (an
// explicit stack of at most 41 intervals).
__device__ double seg_integrand(double Ea, double Eb, double da, double db, double h, double w, double s)
{
    double t = s / h, t2 = dmul(t, t);
    double c6 = dadd(dmul(6.0, t2), -dmul(6.0, t));  // 6 t^2 - 6 t
    double ce = dadd(dmul(c6, Ea), dmul(-c6, Eb)) / h;
    double ca = dadd(dadd(dmul(3.0, t2), -dmul(4.0, t)), 1.0);  // 3 t^2 - 4 t + 1
    double cb = dadd(dmul(3.0, t2), -dmul(2.0, t));            // 3 t^2 - 2 t
    double dE = dadd(dadd(ce, dmul(ca, da)), dmul(cb, db));
    double u = 1.0 - w;
    return sqrt(dadd(dmul(u, u), dmul(dmul(w, w), dmul(dE, dE))));
}

__device__ double seg_length(double Ea, double Eb, double da, double db, double h, double w)
{
    if (w == 0.0) return h;
    if (!(h > 0)) return 0.0;
    struct Iv {
        double a, b, fa, fm, fb, whole, eps;
        int depth;
    } stk[44];
    int sp = 0;
    double fa = seg_integrand(Ea, Eb, da, db, h, w, 0.0), fm = seg_integrand(Ea, Eb, da, db, h, w, 0.5 * h),
           fb = seg_integrand(Ea, Eb, da, db, h, w, h);
    stk[sp++] = Iv{0.0, h, fa, fm, fb, dmul(h / 6, dadd(dadd(fa, dmul(4.0, fm)), fb)), 1e-13 * h, 40};
    double total = 0.0;
    while (sp > 0) {
        Iv c = stk[--sp];
        double m = 0.5 * (c.a + c.b), lm = 0.5 * (c.a + m), rm = 0.5 * (m + c.b);
        double flm = seg_integrand(Ea, Eb, da, db, h, w, lm), frm = seg_integrand(Ea, Eb, da, db, h, w, rm);
        double left = dmul((m - c.a) / 6, dadd(dadd(c.fa, dmul(4.0, flm)), c.fm));
        double right = dmul((c.b - m) / 6, dadd(dadd(c.fm, dmul(4.0, frm)), c.fb));
        double d = dadd(dadd(left, right), -c.whole);
        if (c.depth <= 0 || fabs(d) <= 15 * c.eps) {
            total = dadd(total, dadd(dadd(left, right), d / 15));
        } else {
            // right half below the left one: the left half is finished first
            stk[sp++] = Iv{m, c.b, c.fm, frm, c.fb, right, 0.5 * c.eps, c.depth - 1};
            stk[sp++] = Iv{c.a, m, c.fa, flm, c.fm, left, 0.5 * c.eps, c.depth - 1};
        }
    }
    return total;
}

struct CoefArgs {
    double kspring, w;
    int climbing, weighted;
};

// What image nu of a chain does: its own kind, or normal / climbing (ci).
__device__ __forceinline__ int im_kind(int kind, int nu, int ci)
{
    return kind >= 0 ? kind : (nu == ci ? SP_IMAGE_CLIMBING : SP_IMAGE_NORMAL);
}

// After the field pass: tangents, segment lengths and force coefficients of
// the chain whose first image is g, by one warp, a lane per image.
// The force coefficient a of an interior image (F = -Pg + a tau): climbing
// image (the chain's highest interior image when climbing is on, and the image
// has no fixed kind): a = 2 Pg.tau / |tau|^2; falling image: 0; otherwise
// (Pg.tau / |tau| + k (l_g - l_{g-1})) / |tau|, l the geodesic or
// energy-weighted segment lengths.
// What bounds it: one trip to memory and the FP64 divisions and square roots
// of one image (a thread per image whose search for the highest image read the
// energies one after another took as long, and the tangent weights a launch of
// 3 us before it).
template <typename T>
__device__ void chain_coefs(int g0, const ImgInfo *img, double *scal, CoefArgs ca)
{
    const ImgInfo im = img[g0];
    if (im.nu != 0 || threadIdx.x >= 32) return;
    const int l = threadIdx.x, M = im.M;
    // the highest interior image, the first of equals
    int ci = 1;
    if (M > 2) {
        double best = __ldcg(scal + kS * (g0 + 1) + kE);
        for (int nu = 2 + l; nu < M - 1; nu += 32) {
            const double e = __ldcg(scal + kS * (g0 + nu) + kE);
            if (e > best) {
                best = e;
                ci = nu;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double e = xor_of(best, o);
            const int n = __shfl_xor_sync(0xffffffffu, ci, o);
            if (e > best || (e == best && n < ci)) {
                best = e;
                ci = n;
            }
        }
    }
    if (!ca.climbing) ci = -1;
    // |tau|^2 and Pg.tau with the weights as the force pass uses them; at the
    // endpoints one-sided differences (for the slopes)
    for (int nu = l; nu < M; nu += 32) {
        double *sc = scal + kS * (g0 + nu);
        const double *sm = nu > 0 ? sc - kS : sc, *sp = nu < M - 1 ? sc + kS : sc;
        const double E0 = __ldcg(sc + kE), Em = __ldcg(sm + kE), Ep = __ldcg(sp + kE), L = __ldcg(sc + kL2),
                     Lm = __ldcg(sm + kL2), pp = __ldcg(sc + kPP), pm = __ldcg(sc + kPM), mm = __ldcg(sc + kMM),
                     gp = __ldcg(sc + kGP), gm = __ldcg(sc + kGM);
        double wp = 1.0, wm = 0.0;
        if (nu == M - 1) {
            wp = 0.0;
            wm = 1.0;
        } else if (nu > 0) {
            tangent_weights(Em, E0, Ep, &wp, &wm);
        }
        wp = (double)(T)wp;
        wm = (double)(T)wm;
        const double tt = dadd(dadd(dmul(dmul(wp, wp), pp), dmul(dmul(wm, wm), mm)), dmul(dmul(2.0 * wp, wm), pm));
        const double gt = dadd(dmul(wp, gp), dmul(wm, gm)), inv = tt > 0 ? 1.0 / sqrt(tt) : 0.0;
        sc[kWP] = wp;
        sc[kWM] = wm;
        sc[kTT] = tt;
        sc[kGT] = gt;
        const int kind = im_kind(img[g0 + nu].kind, nu, ci);
        // climbing: tangential component inverted, no spring; falling: the full
        // projected gradient, no spring (descends to a minimum along the path)
        const double gn = dmul(gt, inv);
        double coef = kind == SP_IMAGE_CLIMBING ? 2.0 * gn : (kind == SP_IMAGE_FALLING ? 0.0 : gn);
        if (kind == SP_IMAGE_NORMAL && !ca.weighted) coef = dadd(gn, dmul(ca.kspring, sqrt(L) - sqrt(Lm)));
        sc[kA] = dmul(coef, inv);
    }
    if (!ca.weighted) return;
    // energy-weighted springs: the lengths need the slopes of both ends
    __threadfence_block();
    __syncwarp();
    auto at = [&](int nu, int k) { return *(const volatile double *)(scal + kS * (g0 + nu) + k); };
    auto slope = [&](int nu) {
        const double tt = at(nu, kTT);
        return tt > 0 ? at(nu, kGT) / sqrt(tt) : 0.0;
    };
    for (int nu = l; nu < M - 1; nu += 32)
        scal[kS * (g0 + nu) + kLW] =
            seg_length(at(nu, kE), at(nu + 1, kE), slope(nu), slope(nu + 1), sqrt(at(nu, kL2)), ca.w);
    __threadfence_block();
    __syncwarp();
    for (int nu = 1 + l; nu < M - 1; nu += 32) {
        if (im_kind(img[g0 + nu].kind, nu, ci) != SP_IMAGE_NORMAL) continue;
        const double tt = at(nu, kTT), inv = tt > 0 ? 1.0 / sqrt(tt) : 0.0;
        const double fs = dmul(ca.kspring, at(nu, kLW) - at(nu - 1, kLW));
        scal[kS * (g0 + nu) + kA] = dmul(dadd(dmul(at(nu, kGT), inv), fs), inv);
    }
}
template <typename T>
__global__ void k_g_coefs(const ImgInfo *__restrict__ img, double *scal, const CoefArgs ca)
{
    chain_coefs<T>(blockIdx.x, img, scal, ca);
}

struct NoPost2 {
    __device__ void operator()(int) const {}
};

template <typename T, Nbr LOOPS = Nbr::ALL, typename R>
__device__ __forceinline__ void g_field_body(int vb, const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img,
                                             const Stencil<T> *__restrict__ S, const R *x, R *G, double *part,
                                             unsigned *cnt, double *scal)
{
    BlkInfo bi = blk[vb];
    ImgInfo im = img[bi.g];
    // the chain's stencil, staged in shared memory for the neighbour loop
    __shared__ __align__(16) unsigned char st_raw[sizeof(Stencil<T>)];
    Stencil<T> &St = *reinterpret_cast<Stencil<T> *>(st_raw);
    copy_stencil(S + bi.chain, &St, bi.ne);
    __syncthreads();
    const long long base = im.spin0 + (long long)im.nu * im.N;
    const R *xb = x + base;
    const bool has_p = im.nu < im.M - 1, has_m = im.nu > 0;
    // every sum in FP64, or float-float for FP32 (the same sums of the same
    // products to ~1e-14, off the FP64 pipe)
    using A = typename Acc<T>::type;
    A r[8] = {};
    for (int s = 0; s < im.spt; ++s) {
        const int i = (bi.t * im.spt + s) * kBlock + (int)threadIdx.x;
        if (i >= im.N) break;
        int b;
        const v3<T> ni = ld(xb, i);
        v3<T> B;
        if constexpr (std::is_same<T, float>::value) {
            v3<T> lo;
            B = local_field_comp<LOOPS>(St, xb, i, ni, b, lo);
            // r[0] collects n.(B + Bz), B = hi + lo; the -1/2 follows at the end
            acc_add(r[0], ni, B);
            acc_add(r[0], ni, mk(St.Bz[b][0], St.Bz[b][1], St.Bz[b][2]));
            r[0].lo += xdot(ni, lo);
            B = B + lo;
        } else {
            B = local_field(St, xb, i, ni, b);
            r[0] += xdot(ni, B + mk(St.Bz[b][0], St.Bz[b][1], St.Bz[b][2]));
        }
        const v3<T> pg = minus_tangent(B, ni);  // tangent-space part of dH/dn = -B
        st(G, base + i, pg);
        asm volatile("" ::: "memory");  // the neighbours' registers first, then those of the images
        const v3<T> np = has_p ? ldc(xb + im.N, i) : ni, nm = has_m ? ldc(xb - im.N, i) : ni;
        v3<T> dp = np - ni, dm = ni - nm;
        dp = tangent(dp, ni);
        dm = tangent(dm, ni);
        if (has_p) {
            const v3<T> c = xcross(ni, np);
            const T th = atan2(sqrt(xdot(c, c)), xdot(ni, np));
            acc_add(r[1], th, th);
            acc_add(r[kPP], dp, dp);
            acc_add(r[kGP], pg, dp);
        }
        if (has_m) {
            acc_add(r[kMM], dm, dm);
            acc_add(r[kGM], pg, dm);
        }
        if (has_p && has_m) acc_add(r[kPM], dp, dm);
    }
    if constexpr (std::is_same<T, float>::value)
        r[0] = f2sum{-0.5f * r[0].hi, -0.5f * r[0].lo};
    else
        r[0] *= -0.5;
    image_sums<8, false>(r, A{}, part, vb, im.blk0, im.bpi, cnt + bi.g, scal + kS * bi.g, NoPost2());
}
static_assert(kE == 0 && kL2 == 1 && kGM == 6 && kVF == 7, "the field pass writes slots 0..7 (7: padding)");

template <typename T, Nbr LOOPS>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? SPGB_GF_MINB : 1)
    k_g_field(const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img, const Stencil<T> *__restrict__ S,
              const rec_t<T> *__restrict__ x, rec_t<T> *__restrict__ G, double *part, unsigned *cnt, double *scal)
{
    g_field_body<T, LOOPS>(blockIdx.x, blk, img, S, x, G, part, cnt, scal);
}

// mode 0: F only; 1: v from memory (the call's first iteration); 2: v = c F,
// c the projection coefficient of the previous force pass (read before this
// block's ticket, so before the image's last block replaces it).
template <typename T, typename R>
__device__ __forceinline__ void g_force_body(int vb, const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img,
                                             const R *x, const R *v, R *F, const R *G, T dth_m, int mode, double *part,
                                             unsigned *cnt, double *scal)
{
    BlkInfo bi = blk[vb];
    ImgInfo im = img[bi.g];
    if (im.nu == 0 || im.nu == im.M - 1) return;
    double *sc = scal + kS * bi.g;
    const T a = (T)sc[kA], wp = (T)sc[kWP], wm = (T)sc[kWM], c = mode == 2 ? (T)sc[kC] : T(0);
    const long long base = im.spin0 + (long long)im.nu * im.N;
    using A = typename Acc<T>::type;
    A r[2] = {}, mx{};
    for (int s = 0; s < im.spt; ++s) {
        const int i = (bi.t * im.spt + s) * kBlock + (int)threadIdx.x;
        if (i >= im.N) break;
        const long long p = base + i;
        const v3<T> xi = ld(x, p), xp = ld(x, p + im.N), xm = ld(x, p - im.N);
        v3<T> t = axpy(wp, xp - xi, wm * (xi - xm));
        t = tangent(t, xi);
        const v3<T> Fn = axpy(a, t, -ldc(G, p));
        if (mode) {
            const v3<T> Fo = ldc((const R *)F, p);
            const v3<T> vi = axpy(dth_m, Fo + Fn, mode == 1 ? ldc(v, p) : c * Fo);
            acc_add(r[0], vi, Fn);
        }
        st(F, p, Fn);
        const A f2 = acc_dot(Fn, Fn);
        r[1] = r[1] + f2;
        mx = nan_max(mx, f2);  // max |F|^2; the image's max |F| is its square root
    }
    image_sums<2, true>(r, mx, part, vb, im.blk0, im.bpi, cnt + bi.g, sc + kVF, ForcePost{sc + kVF});
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_g_force(const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img,
                                                    const rec_t<T> *__restrict__ x, const rec_t<T> *__restrict__ v,
                                                    rec_t<T> *__restrict__ F, const rec_t<T> *__restrict__ G, T dth_m,
                                                    int mode, double *part, unsigned *cnt, double *scal)
{
    g_force_body<T>(blockIdx.x, blk, img, x, v, F, G, dth_m, mode, part, cnt, scal);
}

// mode 0: move with the stored v; 1: move with v = c F; 2: store v = c F
template <typename T, typename R>
__device__ __forceinline__ void g_move_body(int vb, const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img,
                                            R *x, R *v, const R *F, T dt, T dt2_2m, int mode, const double *scal)
{
    BlkInfo bi = blk[vb];
    ImgInfo im = img[bi.g];
    if (im.nu == 0 || im.nu == im.M - 1) return;
    // projection coefficient of the last force pass: every thread reads the
    // image's slot (one broadcast load, no block barrier)
    const T c = mode >= 1 ? (T)scal[kS * bi.g + kC] : T(0);
    const long long base = im.spin0 + (long long)im.nu * im.N;
    for (int s = 0; s < im.spt; ++s) {
        const int i = (bi.t * im.spt + s) * kBlock + (int)threadIdx.x;
        if (i >= im.N) break;
        const long long p = base + i;
        const v3<T> Fi = ldc(F, p), vi = mode >= 1 ? c * Fi : ldc((const R *)v, p);
        if (mode == 2)
            st(v, p, vi);
        else
            st(x, p, xunit(axpy(dt2_2m, Fi, axpy(dt, vi, ldc((const R *)x, p)))));
    }
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_g_move(const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img,
                                                   rec_t<T> *__restrict__ x, rec_t<T> *__restrict__ v,
                                                   const rec_t<T> *__restrict__ F, T dt, T dt2_2m, int mode,
                                                   const double *scal)
{
    g_move_body<T>(blockIdx.x, blk, img, x, v, F, dt, dt2_2m, mode, scal);
}

// ------------------------------------------------------------ persistent GNEB
// Grid-wide barrier of a cooperative launch, with a bounded wait: the arrival
// counter *bar only grows (by gridDim.x per barrier; the host zeroes it before
// the launch).  A block polls at most `limit` times; a block that gives up
// raises *abort_flag and ORs `site` into status[1] (the context's status word,
// timeouts), and every block that sees the abort flag while waiting leaves
// too, so no block waits unboundedly.  Returns false when the kernel must
// return.
__device__ bool grid_sync(unsigned *bar, unsigned *abort_flag, unsigned &gen, long long limit, unsigned *status,
                          unsigned site)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        gen += 1;
        const unsigned target = gen * gridDim.x;
        __threadfence();  // this block's writes before its arrival
        atomicAdd(bar, 1u);
        int ok = 1;
        long long polls = 0;
        while (*(volatile unsigned *)bar < target) {
            if (*(volatile unsigned *)abort_flag) {
                ok = 0;
                break;
            }
            if (++polls > limit) {
                ok = 0;
                atomicExch(abort_flag, 1u);
                if (status) atomicOr_system(status + 1, site);
                break;
            }
            __nanosleep(64);
        }
        __threadfence();  // the other blocks' writes after the barrier
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <typename T> struct PersistArgs {
    const BlkInfo *blk;
    const ImgInfo *img;
    const Stencil<T> *S;
    rec_t<T> *x, *v, *F, *G;
    double *part, *scal;
    unsigned *cnt;
    T dt, dt2_2m, dth_m;
    int n_blk, n_img, n_iter;
    CoefArgs ca;
    unsigned *bar, *abort_flag, *status;
    long long limit;
};

// n_iter GNEB iterations (move, field, coefs, force) of every image of every chain in
// one cooperative launch (coefs: a warp per chain): each pass is a grid-stride loop over the block
// table, the passes are separated by grid barriers.  The bodies are those of
// the per-pass kernels, so the iterates are bit-identical.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_g_persistent(const __grid_constant__ PersistArgs<T> a)
{
    // every spin, velocity and pass buffer is read with plain (coherent)
    // loads: other blocks wrote them earlier in this launch
    using R = typename ShRec<T>::type;
    static_assert(sizeof(R) == sizeof(rec_t<T>), "plain-load records have the record layout");
    R *x = reinterpret_cast<R *>(a.x), *v = reinterpret_cast<R *>(a.v), *F = reinterpret_cast<R *>(a.F),
      *G = reinterpret_cast<R *>(a.G);
    unsigned gen = 0;
    for (int it = 0; it < a.n_iter; ++it) {
        for (int vb = blockIdx.x; vb < a.n_blk; vb += gridDim.x) {
            g_move_body<T>(vb, a.blk, a.img, x, v, (const R *)F, a.dt, a.dt2_2m, it ? 1 : 0, a.scal);
            __syncthreads();
        }
        if (!grid_sync(a.bar, a.abort_flag, gen, a.limit, a.status, 1u)) return;
        for (int vb = blockIdx.x; vb < a.n_blk; vb += gridDim.x) {
            g_field_body<T>(vb, a.blk, a.img, a.S, (const R *)x, G, a.part, a.cnt, a.scal);
            __syncthreads();
        }
        if (!grid_sync(a.bar, a.abort_flag, gen, a.limit, a.status, 1u)) return;
        for (int g = blockIdx.x; g < a.n_img; g += gridDim.x) chain_coefs<T>(g, a.img, a.scal, a.ca);
        if (!grid_sync(a.bar, a.abort_flag, gen, a.limit, a.status, 1u)) return;
        for (int vb = blockIdx.x; vb < a.n_blk; vb += gridDim.x) {
            g_force_body<T>(vb, a.blk, a.img, (const R *)x, (const R *)v, F, (const R *)G, a.dth_m, it ? 2 : 1, a.part,
                            a.cnt, a.scal);
            __syncthreads();
        }
        if (!grid_sync(a.bar, a.abort_flag, gen, a.limit, a.status, 1u)) return;
    }
}

__global__ void k_g_finish(const ImgInfo *__restrict__ img, int n_img, const double *scal, double *E, double *fmax_out,
                           int n_chains)
{
    // one thread per image; the thread of each chain's image 0 also takes the
    // chain's max force over its interior images (in image order)
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n_img; g += gridDim.x * blockDim.x) {
        E[g] = scal[kS * g + kE];
        const ImgInfo im = img[g];
        if (im.nu != 0 || im.chain >= n_chains) continue;
        double m = 0;
        for (int nu = 1; nu < im.M - 1; ++nu) m = nan_max(m, scal[kS * (im.g0 + nu) + kFMAX]);
        fmax_out[im.chain] = sqrt(m);  // the slot holds max |F|^2
    }
}

}  // namespace

// ------------------------------------------------------------ VP host loop
template <typename T>
int vp_minimise(MinScratch **sp, const Stencil<T> &S, void *n, void *v, const MinArgs &a, int *iters, double *max_torque,
                cudaStream_t st)
{
    int rc = scratch(sp);
    if (rc) return rc;
    MinScratch *s = *sp;
    int N = S.N;
    int nblk = blocks_for(N > 0 ? N : 1);
    if (grow(s->F, sizeof(rec_t<T>) * (size_t)(N > 0 ? N : 1)) || grow(s->scal, kS * sizeof(double)) ||
        grow(s->part, kPartRow * sizeof(double) * (size_t)nblk) || grow_counters(s->cnt, 1, st) ||
        grow(s->state, 4 * sizeof(int)))
        return SP_ERR_CUDA;
    rec_t<T> *x = (rec_t<T> *)n, *vv = (rec_t<T> *)v, *F = (rec_t<T> *)s->F.p;
    double *scal = (double *)s->scal.p, *part = (double *)s->part.p;
    unsigned *cnt = (unsigned *)s->cnt.p;
    int *state = (int *)s->state.p;
    double dth_m = a.dt / (2.0 * a.mass), dt2_2m = a.dt * a.dt / (2.0 * a.mass);
    if (cudaMemsetAsync(state, 0, 4 * sizeof(int), st) != cudaSuccess) return SP_ERR_CUDA;
    launch_pdl(k_vp_force<T>, dim3(nblk), dim3(kBlock), 0, st, S, (const rec_t<T> *)x, (const rec_t<T> *)vv, F, (T)dth_m, 0,
               part, cnt, scal, (const int *)state);
    int k = 0;
    while (k < a.max_iter) {
        int chunk = std::min(a.check_every, a.max_iter - k);
        for (int c = 0; c < chunk; ++c, ++k) {
            launch_pdl(k_vp_move<T>, dim3(nblk), dim3(kBlock), 0, st, N, x, vv, (const rec_t<T> *)F, (T)a.dt, (T)dt2_2m,
                       a.tol, k, a.max_iter, (const double *)scal, state);
            launch_pdl(k_vp_force<T>, dim3(nblk), dim3(kBlock), 0, st, S, (const rec_t<T> *)x, (const rec_t<T> *)vv, F,
                       (T)dth_m, k == 0 ? 1 : 2, part, cnt, scal, (const int *)state);
        }
        if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
        if (cudaMemcpyAsync(s->host_state, state, 2 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return SP_ERR_CUDA;
        if (s->host_state[1] == 0) break;
    }
    // final projection of the velocity (or nothing when no iteration ran)
    launch_pdl(k_vp_move<T>, dim3(nblk), dim3(kBlock), 0, st, N, x, vv, (const rec_t<T> *)F, (T)a.dt, (T)dt2_2m, a.tol,
               a.max_iter, a.max_iter, (const double *)scal, state);
    if (cudaMemcpyAsync(s->host_state, state, 2 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(s->host_fmax, scal + kFMAX, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SP_ERR_CUDA;
    *iters = s->host_state[0];
    *max_torque = sqrt(*s->host_fmax);
    return 0;
}

// ------------------------------------------------------------ batched VP
// One image per system.  Per system g: the slots kVF.. from the last force
// pass, state[2g] iterations moved, state[2g+1] active flag, proj[g] whether
// the last force pass had a velocity.
// 1 M spins in 64 systems: 56 -> 50 us an iteration; bound by the chain of a
// block (tables, state, neighbours, block sum, ticket) with 6 blocks per SM
// in flight (5: 53, 4: 56).
template <typename T>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? SPGB_VP_MINB : 1)
    k_bvp_force(const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img, const Stencil<T> *__restrict__ S,
                const rec_t<T> *__restrict__ x, const rec_t<T> *__restrict__ v, rec_t<T> *__restrict__ F, T dth_m, int mode,
                double *part, unsigned *cnt, double *scal, const int *state, int *proj)
{
    // the tables and stencils do not change while kernels are in flight
    const BlkInfo bi = blk[blockIdx.x];
    const ImgInfo im = img[bi.g];
    __shared__ __align__(16) unsigned char st_raw[sizeof(Stencil<T>)];
    Stencil<T> &St = *reinterpret_cast<Stencil<T> *>(st_raw);
    copy_stencil(S + bi.chain, &St, bi.ne);
    __syncthreads();
    allow_dependents();
    wait_prerequisite(x, v, F, scal, state);  // state, scalars and records come from the kernels before
    if (mode && state[2 * bi.g + 1] == 0) return;
    double *sc = scal + kS * bi.g;
    const T c = mode == 2 ? (T)sc[kC] : T(0);
    const int i = bi.t * kBlock + threadIdx.x;
    T r[2] = {0, 0}, mx = 0;
    if (i < im.N) vp_force(St, x + im.spin0, v + im.spin0, F + im.spin0, i, dth_m, mode, c, r, mx);
    image_sums<2, true>(r, mx, part, blockIdx.x, im.blk0, im.bpi, cnt + bi.g, sc + kVF, ForcePost{sc + kVF});
    if (bi.t == 0 && threadIdx.x == 0) proj[bi.g] = mode;
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_bvp_move(const BlkInfo *__restrict__ blk, const ImgInfo *__restrict__ img,
                                                     rec_t<T> *__restrict__ x, rec_t<T> *__restrict__ v,
                                                     const rec_t<T> *__restrict__ F, T dt, T dt2_2m, double tol,
                                                     int k, int max_iter, const double *scal, int *state,
                                                     const int *proj)
{
    const BlkInfo bi = blk[blockIdx.x];
    const ImgInfo im = img[bi.g];
    allow_dependents();
    wait_prerequisite(x, v, F, scal, state, proj);  // state, scalars and records come from the kernels before
    const double *sc = scal + kS * bi.g;
    const bool done = sc[kFN] < tol || k >= max_iter;
    const int i = bi.t * kBlock + threadIdx.x;
    if (i < im.N)
        vp_move(x + im.spin0, v + im.spin0, F + im.spin0, i, dt, dt2_2m, proj[bi.g] != 0, (T)sc[kC], done,
                k >= max_iter);
    if (bi.t == 0 && threadIdx.x == 0) {
        state[2 * bi.g + 1] = done ? 0 : 1;
        if (!done) state[2 * bi.g] = k + 1;
    }
}

template <typename T>
int vp_batch_run(MinScratch **sp, const std::vector<Stencil<T>> &stencils, const std::vector<long long> &spin0,
                 void *spins, void *vel, const MinArgs &a, int *iters, double *max_torque, cudaStream_t st)
{
    int rc = scratch(sp);
    if (rc) return rc;
    MinScratch *s = *sp;
    int C = (int)stencils.size();
    std::vector<ImgInfo> img;
    std::vector<BlkInfo> blk;
    long long total = 0;
    for (int c = 0; c < C; ++c) {
        int N = stencils[c].N;
        int bpi = blocks_for(N > 0 ? N : 1);
        ImgInfo im{spin0[c], N, c, 0, 1, c, (int)blk.size(), bpi, -1, 1, 0};
        for (int t = 0; t < bpi; ++t) blk.push_back(BlkInfo{c, t, c, stencils[c].off[stencils[c].nb]});
        img.push_back(im);
        total = std::max(total, spin0[c] + (long long)N);
    }
    int n_full = (int)blk.size();
    size_t rb = sizeof(rec_t<T>) * (size_t)std::max(total, 1LL);
    // blk holds the full table followed by room for a compacted copy
    if (grow(s->F, rb) || grow(s->scal, kS * sizeof(double) * C) || grow(s->part, kPartRow * sizeof(double) * (size_t)n_full) ||
        grow_counters(s->cnt, C, st) || grow(s->blk, 2 * sizeof(BlkInfo) * n_full) ||
        grow(s->img, sizeof(ImgInfo) * C) || grow(s->sten, sizeof(Stencil<T>) * C) ||
        grow(s->state, sizeof(int) * 3 * C))
        return SP_ERR_CUDA;
    BlkInfo *Bfull = (BlkInfo *)s->blk.p, *Bact = Bfull + n_full;
    ImgInfo *I = (ImgInfo *)s->img.p;
    if (cudaMemcpyAsync(Bfull, blk.data(), sizeof(BlkInfo) * n_full, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(Bact, blk.data(), sizeof(BlkInfo) * n_full, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(I, img.data(), sizeof(ImgInfo) * C, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(s->sten.p, stencils.data(), sizeof(Stencil<T>) * C, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemsetAsync(s->state.p, 0, sizeof(int) * 3 * C, st) != cudaSuccess)
        return SP_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SP_ERR_CUDA;
    s->layout.clear();  // the GNEB tables were overwritten
    const Stencil<T> *Sd = (const Stencil<T> *)s->sten.p;
    rec_t<T> *x = (rec_t<T> *)spins, *v = (rec_t<T> *)vel, *F = (rec_t<T> *)s->F.p;
    double *scal = (double *)s->scal.p, *part = (double *)s->part.p;
    unsigned *cnt = (unsigned *)s->cnt.p;
    int *state = (int *)s->state.p, *proj = state + 2 * C;
    double dth_m = a.dt / (2.0 * a.mass), dt2_2m = a.dt * a.dt / (2.0 * a.mass);
    std::vector<int> hs(2 * C);
    launch_pdl(k_bvp_force<T>, dim3(n_full), dim3(kBlock), 0, st, (const BlkInfo *)Bfull, (const ImgInfo *)I, Sd,
               (const rec_t<T> *)x, (const rec_t<T> *)v, F, (T)dth_m, 0, part, cnt, scal, (const int *)state, proj);
    int k = 0, n_act = n_full;
    while (k < a.max_iter) {
        int chunk = std::min(a.check_every, a.max_iter - k);
        for (int c = 0; c < chunk; ++c, ++k) {
            launch_pdl(k_bvp_move<T>, dim3(n_act), dim3(kBlock), 0, st, (const BlkInfo *)Bact, (const ImgInfo *)I, x, v,
                       (const rec_t<T> *)F, (T)a.dt, (T)dt2_2m, a.tol, k, a.max_iter, (const double *)scal, state,
                       (const int *)proj);
            launch_pdl(k_bvp_force<T>, dim3(n_act), dim3(kBlock), 0, st, (const BlkInfo *)Bact, (const ImgInfo *)I, Sd,
                       (const rec_t<T> *)x, (const rec_t<T> *)v, F, (T)dth_m, k == 0 ? 1 : 2, part, cnt, scal,
                       (const int *)state, proj);
        }
        if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
        if (cudaMemcpyAsync(hs.data(), state, sizeof(int) * 2 * C, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return SP_ERR_CUDA;
        // Drop converged systems from the launch tables once a quarter of the
        // launched blocks belongs to them.  A converged system is frozen: its
        // force pass returns at once and its move re-applies the same
        // projection, so leaving it out changes no result.
        std::vector<BlkInfo> act;
        for (int c = 0; c < C; ++c)
            if (hs[2 * c + 1]) {
                img[c].blk0 = (int)act.size();
                for (int t = 0; t < img[c].bpi; ++t) act.push_back(BlkInfo{c, t, c, stencils[c].off[stencils[c].nb]});
            }
        if (act.empty()) break;
        if (4 * (long long)act.size() <= 3LL * n_act) {
            n_act = (int)act.size();
            if (cudaMemcpyAsync(Bact, act.data(), sizeof(BlkInfo) * n_act, cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaMemcpyAsync(I, img.data(), sizeof(ImgInfo) * C, cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess)
                return SP_ERR_CUDA;
        }
    }
    // final projection (where the last force pass updated the velocity)
    launch_pdl(k_bvp_move<T>, dim3(n_full), dim3(kBlock), 0, st, (const BlkInfo *)Bfull, (const ImgInfo *)I, x, v,
               (const rec_t<T> *)F, (T)a.dt, (T)dt2_2m, a.tol, a.max_iter, a.max_iter, (const double *)scal, state,
               (const int *)proj);
    std::vector<double> hsc(kS * C);
    if (cudaMemcpyAsync(hs.data(), state, sizeof(int) * 2 * C, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(hsc.data(), scal, sizeof(double) * kS * C, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SP_ERR_CUDA;
    for (int c = 0; c < C; ++c) {
        iters[c] = hs[2 * c];
        max_torque[c] = sqrt(hsc[kS * c + kFMAX]);
    }
    return 0;
}

// ------------------------------------------------------------ GNEB host side
template <typename T>
int gneb_batch_run(MinScratch **sp, const std::vector<Stencil<T>> &stencils, const std::vector<int> &M,
                   const std::vector<long long> &spin0, void *chain, void *vel, const GnebArgs &a, double *E_dev,
                   double *fmax_dev, cudaStream_t st)
{
    int rc = scratch(sp);
    if (rc) return rc;
    MinScratch *s = *sp;
    int C = (int)stencils.size();
    std::vector<ImgInfo> img;
    std::vector<BlkInfo> blk;
    long long total = 0;
    for (int c = 0; c < C; ++c) {
        int N = stencils[c].N;
        const int spt = gneb_spt((long long)M[c] * N);
        int bpi = blocks_for(N > 0 ? N : 1, kBlock * spt);
        int g0 = (int)img.size();
        for (int nu = 0; nu < M[c]; ++nu) {
            int kind = a.kinds ? a.kinds[g0 + nu] : -1;
            ImgInfo im{spin0[c], N, c, nu, M[c], g0, (int)blk.size(), bpi, kind, spt, 0};
            for (int t = 0; t < bpi; ++t) blk.push_back(BlkInfo{(int)img.size(), t, c, stencils[c].off[stencils[c].nb]});
            img.push_back(im);
        }
        total = std::max(total, spin0[c] + (long long)M[c] * N);
    }
    int n_img = (int)img.size(), n_blk = (int)blk.size();
    size_t rb = sizeof(rec_t<T>) * (size_t)std::max(total, 1LL);
    if (grow(s->F, rb) || grow(s->G, rb) || grow(s->scal, kS * sizeof(double) * n_img) ||
        grow(s->part, kPartRow * sizeof(double) * (size_t)n_blk) || grow_counters(s->cnt, n_img, st) ||
        grow(s->blk, sizeof(BlkInfo) * n_blk) || grow(s->img, sizeof(ImgInfo) * n_img) ||
        grow(s->sten, sizeof(Stencil<T>) * C))
        return SP_ERR_CUDA;
    // upload the tables only when the layout changed (a call with an
    // unchanged layout launches kernels only, so it can be stream-captured)
    std::vector<char> key(sizeof(int) + img.size() * sizeof(ImgInfo) + stencils.size() * sizeof(Stencil<T>));
    int tsz = (int)sizeof(T);
    memcpy(key.data(), &tsz, sizeof(int));
    memcpy(key.data() + sizeof(int), img.data(), img.size() * sizeof(ImgInfo));
    memcpy(key.data() + sizeof(int) + img.size() * sizeof(ImgInfo), stencils.data(), stencils.size() * sizeof(Stencil<T>));
    if (key != s->layout) {
        if (cudaMemcpyAsync(s->blk.p, blk.data(), sizeof(BlkInfo) * n_blk, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(s->img.p, img.data(), sizeof(ImgInfo) * n_img, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(s->sten.p, stencils.data(), sizeof(Stencil<T>) * C, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return SP_ERR_CUDA;
        // the host vectors must outlive the copies above
        if (cudaStreamSynchronize(st) != cudaSuccess) return SP_ERR_CUDA;
        s->layout.swap(key);
    }
    const BlkInfo *B = (const BlkInfo *)s->blk.p;
    const ImgInfo *I = (const ImgInfo *)s->img.p;
    const Stencil<T> *Sd = (const Stencil<T> *)s->sten.p;
    rec_t<T> *x = (rec_t<T> *)chain, *v = (rec_t<T> *)vel;
    rec_t<T> *F = (rec_t<T> *)s->F.p, *G = (rec_t<T> *)s->G.p;
    double *scal = (double *)s->scal.p, *part = (double *)s->part.p;
    unsigned *cnt = (unsigned *)s->cnt.p;
    double dth_m = a.dt / (2.0 * a.mass), dt2_2m = a.dt * a.dt / (2.0 * a.mass);
    const CoefArgs ca{a.k, a.w, a.climbing, a.w != 0.0};
    // FP32 batches of chains without the unrolled neighbour loops take the kernel
    // with the loop over the entries alone, which does not spill (20 images of 128 x
    // 128 spins, 10 iterations: 18 bonds 734 -> 665 us, 12 bonds 623 -> 570, two atoms
    // with nine 546 -> 494)
    bool entries = sizeof(T) == 4;
    for (const Stencil<T> &sc : stencils) entries = entries && !sc.fixed;
    const auto field = entries ? k_g_field<T, sizeof(T) == 4 ? Nbr::ENTRIES : Nbr::ALL> : k_g_field<T, Nbr::ALL>;
    auto forces = [&](int mode, cudaStream_t ss) {
        field<<<n_blk, kBlock, 0, ss>>>(B, I, Sd, x, G, part, cnt, scal);
        k_g_coefs<T><<<n_img, 32, 0, ss>>>(I, scal, ca);
        k_g_force<T><<<n_blk, kBlock, 0, ss>>>(B, I, x, v, F, G, dth_m, mode, part, cnt, scal);
    };
    auto iteration = [&](cudaStream_t ss) {
        k_g_move<T><<<n_blk, kBlock, 0, ss>>>(B, I, x, v, F, a.dt, dt2_2m, 1, scal);
        forces(2, ss);
    };
    forces(0, st);
    int remaining = a.n_iter;
    if (remaining > 0 && a.persistent) {
        // every iteration of the call in one cooperative launch; the barrier
        // counter, abort flag and the image tickets start at zero (a launch
        // that gave up may have left tickets behind)
        if (grow(s->sync, 4 * sizeof(unsigned))) return SP_ERR_CUDA;
        int dev = 0, nsm = 0, per_sm = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_g_persistent<T>, kBlock, 0) != cudaSuccess ||
            per_sm < 1)
            return SP_ERR_CUDA;
        int grid = (int)std::min<long long>((long long)nsm * per_sm, n_blk);
        PersistArgs<T> pa{B, I, Sd, x, v, F, G, part, scal, cnt, (T)a.dt, (T)dt2_2m, (T)dth_m, n_blk, n_img, remaining,
                          ca, (unsigned *)s->sync.p,
                          (unsigned *)s->sync.p + 1, a.status, a.wait_limit > 0 ? a.wait_limit : (1LL << 21)};
        void *args[] = {&pa};
        if (cudaMemsetAsync(s->sync.p, 0, 4 * sizeof(unsigned), st) != cudaSuccess ||
            cudaMemsetAsync(cnt, 0, sizeof(unsigned) * n_img, st) != cudaSuccess ||
            cudaLaunchCooperativeKernel((const void *)k_g_persistent<T>, dim3(grid), dim3(kBlock), args, 0, st) !=
                cudaSuccess)
            return SP_ERR_CUDA;
        // leave the tickets at zero for the next call whatever happened
        if (cudaMemsetAsync(cnt, 0, sizeof(unsigned) * n_img, st) != cudaSuccess) return SP_ERR_CUDA;
        remaining = 0;
    }
    if (remaining > 0) {
        k_g_move<T><<<n_blk, kBlock, 0, st>>>(B, I, x, v, F, a.dt, dt2_2m, 0, scal);
        forces(1, st);
        --remaining;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return SP_ERR_CUDA;
    if (remaining >= kGraphIters && cap == cudaStreamCaptureStatusNone) {
        // replay kGraphIters iterations per graph launch on a private stream
        if (!s->gstream) {
            if (cudaStreamCreateWithFlags(&s->gstream, cudaStreamNonBlocking) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev0, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev1, cudaEventDisableTiming) != cudaSuccess)
                return SP_ERR_CUDA;
        }
        struct GKey {
            const void *x, *v, *F, *G, *scal, *part, *cnt, *blk, *img, *sten;
            double dt, mass, k, w;
            int climbing, n_blk;
        } gk{x, v, F, G, scal, part, cnt, B, I, Sd, a.dt, a.mass, a.k, a.w, a.climbing, n_blk};
        std::vector<char> gkey(sizeof gk + s->layout.size());
        memcpy(gkey.data(), &gk, sizeof gk);
        memcpy(gkey.data() + sizeof gk, s->layout.data(), s->layout.size());
        if (!s->gexec || gkey != s->gkey) {
            if (s->gexec) cudaGraphExecDestroy(s->gexec);
            s->gexec = nullptr;
            cudaGraph_t graph;
            if (cudaStreamBeginCapture(s->gstream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return SP_ERR_CUDA;
            for (int r = 0; r < kGraphIters; ++r) iteration(s->gstream);
            if (cudaStreamEndCapture(s->gstream, &graph) != cudaSuccess) return SP_ERR_CUDA;
            cudaError_t e = cudaGraphInstantiate(&s->gexec, graph, 0);
            cudaGraphDestroy(graph);
            if (e != cudaSuccess) return SP_ERR_CUDA;
            s->gkey.swap(gkey);
        }
        if (cudaEventRecord(s->ev0, st) != cudaSuccess || cudaStreamWaitEvent(s->gstream, s->ev0, 0) != cudaSuccess)
            return SP_ERR_CUDA;
        for (; remaining >= kGraphIters; remaining -= kGraphIters)
            if (cudaGraphLaunch(s->gexec, s->gstream) != cudaSuccess) return SP_ERR_CUDA;
        if (cudaEventRecord(s->ev1, s->gstream) != cudaSuccess || cudaStreamWaitEvent(st, s->ev1, 0) != cudaSuccess)
            return SP_ERR_CUDA;
    }
    for (; remaining > 0; --remaining) iteration(st);
    if (a.n_iter > 0) k_g_move<T><<<n_blk, kBlock, 0, st>>>(B, I, x, v, F, a.dt, dt2_2m, 2, scal);
    k_g_finish<<<(n_img + 255) / 256, 256, 0, st>>>(I, n_img, scal, E_dev, fmax_dev, C);
    return cudaGetLastError() == cudaSuccess ? 0 : SP_ERR_CUDA;
}

template <typename T>
int gneb_run(MinScratch **s, const Stencil<T> &S, void *chain, void *vel, const GnebArgs &a, double *E_dev,
             double *fmax_dev, cudaStream_t st)
{
    std::vector<Stencil<T>> sv(1, S);
    return gneb_batch_run<T>(s, sv, std::vector<int>{a.M}, std::vector<long long>{0}, chain, vel, a, E_dev, fmax_dev, st);
}

template <typename T>
int gneb_path_scalars(MinScratch **sp, const Stencil<T> &S, const void *chain, int M, double *E, double *dist,
                      double *slope, cudaStream_t st)
{
    int rc = scratch(sp);
    if (rc) return rc;
    if (grow((*sp)->aux, sizeof(double) * (size_t)(M + 1))) return SP_ERR_CUDA;
    double *Ed = (double *)(*sp)->aux.p;
    // zero iterations: energies, distances, tangents and slopes of every
    // image are evaluated and nothing moves (the velocity is not touched)
    GnebArgs a{0.1, 1.0, 0.0, 0, M, 0, nullptr, 0.0};
    std::vector<Stencil<T>> sv(1, S);
    rc = gneb_batch_run<T>(sp, sv, std::vector<int>{M}, std::vector<long long>{0}, const_cast<void *>(chain),
                           const_cast<void *>(chain), a, Ed, Ed + M, st);
    if (rc) return rc;
    std::vector<double> sc(kS * (size_t)M);
    if (cudaMemcpyAsync(sc.data(), (*sp)->scal.p, sizeof(double) * kS * M, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SP_ERR_CUDA;
    for (int g = 0; g < M; ++g) {
        E[g] = sc[kS * g + kE];
        if (g + 1 < M) dist[g] = sqrt(sc[kS * g + kL2]);
        double tt = sc[kS * g + kTT];
        slope[g] = tt > 0 ? sc[kS * g + kGT] / sqrt(tt) : 0.0;
    }
    return 0;
}

#define SPGB_MIN_INST(T)                                                                                               \
    template int gneb_path_scalars<T>(MinScratch **, const Stencil<T> &, const void *, int, double *, double *,         \
                                      double *, cudaStream_t);                                                         \
    template int vp_batch_run<T>(MinScratch **, const std::vector<Stencil<T>> &, const std::vector<long long> &, void *, \
                                 void *, const MinArgs &, int *, double *, cudaStream_t);                              \
    template int vp_minimise<T>(MinScratch **, const Stencil<T> &, void *, void *, const MinArgs &, int *, double *,    \
                                cudaStream_t);                                                                         \
    template int gneb_run<T>(MinScratch **, const Stencil<T> &, void *, void *, const GnebArgs &, double *, double *,   \
                             cudaStream_t);                                                                            \
    template int gneb_batch_run<T>(MinScratch **, const std::vector<Stencil<T>> &, const std::vector<int> &,           \
                                   const std::vector<long long> &, void *, void *, const GnebArgs &, double *,          \
                                   double *, cudaStream_t);
SPGB_MIN_INST(float)
SPGB_MIN_INST(double)

}  // namespace spgb
