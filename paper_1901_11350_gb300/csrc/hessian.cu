// hessian.cu -- covariant Hessian on the spin manifold, its lowest mode and
// minimum mode following (Sec. MMF and the appendix on the manifold of
// constant-length spins): sp_hessian_apply, sp_lowest_mode, sp_mmf.
//
// Hessian-vector product, per spin i, for a tangent field w:
//   H w|_i = P_i (Hbar w)_i - (n_i . grad_i Hbar) w_i
// where Hbar are the second derivatives of the Hamiltonian continued to
// R^{3N}: (Hbar w)_i = -(sum_j J_ij w_j + w_j x D_ij + 2 K (Khat.w_i) Khat),
// i.e. minus the local field evaluated on w without the Zeeman term, and
// grad_i Hbar = -B_i.  The lowest mode comes from Lanczos with full
// reorthogonalisation (all of a run on the device; the small tridiagonal
// eigenproblem on the host by bisection and inverse iteration).  MMF
// moves with the effective force F - 2 (F.l) l (-(F.l) l where the lowest
// eigenvalue is not negative) by the velocity projection of Appendix D.
#include <algorithm>
#include <cmath>
#include <initializer_list>
#include <vector>

#include "ctx.h"

constexpr int kMaxKrylov = 256;

// What a Lanczos run leaves on the device: the tridiagonal matrix, the running
// estimate of its norm, and per step whether its vector was taken (0: the
// Krylov space had closed, and the remaining kernels of the run return).
struct LzRun {
    double alpha[kMaxKrylov], beta[kMaxKrylov], tnorm[kMaxKrylov];
    int go[kMaxKrylov];
    int nan_start;  // the start vector or the state is not finite
};
struct LzHost {  // pinned
    LzRun run;
    double y[kMaxKrylov];  // Ritz coefficients
};

struct HessScratch {
    DevBuf Q, w, w2, F, Fe, F2, Fe2, y, nB, part, dots, run, coef;
    LzHost *host = nullptr;
};

namespace {

constexpr int kHB = 256;
int grow_h(DevBuf &b, size_t bytes)
{
    if (b.p && b.bytes >= bytes) return 0;
    if (b.p) cudaFree(b.p);
    b.p = nullptr;
    b.bytes = 0;
    if (cudaMalloc(&b.p, bytes) != cudaSuccess) return SP_ERR_CUDA;
    b.bytes = bytes;
    return 0;
}

// H v with v projected onto the tangent planes on the fly: one pass over
// the stencil loads n_j and v_j together and accumulates the field of n and
// the field of the projected w without the Zeeman term.
template <typename T>
__global__ void __launch_bounds__(kHB) k_hvp(const __grid_constant__ Stencil<T> S, const rec_t<T> *__restrict__ n,
                                             const rec_t<T> *__restrict__ v, rec_t<T> *__restrict__ out,
                                             unsigned *status = nullptr)
{
    allow_dependents();
    wait_prerequisite(n, v);  // they may come from the kernels before
    int i = blockIdx.x * kHB + threadIdx.x;
    if (i >= S.N) return;
    int b, c0, c1, c2;
    decode_site(S, i, b, c0, c1, c2);
    const bool inner = interior_site(S, c0, c1, c2);
    v3<T> ni = ld(n, i), vi = ld(v, i);
    v3<T> wi = vi - dot(vi, ni) * ni;
    v3<T> kh = mk(S.Kh[b][0], S.Kh[b][1], S.Kh[b][2]);
    v3<T> Bn = mk(S.Bz[b][0], S.Bz[b][1], S.Bz[b][2]) + (T(2) * S.K[b] * dot(kh, ni)) * kh;
    v3<T> Lw = (T(2) * S.K[b] * dot(kh, wi)) * kh;
    for (int q = S.off[b]; q < S.off[b + 1]; ++q) {
        const NbrEntry<T> &E = S.e[q];
        int j = nbr_index(S, E, i, inner, c0, c1, c2);
        if (j < 0) continue;
        v3<T> nj = ld(n, j), vj = ld(v, j);
        v3<T> wj = vj - dot(vj, nj) * nj;
        v3<T> D = mk(E.Dx, E.Dy, E.Dz);
        Bn = axpy(E.J, nj, Bn + cross(nj, D));
        Lw = axpy(E.J, wj, Lw + cross(wj, D));
    }
    // P (Hbar w) with Hbar w = -Lw, plus the Weingarten term (n . B) w
    v3<T> r3 = (dot(Lw, ni) * ni - Lw) + dot(ni, Bn) * wi;
    st(out, i, r3);
    // status != null: a non-finite product sets the Hessian bit of the
    // context's status word (the check of the output, without a second pass)
    if (status) {
        const bool bad = !(isfinite(r3.x) && isfinite(r3.y) && isfinite(r3.z));
        const unsigned act = __activemask();
        if (__any_sync(act, bad) && (threadIdx.x & 31) == __ffs(act) - 1) atomicOr_system(status, (unsigned)SITE_HESSIAN);
    }
}

// part[blk] = sum over the block's spins of a . q
template <typename T>
__global__ void __launch_bounds__(kHB) k_dot(int N, const rec_t<T> *__restrict__ a, const rec_t<T> *__restrict__ q,
                                             double *__restrict__ part)
{
    __shared__ double sh[kHB / 32];
    int i = blockIdx.x * kHB + threadIdx.x;
    double v = i < N ? ddot(ld(a, i), ld(q, i)) : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int w = 0; w < kHB / 32; ++w) s += sh[w];
        part[blockIdx.x] = s;
    }
}

__global__ void k_dot_final(const double *__restrict__ part, int nblk, double *__restrict__ out)
{
    double s = 0;
    for (int b = 0; b < nblk; ++b) s += part[b];
    *out = s;
}

// ---------------------------------------------------------------- Lanczos
// One Lanczos step is three launches, and nothing returns to the host until
// the run is over (once the Krylov space has closed the launches that are left
// return at once):
//   k_lz_apply  closes the previous step (its coupling b_{k-1} from the norm
//               partials), q_k = w / b, w' = H q_k, partials of alpha_k
//   k_lz_dots   w' -= alpha_k q_k + b_{k-1} q_{k-1}, partials of w' . q_j, j <= k
//   k_lz_sub    w' -= sum_j (w' . q_j) q_j, partials of |w'|^2
// The three-term subtraction leaves w' at its final size, so one further
// Gram-Schmidt pass against every vector brings the overlaps to rounding
// level, as two passes from the full w' did, for half their FP64 work.  Every
// block sums the partials it needs itself, in one order, so all blocks hold
// the same bits.
// What bounds it (FP64): the part's FP64 rate, 2 multiply-adds per clock and
// SM -- 6 per spin, vector and step here, 0.7 ms at 128 x 128 spins and 64
// vectors -- and the chain of three launches a step, each of them four to
// five dependent accesses to L2 and two FP64 reductions long (9 to 11 us even
// for one vector).  That run takes 2.9 ms; with a host round trip per
// reduction, two passes and a Jacobi diagonalisation on the host it took 16.1.
constexpr int kLzB = 128;            // spins per tile; threads per block of the per-spin kernels
constexpr int kLzG = 4;              // groups of kLzB threads in k_lz_dots and k_lz_sub: each takes its share of the
                                     // vectors for the block's tile (one thread per spin left 4 warps per SM waiting
                                     // on the reads of the basis: 22 and 35 us a launch at 64 vectors,
                                     // 19 and 18 us with the groups)
constexpr int kLzBlocks = 152;       // blocks of those two at most: one per SM
constexpr int kLzSpinBlocks = 1216;  // blocks of the per-spin kernels at most
constexpr int kLzChunk = 16;         // basis vectors per transposing warp reduction
static_assert(kMaxKrylov % kLzChunk == 0, "whole chunks");

// dot products: plain FP64, or float-float for FP32 records
template <typename T> struct LzAcc {
    using type = double;
};
template <> struct LzAcc<float> {
    using type = f2sum;
};
__device__ __forceinline__ f2sum lz_dot(v3<float> a, v3<float> b) { return exact_dot(a, b); }
__device__ __forceinline__ double lz_dot(v3<double> a, v3<double> b) { return dot(a, b); }
__device__ __forceinline__ double lz_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ f2sum lz_xor(f2sum v, int o)
{
    return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// Sum over a warp of kLzChunk = 16 values per lane; lanes l and l + 16 receive
// the sum of value l.  31 additions in all (a butterfly that halves the values
// at every step), not 5 per value: additions in FP64 are what a reduction
// costs here.
template <typename A> __device__ __forceinline__ A warp_sums(A (&v)[kLzChunk])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < kLzChunk; ++i) v[i] = v[i] + lz_xor(v[i], 16);
#pragma unroll
    for (int o = kLzChunk / 2; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const A send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
            v[i] = keep + lz_xor(send, o);
        }
    }
    return v[0];
}

// Sum of one value per thread over the block (all threads call it; thread 0
// holds the result).
template <typename A> __device__ __forceinline__ double block_sum(A v)
{
    __shared__ double sh[kLzB * kLzG / 32];
    for (int o = 16; o > 0; o >>= 1) v = v + lz_xor(v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = to_double(v);
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)blockDim.x / 32; ++w) s += sh[w];
    return s;
}

// Sum of n block partials by one warp, the same bits in every block (lane 0
// holds it).
__device__ __forceinline__ double partial_sum(const double *part, int n)
{
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    int p = threadIdx.x & 31;
    for (; p + 96 < n; p += 128) {
        s0 += __ldcg(part + p);
        s1 += __ldcg(part + p + 32);
        s2 += __ldcg(part + p + 64);
        s3 += __ldcg(part + p + 96);
    }
    for (; p < n; p += 32) s0 += __ldcg(part + p);
    double s = (s0 + s1) + (s2 + s3);
    for (int o = 16; o > 0; o >>= 1) s += lz_xor(s, o);
    return s;
}

__device__ __forceinline__ v3<float> ldg2(const float4 *p, long i)
{
    const float4 v = __ldcg(p + i);
    return {v.x, v.y, v.z};
}
__device__ __forceinline__ v3<double> ldg2(const dq4 *p, long i)
{
    const double2 *q = reinterpret_cast<const double2 *>(p + i);
    const double2 a = __ldcg(q), b = __ldcg(q + 1);
    return {a.x, a.y, b.x};
}

// component i of the fixed pseudo-random field (integer hash of the index)
// that starts a run without a start vector
template <typename T> __device__ __forceinline__ v3<T> seed_field(int i)
{
    uint32_t h[3];
    for (int k = 0; k < 3; ++k) {
        uint32_t z = (uint32_t)i * 2654435761u + (uint32_t)k * 40503u + 12345u;
        z ^= z >> 16;
        z *= 2246822519u;
        z ^= z >> 13;
        h[k] = z;
    }
    return mk((T)((int)(h[0] >> 8) - (1 << 23)), (T)((int)(h[1] >> 8) - (1 << 23)), (T)((int)(h[2] >> 8) - (1 << 23)));
}

// part[block] = the largest |component| of v in the block's share (NaN if one
// is).  The start vector is scaled by a power of two near its inverse before
// anything is squared: a start of any size gives the bits of a start of unit
// size, also where squares of FP32 records would under- or overflow.
template <typename T> __global__ void __launch_bounds__(kLzB) k_lz_size(int N, const rec_t<T> *v, double *part)
{
    __shared__ T sh[kLzB / 32];
    wait_prerequisite();
    T m = 0;
    for (int i = blockIdx.x * kLzB + threadIdx.x; i < N; i += gridDim.x * kLzB) {
        const v3<T> a = ldc(v, i);
        m = nan_max(m, nan_max(fabs(a.x), nan_max(fabs(a.y), fabs(a.z))));
    }
    allow_dependents();
    for (int o = 16; o > 0; o >>= 1) m = nan_max(m, shfl_down(m, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kLzB / 32; ++w) m = nan_max(m, sh[w]);
        part[blockIdx.x] = (double)m;
    }
}

// w = start, scaled, projected onto the tangent planes of n (a zero start, by
// the nS partials startS of its size: the fixed pseudo-random field where
// allow_seed), partN its norm, nB_i = n_i . B_i (the Weingarten term of every
// product of the run).
template <typename T>
__global__ void __launch_bounds__(kLzB) k_lz_begin(const __grid_constant__ Stencil<T> S, const rec_t<T> *__restrict__ n,
                                                   const rec_t<T> *start, int allow_seed, const double *startS, int nS,
                                                   rec_t<T> *w, T *nB, double *partN)
{
    __shared__ int s_seed;
    __shared__ T s_scale[2];
    wait_prerequisite();
    if (threadIdx.x < 32) {
        double z = 0;
        for (int p = threadIdx.x; p < nS; p += 32) z = nan_max(z, __ldcg(startS + p));
        for (int o = 16; o > 0; o >>= 1) z = nan_max(z, lz_xor(z, o));
        if (threadIdx.x == 0) {
            s_seed = allow_seed && !(z > 0);
            // in two factors: 2^-e alone can be out of T's range
            const int e = z > 0 && isfinite(z) ? ilogb(z) : 0;
            s_scale[0] = (T)scalbn(1.0, -(e / 2));
            s_scale[1] = (T)scalbn(1.0, -(e - e / 2));
        }
    }
    __syncthreads();
    const bool seed = s_seed;
    const T s0 = s_scale[0], s1 = s_scale[1];
    typename LzAcc<T>::type s{};
    for (int i = blockIdx.x * kLzB + threadIdx.x; i < S.N; i += gridDim.x * kLzB) {
        int b;
        const v3<T> ni = ldc(n, i), vi = seed ? seed_field<T>(i) : s1 * (s0 * ldc(start, i));
        const v3<T> wi = vi - dot(vi, ni) * ni;
        st(w, i, wi);
        nB[i] = dot(ni, local_field(S, n, i, ni, b));
        s = s + lz_dot(wi, wi);
    }
    allow_dependents();
    const double r = block_sum(s);
    if (threadIdx.x == 0) partN[blockIdx.x] = r;
}

// H u for u = scale w, w tangent: -P (sum_j J u_j + u_j x D + 2 K (Kh.u) Kh) + (n.B) u; u: that of spin i
template <typename T>
__device__ __forceinline__ v3<T> lz_product(const Stencil<T> &S, const rec_t<T> *w, int i, v3<T> ni, v3<T> u, T nB,
                                            T scale)
{
    int bs, c0, c1, c2;
    decode_site(S, i, bs, c0, c1, c2);
    const v3<T> kh = mk(S.Kh[bs][0], S.Kh[bs][1], S.Kh[bs][2]);
    v3<T> L = (T(2) * S.K[bs] * dot(kh, u)) * kh;
    auto load = [&](int j) { return sizeof(T) == 4 ? scale * ldg2(w, j) : ldg2(w, j); };  // tangent: no projection here
    for_neighbours(S, i, bs, c0, c1, c2, load,
                   [&](const NbrEntry<T> &E, v3<T> v) {
                       L.x = fma(-v.z, E.Dy, fma(v.y, E.Dz, fma(E.J, v.x, L.x)));
                       L.y = fma(-v.x, E.Dz, fma(v.z, E.Dx, fma(E.J, v.y, L.y)));
                       L.z = fma(-v.y, E.Dx, fma(v.x, E.Dy, fma(E.J, v.z, L.z)));
                   });
    return axpy(nB, u, axpy(dot(L, ni), ni, -L));
}

template <typename T>
__global__ void __launch_bounds__(kLzB) k_lz_apply(const __grid_constant__ Stencil<T> S, const rec_t<T> *__restrict__ n,
                                                   const T *nB, const rec_t<T> *w, rec_t<T> *wn, rec_t<T> *Q, int k,
                                                   double brk, const double *partN, int nN, double *partA, LzRun *run)
{
    __shared__ double s_inv;
    wait_prerequisite();
    if (k && !run->go[k - 1]) return;
    if (threadIdx.x < 32) {
        const double b2 = partial_sum(partN, nN);
        if (threadIdx.x == 0) {
            // the coupling that closes step k - 1: a residual at the rounding
            // level of the stored records (relative to the running estimate of
            // |T|) is an invariant subspace, not a new direction: normalising
            // it would add a dependent vector
            const double b = sqrt(b2);
            double tnorm = 0;
            if (k > 0) tnorm = fabs(run->alpha[k - 1]) + b;
            if (k > 1) tnorm = fmax(run->tnorm[k - 1], tnorm + run->beta[k - 2]);
            const bool go = k ? b > brk * tnorm : b2 > 0 && isfinite(b2);
            s_inv = go ? 1.0 / b : 0.0;
            if (blockIdx.x == 0) {
                if (go) {
                    run->go[k] = 1;
                    run->tnorm[k] = tnorm;
                    if (k) run->beta[k - 1] = b;
                } else if (k == 0) {
                    run->nan_start = !isfinite(b2);
                }
            }
        }
    }
    rec_t<T> *q = Q + (size_t)k * S.N;
    typename LzAcc<T>::type s{};
    int i = blockIdx.x * kLzB + threadIdx.x;
    if constexpr (sizeof(T) == 4) {
        // FP32: the product of the vector as it is stored.  That of the unscaled w
        // (below) is not its product to the last bits, and shows in the mode:
        // 8.5e-7 off (geometric mean of 150 states, 50 x 50, 40 vectors), 7.6e-7
        // with the product of q; 1.02e-6 and 0.91e-6 at 64 x 64 and 64 vectors (128 x
        // 128, 64 vectors: 1.59 ms, and 1.67 for the norm that comes first)
        __syncthreads();
        const T inv = (T)s_inv;
        if (inv == T(0)) return;
        for (; i < S.N; i += gridDim.x * kLzB) {
            const v3<T> qi = inv * ldg2(w, i), r = lz_product(S, w, i, ldc(n, i), qi, nB[i], inv);
            st(q, i, qi);
            st(wn, i, r);
            s = s + lz_dot(qi, r);
        }
    } else {
        // FP64: the product is linear, and is formed from the unscaled w while the
        // norm is being summed
        v3<T> u = mk(T(0), T(0), T(0)), h = u;
        if (i < S.N) {
            u = ldg2(w, i);
            h = lz_product(S, w, i, ldc(n, i), u, nB[i], T(1));
        }
        __syncthreads();
        const T inv = (T)s_inv;
        if (inv == T(0)) return;
        while (i < S.N) {
            const v3<T> qi = inv * u, r = inv * h;
            st(q, i, qi);
            st(wn, i, r);
            s = s + lz_dot(qi, r);
            i += gridDim.x * kLzB;
            if (i >= S.N) break;
            u = ldg2(w, i);
            h = lz_product(S, w, i, ldc(n, i), u, nB[i], T(1));
        }
    }
    allow_dependents();
    const double r = block_sum(s);
    if (threadIdx.x == 0) partA[blockIdx.x] = r;
}

template <typename T>
__global__ void __launch_bounds__(kLzB *kLzG) k_lz_dots(int N, const rec_t<T> *__restrict__ n, rec_t<T> *w,
                                                        const rec_t<T> *Q, int k, int last, const double *partA, int nA,
                                                        double *partD, LzRun *run)
{
    using A = typename LzAcc<T>::type;
    __shared__ double sh[kLzB / 32][kMaxKrylov];
    __shared__ double s_al;
    wait_prerequisite();
    if (!run->go[k]) return;
    if (threadIdx.x < 32) {
        const double al = partial_sum(partA, nA);
        if (threadIdx.x == 0) {
            s_al = al;
            if (blockIdx.x == 0) run->alpha[k] = al;
        }
    }
    __syncthreads();
    if (last) return;  // no vector follows: only the diagonal entry is wanted
    const T a = (T)s_al, be = k ? (T)run->beta[k - 1] : T(0);
    const int lane = threadIdx.x & 31, t = threadIdx.x % kLzB, grp = threadIdx.x / kLzB;
    const rec_t<T> *qk = Q + (size_t)k * N, *qm = k ? qk - N : qk;
    auto three_term = [&](int i) {
        const v3<T> ni = ldc(n, i);
        const v3<T> u = axpy(-be, ldc(qm, i), axpy(-a, ldc(qk, i), ldc((const rec_t<T> *)w, i)));
        return u - dot(u, ni) * ni;
    };
    // every group forms the w of the block's first tile for itself (the first
    // group stores it once all have); further tiles are formed by one group
    // each and read back from memory
    const int stride = gridDim.x * kLzB, i0 = blockIdx.x * kLzB + t;
    v3<T> u = i0 < N ? three_term(i0) : mk(T(0), T(0), T(0));
    for (int i = i0 + stride, c = 1; i < N; i += stride, ++c)
        if (c % kLzG == grp) st(w, i, three_term(i));
    __syncthreads();
    if (grp == 0 && i0 < N) st(w, i0, u);
    for (int j0 = grp * kLzChunk; j0 <= k; j0 += kLzG * kLzChunk) {
        A tot{};
        const int m = min(kLzChunk, k + 1 - j0);
        // whole warps walk the tiles together: a thread past the end adds zeros
        for (int b0 = blockIdx.x * kLzB; b0 < N; b0 += stride) {
            const int i = b0 + t;
            A v[kLzChunk];
            const v3<T> x = b0 == (int)blockIdx.x * kLzB ? u : (i < N ? ldc((const rec_t<T> *)w, i) : mk(T(0), T(0), T(0)));
            const rec_t<T> *qj = Q + (size_t)j0 * N + min(i, N - 1);
            if (m == kLzChunk) {
#pragma unroll
                for (int j = 0; j < kLzChunk; ++j) v[j] = lz_dot(x, ldc(qj, (long)j * N));
            } else {
#pragma unroll
                for (int j = 0; j < kLzChunk; ++j) v[j] = j < m ? lz_dot(x, ldc(qj, (long)j * N)) : A{};
            }
            tot = tot + warp_sums(v);
        }
        if (lane < kLzChunk) sh[t >> 5][j0 + lane] = to_double(tot);
    }
    allow_dependents();
    __syncthreads();
    for (int j = threadIdx.x; j <= k; j += kLzB * kLzG)
        partD[(size_t)blockIdx.x * kMaxKrylov + j] = (sh[0][j] + sh[1][j]) + (sh[2][j] + sh[3][j]);
}
static_assert(kLzB == 128, "k_lz_dots adds four warps' sums");

// w -= sum_j c_j q_j with c_j summed from the nD blocks' partials; or (ritz)
// w = sum_j c_j q_j with the m coefficients given.  Projected, partials of
// |w|^2.
template <typename T>
__global__ void __launch_bounds__(kLzB *kLzG) k_lz_sub(int N, const rec_t<T> *__restrict__ n, rec_t<T> *w,
                                                       const rec_t<T> *Q, int m, const double *partD, int nD,
                                                       const double *ritz, double *partN, const LzRun *run)
{
    __shared__ double c8[8][64];
    __shared__ T cs[kMaxKrylov];
    __shared__ v3<T> part[kLzG - 1][kLzB];
    wait_prerequisite();
    if (!ritz && !run->go[m - 1]) return;
    if (ritz) {
        for (int j = threadIdx.x; j < m; j += kLzB * kLzG) cs[j] = (T)ritz[j];
        __syncthreads();
    } else {
        // 64 vectors at a time: thread (g, j) sums every eighth block's partials of vector j
        for (int j0 = 0; j0 < m; j0 += 64) {
            const int j = threadIdx.x & 63, g = threadIdx.x >> 6;
            if (j0 + j < m) {
                const double *pd = partD + j0 + j;
                double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
                int p = g;
                for (; p + 24 < nD; p += 32) {
                    s0 += __ldcg(pd + (size_t)p * kMaxKrylov);
                    s1 += __ldcg(pd + (size_t)(p + 8) * kMaxKrylov);
                    s2 += __ldcg(pd + (size_t)(p + 16) * kMaxKrylov);
                    s3 += __ldcg(pd + (size_t)(p + 24) * kMaxKrylov);
                }
                for (; p < nD; p += 8) s0 += __ldcg(pd + (size_t)p * kMaxKrylov);
                c8[g][j] = (s0 + s1) + (s2 + s3);
            }
            __syncthreads();
            if (g == 0 && j0 + j < m)
                cs[j0 + j] = (T)-(((c8[0][j] + c8[1][j]) + (c8[2][j] + c8[3][j])) +
                                  ((c8[4][j] + c8[5][j]) + (c8[6][j] + c8[7][j])));
            __syncthreads();
        }
    }
    const int t = threadIdx.x % kLzB, grp = threadIdx.x / kLzB;
    const int per = (m + kLzG - 1) / kLzG, ja = min(m, grp * per), jb = min(m, ja + per);
    typename LzAcc<T>::type s{};
    for (int b0 = blockIdx.x * kLzB; b0 < N; b0 += gridDim.x * kLzB) {
        const int i = b0 + t;
        v3<T> u = mk(T(0), T(0), T(0));
        if (i < N) {
            if (grp == 0 && !ritz) u = ldc((const rec_t<T> *)w, i);
            const rec_t<T> *qi = Q + i;
#pragma unroll 8
            for (int j = ja; j < jb; ++j) u = axpy(cs[j], ldc(qi, (long)j * N), u);
        }
        if (grp) part[grp - 1][t] = u;
        __syncthreads();
        if (grp == 0 && i < N) {
            u = (u + part[0][t]) + (part[1][t] + part[2][t]);
            const v3<T> ni = ldc(n, i);
            u = u - dot(u, ni) * ni;
            st(w, i, u);
            s = s + lz_dot(u, u);
        }
        __syncthreads();
    }
    allow_dependents();
    const double r = block_sum(s);
    if (threadIdx.x == 0) partN[blockIdx.x] = r;
}
static_assert(kLzG == 4, "k_lz_sub adds four groups' sums");

// v *= 1 / |v| (from its norm partials)
template <typename T> __global__ void __launch_bounds__(kLzB) k_lz_unit(int N, rec_t<T> *v, const double *partN, int nN)
{
    __shared__ double s_inv;
    wait_prerequisite();
    if (threadIdx.x < 32) {
        const double s = partial_sum(partN, nN);
        if (threadIdx.x == 0) s_inv = 1.0 / sqrt(s);
    }
    __syncthreads();
    const T inv = (T)s_inv;
    for (int i = blockIdx.x * kLzB + threadIdx.x; i < N; i += gridDim.x * kLzB)
        st(v, i, inv * ldc((const rec_t<T> *)v, i));
}

// F = B - (B.n) n
template <typename T>
__global__ void __launch_bounds__(kHB) k_force(const __grid_constant__ Stencil<T> S, const rec_t<T> *__restrict__ n,
                                               rec_t<T> *__restrict__ F)
{
    int i = blockIdx.x * kHB + threadIdx.x;
    if (i >= S.N) return;
    int b;
    v3<T> ni = ld(n, i);
    v3<T> B = local_field(S, n, i, ni, b);
    st(F, i, B - dot(B, ni) * ni);
}

// y = normalise(x + dt v + dt^2/(2m) Fe)
template <typename T>
__global__ void k_mmf_move(int N, const rec_t<T> *__restrict__ x, const rec_t<T> *__restrict__ v,
                           const rec_t<T> *__restrict__ Fe, rec_t<T> *__restrict__ y, double dt, double dt2_2m)
{
    int i = blockIdx.x * kHB + threadIdx.x;
    if (i >= N) return;
    st(y, i, normalised(axpy((T)dt2_2m, ld(Fe, i), axpy((T)dt, ld(v, i), ld(x, i)))));
}

// v += dt/(2m) (Fe + Fe2)
template <typename T>
__global__ void k_mmf_vel(int N, rec_t<T> *__restrict__ v, const rec_t<T> *__restrict__ Fe,
                          const rec_t<T> *__restrict__ Fe2, double dth_m)
{
    int i = blockIdx.x * kHB + threadIdx.x;
    if (i >= N) return;
    st(v, i, axpy((T)dth_m, ld(Fe, i) + ld(Fe2, i), ld(v, i)));
}

// out = a u + b z (plain records)
template <typename T>
__global__ void k_lin(int N, rec_t<T> *__restrict__ out, double a, const rec_t<T> *__restrict__ u, double b,
                      const rec_t<T> *__restrict__ z)
{
    int i = blockIdx.x * kHB + threadIdx.x;
    if (i >= N) return;
    st(out, i, axpy((T)b, ld(z, i), (T)a * ld(u, i)));
}

// max_i |F_i|
template <typename T>
__global__ void k_maxnorm(int N, const rec_t<T> *__restrict__ F, double *__restrict__ part)
{
    __shared__ double sh[kHB / 32];
    int i = blockIdx.x * kHB + threadIdx.x;
    double v = i < N ? sqrt(ddot(ld(F, i), ld(F, i))) : 0.0;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int w = 0; w < kHB / 32; ++w) s = fmax(s, sh[w]);
        part[blockIdx.x] = s;
    }
}

// Lowest eigenvalue of the symmetric tridiagonal matrix (alpha, beta) by
// bisection on the Sturm count (a negative pivot of T - x I: x lies above the
// lowest eigenvalue), down to adjacent floating-point numbers.  NaN where the
// matrix is not finite.
double tri_lowest(const std::vector<double> &alpha, const std::vector<double> &beta)
{
    const int m = (int)alpha.size();
    double lo = 1e300, hi = 1e300, scale = 0;
    for (int i = 0; i < m; ++i) {
        const double r = (i ? fabs(beta[i - 1]) : 0.0) + (i + 1 < m ? fabs(beta[i]) : 0.0);
        if (!std::isfinite(alpha[i]) || !std::isfinite(r)) return NAN;
        lo = std::min(lo, alpha[i] - r);
        hi = std::min(hi, alpha[i]);  // a diagonal entry bounds it from above
        scale = std::max(scale, fabs(alpha[i]) + r);
    }
    const double pivmin = std::max(1e-300, 1e-290 * scale * scale);
    lo -= 1e-14 * scale;
    for (int it = 0; it < 200; ++it) {
        const double x = 0.5 * (lo + hi);
        if (!(x > lo && x < hi)) break;
        bool above = false;
        double d = 1.0;
        for (int i = 0; i < m && !above; ++i) {
            d = alpha[i] - x - (i ? beta[i - 1] * beta[i - 1] / d : 0.0);
            if (fabs(d) < pivmin) d = -pivmin;
            above = d < 0;
        }
        (above ? hi : lo) = x;
    }
    return 0.5 * (lo + hi);
}

unsigned hblocks(long long n) { return (unsigned)((n + kHB - 1) / kHB); }

template <typename T>
struct Ops {
    const Stencil<T> &S;
    HessScratch &h;
    cudaStream_t st;
    int N;
    unsigned nb;

    rec_t<T> *q(int k) { return (rec_t<T> *)h.Q.p + (size_t)k * N; }

    // a . b, copied to the host
    int dot1(const rec_t<T> *a, const rec_t<T> *b, double *host)
    {
        k_dot<T><<<nb, kHB, 0, st>>>(N, a, b, (double *)h.part.p);
        k_dot_final<<<1, 1, 0, st>>>((const double *)h.part.p, (int)nb, (double *)h.dots.p);
        if (cudaMemcpyAsync(host, h.dots.p, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return SP_ERR_CUDA;
        return 0;
    }

    // Lowest eigenpair of H at n by m Lanczos steps from `start` (allow_seed:
    // a zero start selects a fixed pseudo-random tangent field).  mode
    // receives the unit Ritz vector.  One synchronisation, for the
    // tridiagonal matrix: on return the launches that form the mode are queued.
    int lowest(const rec_t<T> *n, const rec_t<T> *start, bool allow_seed, rec_t<T> *mode, int m, double *lam)
    {
        // the Krylov space cannot outgrow the 2N-dimensional tangent space
        m = (int)std::min<long long>(m, 2LL * N);
        const int nt = (N + kLzB - 1) / kLzB, nS = std::min(nt, kLzSpinBlocks), nD = std::min(nt, kLzBlocks);
        const dim3 gs(nS), bs(kLzB), gd(nD), bd(kLzB * kLzG);
        rec_t<T> *W[2] = {(rec_t<T> *)h.w.p, (rec_t<T> *)h.w2.p};
        T *nB = (T *)h.nB.p;
        double *pN = (double *)h.part.p, *pA = pN + kLzSpinBlocks, *pD = pA + kLzSpinBlocks;
        LzRun *run = (LzRun *)h.run.p;
        const double brk = sizeof(T) == 4 ? 1e-5 : 1e-13;
        if (cudaMemsetAsync(run, 0, sizeof(LzRun), st) != cudaSuccess) return SP_ERR_CUDA;
        // launched plainly: all that was written before the run is in place
        // before any kernel of the run begins
        k_lz_size<T><<<gs, bs, 0, st>>>(N, start, pA);
        cudaError_t e = launch_pdl(k_lz_begin<T>, gs, bs, 0, st, S, n, start, (int)allow_seed, (const double *)pA, nS,
                                   W[0], nB, pN);
        for (int k = 0; k < m && e == cudaSuccess; ++k) {
            rec_t<T> *w = W[(k + 1) & 1];
            e = launch_pdl(k_lz_apply<T>, gs, bs, 0, st, S, n, (const T *)nB, (const rec_t<T> *)W[k & 1], w, q(0), k,
                           brk, (const double *)pN, k ? nD : nS, pA, run);
            if (e == cudaSuccess)
                e = launch_pdl(k_lz_dots<T>, gd, bd, 0, st, N, n, w, (const rec_t<T> *)q(0), k, (int)(k == m - 1),
                               (const double *)pA, nS, pD, run);
            if (e == cudaSuccess && k < m - 1)
                e = launch_pdl(k_lz_sub<T>, gd, bd, 0, st, N, n, w, (const rec_t<T> *)q(0), k + 1, (const double *)pD,
                               nD, (const double *)nullptr, pN, (const LzRun *)run);
        }
        if (e != cudaSuccess ||
            cudaMemcpyAsync(&h.host->run, run, sizeof(LzRun), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return SP_ERR_CUDA;
        const LzRun &r = h.host->run;
        if (!r.go[0]) return r.nan_start ? SP_ERR_NAN : SP_ERR_ARG;
        int used = 0;
        while (used < m && r.go[used]) ++used;
        const std::vector<double> al(r.alpha, r.alpha + used), be(r.beta, r.beta + used);
        *lam = tri_lowest(al, be);
        std::vector<double> y;
        if (std::isfinite(*lam))
            tri_eigenvector(al, be, *lam, y);
        else
            y.assign(used, NAN);
        std::copy(y.begin(), y.end(), h.host->y);
        if (cudaMemcpyAsync(h.coef.p, h.host->y, sizeof(double) * used, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return SP_ERR_CUDA;
        e = launch_pdl(k_lz_sub<T>, gd, bd, 0, st, N, n, mode, (const rec_t<T> *)q(0), used, (const double *)pD, nD,
                       (const double *)h.coef.p, pN, (const LzRun *)run);
        if (e == cudaSuccess) e = launch_pdl(k_lz_unit<T>, gs, bs, 0, st, N, mode, (const double *)pN, nD);
        return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : SP_ERR_CUDA;
    }

    // F, the lowest mode (warm-started from `mode`, updated) and Fe at x
    int effective(const rec_t<T> *x, rec_t<T> *F, rec_t<T> *mode, bool allow_seed, rec_t<T> *Fe, int m, double *lam)
    {
        k_force<T><<<nb, kHB, 0, st>>>(S, x, F);
        int rc = lowest(x, mode, allow_seed, mode, m, lam);
        if (rc) return rc;
        double fl;
        if ((rc = dot1(F, mode, &fl))) return rc;
        if (*lam < 0)
            k_lin<T><<<nb, kHB, 0, st>>>(N, Fe, 1.0, F, -2.0 * fl, mode);
        else
            k_lin<T><<<nb, kHB, 0, st>>>(N, Fe, 0.0, F, -fl, mode);
        return cudaGetLastError() == cudaSuccess ? 0 : SP_ERR_CUDA;
    }
};

template <typename T>
int setup(sp_ctx *c, int m)
{
    HessScratch *&h = c->hess;
    if (!h) h = new HessScratch;
    size_t rec = sizeof(rec_t<T>) * (size_t)c->N;
    unsigned nb = hblocks(c->N);
    // partials: per block a norm, an alpha and kMaxKrylov dot products of the
    // Lanczos kernels, or one dot product or maximum per block of kHB spins
    size_t part = sizeof(double) * std::max<size_t>(nb, 2 * kLzSpinBlocks + (size_t)kLzBlocks * kMaxKrylov);
    if (grow_h(h->Q, rec * m) || grow_h(h->w, rec) || grow_h(h->w2, rec) || grow_h(h->nB, sizeof(T) * (size_t)c->N) ||
        grow_h(h->part, part) || grow_h(h->dots, sizeof(double)) || grow_h(h->run, sizeof(LzRun)) ||
        grow_h(h->coef, sizeof(double) * kMaxKrylov))
        return SP_ERR_CUDA;
    if (!h->host && cudaMallocHost(&h->host, sizeof(LzHost)) != cudaSuccess) {
        h->host = nullptr;
        return SP_ERR_CUDA;
    }
    return 0;
}

template <typename T>
int lowest_mode_run(sp_ctx *c, const Stencil<T> &S, const void *n, void *mode, int m, double *lam, cudaStream_t st)
{
    int rc = setup<T>(c, m);
    if (rc) return rc;
    Ops<T> op{S, *c->hess, st, c->N, hblocks(c->N)};
    rec_t<T> *md = (rec_t<T> *)mode;
    if ((rc = op.lowest((const rec_t<T> *)n, md, true, md, m, lam))) return rc;
    // the launches that form the mode read the context's scratch, and the next
    // call may come on another stream
    return cudaStreamSynchronize(st) == cudaSuccess ? 0 : SP_ERR_CUDA;
}

template <typename T>
int mmf_run(sp_ctx *c, const Stencil<T> &S, void *n, void *vel, void *mode, const sp_mmf_params *p, int n_iter,
            double *max_force, double *lam, cudaStream_t st)
{
    int rc = setup<T>(c, p->krylov);
    if (rc) return rc;
    HessScratch &h = *c->hess;
    const size_t rec = sizeof(rec_t<T>) * (size_t)c->N;
    if (grow_h(h.F, rec) || grow_h(h.Fe, rec) || grow_h(h.F2, rec) || grow_h(h.Fe2, rec) || grow_h(h.y, rec))
        return SP_ERR_CUDA;
    Ops<T> op{S, h, st, c->N, hblocks(c->N)};
    int N = c->N;
    rec_t<T> *x = (rec_t<T> *)n, *v = (rec_t<T> *)vel, *md = (rec_t<T> *)mode;
    rec_t<T> *F = (rec_t<T> *)h.F.p, *Fe = (rec_t<T> *)h.Fe.p, *F2 = (rec_t<T> *)h.F2.p, *Fe2 = (rec_t<T> *)h.Fe2.p,
             *y = (rec_t<T> *)h.y.p;
    double dth_m = p->dt / (2.0 * p->mass), dt2_2m = p->dt * p->dt / (2.0 * p->mass);
    if ((rc = op.effective(x, F, md, true, Fe, p->krylov, lam))) return rc;
    for (int it = 0; it < n_iter; ++it) {
        k_mmf_move<T><<<op.nb, kHB, 0, st>>>(N, x, v, Fe, y, p->dt, dt2_2m);
        if ((rc = op.effective(y, F2, md, false, Fe2, p->krylov, lam))) return rc;
        k_mmf_vel<T><<<op.nb, kHB, 0, st>>>(N, v, Fe, Fe2, dth_m);
        double vf, ff;
        if ((rc = op.dot1(v, Fe2, &vf)) || (rc = op.dot1(Fe2, Fe2, &ff))) return rc;
        double cpr = (vf > 0 && ff > 0) ? vf / ff : 0.0;
        k_lin<T><<<op.nb, kHB, 0, st>>>(N, v, 0.0, v, cpr, Fe2);
        if (cudaMemcpyAsync(x, y, sizeof(rec_t<T>) * (size_t)N, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(F, F2, sizeof(rec_t<T>) * (size_t)N, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(Fe, Fe2, sizeof(rec_t<T>) * (size_t)N, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            return SP_ERR_CUDA;
    }
    k_maxnorm<T><<<op.nb, kHB, 0, st>>>(N, F, (double *)h.part.p);
    std::vector<double> pm(op.nb);
    if (cudaMemcpyAsync(pm.data(), h.part.p, sizeof(double) * op.nb, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SP_ERR_CUDA;
    *max_force = *std::max_element(pm.begin(), pm.end());
    return 0;
}

int hfail(sp_ctx *c, int code, const char *msg)
{
    c->err = msg;
    return code;
}

int hcheck(sp_ctx *c)
{
    if (!c) return SP_ERR_ARG;
    if (!c->have_geom || !c->have_ham) return hfail(c, SP_ERR_STATE, "context not configured");
    if (c->h.dipole != SP_DIPOLE_NONE) return hfail(c, SP_ERR_UNSUPPORTED, "Hessian with the dipole term");
    return status_enter(c);
}

// Device record arrays start on a record boundary (16 B in FP32, 32 B in FP64).
bool hrecords_aligned(const sp_ctx *c, std::initializer_list<const void *> ptrs)
{
    const uintptr_t a = c->prec == SP_F64 ? 32 : 16;
    for (const void *p : ptrs)
        if ((uintptr_t)p % a) return false;
    return true;
}

}  // namespace

namespace spgb {
template <typename T>
cudaError_t launch_hvp(const Stencil<T> &S, const rec_t<T> *n, const rec_t<T> *v, rec_t<T> *out, cudaStream_t st)
{
    if (S.N <= 0) return cudaSuccess;
    k_hvp<T><<<hblocks(S.N), kHB, 0, st>>>(S, n, v, out);
    return cudaGetLastError();
}
template cudaError_t launch_hvp<float>(const Stencil<float> &, const float4 *, const float4 *, float4 *, cudaStream_t);
template cudaError_t launch_hvp<double>(const Stencil<double> &, const dq4 *, const dq4 *, dq4 *, cudaStream_t);
}  // namespace spgb

void hess_scratch_destroy(HessScratch *h)
{
    if (!h) return;
    DevBuf *bufs[] = {&h->Q, &h->w, &h->w2, &h->F, &h->Fe, &h->F2, &h->Fe2, &h->y, &h->nB, &h->part, &h->dots,
                      &h->run, &h->coef};
    for (DevBuf *b : bufs)
        if (b->p) cudaFree(b->p);
    if (h->host) cudaFreeHost(h->host);
    delete h;
}

extern "C" {

int sp_hessian_apply(sp_ctx *c, const void *n_dev, const void *v_dev, void *out_dev, void *stream)
{
    int rc = hcheck(c);
    if (rc) return rc;
    if (!n_dev || !v_dev || !out_dev) return hfail(c, SP_ERR_ARG, "NULL argument");
    if (v_dev == out_dev) return hfail(c, SP_ERR_ARG, "v and out must differ");
    if (!hrecords_aligned(c, {n_dev, v_dev, out_dev})) return hfail(c, SP_ERR_ARG, "misaligned record array");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned nb = hblocks(c->N);
    unsigned *w = status_word(c);
    if (!w) return hfail(c, SP_ERR_CUDA, "status word");
    cudaError_t e = c->prec == SP_F64 ? launch_pdl(k_hvp<double>, dim3(nb), dim3(kHB), 0, st, c->Sd, (const dq4 *)n_dev,
                                                   (const dq4 *)v_dev, (dq4 *)out_dev, w)
                                      : launch_pdl(k_hvp<float>, dim3(nb), dim3(kHB), 0, st, c->Sf,
                                                   (const float4 *)n_dev, (const float4 *)v_dev, (float4 *)out_dev, w);
    if (e != cudaSuccess) return hfail(c, SP_ERR_CUDA, "Hessian launch failed");
    return SP_OK;
}

int sp_lowest_mode(sp_ctx *c, const void *n_dev, void *mode_dev, int krylov, double *lambda, void *stream)
{
    int rc = hcheck(c);
    if (rc) return rc;
    if (!n_dev || !mode_dev || !lambda) return hfail(c, SP_ERR_ARG, "NULL argument");
    if (krylov < 1 || krylov > kMaxKrylov) return hfail(c, SP_ERR_ARG, "krylov must be in 1..256");
    if (!hrecords_aligned(c, {n_dev, mode_dev})) return hfail(c, SP_ERR_ARG, "misaligned record array");
    cudaStream_t st = (cudaStream_t)stream;
    rc = c->prec == SP_F64 ? lowest_mode_run<double>(c, c->Sd, n_dev, mode_dev, krylov, lambda, st)
                           : lowest_mode_run<float>(c, c->Sf, n_dev, mode_dev, krylov, lambda, st);
    if (rc == SP_ERR_NAN) return hfail(c, rc, "lowest mode: a non-finite value in the state or the start vector");
    if (rc) return hfail(c, rc, "Lanczos failed");
    return std::isfinite(*lambda) ? SP_OK : hfail(c, SP_ERR_NAN, "lowest mode: the eigenvalue is not finite");
}

int sp_mmf(sp_ctx *c, void *n_dev, void *vel_dev, void *mode_dev, const sp_mmf_params *p, int n_iter,
           double *max_force, double *lambda, void *stream)
{
    int rc = hcheck(c);
    if (rc) return rc;
    if (!n_dev || !vel_dev || !mode_dev || !p || !max_force || !lambda) return hfail(c, SP_ERR_ARG, "NULL argument");
    if (!(p->dt > 0) || !(p->mass > 0) || p->krylov < 1 || p->krylov > kMaxKrylov || n_iter < 0)
        return hfail(c, SP_ERR_ARG, "bad MMF parameters");
    if (!hrecords_aligned(c, {n_dev, vel_dev, mode_dev})) return hfail(c, SP_ERR_ARG, "misaligned record array");
    cudaStream_t st = (cudaStream_t)stream;
    rc = c->prec == SP_F64 ? mmf_run<double>(c, c->Sd, n_dev, vel_dev, mode_dev, p, n_iter, max_force, lambda, st)
                           : mmf_run<float>(c, c->Sf, n_dev, vel_dev, mode_dev, p, n_iter, max_force, lambda, st);
    if (rc == SP_ERR_NAN) return hfail(c, rc, "minimum mode following: a non-finite value");
    if (rc) return hfail(c, rc, "minimum mode following failed");
    return std::isfinite(*max_force) && std::isfinite(*lambda)
               ? SP_OK
               : hfail(c, SP_ERR_NAN, "minimum mode following: the force or eigenvalue is not finite");
}

}  // extern "C"
