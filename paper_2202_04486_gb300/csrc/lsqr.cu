// Full-gradient MDD by LSQR (Paige & Saunders 1982), the baseline the paper compares stochastic MDD
// against: every source at once, on the preconditioned operator A = P C (Eq. 3-4).
//
// The vectors are FP32 device arrays, every norm is reduced in a fixed order to FP64 accuracy (runs of a thread's
// elements in FP32 words that are no less exact, SumSq; then threads, blocks and one block over them in FP64), and
// the scalar recurrence of the bidiagonalisation and of the plane rotations runs on the device (one thread), so an
// iteration is a fixed sequence of launches with no host round trip.  The operator's forward and adjoint are the plan's own kernels with nb = ns.
#include <cmath>
#include <cstring>

#include "smdd_fft.cuh"
#include "smdd_internal.h"

namespace smdd {

namespace {

constexpr int VEC_THREADS = 256;
constexpr int VEC_BLOCKS = 2 * 152;   // a multiple of the SM count; grid-stride loops

// LSQR scalars (device)
struct LsqrScalars {
    double alpha, beta, rho_bar, phi_bar;
    double cx, cw;        // x += cx w;  w = v - cw w
    double inv;           // 1 / (the norm just reduced), 0 for a zero vector
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Element-wise passes.  Four elements per thread and access where every vector is 16-byte aligned (a tail and
// unaligned vectors element by element), and the norm of what a pass writes in the same pass: one FP64 partial of the
// sum of squares per block (fixed assignment of elements to blocks and threads).
//
// A thread's share of a long vector has hundreds of squares in each half of its FP32 pair, so the sum in the pair goes
// to the FP64 sum after the NORM_RUN groups (eight squares a half and group) that SumSq takes, and when a larger value
// than its bound comes.  Groups of 16 elements, whose loads are all issued before the first is used: one range check a
// group, and the loads do not wait for the sum of the elements before (with groups of 4: +38 us a pass at 4.6e7 elements).
constexpr int NORM_GROUP = 4;   // accesses of four elements
constexpr int NORM_RUN = SumSq::SQUARES / (2 * NORM_GROUP);

struct NormSum {
    SumSq q{0.f};
    float bound = 0.f;
    double d = 0.0;
    int run = 0;
    __device__ __forceinline__ void add(const float4 (&v)[NORM_GROUP]) {
        float top = 0.f;
#pragma unroll
        for (int u = 0; u < NORM_GROUP; ++u)
            top = fmaxf(top, fmaxf(fmaxf(fabsf(v[u].x), fabsf(v[u].y)), fmaxf(fabsf(v[u].z), fabsf(v[u].w))));
        if (SumSq::in_range(top)) {   // (a NaN passes and reaches the sum)
            if (run == NORM_RUN || SumSq::pow2(top) > bound) {
                d += q.total();
                bound = fmaxf(bound, SumSq::pow2(top));
                q = SumSq(bound);
                run = 0;
            }
            ++run;
#pragma unroll
            for (int u = 0; u < NORM_GROUP; ++u) {
                q.add(pk2(v[u].x, v[u].y));
                q.add(pk2(v[u].z, v[u].w));
            }
        } else {
#pragma unroll
            for (int u = 0; u < NORM_GROUP; ++u)
                d += (double)v[u].x * v[u].x + (double)v[u].y * v[u].y + (double)v[u].z * v[u].z + (double)v[u].w * v[u].w;
        }
    }
    __device__ __forceinline__ double total() const { return q.total() + d; }
};

__device__ __forceinline__ void block_partial(double s, double *partials) {
    __shared__ double red[VEC_THREADS / 32];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < VEC_THREADS / 32; ++w) t += red[w];
        partials[blockIdx.x] = t;
    }
}

// y = t - coef y (coef: alpha or beta of the scalars, or 1, by `which` = 0, 1, 2; 3: y = t), t muted, and the partials
// of sum(y^2)
__global__ void __launch_bounds__(VEC_THREADS) k_combine_norm(float *__restrict__ y, const float *__restrict__ t, long long n, int vec,
                                                                const LsqrScalars *sc, int which, const int32_t *__restrict__ mute,
                                                                int nt, double *__restrict__ partials) {
    const float cf = which == 0 ? (float)sc->alpha : which == 1 ? (float)sc->beta : 1.f;
    const long long first = blockIdx.x * (long long)VEC_THREADS + threadIdx.x, step = (long long)gridDim.x * VEC_THREADS;
    NormSum sum;
    auto muted = [&](float x, long long i) { return (mute && (int)(i % nt) < mute[i / nt]) ? 0.f : x; };
    const long long n4 = vec ? n / 4 : 0;
    for (long long i = first; i < n4; i += NORM_GROUP * step) {
        float4 a[NORM_GROUP], b[NORM_GROUP];
#pragma unroll
        for (int u = 0; u < NORM_GROUP; ++u) {
            const long long j = i + u * step;
            a[u] = b[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < n4) {
                a[u] = reinterpret_cast<const float4 *>(t)[j];
                if (which < 3) b[u] = reinterpret_cast<const float4 *>(y)[j];
            }
        }
#pragma unroll
        for (int u = 0; u < NORM_GROUP; ++u) {
            const long long j = i + u * step;
            if (j >= n4) continue;
            if (mute) a[u] = make_float4(muted(a[u].x, 4 * j), muted(a[u].y, 4 * j + 1), muted(a[u].z, 4 * j + 2), muted(a[u].w, 4 * j + 3));
            if (which < 3) a[u] = make_float4(a[u].x - cf * b[u].x, a[u].y - cf * b[u].y, a[u].z - cf * b[u].z, a[u].w - cf * b[u].w);
            reinterpret_cast<float4 *>(y)[j] = a[u];
        }
        sum.add(a);
    }
    for (long long i = 4 * n4 + first; i < n; i += NORM_GROUP * step) {   // the tail, or unaligned vectors
        float a[NORM_GROUP];
        float4 g[NORM_GROUP];
#pragma unroll
        for (int u = 0; u < NORM_GROUP; ++u) a[u] = i + u * step < n ? t[i + u * step] : 0.f;
#pragma unroll
        for (int u = 0; u < NORM_GROUP; ++u) {
            const long long j = i + u * step;
            if (j < n) {
                a[u] = muted(a[u], j);
                if (which < 3) a[u] = a[u] - cf * y[j];
                y[j] = a[u];
            }
            g[u] = make_float4(a[u], 0.f, 0.f, 0.f);
        }
        sum.add(g);
    }
    block_partial(sum.total(), partials);
}

// the norm from the partials (summed in a fixed order), then the scalar step `what`:
//   0: beta_1 = ||u||, phi_bar = beta                       (start)
//   1: alpha_1 = ||v||, rho_bar = alpha                     (start)
//   2: beta = ||u||                                          (iteration, after u = A v - alpha u)
//   3: alpha = ||v||, then the plane rotation; norms[it] = phi_bar   (iteration, after v = A^T u - beta v)
constexpr int NORM_THREADS = 256;

__global__ void __launch_bounds__(NORM_THREADS) k_norm_step(const double *__restrict__ partials, int nparts, LsqrScalars *sc, int what,
                                                              double *norms, int it) {
    __shared__ double red[NORM_THREADS / 32];
    double t = 0.0;
    for (int b = threadIdx.x; b < nparts; b += NORM_THREADS) t += partials[b];
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x != 0) return;
    t = 0.0;
    for (int w = 0; w < NORM_THREADS / 32; ++w) t += red[w];
    const double nrm = sqrt(t);
    sc->inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
    if (what == 0) {
        sc->beta = nrm;
        sc->phi_bar = nrm;
        if (norms) norms[0] = nrm;
    } else if (what == 1) {
        sc->alpha = nrm;
        sc->rho_bar = nrm;
    } else if (what == 2) {
        sc->beta = nrm;
    } else {
        sc->alpha = nrm;
        const double rho = hypot(sc->rho_bar, sc->beta);
        const double c = rho > 0.0 ? sc->rho_bar / rho : 0.0, s = rho > 0.0 ? sc->beta / rho : 0.0;
        const double theta = s * nrm;
        const double phi = c * sc->phi_bar;
        sc->rho_bar = -c * nrm;
        sc->phi_bar = s * sc->phi_bar;
        sc->cx = rho > 0.0 ? phi / rho : 0.0;
        sc->cw = rho > 0.0 ? theta / rho : 0.0;
        if (norms) norms[it] = sc->phi_bar;
    }
}

// a *= inv (the reciprocal of the last norm), and a copy to w (or null)
__global__ void __launch_bounds__(VEC_THREADS) k_scale_inv(float *__restrict__ a, float *__restrict__ w, long long n, const LsqrScalars *sc) {
    const float inv = (float)sc->inv;
    const long long first = blockIdx.x * (long long)VEC_THREADS + threadIdx.x, step = (long long)gridDim.x * VEC_THREADS;
    for (long long i = first; i < n / 4; i += step) {
        float4 v = reinterpret_cast<const float4 *>(a)[i];
        v = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
        reinterpret_cast<float4 *>(a)[i] = v;
        if (w) reinterpret_cast<float4 *>(w)[i] = v;
    }
    for (long long i = (n & ~3LL) + first; i < n; i += step) {
        a[i] *= inv;
        if (w) w[i] = a[i];
    }
}

// v *= inv; then x += cx w; w = v - cw w   (the normalisation of v fused with the solution update)
__global__ void __launch_bounds__(VEC_THREADS) k_update_xw(float *__restrict__ x, float *__restrict__ w, float *__restrict__ v,
                                                             long long n, int vec, const LsqrScalars *sc) {
    const float inv = (float)sc->inv, cx = (float)sc->cx, cw = (float)sc->cw;
    const long long first = blockIdx.x * (long long)VEC_THREADS + threadIdx.x, step = (long long)gridDim.x * VEC_THREADS;
    auto one = [&](float &xv, float &wv, float &vv) {
        vv *= inv;
        xv = fmaf(cx, wv, xv);
        wv = fmaf(-cw, wv, vv);
    };
    const long long n4 = vec ? n / 4 : 0;
    for (long long i = first; i < n4; i += step) {
        float4 a = reinterpret_cast<const float4 *>(x)[i], b = reinterpret_cast<const float4 *>(w)[i], c = reinterpret_cast<const float4 *>(v)[i];
        one(a.x, b.x, c.x);
        one(a.y, b.y, c.y);
        one(a.z, b.z, c.z);
        one(a.w, b.w, c.w);
        reinterpret_cast<float4 *>(x)[i] = a;
        reinterpret_cast<float4 *>(w)[i] = b;
        reinterpret_cast<float4 *>(v)[i] = c;
    }
    for (long long i = 4 * n4 + first; i < n; i += step) one(x[i], w[i], v[i]);
}

}  // namespace

LsqrWork::~LsqrWork() { release(); }

void LsqrWork::release() {
    cudaFree(u);
    cudaFree(t);
    cudaFree(v);
    cudaFree(w);
    cudaFree(g);
    cudaFree(idx);
    cudaFree(partials);
    cudaFree(scalars);
    u = t = v = w = g = nullptr;
    idx = nullptr;
    partials = nullptr;
    scalars = nullptr;
    nd = nm = 0;
}

cudaError_t LsqrWork::ensure(long long n_data, long long n_model, int ns) {
    if (u && n_data == nd && n_model == nm) return cudaSuccess;
    release();
    cudaError_t e;
    if ((e = cudaMalloc(&u, n_data * sizeof(float))) || (e = cudaMalloc(&t, n_data * sizeof(float))) ||
        (e = cudaMalloc(&v, n_model * sizeof(float))) || (e = cudaMalloc(&w, n_model * sizeof(float))) ||
        (e = cudaMalloc(&g, n_model * sizeof(float))) || (e = cudaMalloc(&idx, ns * sizeof(int32_t))) ||
        (e = cudaMalloc(&partials, VEC_BLOCKS * sizeof(double))) || (e = cudaMalloc(&scalars, sizeof(LsqrScalars)))) {
        release();
        return e;
    }
    nd = n_data;
    nm = n_model;
    return cudaSuccess;
}

// The LSQR iteration; apply_fwd(x, out) and apply_adj(r, out) launch the plan's operator (all
// sources; the adjoint with the reciprocity projection when asked), mute is the causality table or null.
cudaError_t lsqr_run(LsqrWork &wk, float *x, const float *b, long long nd, long long nm, int nt, int n_iter,
                     const int32_t *mute, double *norms, cudaStream_t st, const OperatorFn &apply_fwd,
                     const OperatorFn &apply_adj, long long *launches) {
    LsqrScalars *sc = reinterpret_cast<LsqrScalars *>(wk.scalars);
    long long nl = 0;
    const auto aligned = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 ? 1 : 0; };
    // y = t - coef y (or y = t) with its norm, and the scalar step `what`
    auto combine = [&](float *y, const float *t, long long n, int which, const int32_t *m, int what, int it) {
        k_combine_norm<<<VEC_BLOCKS, VEC_THREADS, 0, st>>>(y, t, n, aligned(y) && aligned(t), sc, which, m, nt, wk.partials);
        k_norm_step<<<1, NORM_THREADS, 0, st>>>(wk.partials, VEC_BLOCKS, sc, what, norms, it);
        nl += 2;
        return cudaGetLastError();
    };
    cudaError_t e;
    // u = b - A x0; beta = ||u||; u /= beta
    if ((e = apply_fwd(x, wk.u))) return e;
    if ((e = combine(wk.u, b, nd, 2, nullptr, 0, 0))) return e;
    k_scale_inv<<<VEC_BLOCKS, VEC_THREADS, 0, st>>>(wk.u, nullptr, nd, sc);
    ++nl;
    // v = C A^T u; alpha = ||v||; v /= alpha; w = v
    if ((e = apply_adj(wk.u, wk.g))) return e;
    if ((e = combine(wk.v, wk.g, nm, 3, mute, 1, 0))) return e;
    k_scale_inv<<<VEC_BLOCKS, VEC_THREADS, 0, st>>>(wk.v, wk.w, nm, sc);
    ++nl;
    for (int it = 1; it <= n_iter; ++it) {
        // u = A v - alpha u; beta = ||u||; u /= beta
        if ((e = apply_fwd(wk.v, wk.t))) return e;
        if ((e = combine(wk.u, wk.t, nd, 0, nullptr, 2, it))) return e;
        k_scale_inv<<<VEC_BLOCKS, VEC_THREADS, 0, st>>>(wk.u, nullptr, nd, sc);
        ++nl;
        // v = C A^T u - beta v; alpha = ||v||; rotation; v /= alpha; x, w updates
        if ((e = apply_adj(wk.u, wk.g))) return e;
        if ((e = combine(wk.v, wk.g, nm, 1, mute, 3, it))) return e;
        k_update_xw<<<VEC_BLOCKS, VEC_THREADS, 0, st>>>(x, wk.w, wk.v, nm, aligned(x), sc);
        ++nl;
    }
    if (launches) *launches += nl;
    return cudaGetLastError();
}

}  // namespace smdd
