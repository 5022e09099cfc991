// Trace-parallel FFT kernels of the MDC hot path: model / residual / kernel spectra (rfft), the
// residual step (inverse FFT, causal window, subtraction of the observed data, loss to FP64 accuracy, forward FFT),
// the SGD update (inverse FFT of the gradient spectrum, window, X <- X - alpha g, optional forward FFT
// of the new model) and plain inverse transforms for the operator outputs.
//
// Appendix A: MDC = FFT along time -> batched per-frequency products -> inverse FFT.  The causal
// window keeps t in [0, nt) of the length-N result; with N >= 2 nt - 1 this equals the linear
// convolution (forward) and the linear cross-correlation at non-negative lags (adjoint, Eq. 6).
//
// Memory behaviour: a CTA owns TR traces whose spectra are adjacent along the contiguous axis; its threads
// read and write the bins of those traces straight from the edge passes of the FFT (smdd_fft.cuh): 8 traces x
// SPEC_F bins are 256 contiguous bytes (smdd_internal.h), all loads of a thread are issued together.
// Time-domain inputs needed after an inverse FFT (the model for the update, the observed data for the
// residual) are loaded into registers before its middle passes, so their latency overlaps them (after the inverse
// where the registers do not reach, Team::LATE).
//
// This header holds the device code and the per-length launchers FftLaunch<M>; each complex length M is
// instantiated in a translation unit of its own (fft_m*.cu) so the library compiles in parallel, and
// fft_kernels.cu dispatches on M at run time.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "smdd_fft.cuh"
#include "smdd_internal.h"
#include "work_queue.cuh"

namespace smdd {

struct TileCoord {
    int i, j;
    bool valid;
};

// trace tr of tile bid of the grid (blockIdx.x in a plain launch, the dequeued tile in a work-queue launch)
template <int M>
__device__ __forceinline__ TileCoord coord_of(const TraceGrid &g, int tr, int bid) {
    constexpr int TR = Team<M>::TR;
    const int ti = 1 << g.ti_log2;
    const int tj = TR >> g.ti_log2;
    const int ntile_i = (g.ni + ti - 1) / ti;
    const int bi = bid % ntile_i, bj = bid / ntile_i;
    TileCoord c;
    c.i = bi * ti + (tr & (ti - 1));
    c.j = bj * tj + (tr >> g.ti_log2);
    c.valid = c.i < g.ni && c.j < g.nj;
    return c;
}

// Upper enumeration of a square grid (TraceGrid::sym): tile number bid -> the number of the same tile in
// the full enumeration (bi + nbi j).  Rows j = TR g .. TR g + TR - 1 form group g, each row holding the
// tiles bi = g .. nbi - 1, so group g starts at G(g) = TR (g nbi - g (g - 1) / 2).
__host__ __device__ __forceinline__ int sym_tile_to_full(const TraceGrid &g, int TR, int bid) {
    const int nbi = (g.ni + TR - 1) / TR;
    auto G = [&](long long q) { return (long long)TR * (q * nbi - q * (q - 1) / 2); };
    const float h = nbi + 0.5f;
    int q = (int)(h - sqrtf(fmaxf(h * h - 2.f * (float)bid / (float)TR, 0.f)));
    q = q < 0 ? 0 : (q > nbi - 1 ? nbi - 1 : q);
    while (q > 0 && G(q) > bid) --q;
    while (q + 1 < nbi && G(q + 1) <= bid) ++q;
    const int off = (int)(bid - G(q)), w = nbi - q;
    const int j = q * TR + off / w, bi = q + off % w;
    return j * nbi + bi;
}

// The two traces of a thread's pair, its place in the group, and its shared-memory buffer.
template <int M>
struct PairCtx {
    int s;              // thread of the pair: 0 .. T - 1
    TileCoord c[2];     // traces A, B
    float4 *buf;
};

template <int M>
__device__ __forceinline__ PairCtx<M> pair_ctx(const TraceGrid &g, int bid) {
    using TM = Team<M>;
    extern __shared__ __align__(16) float4 fft_smem[];
    const int p = threadIdx.x % TM::PL, grp = TM::G == 1 ? 0 : threadIdx.x / TM::GT;
    PairCtx<M> x;
    x.s = (threadIdx.x / TM::PL) % TM::T;
    const int tr = grp * 2 * TM::PL + 2 * p;
    x.c[0] = coord_of<M>(g, tr, bid);
    x.c[1] = coord_of<M>(g, tr + 1, bid);
    x.buf = fft_smem + grp * (TM::ELEMS * TM::PL) + p;
    return x;
}

// The pair's traces are adjacent along the contiguous spectrum axis and 16-byte aligned (rows have an even
// length): one 16-byte access per bin (a grid with a single trace along i takes two 8-byte accesses).
__device__ __forceinline__ bool pair_io(const TraceGrid &g) { return g.ti_log2 >= 1; }

// bin 0 of a trace
__device__ __forceinline__ long long spec_trace(const TraceGrid &g, const TileCoord &c) {
    return (((long long)(c.i >> 3) << (3 + g.fl2)) + (c.i & 7)) + (long long)c.j * g.ssj;
}
// bin f of a trace relative to its bin 0
__device__ __forceinline__ long long spec_at(const TraceGrid &g, int f) {
    return (long long)(f >> g.fl2) * g.ssf + ((f & ((1 << g.fl2) - 1)) << 3);
}

__device__ __forceinline__ C2 join(float2 a, float2 b) { return C2{pk2(a.x, b.x), pk2(a.y, b.y)}; }

// bins f0 + r fs (r < 8) of the pair; a trace outside the grid reads as zero (its neighbour's 16-byte access
// covers the padding column of the spectra, which is dropped)
template <int M>
__device__ __forceinline__ void bins_load(C2 (&z)[8], const float2 *__restrict__ spec, const TraceGrid &g, const PairCtx<M> &x,
                                          int f0, int fs) {
    const float2 *a = spec + spec_trace(g, x.c[0]) + spec_at(g, f0);
    const long long st = spec_at(g, fs);   // fs is a multiple of the bins of a block
    if (pair_io(g)) {
        float4 v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r)
            v[r] = x.c[0].valid ? __ldcs(reinterpret_cast<const float4 *>(a + r * st)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int r = 0; r < 8; ++r)
            z[r] = join(make_float2(v[r].x, v[r].y), x.c[1].valid ? make_float2(v[r].z, v[r].w) : make_float2(0.f, 0.f));
    } else {
        const float2 *b = spec + spec_trace(g, x.c[1]) + spec_at(g, f0);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float2 va = x.c[0].valid ? __ldcs(a + r * st) : make_float2(0.f, 0.f);
            const float2 vb = x.c[1].valid ? __ldcs(b + r * st) : make_float2(0.f, 0.f);
            z[r] = join(va, vb);
        }
    }
}

template <int M>
__device__ __forceinline__ void bins_store(const C2 (&z)[8], float2 *__restrict__ spec, const TraceGrid &g, const PairCtx<M> &x,
                                           int f0, int fs) {
    float2 *a = spec + spec_trace(g, x.c[0]) + spec_at(g, f0);
    const long long st = spec_at(g, fs);
    if (pair_io(g) && x.c[1].valid) {   // (the first trace of a pair is valid if the second is)
#pragma unroll
        for (int r = 0; r < 8; ++r)
            *reinterpret_cast<float4 *>(a + r * st) = make_float4(lo2(z[r].re), lo2(z[r].im), hi2(z[r].re), hi2(z[r].im));
    } else {
        float2 *b = spec + spec_trace(g, x.c[1]) + spec_at(g, f0);
        if (x.c[0].valid) {
#pragma unroll
            for (int r = 0; r < 8; ++r) a[r * st] = make_float2(lo2(z[r].re), lo2(z[r].im));
        }
        if (x.c[1].valid) {
#pragma unroll
            for (int r = 0; r < 8; ++r) b[r * st] = make_float2(hi2(z[r].re), hi2(z[r].im));
        }
    }
}

template <int M>
__device__ __forceinline__ long long time_off(const TraceGrid &g, const TileCoord &c) {
    return c.valid ? (long long)c.i * g.tsi + (long long)c.j * g.tsj : 0;
}

__device__ __forceinline__ void bulk_prefetch_l2(const void *p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

// The spectra of tile bid + `ahead` (the CTAs resident on the GPU, so about the tile that starts when this one ends)
// into L2, 256 contiguous bytes of four bins at a time, while this tile is transformed.  Only for 256 <= M <= 512 and whole tiles of
// 8 columns: update 432 -> 409 us at nt 512, 400 x 400, 478 -> 462 us at nt 256, 600 x 600; at M = 1024 and 1536, whose tiles
// take longer, 1 % slower to 5 % faster by shape, at M = 128 no change.
template <int M>
constexpr bool prefetches() { return M >= 256 && M <= 512; }
template <int M>
__device__ __forceinline__ void tile_prefetch(const FftArgs &a, int bid) {
    if ((1 << a.g.ti_log2) != 8) return;
    const TileCoord c = coord_of<M>(a.g, 0, bid);
    if (!c.valid) return;
    const float2 *s = a.spec + spec_trace(a.g, c);   // (a column tile is a whole block of 8: 256 bytes, 256-byte aligned)
    for (int b = threadIdx.x; b < spec_blocks(M + 1); b += Team<M>::THREADS) bulk_prefetch_l2(s + (long long)b * a.g.ssf, 64 * SPEC_F);
}

// spectra in global memory -> first inverse pass in shared memory (no barrier at the end)
template <int M>
__device__ __forceinline__ void spec_to_smem(const FftArgs &a, const PairCtx<M> &x) {
    constexpr int S = M / 8;
    const int s = x.s;
    C2 A[8], B[8];
    bins_load<M>(A, a.spec, a.g, x, s, S);
    bins_load<M>(B, a.spec, a.g, x, s ? S - s : S / 2, S);
    f32x2 nyq = 0;
    if (s == 0) {
        const float2 *b = a.spec + spec_at(a.g, M);
        const float n0 = x.c[0].valid ? b[spec_trace(a.g, x.c[0])].x : 0.f;
        const float n1 = x.c[1].valid ? b[spec_trace(a.g, x.c[1])].x : 0.f;
        nyq = pk2(n0, n1);
    }
    EdgeRoots<M> t;
    t.load(a.tw, s);
    edge_inv<M>(A, B, nyq, x.buf, s, a.tw, t);
}

// last forward pass -> spectra in global memory
template <int M>
__device__ __forceinline__ void smem_to_spec(const FftArgs &a, const PairCtx<M> &x) {
    constexpr int S = M / 8;
    const int s = x.s;
    C2 A[8], B[8];
    f32x2 nyq;
    edge_fwd<M>(A, B, nyq, x.buf, s, a.tw);
    bins_store<M>(A, a.spec, a.g, x, s, S);
    bins_store<M>(B, a.spec, a.g, x, s ? S - s : S / 2, S);
    if (s == 0) {
        float2 *b = a.spec + spec_at(a.g, M);
        if (x.c[0].valid) b[spec_trace(a.g, x.c[0])] = make_float2(lo2(nyq), 0.f);
        if (x.c[1].valid) b[spec_trace(a.g, x.c[1])] = make_float2(hi2(nyq), 0.f);
    }
}

// Time samples of one trace in first-pass order: slot q R1/2 + r (r < R1/2) holds z[n] = (x[2n], x[2n+1]) with
// n = first_jj(q) + r L1.  Only these positions can hold samples (the upper half is the zero padding since
// nt <= M).  vec: 2 = float4 accesses where a thread's butterflies are adjacent (16-byte aligned traces),
// 1 = float2 accesses (8-byte aligned), 0 = scalar.
constexpr int NSLOT = FFT_P / 2;

template <int M>
__device__ __forceinline__ int slot_sample(int s, int h) {
    constexpr int R = Team<M>::R1, L = Team<M>::L1;
    return 2 * (first_jj<M>(s, h / (R / 2)) + (h % (R / 2)) * L);
}

template <int M>
__device__ __forceinline__ void time_load(float2 (&h)[NSLOT], const float *__restrict__ x, int nt, bool valid, int vec, int s) {
    constexpr int R = Team<M>::R1, HR = R / 2;
#pragma unroll
    for (int i = 0; i < NSLOT; ++i) h[i] = make_float2(0.f, 0.f);
    if (!valid) return;
    if (R < 16 && vec == 2) {
#pragma unroll
        for (int q = 0; q < FFT_P / R; q += 2)
#pragma unroll
            for (int r = 0; r < HR; ++r) {
                const int i0 = slot_sample<M>(s, q * HR + r);
                if (i0 < nt) {   // nt % 4 == 0 and i0 % 4 == 0: the quad lies inside the trace
                    const float4 v = __ldcs(reinterpret_cast<const float4 *>(x + i0));
                    h[q * HR + r] = make_float2(v.x, v.y);
                    h[((q + 1) * HR + r) % NSLOT] = make_float2(v.z, v.w);
                }
            }
    } else if (vec >= 1) {
#pragma unroll
        for (int i = 0; i < NSLOT; ++i) {
            const int i0 = slot_sample<M>(s, i);
            if (i0 < nt) h[i] = __ldcs(reinterpret_cast<const float2 *>(x + i0));
        }
    } else {
#pragma unroll
        for (int i = 0; i < NSLOT; ++i) {
            const int i0 = slot_sample<M>(s, i);
            if (i0 < nt) h[i].x = x[i0];
            if (i0 + 1 < nt) h[i].y = x[i0 + 1];
        }
    }
}

template <int M>
__device__ __forceinline__ void time_store(const float2 (&h)[NSLOT], float *__restrict__ x, int nt, int vec, int s) {
    constexpr int R = Team<M>::R1, HR = R / 2;
    if (R < 16 && vec == 2) {
#pragma unroll
        for (int q = 0; q < FFT_P / R; q += 2)
#pragma unroll
            for (int r = 0; r < HR; ++r) {
                const int i0 = slot_sample<M>(s, q * HR + r);
                const float2 u = h[q * HR + r], v = h[((q + 1) * HR + r) % NSLOT];
                if (i0 < nt) *reinterpret_cast<float4 *>(x + i0) = make_float4(u.x, u.y, v.x, v.y);
            }
    } else if (vec >= 1) {
#pragma unroll
        for (int i = 0; i < NSLOT; ++i) {
            const int i0 = slot_sample<M>(s, i);
            if (i0 < nt) *reinterpret_cast<float2 *>(x + i0) = h[i];
        }
    } else {
#pragma unroll
        for (int i = 0; i < NSLOT; ++i) {
            const int i0 = slot_sample<M>(s, i);
            if (i0 < nt) x[i0] = h[i].x;
            if (i0 + 1 < nt) x[i0 + 1] = h[i].y;
        }
    }
}

// registers of the first forward pass <-> the slots of the two traces
template <int M>
__device__ __forceinline__ void slots_to_regs(C2 (&a)[FFT_P], const float2 (&ha)[NSLOT], const float2 (&hb)[NSLOT]) {
    constexpr int R = Team<M>::R1, HR = R / 2;
#pragma unroll
    for (int i = 0; i < NSLOT; ++i) a[(i / HR) * R + i % HR] = join(ha[i], hb[i]);
}
template <int M>
__device__ __forceinline__ float2 slot_of(const C2 (&a)[FFT_P], int i, int which) {
    constexpr int R = Team<M>::R1, HR = R / 2;
    const C2 z = a[(i / HR) * R + i % HR];
    return which ? make_float2(hi2(z.re), hi2(z.im)) : make_float2(lo2(z.re), lo2(z.im));
}

// ------------------------------------------------------------------------------------------------
// kernels
// ------------------------------------------------------------------------------------------------
// forward transform of the slots and store of the spectra (in place over the buffer of the inverse: the first
// pass writes the locations that this thread read last, so no barrier precedes it)
template <int M>
__device__ __forceinline__ void slots_to_spec(const FftArgs &a, const PairCtx<M> &x, const float2 (&ha)[NSLOT], const float2 (&hb)[NSLOT]) {
    C2 v[FFT_P];
    slots_to_regs<M>(v, ha, hb);
    fwd_first<M>(v, x.buf, x.s);
    mid_passes<M, false, 1>(x.buf, x.s, a.tw);
    smem_to_spec<M>(a, x);
}

template <int M>
__device__ __forceinline__ void rfft_body(const FftArgs &a, int bid) {
    const PairCtx<M> x = pair_ctx<M>(a.g, bid);
    float2 h[2][NSLOT];
#pragma unroll
    for (int k = 0; k < 2; ++k) time_load<M>(h[k], a.tin + time_off<M>(a.g, x.c[k]), a.nt, x.c[k].valid, a.vec, x.s);
    slots_to_spec<M>(a, x, h[0], h[1]);
}

template <int M>
__global__ void __launch_bounds__(Team<M>::THREADS, Team<M>::MINB) k_rfft(FftArgs a) {
    rfft_body<M>(a, blockIdx.x);
}

// spectra -> s * irfft, causal window [0, nt)
template <int M>
__global__ void __launch_bounds__(Team<M>::THREADS, Team<M>::MINB) k_irfft_out(FftArgs a) {
    const PairCtx<M> x = pair_ctx<M>(a.g, blockIdx.x);
    spec_to_smem<M>(a, x);
    mid_passes<M, true, fft_npass(M) - 2>(x.buf, x.s, a.tw);
    group_sync<M>();
    C2 v[FFT_P];
    inv_last<M>(v, x.buf, x.s);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (!x.c[k].valid) continue;
        float2 h[NSLOT];
#pragma unroll
        for (int i = 0; i < NSLOT; ++i) {
            const float2 z = slot_of<M>(v, i, k);
            h[i] = make_float2(z.x * a.s, z.y * a.s);
        }
        time_store<M>(h, a.tout + time_off<M>(a.g, x.c[k]), a.nt, a.vec, x.s);
    }
}

__device__ __forceinline__ double block_sum(double v, double *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();   // red may still be read by a previous call
    if (l == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) s += red[i];
    return s;   // valid in thread 0
}

// Residual step: R = s * irfft(Uh)[0:nt] - U_obs[row], loss partial 1/2 sum R^2 (SumSq, then FP64), Rh = rfft(R)
// written in place over Uh.  Trace grid: i = batch entry b, j = virtual source v.
// tile bid of nblk tiles; the last tile to finish (atomic ticket) sums the partials of all nblk
template <int M>
__device__ __forceinline__ void residual_body(const FftArgs &a, int bid, int nblk) {
    __shared__ double red[32];
    __shared__ bool am_last;
    const PairCtx<M> x = pair_ctx<M>(a.g, bid);

    const float *uo[2] = {nullptr, nullptr};   // observed row of each trace
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (x.c[k].valid) {
            int row = x.c[k].i;
            if (!a.gathered) {
                row = a.idx[row];
                if (row < 0 || row >= a.ns) {
                    atomicOr(a.status, 1);
                    row = -1;
                }
            }
            if (row >= 0) uo[k] = a.uobs + (long long)row * a.uo_si + (long long)x.c[k].j * a.uo_sj;
        }
    spec_to_smem<M>(a, x);
    float2 o[2][NSLOT];   // observed rows, loaded before the middle passes (their latency overlaps the rest)
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (!Team<M>::LATE) time_load<M>(o[k], uo[k] ? uo[k] : a.uobs, a.nt, uo[k] != nullptr, a.vec, x.s);
    mid_passes<M, true, fft_npass(M) - 2>(x.buf, x.s, a.tw);
    group_sync<M>();
    C2 v[FFT_P];
    inv_last<M>(v, x.buf, x.s);
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (Team<M>::LATE) time_load<M>(o[k], uo[k] ? uo[k] : a.uobs, a.nt, uo[k] != nullptr, a.vec, x.s);
    // z = s p - o inside the window [0, nt), zero outside
    float top = 0.f;
#pragma unroll
    for (int i = 0; i < NSLOT; ++i) {
        const int i0 = slot_sample<M>(x.s, i);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float2 p = slot_of<M>(v, i, k);
            const bool in0 = x.c[k].valid && i0 < a.nt, in1 = x.c[k].valid && i0 + 1 < a.nt;
            o[k][i] = make_float2(in0 ? fmaf(p.x, a.s, -o[k][i].x) : 0.f, in1 ? fmaf(p.y, a.s, -o[k][i].y) : 0.f);
            top = fmaxf(top, fmaxf(fabsf(o[k][i].x), fabsf(o[k][i].y)));
        }
    }
    double l2;
    if (SumSq::in_range(top)) {   // (a NaN passes and reaches the sum)
        static_assert(2 * NSLOT <= SumSq::SQUARES, "one sum for a thread's samples");
        SumSq q(SumSq::pow2(top));
#pragma unroll
        for (int i = 0; i < NSLOT; ++i) {
            const C2 z = join(o[0][i], o[1][i]);
            q.add(z.re);
            q.add(z.im);
        }
        l2 = q.total();
    } else {
        l2 = 0.0;
#pragma unroll
        for (int i = 0; i < NSLOT; ++i)
#pragma unroll
            for (int k = 0; k < 2; ++k) l2 += (double)o[k][i].x * o[k][i].x + (double)o[k][i].y * o[k][i].y;
    }
    slots_to_spec<M>(a, x, o[0], o[1]);

    // deterministic loss: per-block partials, summed in block order by the last block to finish
    const double bs = block_sum(l2, red);
    if (threadIdx.x == 0) {
        a.partials[bid] = bs;
        __threadfence();
        const unsigned prev = atomicAdd(a.counter, 1u);
        am_last = (prev == (unsigned)(nblk - 1));
    }
    __syncthreads();
    if (am_last) {   // block-uniform
        __threadfence();
        double s = 0.0;
        for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += __ldcg(&a.partials[b]);
        s = block_sum(s, red);   // fixed assignment and order: deterministic
        if (threadIdx.x == 0) {
            if (a.loss) *a.loss = 0.5 * s;
            *a.counter = 0u;
        }
    }
}

template <int M>
__global__ void __launch_bounds__(Team<M>::THREADS, Team<M>::MINB) k_residual(FftArgs a) {
    residual_body<M>(a, blockIdx.x, gridDim.x);
}

// Update: g = s * irfft(Gh)[0:nt];  X <- X - alpha g (SGD), or with the causality mute and/or Nesterov
// momentum (see the else branch);  optionally Gh <- rfft(X_new) (in place).
// Trace grid: i = receiver r, j = virtual source v (model layout [nv][nr][nt]).
//
// Symmetric model (a.g.sym, reciprocity on a square grid with X[v][r] = X[r][v], and so the velocity or the
// moments of a symmetric start): only the tiles on or above the TR-block diagonal run; a trace (v, r) of a
// tile above it (r >= TR (v / TR + 1)) also writes its mirror (r, v) of each array, which it equals, and the
// spectra below the block diagonal are left to launch_mirror_lower or to the transposed read of the
// forward product.  Traces of the diagonal blocks run in both orders (their mirrors are in the same
// block row and column), so every element of X is written once.
//
// EXT: 0 SGD, 1 SGD with the causality mute, 2 with a velocity or Adam moments (and the mute).  (The mute without the code
// of the others: update 1200 -> 1030 us at nt 1500, 300 x 300, 330 -> 243 us at nt 1024, 201 x 201.)
//
// At M = 1536 a thread with a velocity or moments has 24 to 32 more values to hold than 80 registers take: one CTA per SM
// at 168 registers there, without spills and with the model loaded early (two CTAs at 80 registers spill 468 to 716 bytes a
// thread; us at nt 1500, two / one CTA: 300 x 300 N-SGD 1389 / 1366, Adam 1730 / 1630; 600 x 600 symmetric N-SGD 3611 /
// 3121, Adam 4939 / 3779).
template <int M, int EXT>
constexpr bool one_cta() { return M == 1536 && EXT == 2; }
template <int M, int EXT>
constexpr int update_minb() { return one_cta<M, EXT>() ? 1 : Team<M>::MINB; }

template <int M, bool KEEP, int EXT>
__device__ __forceinline__ void update_body(const FftArgs &a, int bid_in) {
    constexpr int TR = Team<M>::TR;
    constexpr bool LATE = Team<M>::LATE && !one_cta<M, EXT>();
    const int bid = a.g.sym ? sym_tile_to_full(a.g, TR, bid_in) : bid_in;
    const PairCtx<M> x = pair_ctx<M>(a.g, bid);
    spec_to_smem<M>(a, x);
    if constexpr (prefetches<M>()) {
        const int nxt = bid_in + a.ahead;
        if (a.ahead > 0 && nxt < (int)gridDim.x) tile_prefetch<M>(a, a.g.sym ? sym_tile_to_full(a.g, TR, nxt) : nxt);
    }
    float2 xo[2][NSLOT];   // model samples, loaded before the middle passes (their latency overlaps the rest)
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (!LATE) time_load<M>(xo[k], a.tout + time_off<M>(a.g, x.c[k]), a.nt, x.c[k].valid, a.vec, x.s);
    mid_passes<M, true, fft_npass(M) - 2>(x.buf, x.s, a.tw);
    group_sync<M>();
    C2 v[FFT_P];
    inv_last<M>(v, x.buf, x.s);
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (LATE) time_load<M>(xo[k], a.tout + time_off<M>(a.g, x.c[k]), a.nt, x.c[k].valid, a.vec, x.s);
    const float nas = -a.alpha * a.s;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const TileCoord &c = x.c[k];
        const long long off = time_off<M>(a.g, c);
        // the mirror trace (r, v) of a trace above the block diagonal
        const bool mir = a.g.sym && c.valid && c.i / TR > c.j / TR;
        const long long moff = mir ? (long long)c.j * a.g.tsi + (long long)c.i * a.g.tsj : 0;
        if constexpr (EXT == 0) {
            // SGD: X <- X - alpha g
#pragma unroll
            for (int i = 0; i < NSLOT; ++i) {
                const int i0 = slot_sample<M>(x.s, i);
                const float2 g = slot_of<M>(v, i, k);
                xo[k][i] = make_float2((i0 < a.nt) ? fmaf(nas, g.x, xo[k][i].x) : 0.f,
                                       (i0 + 1 < a.nt) ? fmaf(nas, g.y, xo[k][i].y) : 0.f);
            }
        } else {
            // causality mute (the step is zero before the first kept sample) and, with a velocity,
            // Nesterov momentum on the look-ahead point: V <- mu V + step, X <- X + mu V + step;
            // or, with Adam moments m and v (Kingma & Ba, Algorithm 1) of the preconditioned gradient g:
            // m <- b1 m + (1-b1) g, v <- b2 v + (1-b2) g^2, X <- X - alpha (c1 m) / (sqrt(c2 v) + eps)
            const int first = (a.mute && c.valid) ? __ldg(a.mute + (long long)c.j * a.g.ni + c.i) : 0;
            float2 m0[NSLOT], m1[NSLOT];   // velocity, or the moments
            if (EXT == 2 && a.adam_m) {
                time_load<M>(m0, a.adam_m + off, a.nt, c.valid, a.vec, x.s);
                time_load<M>(m1, a.adam_v + off, a.nt, c.valid, a.vec, x.s);
            } else if (EXT == 2 && a.vel) {
                time_load<M>(m0, a.vel + off, a.nt, c.valid, a.vec, x.s);
            }
            auto sample = [&](int t, float g0, float xv, float &p, float &q) {
                float z;
                if (EXT == 2 && a.adam_m) {
                    const float g = (t >= first) ? a.s * g0 : 0.f;
                    p = fmaf(a.beta1, p, (1.f - a.beta1) * g);
                    q = fmaf(a.beta2, q, (1.f - a.beta2) * (g * g));
                    z = xv - a.alpha * (p * a.c1) / (sqrtf(q * a.c2) + a.eps);
                } else {
                    const float st = (t >= first) ? nas * g0 : 0.f;
                    if (EXT == 2 && a.vel) {
                        p = fmaf(a.mu, p, st);
                        z = fmaf(a.mu, p, xv + st);
                    } else {
                        z = xv + st;
                    }
                }
                return t < a.nt ? z : 0.f;
            };
#pragma unroll
            for (int i = 0; i < NSLOT; ++i) {
                const int i0 = slot_sample<M>(x.s, i);
                const float2 g = slot_of<M>(v, i, k);
                xo[k][i] = make_float2(sample(i0, g.x, xo[k][i].x, m0[i].x, m1[i].x),
                                       sample(i0 + 1, g.y, xo[k][i].y, m0[i].y, m1[i].y));
            }
            if (c.valid) {
                if (EXT == 2 && a.adam_m) {
                    time_store<M>(m0, a.adam_m + off, a.nt, a.vec, x.s);
                    time_store<M>(m1, a.adam_v + off, a.nt, a.vec, x.s);
                } else if (EXT == 2 && a.vel) {
                    time_store<M>(m0, a.vel + off, a.nt, a.vec, x.s);
                }
                if (mir) {   // the mirror trace of the velocity or of the moments
                    if (EXT == 2 && a.adam_m) {
                        time_store<M>(m0, a.adam_m + moff, a.nt, a.vec, x.s);
                        time_store<M>(m1, a.adam_v + moff, a.nt, a.vec, x.s);
                    } else if (EXT == 2 && a.vel) {
                        time_store<M>(m0, a.vel + moff, a.nt, a.vec, x.s);
                    }
                }
            }
        }
        if (c.valid) time_store<M>(xo[k], a.tout + off, a.nt, a.vec, x.s);
        if (mir) time_store<M>(xo[k], a.tout + moff, a.nt, a.vec, x.s);
    }
    if constexpr (KEEP) slots_to_spec<M>(a, x, xo[0], xo[1]);
}

template <int M, bool KEEP, int EXT>
__global__ void __launch_bounds__(Team<M>::THREADS, update_minb<M, EXT>()) k_update(FftArgs a) {
    update_body<M, KEEP, EXT>(a, blockIdx.x);
}

// work-queue forms: persistent CTAs taking (problem, tile) items until the queue is empty
template <int M>
__global__ void __launch_bounds__(Team<M>::THREADS, Team<M>::MINB) k_rfft_q(WorkQueue q) {
    const FftArgs *args = static_cast<const FftArgs *>(q.args);
    int m = 0, tile = 0;
    __shared__ FftArgs sa;
    while (queue_next(q, m, tile) >= 0) {
        queue_args(args + m, sa);
        __syncthreads();
        rfft_body<M>(sa, tile);
    }
}

template <int M>
__global__ void __launch_bounds__(Team<M>::THREADS, Team<M>::MINB) k_residual_q(WorkQueue q) {
    const FftArgs *args = static_cast<const FftArgs *>(q.args);
    int m = 0, tile = 0;
    __shared__ FftArgs sa;
    while (queue_next(q, m, tile) >= 0) {
        queue_args(args + m, sa);
        __syncthreads();
        residual_body<M>(sa, tile, __ldg(q.start + m + 1) - __ldg(q.start + m));
    }
}

template <int M>
__global__ void __launch_bounds__(Team<M>::THREADS, Team<M>::MINB) k_update_q(WorkQueue q) {
    const FftArgs *args = static_cast<const FftArgs *>(q.args);
    int m = 0, tile = 0;
    __shared__ FftArgs sa;
    while (queue_next(q, m, tile) >= 0) {
        queue_args(args + m, sa);
        __syncthreads();
        update_body<M, true, 0>(sa, tile);
    }
}

// ------------------------------------------------------------------------------------------------
// launchers of one complex length M (instantiated in fft_m*.cu)
// ------------------------------------------------------------------------------------------------
template <int M>
int blocks_for(const TraceGrid &g) {
    // -1: the grid was laid out for CTAs of another trace count (more traces along i than a CTA holds), or
    // an upper enumeration of a grid that is not square with whole CTAs along i
    const int ti = 1 << g.ti_log2, tj = Team<M>::TR >> g.ti_log2;
    if (tj < 1) return -1;
    if (g.sym) return (tj == 1 && g.ni == g.nj) ? (int)sym_tiles(g.ni, Team<M>::TR) : -1;
    return ((g.ni + ti - 1) / ti) * ((g.nj + tj - 1) / tj);
}

template <int M>
struct FftLaunch {
    static cudaError_t prepare();
    static cudaError_t rfft(const FftArgs &a, cudaStream_t st);
    static cudaError_t irfft_out(const FftArgs &a, cudaStream_t st);
    static cudaError_t residual(const FftArgs &a, int nblocks_expected, cudaStream_t st);
    static cudaError_t update(bool keep, const FftArgs &a, cudaStream_t st);
    static int update_ahead();
    static cudaError_t queue_rfft(const WorkQueue &q, cudaStream_t st);
    static cudaError_t queue_residual(const WorkQueue &q, cudaStream_t st);
    static cudaError_t queue_update(const WorkQueue &q, cudaStream_t st);
};

#ifdef SMDD_FFT_INSTANTIATE
template <int M>
cudaError_t FftLaunch<M>::prepare() {
    const void *kernels[] = {(const void *)k_rfft<M>, (const void *)k_irfft_out<M>, (const void *)k_residual<M>,
                             (const void *)k_update<M, false, 0>, (const void *)k_update<M, true, 0>,
                             (const void *)k_update<M, false, 1>, (const void *)k_update<M, true, 1>,
                             (const void *)k_update<M, false, 2>, (const void *)k_update<M, true, 2>,
                             (const void *)k_rfft_q<M>, (const void *)k_residual_q<M>, (const void *)k_update_q<M>};
    for (const void *k : kernels) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Team<M>::SMEM);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int M>
cudaError_t FftLaunch<M>::rfft(const FftArgs &a, cudaStream_t st) {
    const int nb = blocks_for<M>(a.g);
    if (nb < 0) return cudaErrorInvalidValue;
    if (nb == 0) return cudaSuccess;
    k_rfft<M><<<nb, Team<M>::THREADS, Team<M>::SMEM, st>>>(a);
    return cudaGetLastError();
}

template <int M>
cudaError_t FftLaunch<M>::irfft_out(const FftArgs &a, cudaStream_t st) {
    const int nb = blocks_for<M>(a.g);
    if (nb < 0) return cudaErrorInvalidValue;
    if (nb == 0) return cudaSuccess;
    k_irfft_out<M><<<nb, Team<M>::THREADS, Team<M>::SMEM, st>>>(a);
    return cudaGetLastError();
}

template <int M>
cudaError_t FftLaunch<M>::residual(const FftArgs &a, int nblocks_expected, cudaStream_t st) {
    const int nb = blocks_for<M>(a.g);
    if (nb <= 0 || nb > nblocks_expected) return cudaErrorInvalidValue;
    k_residual<M><<<nb, Team<M>::THREADS, Team<M>::SMEM, st>>>(a);
    return cudaGetLastError();
}

template <int M>
cudaError_t FftLaunch<M>::update(bool keep, const FftArgs &a, cudaStream_t st) {
    const int nb = blocks_for<M>(a.g);
    if (nb < 0) return cudaErrorInvalidValue;
    if (nb == 0) return cudaSuccess;
    auto kern = (a.vel || a.adam_m) ? (keep ? k_update<M, true, 2> : k_update<M, false, 2>)
                : a.mute            ? (keep ? k_update<M, true, 1> : k_update<M, false, 1>)
                                    : (keep ? k_update<M, true, 0> : k_update<M, false, 0>);
    kern<<<nb, Team<M>::THREADS, Team<M>::SMEM, st>>>(a);
    return cudaGetLastError();
}

template <int M>
int FftLaunch<M>::update_ahead() {
    int dev = 0, sms = 0, ctas = 0;
    if (!prefetches<M>() || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, k_update<M, true, 0>, Team<M>::THREADS, Team<M>::SMEM) != cudaSuccess)
        return 0;
    return sms * ctas;
}

// work-queue launches: resident CTAs on every SM take (problem, tile) items until the queue is empty
template <class KF>
static cudaError_t launch_queue_kernel(KF kern, int threads, size_t smem, const WorkQueue &q, cudaStream_t st) {
    if (q.total <= 0) return cudaSuccess;
    const int grid = queue_grid(kern, threads, smem, q.total);
    kern<<<grid, threads, smem, st>>>(q);
    return cudaGetLastError();
}

template <int M>
cudaError_t FftLaunch<M>::queue_rfft(const WorkQueue &q, cudaStream_t st) {
    return launch_queue_kernel(k_rfft_q<M>, Team<M>::THREADS, Team<M>::SMEM, q, st);
}

template <int M>
cudaError_t FftLaunch<M>::queue_residual(const WorkQueue &q, cudaStream_t st) {
    return launch_queue_kernel(k_residual_q<M>, Team<M>::THREADS, Team<M>::SMEM, q, st);
}

template <int M>
cudaError_t FftLaunch<M>::queue_update(const WorkQueue &q, cudaStream_t st) {
    return launch_queue_kernel(k_update_q<M>, Team<M>::THREADS, Team<M>::SMEM, q, st);
}
#endif  // SMDD_FFT_INSTANTIATE

}  // namespace smdd
