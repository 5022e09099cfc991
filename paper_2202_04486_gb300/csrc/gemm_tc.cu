// Per-frequency complex products on the tensor cores (tcgen05) with split-BF16 operands: the
// mixed-precision form of the batched MMM of Appendix A (Eq. 2 forward, Eq. 6 adjoint).
//
// Every FP32 operand value x is written to shared memory as two BF16 numbers, hi = bf16(x) and
// lo = bf16(x - hi); a real product is x*y ~ hi_x hi_y + hi_x lo_y + lo_x hi_y (the lo*lo term is
// dropped), accumulated in FP32 in tensor memory.  A complex product uses the four real products
// (re*re - im*im, re*im + im*re), the subtraction through the negate-B bit of the instruction
// descriptor.  So each K-step of 16 issues 12 MMAs of M = 128 rows into two accumulators (re, im).
//
// Tile kernels (work-queue epochs, the mirrored tiles of reciprocity steps, the products that launch_tc_fwd_p and
// adj_persistent leave to them, and where no tensor maps are to be had): the CUDA threads of a CTA load the FP32 complex spectra (coalesced rows), split them and store the
// four BF16 planes (re hi, re lo, im hi, im lo) in the 128-byte swizzled layouts of tc_common.cuh -- or,
// for the adjoint of a plan that holds them, copy the planes from operand images split once per step
// (k_tc_adj_images); thread 0 issues the MMAs and commits them to an mbarrier.  The persistent kernels k_tc_fwd_p and
// k_tc_adj_p run the same products with their roles on different warps.  Every wait is bounded.
// Status bits: 1 = a source index out of range, 2 = a bounded wait gave up.
#include <algorithm>
#include <cstdint>
#include <cstring>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "smdd_fft.cuh"
#include "smdd_internal.h"
#include "tc_common.cuh"
#include "work_queue.cuh"

namespace smdd {

constexpr int TC_THREADS = 256;
#ifndef SMDD_TC_FWD_STAGES
#define SMDD_TC_FWD_STAGES 1   // one stage: two CTAs share an SM and hide each other's load latency
#endif
constexpr int TC_FWD_STAGES = SMDD_TC_FWD_STAGES;

__device__ __forceinline__ uint8_t *align1024(uint8_t *p) {
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// load the 8 complex columns k .. k+7 (k a multiple of 8) of a row in the layout of F bins, zero past n (row may be
// null: all zero)
template <int F = 1>
__device__ __forceinline__ void load8(const float2 *row, int k, int n, float2 (&z)[8]) {
    row += row ? (long long)k * (F - 1) : 0;
    if (row && k + 7 < n) {
        const float4 *p = reinterpret_cast<const float4 *>(row + k);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = __ldg(p + i);
            z[2 * i] = make_float2(v.x, v.y);
            z[2 * i + 1] = make_float2(v.z, v.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = (row && k + i < n) ? row[k + i] : make_float2(0.f, 0.f);
    }
}

// Row v of a symmetric model's spectra, elements k .. k+8 (zero past n), when only the part on and above
// the TR-block diagonal is stored: element r < lo = TR floor(v / TR) is read at (r, v) (column v of row r).
// (ld: float2 of a row over its bins)
__device__ __forceinline__ void load8_sym(const float2 *Af, long long ld, int v, int k, int n, int lo, float2 (&z)[8]) {
    if (k >= lo) {
        load8<SPEC_F>(Af + (long long)v * ld, k, n, z);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = k + i;
            z[i] = r < n ? __ldg(r >= lo ? Af + (long long)v * ld + spec_col(r) : Af + (long long)r * ld + spec_col(v)) : make_float2(0.f, 0.f);
        }
    }
}

// store one 16-byte chunk of each plane; planes are `pstride` bytes apart
__device__ __forceinline__ void store_planes(uint8_t *base, int off, int pstride, const Chunk4 &c) {
    *reinterpret_cast<uint4 *>(base + off) = c.rh;
    *reinterpret_cast<uint4 *>(base + pstride + off) = c.rl;
    *reinterpret_cast<uint4 *>(base + 2 * pstride + off) = c.ih;
    *reinterpret_cast<uint4 *>(base + 3 * pstride + off) = c.il;
}

// 12 MMAs of one K-step: acc_re += Ar Br - Ai Bi, acc_im += Ar Bi + Ai Br, each real product split
// into hi*hi + hi*lo + lo*hi.  a[p], b[p]: descriptors of the planes (re hi, re lo, im hi, im lo).
__device__ __forceinline__ void mma_complex_split(uint32_t d_re, uint32_t d_im, const uint64_t (&a)[4],
                                                  const uint64_t (&b)[4], uint32_t idp, uint32_t idn, uint32_t acc) {
    umma_bf16(d_re, a[0], b[0], idp, acc);
    umma_bf16(d_re, a[0], b[1], idp, 1);
    umma_bf16(d_re, a[1], b[0], idp, 1);
    umma_bf16(d_re, a[2], b[2], idn, 1);
    umma_bf16(d_re, a[2], b[3], idn, 1);
    umma_bf16(d_re, a[3], b[2], idn, 1);
    umma_bf16(d_im, a[0], b[2], idp, acc);
    umma_bf16(d_im, a[0], b[3], idp, 1);
    umma_bf16(d_im, a[1], b[2], idp, 1);
    umma_bf16(d_im, a[2], b[0], idp, 1);
    umma_bf16(d_im, a[2], b[1], idp, 1);
    umma_bf16(d_im, a[3], b[0], idp, 1);
}

// ------------------------------------------------------------------------------------------------
// forward: C[f][v][b] = sum_r A[f][v][r] Dh[f][idx_b][r]   (M = 128 rows v, N = NB batch columns)
// K = nr streamed in chunks of 64 through two shared-memory stages.
// ------------------------------------------------------------------------------------------------
template <int NB, int NSTAGE>
struct TcFwd {
    static constexpr int A_PLANE = 128 * 128;           // bytes per plane per stage
    static constexpr int B_PLANE = NB * 128;
    static constexpr int STAGE = 4 * A_PLANE + 4 * B_PLANE;
    static constexpr size_t SMEM = NSTAGE * (size_t)STAGE + 1024;
    static constexpr uint32_t TMEM_COLS = 2 * NB <= 32 ? 32 : 2 * NB;   // power of two >= 32
};

// Tile (bx, by, bz) = (row block of 128 virtual sources, batch block of NB, bin f).  Q: a work-queue
// item of a persistent CTA, which owns its TMEM (tmem_q) for all its items; the barriers are
// invalidated at the end of the item so that the next one can initialise them again.
template <int NB, int NSTAGE, bool Q, bool SYM = false>
__device__ __forceinline__ void tc_fwd_body(const GemmArgs &a, int bx, int by, int bz, uint32_t tmem_q) {
    using G = TcFwd<NB, NSTAGE>;
    extern __shared__ uint8_t tc_raw[];
    __shared__ uint64_t bars[2];
    __shared__ uint32_t tmem_holder;
    __shared__ int drows[NB];
    __shared__ int fail, issued;
    uint8_t *sm = align1024(tc_raw);
    const int f = bz, v0 = bx * 128, b0 = by * NB;
    if (a.nf_active > 0 && f >= a.nf_active) {   // above the band limit: zero products, no TMEM
        zero_tile(a.C + spec_bin(f, a.sCf), (long long)a.ldb * SPEC_F, v0, 128, b0, NB, a.nv, a.nb);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float2 *Af = a.A + spec_bin(f, a.sAf);
    const long long arow = (long long)a.ldr * SPEC_F;
    const float2 *Df = a.Dh + (long long)f * a.sDf;

    for (int j = tid; j < NB; j += TC_THREADS) {
        int s = -1;
        if (b0 + j < a.nb) {
            s = a.idx[b0 + j];
            if (s < 0 || s >= a.ns) {
                atomicOr(a.status, 1);
                s = -1;
            }
        }
        drows[j] = s;
    }
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fail = 0;
        issued = 0;
        fence_mbar_init();
    }
    if (!Q && warp == 0) tmem_alloc(&tmem_holder, G::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = Q ? tmem_q : tmem_holder;
    constexpr uint32_t idp = umma_idesc(128, NB, 0, 0, 0), idn = umma_idesc(128, NB, 0, 0, 1);
    // failure-path check: before any copy or product, wait on a barrier that nothing arrives on (phase
    // 0 of bars[1] never completes here) for a short limit, then take the timeout path below
    if (a.wait_probe > 0) {
        if (tid == 0 && !mbar_wait_limit(&bars[1], 0, a.wait_probe)) fail = 1;
        __syncthreads();
    }

    const int nk = fail ? 0 : (a.nr + 63) / 64;
    for (int kc = 0; kc < nk; ++kc) {
        const int s = kc % NSTAGE;
        uint8_t *st = sm + s * G::STAGE;
        // model spectra rows: 128 rows x 8 chunks of 8 complex; every load of the chunk is issued
        // before the first split, so their latencies overlap, and before the wait for the stage, so
        // they also overlap the MMAs of the previous chunk
        {
            constexpr int UA = 128 * 8 / TC_THREADS;
            float2 z[UA][8];
#pragma unroll
            for (int i = 0; i < UA; ++i) {
                const int u = tid + i * TC_THREADS, row = u >> 3, c = u & 7, v = v0 + row;
                if (SYM && v < a.nv)
                    load8_sym(Af, arow, v, kc * 64 + 8 * c, a.nr, a.sym_tr * (v / a.sym_tr), z[i]);
                else
                    load8<SPEC_F>(v < a.nv ? Af + v * arow : nullptr, kc * 64 + 8 * c, a.nr, z[i]);
            }
            // stage s is free again once the MMAs of chunk kc - NSTAGE (the previous use of bars[s]) are done
            if (kc >= NSTAGE && !mbar_wait_bounded(&bars[s], ((kc - NSTAGE) / NSTAGE) & 1)) fail = 1;
#pragma unroll
            for (int i = 0; i < UA; ++i) {
                const int u = tid + i * TC_THREADS, row = u >> 3, c = u & 7;
                store_planes(st, row * 128 + ((c ^ (row & 7)) << 4), G::A_PLANE, split8(z[i], false));
            }
        }
        // gathered kernel rows of the batch
        for (int u = tid; u < NB * 8; u += TC_THREADS) {
            const int row = u >> 3, c = u & 7, srow = drows[row];
            float2 z[8];
            load8(srow >= 0 ? Df + (long long)srow * a.ldd : nullptr, kc * 64 + 8 * c, a.nr, z);
            store_planes(st + 4 * G::A_PLANE, row * 128 + ((c ^ (row & 7)) << 4), G::B_PLANE, split8(z, false));
        }
        fence_async_smem();
        __syncthreads();
        if (fail) break;
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint64_t ad[4], bd[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    ad[p] = umma_desc(smem_u32(st + p * G::A_PLANE + ks * 32), 16, 1024);
                    bd[p] = umma_desc(smem_u32(st + 4 * G::A_PLANE + p * G::B_PLANE + ks * 32), 16, 1024);
                }
                mma_complex_split(tmem, tmem + NB, ad, bd, idp, idn, (kc > 0 || ks > 0) ? 1u : 0u);
            }
            umma_commit(&bars[s]);
            issued = 1;
        }
    }
    const int last = nk - 1;
    if (!fail && !mbar_wait_bounded(&bars[last % NSTAGE], (last / NSTAGE) & 1)) fail = 1;
    __syncthreads();
    const bool ok = !fail;
    // after a timeout, give products still in flight one more bounded wait before TMEM is freed
    if (!ok && issued) mbar_wait_bounded(&bars[last % NSTAGE], (last / NSTAGE) & 1);
    tc_fence_after();
    __syncthreads();
    // epilogue: TMEM -> shared staging [128][NB] complex -> coalesced rows of C
    float2 *out = reinterpret_cast<float2 *>(sm);
    if (ok && warp < 4) {
        const int row = 32 * warp + lane;
#pragma unroll
        for (int c0 = 0; c0 < NB; c0 += 16) {
            float re[16], im[16];
            tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + c0, re);
            tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + NB + c0, im);
#pragma unroll
            for (int j = 0; j < 16; ++j) out[row * (NB + 1) + c0 + j] = make_float2(re[j], im[j]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (ok) {
        float2 *Cf = a.C + spec_bin(f, a.sCf);
        for (int e = tid; e < 128 * NB; e += TC_THREADS) {
            const int row = e / NB, j = e % NB, v = v0 + row, b = b0 + j;
            if (v < a.nv && b < a.nb) Cf[(long long)v * a.ldb * SPEC_F + spec_col(b)] = out[row * (NB + 1) + j];
        }
    } else if (tid == 0) {
        atomicOr(a.status, 2);
    }
    if constexpr (Q) {
        __syncthreads();   // every wait on the barriers of this item is over
        if (tid == 0) {
            mbar_inval(&bars[0]);
            mbar_inval(&bars[1]);
        }
    } else {
        if (warp == 0) tmem_dealloc(tmem, G::TMEM_COLS);
    }
}

// SYM: the model spectra hold a symmetric model on and above the a.sym_tr-block diagonal only (load8_sym)
template <int NB, int NSTAGE, bool SYM = false>
__global__ void __launch_bounds__(TC_THREADS, NSTAGE == 1 ? 2 : 1) k_tc_fwd(GemmArgs a) {
    tc_fwd_body<NB, NSTAGE, false, SYM>(a, blockIdx.x, blockIdx.y, blockIdx.z, 0);
}

// work-queue form: persistent CTAs (TMEM allocated once) taking (problem, tile) items; tile t of a
// problem is (bx, by, bz) with t = (bz gy + by) gx + bx, gx = ceil(nv / 128), gy = ceil(nb / NB)
template <int NB>
__global__ void __launch_bounds__(TC_THREADS, 2) k_tc_fwd_q(WorkQueue q) {
    using G = TcFwd<NB, 1>;
    __shared__ uint32_t holder;
    const int warp = threadIdx.x >> 5;
    if (warp == 0) tmem_alloc(&holder, G::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = holder;
    const GemmArgs *args = static_cast<const GemmArgs *>(q.args);
    int m = 0, tile = 0;
    __shared__ GemmArgs sa;
    while (queue_next(q, m, tile) >= 0) {
        queue_args(args + m, sa);
        __syncthreads();
        const GemmArgs &a = sa;
        const int gx = (a.nv + 127) / 128, gy = (a.nb + NB - 1) / NB;
        const int bx = tile % gx, r = tile / gx;
        tc_fwd_body<NB, 1, true>(a, bx, r % gy, r / gy, tmem);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, G::TMEM_COLS);
}

// ------------------------------------------------------------------------------------------------
// adjoint: C[f][v][r] = outscale * sum_k A'[v][k] B'[k][r] on 128 x 128 tiles, K = nb in chunks of 32:
//   first half  A' = Rh[f][v][b],                 B' = conj(Dh[f][idx_b][r])
//   second half A' = conj(Dh[f][idx_b][v]),       B' = Rh[f][r][b]          (reciprocity)
// Both operands are stored MN-major (rows k, 128 contiguous m / n), so every plane is 32 x 256 bytes:
// the kernel rows of Dh are MN-major as loaded, and the residual rows (b contiguous in HBM) are copied
// by cp.async into a staging tile and transposed while they are split.  About 100 KB of shared memory:
// two CTAs share an SM, one CTA's epilogue overlapping the other's loads and products; the loads of
// the next chunk are issued before the wait for the previous chunk's products.
// With reciprocity only the upper-triangular tiles run and the transposed tile is mirrored.
// ------------------------------------------------------------------------------------------------
struct TcAdj {
    static constexpr int KC = 32;                       // K chunk
    static constexpr int PLANE = 2 * KC * 128;          // bytes: 2 atoms of 64 m/n x KC rows x 128 B
    static constexpr int OPER = 8 * PLANE;              // A' and B' planes (64 KB)
    static constexpr int SLD = KC + 2;                  // staging row pitch in float2 (16-byte multiple)
    static constexpr int STAGE = 128 * SLD * 8;         // residual staging tile (34 KB)
    static constexpr int OUT = 128 * 65 * 8;            // epilogue staging: 64 columns per pass
    static constexpr size_t BODY = (size_t)OPER + STAGE;
    static constexpr size_t SMEM = (BODY > OUT ? BODY : OUT) + 1024;
    static constexpr uint32_t TMEM_COLS = 256;
};

__device__ __forceinline__ void cp_async16_zfill(void *smem_dst, const void *gsrc, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(gsrc), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit_wait_all() {
    asm volatile("cp.async.commit_group;\n" ::);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Operand images: per bin f and K chunk kc, for every 128-wide block of the virtual sources (R, from the
// residual spectra) and of the receivers (D, from the conjugated kernel rows of the batch), the four
// split-BF16 planes exactly as the tile kernel's shared memory holds them (MN-major, 128-byte swizzle):
// R image of block b at [f][kc][b], D image of block b at [f][kc][tiles_v + b], TC_ADJ_IMG bytes each.
// The adjoint then copies two images per half instead of loading, transposing and splitting its operands
// (every operand block serves a whole row or column of output tiles).
constexpr int TC_ADJ_IMG = 4 * TcAdj::PLANE;

__global__ void __launch_bounds__(TC_THREADS) k_tc_adj_images(GemmArgs a, uint8_t *img) {
    using G = TcAdj;
    constexpr int KC = G::KC;
    extern __shared__ __align__(16) float2 stg[];   // residual staging [128][SLD]
    __shared__ int sidx[KC];
    const int blk = blockIdx.x, kc = blockIdx.y, f = blockIdx.z, tid = threadIdx.x;
    const int k0 = kc * KC, kn = min(KC, a.nb - k0);
    const int nbl = a.tiles_v + a.tiles_r;
    uint8_t *dst = img + (((long long)f * a.img_nkc + kc) * nbl + blk) * (long long)TC_ADJ_IMG;
    if (blk < a.tiles_v) {
        // R image: residual rows cr .. cr + 127 (b contiguous), staged, then transposed and split
        const int cr = blk * 128;
        const float2 *Rf = a.A + spec_bin(f, a.sAf);
        for (int u = tid; u < 128 * (KC / 2); u += TC_THREADS) {
            const int row = u / (KC / 2), pr = u % (KC / 2), k = k0 + 2 * pr, rr = cr + row;
            int bytes = 0;
            const float2 *src = Rf;
            if (rr < a.nv && k < a.nb) {
                bytes = (k + 1 < a.nb) ? 16 : 8;
                src = Rf + (long long)rr * a.ldb * SPEC_F + spec_col(k);
            }
            cp_async16_zfill(stg + row * G::SLD + 2 * pr, src, bytes);
        }
        cp_async_commit_wait_all();
        __syncthreads();
        for (int u = tid; u < KC * 16; u += TC_THREADS) {
            const int k = u % KC, ch = u / KC, at = ch >> 3, c = ch & 7;
            float2 z[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) z[j] = stg[(64 * at + 8 * c + j) * G::SLD + k];
            store_planes(dst, at * (KC * 128) + k * 128 + ((c ^ (k & 7)) << 4), G::PLANE, split8(z, false));
        }
    } else {
        // D image: conjugated kernel rows of the batch entries k0 .. k0 + 31, receivers cd .. cd + 127
        const int cd = (blk - a.tiles_v) * 128;
        if (tid < KC) {
            int sr = -1;
            if (tid < kn) {
                sr = a.idx[k0 + tid];
                if (sr < 0 || sr >= a.ns) {
                    atomicOr(a.status, 1);
                    sr = -1;
                }
            }
            sidx[tid] = sr;
        }
        __syncthreads();
        const float2 *Df = a.Dh + (long long)f * a.sDf;
        for (int u = tid; u < KC * 16; u += TC_THREADS) {
            const int k = u >> 4, ch = u & 15, at = ch >> 3, c = ch & 7;
            const int srow = sidx[k];
            float2 z[8];
            load8(srow >= 0 ? Df + (long long)srow * a.ldd : nullptr, cd + 64 * at + 8 * c, a.nr, z);
            store_planes(dst, at * (KC * 128) + k * 128 + ((c ^ (k & 7)) << 4), G::PLANE, split8(z, true));
        }
    }
}

// Tile bx of bin by (the upper-triangular enumeration with reciprocity); Q as for tc_fwd_body.  IMG: the
// operands come from the images of k_tc_adj_images (a.img).
template <bool RECIP, bool Q, bool TMA = false, bool IMG = false>
__device__ __forceinline__ void tc_adj_body(const GemmArgs &a, int bx, int by, uint32_t tmem_q,
                                            const CUtensorMap *tmap = nullptr) {
    using G = TcAdj;
    constexpr int KC = G::KC;
    extern __shared__ uint8_t tc_raw[];
    __shared__ uint64_t bar, probe_bar;
    __shared__ uint32_t tmem_holder;
    __shared__ int sidx[1024];
    __shared__ int fail, issued;
    uint8_t *sm = align1024(tc_raw);
    uint8_t *sA = sm, *sB = sm + 4 * G::PLANE;
    float2 *stg = reinterpret_cast<float2 *>(sm + G::OPER);
    const int f = by;
    int vb, rb;
    if (RECIP && a.diag_only) {
        vb = rb = bx;
    } else if (RECIP) {
        int t = bx, row = 0, len = a.tiles_v;
        while (t >= len) { t -= len; ++row; --len; }
        vb = row;
        rb = row + t;
    } else {
        vb = bx / a.tiles_r;
        rb = bx % a.tiles_r;
    }
    const int v0 = vb * 128, r0 = rb * 128;
    if (a.nf_active > 0 && f >= a.nf_active) {   // above the band limit: zero products, no TMEM
        const long long row = (long long)a.ldr * SPEC_F;
        zero_tile(a.C + spec_bin(f, a.sCf), row, v0, 128, r0, 128, a.nv, a.nr);
        if (RECIP) zero_tile(a.C + spec_bin(f, a.sCf), row, r0, 128, v0, 128, a.nr, a.nv);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float2 *Rf = a.A + spec_bin(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf;

    if constexpr (!IMG) {
        for (int b = tid; b < a.nb; b += TC_THREADS) {
            int s = a.idx[b];
            if (s < 0 || s >= a.ns) {
                atomicOr(a.status, 1);
                s = -1;
            }
            sidx[b] = s;
        }
    }
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init(&probe_bar, 1);
        fail = 0;
        issued = 0;
        fence_mbar_init();
    }
    if (!Q && warp == 0) tmem_alloc(&tmem_holder, G::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = Q ? tmem_q : tmem_holder;
    constexpr uint32_t idp = umma_idesc(128, 128, 1, 1, 0), idn = umma_idesc(128, 128, 1, 1, 1);
    // failure-path check: before any copy or product, wait on a barrier that nothing arrives on for a
    // short limit, then take the timeout path below
    if (a.wait_probe > 0) {
        if (tid == 0 && !mbar_wait_limit(&probe_bar, 0, a.wait_probe)) fail = 1;
        __syncthreads();
    }

    const int nkc = (a.nb + KC - 1) / KC;
    const int nhalf = RECIP ? 2 : 1;
    const int njobs = fail ? 0 : nkc * nhalf;
    constexpr int UD = KC * 16 / TC_THREADS;            // kernel-row units (8 complex) per thread
    int phase = 0;
    for (int job = 0; job < njobs; ++job) {
        const int kc = job / nhalf, half = job % nhalf;
        const int k0 = kc * KC;
        const int kn = min(KC, a.nb - k0), kpad = (kn + 15) & ~15;
        if constexpr (IMG) {
            // the previous products must be done reading the planes
            if (job > 0) {
                if (!mbar_wait_bounded(&bar, phase & 1)) fail = 1;
                ++phase;
            }
            tc_fence_after();
            // half 0: A' = R image of the row block, B' = D image of the column block; half 1 the other way
            const int nbl = a.tiles_v + a.tiles_r;
            const uint8_t *base = a.img + ((long long)f * a.img_nkc + kc) * nbl * (long long)TC_ADJ_IMG;
            const uint8_t *ia = base + (long long)(half ? a.tiles_v + vb : vb) * TC_ADJ_IMG;
            const uint8_t *ib = base + (long long)(half ? rb : a.tiles_v + rb) * TC_ADJ_IMG;
            for (int u = tid; u < TC_ADJ_IMG / 16; u += TC_THREADS) {
                cp_async16_zfill(sA + 16 * u, ia + 16 * u, 16);
                cp_async16_zfill(sB + 16 * u, ib + 16 * u, 16);
            }
            cp_async_commit_wait_all();
            fence_async_smem();
            __syncthreads();
        } else {
        const int cr = half ? r0 : v0, ncr = half ? a.nr : a.nv;   // residual rows of this half
        const int cd = half ? v0 : r0, ncd = half ? a.nv : a.nr;   // kernel-row columns of this half
        // residual rows -> staging (cp.async, zero-filled past the matrix); the staging tile was
        // released by the __syncthreads before the previous job's products
        for (int u = tid; u < 128 * (KC / 2); u += TC_THREADS) {
            const int row = u / (KC / 2), pr = u % (KC / 2), k = k0 + 2 * pr, rr = cr + row;
            int bytes = 0;
            const float2 *src = Rf;
            if (rr < ncr && k < a.nb) {
                bytes = (k + 1 < a.nb) ? 16 : 8;
                src = Rf + (long long)rr * a.ldb * SPEC_F + spec_col(k);
            }
            cp_async16_zfill(stg + row * G::SLD + 2 * pr, src, bytes);
        }
        // kernel rows (MN-major operand) -> registers
        float2 zd[UD][8];
#pragma unroll
        for (int i = 0; i < UD; ++i) {
            const int u = tid + i * TC_THREADS, k = u >> 4, ch = u & 15, at = ch >> 3, c = ch & 7;
            const int srow = (k < kn) ? sidx[k0 + k] : -1;
            load8(srow >= 0 ? Df + (long long)srow * a.ldd : nullptr, cd + 64 * at + 8 * c, ncd, zd[i]);
        }
        // the previous products must be done reading the planes
        if (job > 0) {
            if (!mbar_wait_bounded(&bar, phase & 1)) fail = 1;
            ++phase;
        }
        tc_fence_after();
        uint8_t *pD = half ? sA : sB, *pR = half ? sB : sA;
#pragma unroll
        for (int i = 0; i < UD; ++i) {
            const int u = tid + i * TC_THREADS, k = u >> 4, ch = u & 15, at = ch >> 3, c = ch & 7;
            store_planes(pD, at * (KC * 128) + k * 128 + ((c ^ (k & 7)) << 4), G::PLANE, split8(zd[i], true));
        }
        cp_async_commit_wait_all();
        __syncthreads();
        // staging -> transposed, split residual planes: thread (k, chunk) takes 8 consecutive rows
        for (int u = tid; u < KC * 16; u += TC_THREADS) {
            const int k = u % KC, ch = u / KC, at = ch >> 3, c = ch & 7;
            float2 z[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) z[j] = stg[(64 * at + 8 * c + j) * G::SLD + k];
            store_planes(pR, at * (KC * 128) + k * 128 + ((c ^ (k & 7)) << 4), G::PLANE, split8(z, false));
        }
        fence_async_smem();
        __syncthreads();
        }
        if (fail) break;
        if (tid == 0) {
            tc_fence_after();
            for (int ks = 0; ks < kpad / 16; ++ks) {
                uint64_t ad[4], bd[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    ad[p] = umma_desc(smem_u32(sA + p * G::PLANE + ks * 16 * 128), KC * 128, 1024);
                    bd[p] = umma_desc(smem_u32(sB + p * G::PLANE + ks * 16 * 128), KC * 128, 1024);
                }
                mma_complex_split(tmem, tmem + 128, ad, bd, idp, idn, (job > 0 || ks > 0) ? 1u : 0u);
            }
            umma_commit(&bar);
            issued = 1;
        }
    }
    if (!fail && !mbar_wait_bounded(&bar, phase & 1)) fail = 1;
    __syncthreads();
    const bool ok = !fail;
    // after a timeout, give products still in flight one more bounded wait before TMEM is freed
    if (!ok && issued) mbar_wait_bounded(&bar, phase & 1);
    tc_fence_after();
    // epilogue by the tensor memory accelerator for a tile written once (no reciprocity, or an off-diagonal
    // tile of a symmetric model's adjoint, whose mirror is not needed), in two passes of 64 columns: TMEM ->
    // eight staged boxes of 8 complex x 128 rows (64-byte swizzle: granule g of row m at g ^ (m / 2 % 4)) ->
    // eight tiled stores of the tensor map of C (clipped at nv and at the last chunk of 8; the columns past nr of
    // that chunk are padding, which no kernel reads as data)
    if (TMA && (!RECIP || (a.no_mirror && vb != rb))) {
        for (int pass = 0; pass < 2; ++pass) {
            if (ok) {
                const int q = warp & 3, hc = warp >> 2;   // lanes 32q.., columns 32hc.. of this pass
                const int row = 32 * q + lane;
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 16) {
                    const int col = 64 * pass + 32 * hc + c0;
                    float re[16], im[16];
                    tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + col, re);
                    tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + 128 + col, im);
                    uint8_t *box = sm + ((32 * hc + c0) >> 3) * (128 * 64) + row * 64;
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        *reinterpret_cast<float4 *>(box + (g >> 2) * (128 * 64) + (((g & 3) ^ ((row >> 1) & 3)) << 4)) =
                            make_float4(re[2 * g] * a.outscale, im[2 * g] * a.outscale, re[2 * g + 1] * a.outscale,
                                        im[2 * g + 1] * a.outscale);
                }
            }
            fence_async_smem();   // the staged boxes are visible to the tensor memory accelerator
            tc_fence_before();
            __syncthreads();
            if (ok && tid == 0) {
#pragma unroll
                for (int b8 = 0; b8 < 8; ++b8) {
                    const int r = r0 + 64 * pass + 8 * b8;
                    if (r < a.nr) tma_store_5d(tmap, sm + b8 * (128 * 64), 0, f % SPEC_F, r >> 3, v0, f / SPEC_F);
                }
                bulk_commit();
                bulk_wait_read();   // the staging may be written again
            }
            __syncthreads();
        }
        if (ok && tid == 0) bulk_wait_all();
        if (!ok && tid == 0) atomicOr(a.status, 2);
        if constexpr (Q) {
            if (tid == 0) {
                mbar_inval(&bar);
                mbar_inval(&probe_bar);
            }
        } else {
            if (warp == 0) tmem_dealloc(tmem, G::TMEM_COLS);
        }
        return;
    }
    // epilogue in two passes of 64 columns: TMEM -> shared staging [128][65] -> coalesced rows (and
    // the mirror)
    float2 *out = reinterpret_cast<float2 *>(sm);
    float2 *Cf = a.C + spec_bin(f, a.sCf);
    const long long crow = (long long)a.ldr * SPEC_F;
    const bool diag = RECIP && vb == rb;
    for (int pass = 0; pass < 2; ++pass) {
        if (ok) {
            const int q = warp & 3, hc = warp >> 2;   // lanes 32q.., columns 32hc.. of this pass
            const int row = 32 * q + lane;
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += 16) {
                const int col = 64 * pass + 32 * hc + c0;
                float re[16], im[16];
                tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + col, re);
                tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + 128 + col, im);
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    out[row * 65 + 32 * hc + c0 + j] = make_float2(re[j] * a.outscale, im[j] * a.outscale);
            }
        }
        tc_fence_before();
        __syncthreads();
        if (ok) {
            const int rp = r0 + 64 * pass;
            for (int e = tid; e < 128 * 64; e += TC_THREADS) {
                const int row = e >> 6, col = e & 63, v = v0 + row, r = rp + col;
                if (v < a.nv && r < a.nr && (!diag || v <= r)) Cf[v * crow + spec_col(r)] = out[row * 65 + col];
            }
            // the mirror (diagonal tiles always: their lower half is read by the update of a symmetric model)
            if (RECIP && (diag || !a.no_mirror)) {
                for (int e = tid; e < 128 * 64; e += TC_THREADS) {
                    const int rr = e >> 7, vv = e & 127, v = v0 + vv, r = rp + rr;
                    if (v < a.nv && r < a.nr && (!diag || v < r)) Cf[r * crow + spec_col(v)] = out[vv * 65 + rr];
                }
            }
        }
        __syncthreads();
    }
    if (!ok && tid == 0) atomicOr(a.status, 2);
    if constexpr (Q) {
        // the last loop iteration ended with a barrier after every wait: the barriers are free
        if (tid == 0) {
            mbar_inval(&bar);
            mbar_inval(&probe_bar);
        }
    } else {
        if (warp == 0) tmem_dealloc(tmem, G::TMEM_COLS);
    }
}

template <bool RECIP, bool IMG = false>
__global__ void __launch_bounds__(TC_THREADS, 2) k_tc_adj(GemmArgs a) {
    tc_adj_body<RECIP, false, false, IMG>(a, blockIdx.x, blockIdx.y, 0);
}

// the adjoint without reciprocity with its tile written by the tensor memory accelerator (tmap: the
// tensor map of the gradient spectra, i.e. of the model-spectra buffer)
template <bool IMG = false>
__global__ void __launch_bounds__(TC_THREADS, 2) k_tc_adj_tma(GemmArgs a, const __grid_constant__ CUtensorMap tmap) {
    tc_adj_body<false, false, true, IMG>(a, blockIdx.x, blockIdx.y, 0, &tmap);
}

// the adjoint of a symmetric model (reciprocity, a.no_mirror): off-diagonal tiles written by the tensor memory
// accelerator, diagonal tiles with their mirror by the threads
template <bool IMG = false>
__global__ void __launch_bounds__(TC_THREADS, 2) k_tc_adj_sym_tma(GemmArgs a, const __grid_constant__ CUtensorMap tmap) {
    tc_adj_body<true, false, true, IMG>(a, blockIdx.x, blockIdx.y, 0, &tmap);
}

// work-queue form: tile t of a problem is (bx, by) = (t % tiles, t / tiles) with tiles the output tiles
// of one bin (the upper triangle with reciprocity); tiles_v / tiles_r are set in the argument records
template <bool RECIP>
__global__ void __launch_bounds__(TC_THREADS, 2) k_tc_adj_q(WorkQueue q) {
    __shared__ uint32_t holder;
    const int warp = threadIdx.x >> 5;
    if (warp == 0) tmem_alloc(&holder, TcAdj::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = holder;
    const GemmArgs *args = static_cast<const GemmArgs *>(q.args);
    int m = 0, tile = 0;
    __shared__ GemmArgs sa;
    while (queue_next(q, m, tile) >= 0) {
        queue_args(args + m, sa);
        __syncthreads();
        const GemmArgs &a = sa;
        const int tiles = RECIP ? a.tiles_v * (a.tiles_v + 1) / 2 : a.tiles_v * a.tiles_r;
        tc_adj_body<RECIP, true>(a, tile % tiles, tile / tiles, tmem);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TcAdj::TMEM_COLS);
}

// ------------------------------------------------------------------------------------------------
// forward, persistent: the product of tc_fwd_body (same split, same MMAs in the same order, bit-identical) as a
// warp-specialised kernel, one CTA per SM, fed by the tensor memory accelerator, A operand in tensor memory.
// A unit is (two neighbouring bins, 128 rows v, NB batch columns): the SPEC_F layout holds the two bins of 8 columns
// in one 128-byte line.  K = nr runs in chunks of 32 columns (64 KB of both bins).
//  * copy warp (16): tiled copies of boxes of 128 rows x 8 columns x 2 bins (16 KB, 128-byte swizzle), four a chunk,
//    into a ring of RING boxes;
//  * split warps (0-15): thread (row, 8 columns) reads its FP32 values from the staging buffer, splits them and
//    writes the four BF16 planes to tensor memory (tcgen05.st), so the A operand never returns to shared memory:
//    there the product would read every plane three times, 12 x 4 KB a K step, more than the chunk itself.  The
//    gathered kernel rows (in registers one chunk ahead) go to shared-memory planes -Bi, Br, Bi (hi and lo).  Two
//    stages of planes.
//  * MMA warp (17): 6 MMAs of N = 2 NB per K step of 16 and bin, Ar [Br | Bi] and Ai [-Bi | Br] with the accumulators
//    [re | im]: the 12 products of the tile kernel in their order, in half the instructions (the one issuing
//    thread takes about 60 cycles for each, which bound the kernel with 12).
// The split warps also write C: the accumulators of a unit are read after the first chunk of the next one has been
// split (for NB <= 32 there are two sets, so the next unit's products do not wait for it).
// SYM: spectra of a symmetric model, stored on and above the sym_tr-block diagonal.  Chunks wholly below it are copied
// as transposed boxes (8 rows x 128 columns) and read by columns; chunks that straddle it are read from global
// memory by the threads.
// Units go to the CTAs in rounds, so that the CTAs work on neighbouring bins at a time (contiguous ranges of units per
// CTA: 822 against 655 us at nt 1500, 600 columns, 384 rows), rotated by one CTA a round, so that every CTA gets its
// share of ragged last tiles (unrotated, a tile count that divides the grid gives some CTAs none: 842 us for 400
// rows, 655 us for 384).
// Waits (all on mbarriers, all bounded): full (a box landed), empty (a box read), aready (planes written), adone
// (products of a stage finished), ddone (products of a unit finished), dfree (accumulators read).
// ------------------------------------------------------------------------------------------------
constexpr int TCP_SPLIT = 512;                 // split warps 0-15
constexpr int TCP_THREADS = TCP_SPLIT + 64;    // + copy warp, MMA warp
constexpr int TCP_KC = 32;                     // columns of a chunk

template <int NB>
struct TcFwdP {
    static constexpr int BOX = 128 * 128;                    // 128 rows x 8 columns x 2 bins
    // boxes in flight or being read; a multiple of 4, so that a slot always belongs to the same four split warps:
    // their wait for one round of the slot then follows their wait for the round before (a warp that skipped a
    // round would pass the parity test of the next one at once)
    static constexpr int RING = NB <= 32 ? 8 : 4;
    static_assert(RING % 4 == 0, "a slot belongs to one group of split warps");
    static constexpr int B_PLANE = NB * 128;                 // rows b: 32 k of bin 0, 32 k of bin 1
    static constexpr int B_STAGE = 6 * B_PLANE;              // hi: -Bi, Br, Bi; lo: the same
    static constexpr int OUT = 16 * 2048;                    // per split warp: 32 rows x 8 columns
    static constexpr size_t SMEM = RING * (size_t)BOX + 2 * B_STAGE + OUT + 1024;
    static constexpr int DBUF = NB <= 32 ? 2 : 1;            // sets of accumulators
    static constexpr int D_COLS = 4 * NB;                    // two bins x (re, im)
    static constexpr int A_COL = DBUF * D_COLS;              // planes: [stage][bin][plane][16 columns]
    static_assert(A_COL + 256 <= 512, "accumulators and two stages of A planes fill the tensor memory");
    static_assert(SMEM <= 232448, "one CTA per SM");
};

struct FwdUnit {
    int f, v0, b0;   // first bin of the pair, first row, first batch column
};
template <int NB>
__device__ __forceinline__ FwdUnit fwd_unit(int t, int gx, int gy) {
    const int vt = t % gx, r = t / gx;
    return FwdUnit{2 * (r / gy), vt * 128, (r % gy) * NB};
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// A from tensor memory
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint4 v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(taddr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w));
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint4 neg_bf16x8(uint4 v) {
    return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}

// which part of a symmetric model's spectra a chunk (columns k0 .. k0 + 31 of rows v0 .. v0 + 127) lies in
enum { CH_DIRECT = 0, CH_TRANSPOSED = 1, CH_MIXED = 2 };
template <bool SYM>
__device__ __forceinline__ int chunk_kind(const GemmArgs &a, int v0, int k0) {
    if (!SYM) return CH_DIRECT;
    const int vl = min(v0 + 127, a.nv - 1);
    if (k0 + TCP_KC <= a.sym_tr * (v0 / a.sym_tr)) return CH_TRANSPOSED;
    return k0 >= a.sym_tr * (vl / a.sym_tr) ? CH_DIRECT : CH_MIXED;
}

template <int NB, bool SYM>
__global__ void __launch_bounds__(TCP_THREADS, 1)
    k_tc_fwd_p(GemmArgs a, const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap tmap_t, int gx, int gy,
               int nf, int nf_act, int n_units) {
    using G = TcFwdP<NB>;
    extern __shared__ uint8_t tc_raw[];
    __shared__ uint64_t full[G::RING], empty[G::RING], aready[2], adone[2], ddone[G::DBUF], dfree[G::DBUF], probe;
    __shared__ uint32_t tmem_holder;
    __shared__ int fail, s_copies, s_mma;      // copies and stages of products issued, for the failure path
    uint8_t *stg0 = align1024(tc_raw);
    uint8_t *bpl0 = stg0 + G::RING * G::BOX;
    uint8_t *out0 = bpl0 + 2 * G::B_STAGE;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // bins above the band limit: zero products (pairs that hold an active bin are handled with their unit)
    if (nf_act < nf)
        for (int t = gx * gy * ((nf_act + 1) / 2) + blockIdx.x; t < gx * gy * ((nf + 1) / 2); t += gridDim.x) {
            const FwdUnit U = fwd_unit<NB>(t, gx, gy);
            for (int f = U.f; f < min(U.f + 2, nf); ++f)
                zero_tile(a.C + spec_bin(f, a.sCf), (long long)a.ldb * SPEC_F, U.v0, 128, U.b0, NB, a.nv, a.nb);
        }
    const int rounds = n_units / (int)gridDim.x;   // whole rounds; unit i of this CTA is i gridDim + (blockIdx + i) % gridDim
    const int my_units = rounds + (((int)blockIdx.x + rounds) % (int)gridDim.x < n_units % (int)gridDim.x ? 1 : 0);
    if (my_units == 0) return;
    const int nk = (a.nr + TCP_KC - 1) / TCP_KC;

    if (tid == 0) {
        for (int i = 0; i < G::RING; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 4);   // the four split warps that read the box
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&aready[i], TCP_SPLIT / 32);
            mbar_init(&adone[i], 1);
        }
        for (int i = 0; i < G::DBUF; ++i) {
            mbar_init(&ddone[i], 1);
            mbar_init(&dfree[i], TCP_SPLIT / 32);
        }
        mbar_init(&probe, 1);
        fail = 0;
        s_copies = s_mma = 0;
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(&tmem_holder, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_holder;
    // failure-path check: before any copy or product, wait on a barrier that nothing arrives on for a short limit
    if (a.wait_probe > 0) {
        if (tid == 0 && !mbar_wait_limit(&probe, 0, a.wait_probe)) fail = 1;
        __syncthreads();
    }
    volatile int *vfail = &fail;
    auto unit_at = [&](int u) { return fwd_unit<NB>(u * (int)gridDim.x + (int)((blockIdx.x + u) % gridDim.x), gx, gy); };

    if (*vfail) {
        // nothing was issued
    } else if (warp == TCP_SPLIT / 32) {
        // ---------------- copy warp ----------------
        if (lane == 0) {
            int n = 0, slot = 0, round = 0;   // box, its ring slot, times around the ring
            for (int u = 0; u < my_units && !*vfail; ++u) {
                const FwdUnit U = unit_at(u);
                const int pr = (U.f % SPEC_F) / 2, fb = U.f / SPEC_F;
                for (int kc = 0; kc < nk && !*vfail; ++kc) {
                    const int k0 = kc * TCP_KC, kind = chunk_kind<SYM>(a, U.v0, k0);
                    for (int j = 0; j < 4; ++j) {
                        if (round > 0 && !mbar_wait_bounded(&empty[slot], (round - 1) & 1)) fail = 1;
                        if (*vfail) break;
                        if (SYM && kind == CH_MIXED) {
                            mbar_arrive(&full[slot]);
                        } else {
                            mbar_arrive_expect_tx(&full[slot], (uint32_t)G::BOX);
                            if (SYM && kind == CH_TRANSPOSED) tma_load_5d(stg0 + slot * G::BOX, &tmap_t, 0, pr, U.v0 / 8, k0 + 8 * j, fb, &full[slot]);
                            else tma_load_5d(stg0 + slot * G::BOX, &tmap, 0, pr, k0 / 8 + j, U.v0, fb, &full[slot]);
                        }
                        s_copies = ++n;
                        if (++slot == G::RING) {
                            slot = 0;
                            ++round;
                        }
                    }
                }
            }
        }
    } else if (warp == TCP_SPLIT / 32 + 1) {
        // ---------------- MMA warp ----------------
        if (lane == 0) {
            constexpr uint32_t id = umma_idesc(128, 2 * NB, 0, 0, 0);
            const uint64_t bd0 = umma_desc(smem_u32(bpl0), 16, 1024);
            constexpr uint64_t PL = G::B_PLANE >> 4;
            int g = 0;
            for (int u = 0; u < my_units; ++u) {
                const int db = u % G::DBUF;
                if (u >= G::DBUF && !mbar_wait_bounded(&dfree[db], (u / G::DBUF - 1) & 1)) fail = 1;
                for (int kc = 0; kc < nk; ++kc, ++g) {
                    const int s = g & 1;
                    if (!*vfail && !mbar_wait_bounded(&aready[s], (g / 2) & 1)) fail = 1;
                    if (*vfail) break;
                    tc_fence_after();
                    const uint64_t bs = bd0 + (uint64_t)s * (G::B_STAGE >> 4);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {   // the two bins
                        const uint32_t d = tmem + db * G::D_COLS + h * 2 * NB;
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks) {
                            const uint32_t ad = tmem + G::A_COL + s * 128 + h * 64 + ks * 8;   // re hi, re lo, im hi, im lo 16 apart
                            const uint64_t bd = bs + h * 4 + ks * 2;                          // planes -Bi, Br, Bi of hi, then of lo
                            umma_bf16_ts(d, ad, bd + PL, id, (kc > 0 || ks > 0) ? 1u : 0u);
                            umma_bf16_ts(d, ad, bd + 4 * PL, id, 1);
                            umma_bf16_ts(d, ad + 16, bd + PL, id, 1);
                            umma_bf16_ts(d, ad + 32, bd, id, 1);
                            umma_bf16_ts(d, ad + 32, bd + 3 * PL, id, 1);
                            umma_bf16_ts(d, ad + 48, bd, id, 1);
                        }
                    }
                    umma_commit(&adone[s]);
                    if (kc == nk - 1) umma_commit(&ddone[db]);
                    s_mma = g + 1;
                }
                if (*vfail) break;
            }
        }
    } else {
        // ---------------- split warps ----------------
        const int q = warp & 3, cc = warp >> 2, m = 32 * q + lane;   // rows 32q .., columns 8cc .. of a chunk
        const uint32_t lanes = (uint32_t)(32 * q) << 16;
        auto failed = [&] { return __any_sync(0xffffffffu, *vfail) != 0; };   // warp-uniform
        // thread u < 8 NB: kernel row u / 8, bin (u % 8) / 4, columns 8 (u % 4) .. of a chunk
        const bool has_b = tid < NB * 8;
        const int brow = tid >> 3, bc = tid & 7;
        const float2 *brp = nullptr;   // this thread's kernel row, for the unit of the next load
        auto b_row = [&](const FwdUnit &U) {
            brp = nullptr;
            if (!has_b || U.b0 + brow >= a.nb) return;
            const int s = a.idx[U.b0 + brow], f = U.f + (bc >> 2);
            if (s < 0 || s >= a.ns) {
                atomicOr(a.status, 1);
                return;
            }
            if (f < nf_act) brp = a.Dh + (long long)f * a.sDf + (long long)s * a.ldd;
        };
        auto epilogue = [&](int u) {
            const FwdUnit U = unit_at(u);
            const int db = u % G::DBUF;
            if (!mbar_wait_bounded(&ddone[db], (u / G::DBUF) & 1)) fail = 1;
            if (failed()) return;
            tc_fence_after();
            uint8_t *out = out0 + warp * 2048;
            // 8 columns of one bin at a time: TMEM -> 32 rows x 64 bytes -> rows of C
            for (int e = cc; e < 2 * (NB / 8); e += 4) {
                const int h = e & 1, c0 = (e >> 1) * 8, f = U.f + h;
                float re[8], im[8];
                const uint32_t d = tmem + lanes + db * G::D_COLS + h * 2 * NB + c0;
                tmem_ld8(d, re);
                tmem_ld8(d + NB, im);
                const bool live = f < nf_act;   // (a band limit may cut the pair)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<float4 *>(out + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) =
                        live ? make_float4(re[2 * j], im[2 * j], re[2 * j + 1], im[2 * j + 1]) : make_float4(0.f, 0.f, 0.f, 0.f);
                __syncwarp();
                if (f < nf) {
                    const int b = U.b0 + c0 + 2 * (lane & 3);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int row = 8 * i + (lane >> 2), v = U.v0 + 32 * q + row;
                        const float4 w = *reinterpret_cast<const float4 *>(out + row * 64 + (((lane & 3) ^ ((row >> 1) & 3)) << 4));
                        float2 *dst = a.C + spec_bin(f, a.sCf) + (long long)v * a.ldb * SPEC_F + spec_col(b);
                        if (v < a.nv) {
                            if (b + 1 < a.nb) *reinterpret_cast<float4 *>(dst) = w;
                            else if (b < a.nb) *dst = make_float2(w.x, w.y);
                        }
                    }
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dfree[db]);
        };

        float2 zb[8];
        FwdUnit U = unit_at(0);
        b_row(U);
        load8(brp, 8 * (bc & 3), a.nr, zb);
        int g = 0, slot = cc, round = 0;   // chunk, ring slot of this warp's box, times around the ring
        for (int u = 0; u < my_units; ++u) {
            for (int kc = 0; kc < nk; ++kc, ++g) {
                const int s = g & 1, k0 = kc * TCP_KC;
                const int kind = chunk_kind<SYM>(a, U.v0, k0);
                const uint8_t *box = stg0 + slot * G::BOX;
                const int left = a.nr - (k0 + 8 * cc);   // columns of this thread inside the matrix (past it: padding)
                float2 z[2][8];
                if (!mbar_wait_bounded(&full[slot], round & 1)) fail = 1;
                if (!SYM || kind == CH_DIRECT) {
                    const uint8_t *row = box + m * 128;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 w = *reinterpret_cast<const float4 *>(row + ((j ^ (m & 7)) << 4));
                        z[j >> 2][2 * (j & 3)] = make_float2(w.x, w.y);
                        z[j >> 2][2 * (j & 3) + 1] = make_float2(w.z, w.w);
                    }
                } else if (kind == CH_TRANSPOSED) {
                    // row k of the box: 128 columns v in chunks of 8, both bins
                    const int x = (m >> 3) & 7;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            z[h][i] = *reinterpret_cast<const float2 *>(box + i * 2048 + (m >> 3) * 128 +
                                                                        (((h * 4 + ((m & 7) >> 1)) ^ x) << 4) + (m & 1) * 8);
                } else {
                    const int v = U.v0 + m;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int i = 0; i < 8; ++i) z[h][i] = make_float2(0.f, 0.f);
                    if (v < a.nv) {
                        const int lo = a.sym_tr * (v / a.sym_tr);
                        for (int h = 0; h < 2; ++h)   // (the second bin of the last pair lies in the padding of its block)
                            load8_sym(a.A + spec_bin(U.f + h, a.sAf), (long long)a.ldr * SPEC_F, v, k0 + 8 * cc, a.nr, lo, z[h]);
                    }
                }
                if (left < 8) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (i >= left) z[h][i] = make_float2(0.f, 0.f);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[slot]);   // the box has been read
                slot += 4;
                if (slot >= G::RING) {
                    slot -= G::RING;
                    ++round;
                }
                if (g >= 2 && !mbar_wait_bounded(&adone[s], (g / 2 - 1) & 1)) fail = 1;   // planes of stage s free
                if (failed()) break;
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const Chunk4 c = split8(z[h], false);
                    const uint32_t col = tmem + lanes + G::A_COL + s * 128 + h * 64 + (cc >> 1) * 8 + (cc & 1) * 4;
                    tmem_st4(col, c.rh);
                    tmem_st4(col + 16, c.rl);
                    tmem_st4(col + 32, c.ih);
                    tmem_st4(col + 48, c.il);
                }
                if (has_b) {
                    const Chunk4 c = split8(zb, false);
                    uint8_t *p = bpl0 + s * G::B_STAGE + brow * 128 + ((bc ^ (brow & 7)) << 4);
                    *reinterpret_cast<uint4 *>(p) = neg_bf16x8(c.ih);
                    *reinterpret_cast<uint4 *>(p + G::B_PLANE) = c.rh;
                    *reinterpret_cast<uint4 *>(p + 2 * G::B_PLANE) = c.ih;
                    *reinterpret_cast<uint4 *>(p + 3 * G::B_PLANE) = neg_bf16x8(c.il);
                    *reinterpret_cast<uint4 *>(p + 4 * G::B_PLANE) = c.rl;
                    *reinterpret_cast<uint4 *>(p + 5 * G::B_PLANE) = c.il;
                }
                tmem_wait_st();
                fence_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&aready[s]);
                // kernel rows of the next chunk
                if (kc + 1 < nk) {
                    load8(brp, k0 + TCP_KC + 8 * (bc & 3), a.nr, zb);
                } else if (u + 1 < my_units) {
                    U = unit_at(u + 1);
                    b_row(U);
                    load8(brp, 8 * (bc & 3), a.nr, zb);
                }
                if (kc == 0 && u > 0) epilogue(u - 1);
            }
            if (failed()) break;
        }
        if (!failed()) epilogue(my_units - 1);
    }
    __syncthreads();
    if (fail && tid == 0) {
        // copies and products still in flight get one more bounded wait before the CTA frees TMEM and exits
        for (int i = max(0, s_copies - G::RING); i < s_copies; ++i) mbar_wait_bounded(&full[i % G::RING], (i / G::RING) & 1);
        for (int i = max(0, s_mma - 2); i < s_mma; ++i) mbar_wait_bounded(&adone[i & 1], (i / 2) & 1);
        atomicOr(a.status, 2);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------------
// adjoint, persistent: the product of tc_adj_body from the operand images (same MMAs in the same order, bit-identical) for
// tiles that are written once, where it is the faster kernel (adj_persistent): every tile without reciprocity, the off-diagonal ones of a symmetric model (OFF; its
// diagonal tiles, with their mirror, run on k_tc_adj_sym_tma).  One CTA per SM walks its tiles; its roles overlap from
// tile to tile, where the tile kernel runs load, products and stores of a tile one after the other (15 000 cycles a tile
// at two CTAs per SM for 3 700 cycles of output at the HBM rate, nt 1024, 301 x 301, batch 32):
//  * copy warp (8): the two images of a job (a K chunk, a half) by bulk copies of 32 KB into one of two stages;
//  * MMA warp (9): the products of a job; two sets of accumulators fill the tensor memory;
//  * store warps (0-7): 16 columns of 32 rows at a time, tensor memory -> the warp's own staging (two buffers of two
//    boxes of 8 columns x 32 rows, 64-byte swizzle) -> tiled stores (clipped at nv and the last chunk of 8 of nr).
// Tiles go to the CTAs in rounds rotated by one CTA a round, as the forward product's units.
// ------------------------------------------------------------------------------------------------
constexpr int TAP_STORE = 256;                 // store warps 0-7
constexpr int TAP_THREADS = TAP_STORE + 64;    // + copy warp, MMA warp
constexpr int TAP_STAGE = 2 * TC_ADJ_IMG;      // operand planes of a job
constexpr int TAP_OUT = 8 * 8192;
constexpr size_t TAP_SMEM = 2 * (size_t)TAP_STAGE + TAP_OUT + 1024;

__device__ __forceinline__ void bulk_load(void *smem_dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(smem_u32(smem_dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// at most one of this thread's committed bulk stores still reads its shared-memory source
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;\n" ::: "memory"); }

// tile t of nf bins: the bins of a block of SPEC_F fastest (their outputs share 256-byte lines, written by neighbouring
// CTAs at a time), then the tiles of a bin
template <bool OFF>
__device__ __forceinline__ void adj_tile(const GemmArgs &a, int t, int tiles, int nf, int &f, int &vb, int &rb) {
    const int whole = nf / SPEC_F * SPEC_F * tiles;   // tiles of the whole blocks
    int x;
    if (t < whole) {
        x = t / SPEC_F;
        f = x / tiles * SPEC_F + t % SPEC_F;
    } else {
        x = t - whole;
        f = nf / SPEC_F * SPEC_F + x / tiles;
    }
    x %= tiles;
    if (OFF) {   // vb < rb
        int len = a.tiles_v - 1;
        vb = 0;
        while (x >= len) { x -= len; ++vb; --len; }
        rb = vb + 1 + x;
    } else {
        vb = x / a.tiles_r;
        rb = x % a.tiles_r;
    }
}

template <bool OFF>
__global__ void __launch_bounds__(TAP_THREADS, 1)
    k_tc_adj_p(GemmArgs a, const __grid_constant__ CUtensorMap tmap, int tiles, int nf, int nf_act) {
    using G = TcAdj;
    constexpr int KC = G::KC;
    extern __shared__ uint8_t tc_raw[];
    __shared__ uint64_t full[2], adone[2], ddone[2], dfree[2], probe;
    __shared__ uint32_t tmem_holder;
    __shared__ int fail, s_copies, s_mma;
    uint8_t *op0 = align1024(tc_raw), *out0 = op0 + 2 * TAP_STAGE;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    for (int t = blockIdx.x; t < (nf - nf_act) * tiles; t += gridDim.x) {   // above the band limit
        int f, vb, rb;
        adj_tile<OFF>(a, t, tiles, nf - nf_act, f, vb, rb);
        f += nf_act;
        const long long row = (long long)a.ldr * SPEC_F;
        zero_tile(a.C + spec_bin(f, a.sCf), row, vb * 128, 128, rb * 128, 128, a.nv, a.nr);
        if (OFF) zero_tile(a.C + spec_bin(f, a.sCf), row, rb * 128, 128, vb * 128, 128, a.nr, a.nv);
    }
    const int n_tiles = nf_act * tiles, rounds = n_tiles / (int)gridDim.x;
    const int my_tiles = rounds + (((int)blockIdx.x + rounds) % (int)gridDim.x < n_tiles % (int)gridDim.x ? 1 : 0);
    if (my_tiles == 0) return;
    auto tile_at = [&](int u, int &f, int &vb, int &rb) {
        adj_tile<OFF>(a, u * (int)gridDim.x + (int)((blockIdx.x + u) % gridDim.x), tiles, nf_act, f, vb, rb);
    };
    constexpr int NH = OFF ? 2 : 1;
    const int njobs = a.img_nkc * NH;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&adone[i], 1);
            mbar_init(&ddone[i], 1);
            mbar_init(&dfree[i], TAP_STORE / 32);
        }
        mbar_init(&probe, 1);
        fail = 0;
        s_copies = s_mma = 0;
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(&tmem_holder, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_holder;
    if (a.wait_probe > 0) {   // failure-path check, before any copy or product
        if (tid == 0 && !mbar_wait_limit(&probe, 0, a.wait_probe)) fail = 1;
        __syncthreads();
    }
    volatile int *vfail = &fail;

    if (*vfail) {
        // nothing was issued
    } else if (warp == TAP_STORE / 32) {
        // ---------------- copy warp ----------------
        if (lane == 0) {
            const int nbl = a.tiles_v + a.tiles_r;
            int g = 0;
            for (int u = 0; u < my_tiles && !*vfail; ++u) {
                int f, vb, rb;
                tile_at(u, f, vb, rb);
                for (int job = 0; job < njobs; ++job, ++g) {
                    const int s = g & 1, kc = job / NH, half = job % NH;
                    if (g >= 2 && !mbar_wait_bounded(&adone[s], (g / 2 - 1) & 1)) fail = 1;
                    if (*vfail) break;
                    const uint8_t *base = a.img + ((long long)f * a.img_nkc + kc) * nbl * (long long)TC_ADJ_IMG;
                    uint8_t *op = op0 + s * TAP_STAGE;
                    mbar_arrive_expect_tx(&full[s], TAP_STAGE);
                    bulk_load(op, base + (long long)(half ? a.tiles_v + vb : vb) * TC_ADJ_IMG, TC_ADJ_IMG, &full[s]);
                    bulk_load(op + TC_ADJ_IMG, base + (long long)(half ? rb : a.tiles_v + rb) * TC_ADJ_IMG, TC_ADJ_IMG, &full[s]);
                    s_copies = g + 1;
                }
            }
        }
    } else if (warp == TAP_STORE / 32 + 1) {
        // ---------------- MMA warp ----------------
        if (lane == 0) {
            constexpr uint32_t idp = umma_idesc(128, 128, 1, 1, 0), idn = umma_idesc(128, 128, 1, 1, 1);
            const uint64_t a0 = umma_desc(smem_u32(op0), KC * 128, 1024), b0 = umma_desc(smem_u32(op0 + TC_ADJ_IMG), KC * 128, 1024);
            constexpr uint64_t PL = G::PLANE >> 4;
            int g = 0;
            for (int u = 0; u < my_tiles; ++u) {
                const int db = u & 1;
                if (u >= 2 && !mbar_wait_bounded(&dfree[db], (u / 2 - 1) & 1)) fail = 1;
                for (int job = 0; job < njobs; ++job, ++g) {
                    const int s = g & 1, kn = min(KC, a.nb - (job / NH) * KC);
                    if (!*vfail && !mbar_wait_bounded(&full[s], (g / 2) & 1)) fail = 1;
                    if (*vfail) break;
                    tc_fence_after();
                    const uint32_t d_re = tmem + db * 256, d_im = d_re + 128;
                    for (int ks = 0; ks < (kn + 15) / 16; ++ks) {
                        const uint64_t o = (uint64_t)(s * (TAP_STAGE >> 4) + ks * (16 * 128 >> 4));
                        const uint64_t ad[4] = {a0 + o, a0 + o + PL, a0 + o + 2 * PL, a0 + o + 3 * PL};
                        const uint64_t bd[4] = {b0 + o, b0 + o + PL, b0 + o + 2 * PL, b0 + o + 3 * PL};
                        mma_complex_split(d_re, d_im, ad, bd, idp, idn, (job > 0 || ks > 0) ? 1u : 0u);
                    }
                    umma_commit(&adone[s]);
                    if (job == njobs - 1) umma_commit(&ddone[db]);
                    s_mma = g + 1;
                }
                if (*vfail) break;
            }
        }
    } else {
        // ---------------- store warps ----------------
        auto failed = [&] { return __any_sync(0xffffffffu, *vfail) != 0; };   // warp-uniform
        const int q = warp & 3, hc = warp >> 2;   // rows 32q .., columns 64hc .. of a tile
        uint8_t *out = out0 + warp * 8192;
        int nst = 0;   // stores of this warp so far: they alternate between its two buffers
        for (int u = 0; u < my_tiles; ++u) {
            int f, vb, rb;
            tile_at(u, f, vb, rb);
            const int db = u & 1, v = vb * 128 + 32 * q;
            if (!mbar_wait_bounded(&ddone[db], (u / 2) & 1)) fail = 1;
            if (failed()) break;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int col = 64 * hc + 16 * c, r = rb * 128 + col;
                if (v >= a.nv || r >= a.nr) continue;   // warp-uniform
                float re[16], im[16];
                const uint32_t d = tmem + ((uint32_t)(32 * q) << 16) + db * 256 + col;
                tmem_ld16(d, re);
                tmem_ld16(d + 128, im);
                uint8_t *buf = out + (nst++ & 1) * 4096;
                if (lane == 0) bulk_wait_read1();   // the store before the last one has read this buffer
                __syncwarp();
#pragma unroll
                for (int g8 = 0; g8 < 8; ++g8)
                    *reinterpret_cast<float4 *>(buf + (g8 >> 2) * 2048 + lane * 64 + (((g8 & 3) ^ ((lane >> 1) & 3)) << 4)) =
                        make_float4(re[2 * g8] * a.outscale, im[2 * g8] * a.outscale, re[2 * g8 + 1] * a.outscale,
                                    im[2 * g8 + 1] * a.outscale);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_5d(&tmap, buf, 0, f % SPEC_F, r >> 3, v, f / SPEC_F);
                    if (r + 8 < a.nr) tma_store_5d(&tmap, buf + 2048, 0, f % SPEC_F, (r >> 3) + 1, v, f / SPEC_F);
                    bulk_commit();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dfree[db]);
        }
        if (lane == 0) bulk_wait_all();
    }
    __syncthreads();
    if (fail && tid == 0) {
        // copies and products still in flight get one more bounded wait before the CTA frees TMEM and exits
        for (int i = max(0, s_copies - 2); i < s_copies; ++i) mbar_wait_bounded(&full[i & 1], (i / 2) & 1);
        for (int i = max(0, s_mma - 2); i < s_mma; ++i) mbar_wait_bounded(&adone[i & 1], (i / 2) & 1);
        atomicOr(a.status, 2);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------------
cudaError_t tc_prepare() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd<16, TC_FWD_STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<16, TC_FWD_STAGES>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd<32, TC_FWD_STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<32, TC_FWD_STAGES>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd<64, TC_FWD_STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<64, TC_FWD_STAGES>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd<16, TC_FWD_STAGES, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<16, TC_FWD_STAGES>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd<32, TC_FWD_STAGES, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<32, TC_FWD_STAGES>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd<64, TC_FWD_STAGES, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<64, TC_FWD_STAGES>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_p<16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwdP<16>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_p<16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwdP<16>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_p<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwdP<32>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_p<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwdP<32>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_p<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwdP<64>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_p<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwdP<64>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_tma<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_tma<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_sym_tma<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_sym_tma<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_p<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAP_SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_p<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAP_SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_q<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<16, 1>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_q<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<32, 1>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_fwd_q<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcFwd<64, 1>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_q<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(k_tc_adj_q<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcAdj::SMEM))) return e;
    return cudaSuccess;
}

cudaError_t launch_tc_fwd(const GemmArgs &a, int nf, cudaStream_t st) {
    const int gx = (a.nv + 127) / 128;
    constexpr int S = TC_FWD_STAGES;
    if (a.sym_tr > 0) {
        if (a.nb <= 16) k_tc_fwd<16, S, true><<<dim3(gx, 1, nf), TC_THREADS, TcFwd<16, S>::SMEM, st>>>(a);
        else if (a.nb <= 32) k_tc_fwd<32, S, true><<<dim3(gx, 1, nf), TC_THREADS, TcFwd<32, S>::SMEM, st>>>(a);
        else k_tc_fwd<64, S, true><<<dim3(gx, (a.nb + 63) / 64, nf), TC_THREADS, TcFwd<64, S>::SMEM, st>>>(a);
        return cudaGetLastError();
    }
    if (a.nb <= 16) k_tc_fwd<16, S><<<dim3(gx, 1, nf), TC_THREADS, TcFwd<16, S>::SMEM, st>>>(a);
    else if (a.nb <= 32) k_tc_fwd<32, S><<<dim3(gx, 1, nf), TC_THREADS, TcFwd<32, S>::SMEM, st>>>(a);
    else k_tc_fwd<64, S><<<dim3(gx, (a.nb + 63) / 64, nf), TC_THREADS, TcFwd<64, S>::SMEM, st>>>(a);
    return cudaGetLastError();
}

// Tensor maps of the model spectra in the SPEC_F layout, seen as FP32 [nf / F][nv][ceil(nr / 8)][F / BB][16 BB] with
// BB bins in a box: boxes of 8 columns x BB bins times `cblk` column blocks times `rows` rows, swizzled over their
// 64 BB bytes, zero fill outside the tensor (the padding columns of the last block of 8 lie inside it).
static cudaError_t encode_map(void *map_out, const float2 *Xh, int nr, int nv, int ldr, int nf, int bb, int cblk, int rows) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const cuuint64_t row = (cuuint64_t)ldr * SPEC_F * 8;
    const cuuint64_t dims[5] = {(cuuint64_t)16 * bb, (cuuint64_t)SPEC_F / bb, (cuuint64_t)(nr + 7) / 8, (cuuint64_t)nv, (cuuint64_t)spec_blocks(nf)};
    const cuuint64_t strides[4] = {(cuuint64_t)64 * bb, 64 * SPEC_F, row, row * nv};
    const cuuint32_t box[5] = {(cuuint32_t)16 * bb, 1, (cuuint32_t)cblk, (cuuint32_t)rows, 1}, estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = encode(reinterpret_cast<CUtensorMap *>(map_out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5,
                              const_cast<float2 *>(Xh), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              bb == 2 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t tc_encode_maps(TcMaps *m, const float2 *Xh, int nr, int nv, int ldr, int nf) {
    cudaError_t e = encode_map(m->fwd, Xh, nr, nv, ldr, nf, 2, 1, 128);
    if (e == cudaSuccess) e = encode_map(m->fwd_t, Xh, nr, nv, ldr, nf, 2, 16, 8);
    if (e == cudaSuccess) e = encode_map(m->adj, Xh, nr, nv, ldr, nf, 1, 1, 128);
    if (e == cudaSuccess) e = encode_map(m->adj32, Xh, nr, nv, ldr, nf, 1, 1, 32);
    return e;
}

template <int NB>
static cudaError_t launch_fwd_p(const GemmArgs &a, const TcMaps &maps, int nf, int sms, cudaStream_t st) {
    CUtensorMap m, mt;
    memcpy(&m, maps.fwd, sizeof(m));
    memcpy(&mt, maps.fwd_t, sizeof(mt));
    const int gx = (a.nv + 127) / 128, gy = (a.nb + NB - 1) / NB;
    const int nf_act = (a.nf_active > 0 && a.nf_active < nf) ? a.nf_active : nf;
    const int n_units = (nf_act + 1) / 2 * gx * gy;
    const int grid = std::max(1, std::min(std::max(n_units, (nf + 1) / 2 * gx * gy), sms));
    if (a.sym_tr > 0) k_tc_fwd_p<NB, true><<<grid, TCP_THREADS, TcFwdP<NB>::SMEM, st>>>(a, m, mt, gx, gy, nf, nf_act, n_units);
    else k_tc_fwd_p<NB, false><<<grid, TCP_THREADS, TcFwdP<NB>::SMEM, st>>>(a, m, mt, gx, gy, nf, nf_act, n_units);
    return cudaGetLastError();
}

// Tiles of one K chunk that all run at once, one CTA each, take the tile kernel: one bin a CTA, where the persistent
// kernel's units are two bins with nothing after them to overlap with (us, tile / persistent, nf 129: 9.7 / 10.8 at 64 x 64,
// batch 16, 12.1 / 14.1, batch 64; with two chunks, 100 x 100, batch 4, 14.3 / 13.5; at 257 bins, where some SMs get
// two tiles, the persistent kernel is level or ahead).  The results are the same bits.
cudaError_t launch_tc_fwd_p(const GemmArgs &a, const TcMaps &maps, int nf, bool always, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (!always && a.nr <= 64 && tc_fwd_tiles(a, nf) <= sms) return launch_tc_fwd(a, nf, st);
    return a.nb <= 16 ? launch_fwd_p<16>(a, maps, nf, sms, st) : a.nb <= 32 ? launch_fwd_p<32>(a, maps, nf, sms, st) : launch_fwd_p<64>(a, maps, nf, sms, st);
}

int tc_fwd_queue_nb(int nb) { return nb <= 16 ? 16 : nb <= 32 ? 32 : 64; }

int tc_fwd_tiles(const GemmArgs &a, int nf) {
    const int NB = tc_fwd_queue_nb(a.nb);
    return ((a.nv + 127) / 128) * ((a.nb + NB - 1) / NB) * nf;
}

int tc_adj_tiles(GemmArgs &a, bool recip, int nf) {
    a.tiles_v = (a.nv + 127) / 128;
    a.tiles_r = (a.nr + 127) / 128;
    return (recip ? a.tiles_v * (a.tiles_v + 1) / 2 : a.tiles_v * a.tiles_r) * nf;
}

cudaError_t launch_tc_fwd_queue(int NB, const WorkQueue &q, cudaStream_t st) {
    if (q.total <= 0) return cudaSuccess;
    if (NB == 16) k_tc_fwd_q<16><<<queue_grid(k_tc_fwd_q<16>, TC_THREADS, TcFwd<16, 1>::SMEM, q.total), TC_THREADS, TcFwd<16, 1>::SMEM, st>>>(q);
    else if (NB == 32) k_tc_fwd_q<32><<<queue_grid(k_tc_fwd_q<32>, TC_THREADS, TcFwd<32, 1>::SMEM, q.total), TC_THREADS, TcFwd<32, 1>::SMEM, st>>>(q);
    else k_tc_fwd_q<64><<<queue_grid(k_tc_fwd_q<64>, TC_THREADS, TcFwd<64, 1>::SMEM, q.total), TC_THREADS, TcFwd<64, 1>::SMEM, st>>>(q);
    return cudaGetLastError();
}

cudaError_t launch_tc_adj_queue(bool recip, const WorkQueue &q, cudaStream_t st) {
    if (q.total <= 0) return cudaSuccess;
    if (recip) k_tc_adj_q<true><<<queue_grid(k_tc_adj_q<true>, TC_THREADS, TcAdj::SMEM, q.total), TC_THREADS, TcAdj::SMEM, st>>>(q);
    else k_tc_adj_q<false><<<queue_grid(k_tc_adj_q<false>, TC_THREADS, TcAdj::SMEM, q.total), TC_THREADS, TcAdj::SMEM, st>>>(q);
    return cudaGetLastError();
}

// Which products the persistent adjoint takes (K products a tile and its mirror: the batch, twice with reciprocity):
//  * enough tiles for its roles to overlap from tile to tile: two a CTA; sixteen with reciprocity, where the diagonal tiles
//    take a launch of their own (persistent / tile kernel, us, batch 16: 23.6 / 22.0 at nf 257, 128 x 128; symmetric
//    83.6 / 78.5 at nf 257, 300 x 300, 148.9 / 143.1 at nf 513, 300 x 300, 205 / 210 at nf 513, 400 x 400);
//  * and work that hides the writes: two jobs a tile (K > 32: 505 / 650 at nf 1025, 300 x 600, batch 64), or operand images
//    that stay in seven eighths of the L2 (117 / 126 at nf 257, 300 x 600, batch 32; 135 MB of them at nf 513: 254 / 221,
//    batch 16), or output tiles with half as much padding again as
//    outputs, which the tile kernel computes and the persistent one skips (265 / 284 at nf 1025, 301 x 301, batch 32).
//    Otherwise the output bounds both, and the tile kernel's CTAs, which start in the order of the bins, keep the four
//    64-byte pieces of a 256-byte line closer together in time than CTAs that walk lists of tiles (541 / 421 at nf 1025,
//    300 x 600, 764 / 691 at 600 x 600, batch 8; four or two bins of a line on one CTA in turn: 459 and 455, 730 and 721).
static bool adj_persistent(const GemmArgs &a, bool recip, int tiles, int nf, int sms, int l2) {
    if ((long long)tiles * nf < (recip ? 16LL : 2LL) * sms) return false;
    const double images = (double)nf * a.img_nkc * (a.tiles_v + a.tiles_r) * TC_ADJ_IMG;
    const double padded = 128.0 * 128.0 * a.tiles_v * a.tiles_r;
    return a.nb * (recip ? 2 : 1) > TcAdj::KC || images <= 0.875 * l2 || padded >= 1.5 * a.nv * a.nr;
}

cudaError_t launch_tc_adj(const GemmArgs &a0, bool recip, int nf, cudaStream_t st, const TcMaps *maps) {
    const void *map = maps ? maps->adj : nullptr;
    GemmArgs a = a0;
    a.tiles_v = (a.nv + 127) / 128;
    a.tiles_r = (a.nr + 127) / 128;
    const bool img = a.img != nullptr;
    const int tiles = recip ? a.tiles_v * (a.tiles_v - 1) / 2 : a.tiles_v * a.tiles_r;   // of the persistent kernel
    int dev = 0, sms = 0, l2 = 0;
    if (img && maps && (!recip || a.no_mirror)) {
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
        if (e != cudaSuccess) return e;
    }
    if (sms > 0 && adj_persistent(a, recip, tiles, nf, sms, l2)) {
        CUtensorMap m32;
        memcpy(&m32, maps->adj32, sizeof(m32));
        const int nf_act = (a.nf_active > 0 && a.nf_active < nf) ? a.nf_active : nf;
        const int grid = std::min(nf * tiles, sms);
        if (!recip) {
            k_tc_adj_p<false><<<grid, TAP_THREADS, TAP_SMEM, st>>>(a, m32, tiles, nf, nf_act);
        } else {
            k_tc_adj_p<true><<<grid, TAP_THREADS, TAP_SMEM, st>>>(a, m32, tiles, nf, nf_act);
            a.diag_only = 1;
            CUtensorMap tmap;
            memcpy(&tmap, map, sizeof(tmap));
            k_tc_adj_sym_tma<true><<<dim3(a.tiles_v, nf), TC_THREADS, TcAdj::SMEM, st>>>(a, tmap);
        }
        return cudaGetLastError();
    }
    if (recip && map && a.no_mirror) {
        CUtensorMap tmap;
        memcpy(&tmap, map, sizeof(tmap));
        const dim3 grid(a.tiles_v * (a.tiles_v + 1) / 2, nf);
        if (img) k_tc_adj_sym_tma<true><<<grid, TC_THREADS, TcAdj::SMEM, st>>>(a, tmap);
        else k_tc_adj_sym_tma<false><<<grid, TC_THREADS, TcAdj::SMEM, st>>>(a, tmap);
    } else if (recip) {
        if (img) k_tc_adj<true, true><<<dim3(a.tiles_v * (a.tiles_v + 1) / 2, nf), TC_THREADS, TcAdj::SMEM, st>>>(a);
        else k_tc_adj<true><<<dim3(a.tiles_v * (a.tiles_v + 1) / 2, nf), TC_THREADS, TcAdj::SMEM, st>>>(a);
    } else if (map) {
        CUtensorMap tmap;
        memcpy(&tmap, map, sizeof(tmap));
        if (img) k_tc_adj_tma<true><<<dim3(a.tiles_v * a.tiles_r, nf), TC_THREADS, TcAdj::SMEM, st>>>(a, tmap);
        else k_tc_adj_tma<false><<<dim3(a.tiles_v * a.tiles_r, nf), TC_THREADS, TcAdj::SMEM, st>>>(a, tmap);
    } else {
        if (img) k_tc_adj<false, true><<<dim3(a.tiles_v * a.tiles_r, nf), TC_THREADS, TcAdj::SMEM, st>>>(a);
        else k_tc_adj<false><<<dim3(a.tiles_v * a.tiles_r, nf), TC_THREADS, TcAdj::SMEM, st>>>(a);
    }
    return cudaGetLastError();
}

size_t tc_adj_image_bytes(int nv, int nr, int nb, int nf) {
    const int nkc = (nb + TcAdj::KC - 1) / TcAdj::KC;
    if (nkc < 1 || nkc > 2) return 0;
    return (size_t)nf * nkc * (size_t)((nv + 127) / 128 + (nr + 127) / 128) * TC_ADJ_IMG;
}

cudaError_t launch_tc_adj_images(const GemmArgs &a0, uint8_t *img, int nf, cudaStream_t st) {
    GemmArgs a = a0;
    a.tiles_v = (a.nv + 127) / 128;
    a.tiles_r = (a.nr + 127) / 128;
    a.img_nkc = (a.nb + TcAdj::KC - 1) / TcAdj::KC;
    const int nfa = (a.nf_active > 0 && a.nf_active < nf) ? a.nf_active : nf;   // bins above a band limit are zero
    k_tc_adj_images<<<dim3(a.tiles_v + a.tiles_r, a.img_nkc, nfa), TC_THREADS, TcAdj::STAGE, st>>>(a, img);
    return cudaGetLastError();
}

}  // namespace smdd
