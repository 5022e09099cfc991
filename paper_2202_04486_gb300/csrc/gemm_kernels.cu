// Per-frequency complex matrix products of the MDC hot path (FP32 SIMT path).
//
// Eq. 2 states the MDC as one matrix product per frequency; Appendix A calls it the batched MMM.  With
// the model spectra Xh_f [nv x nr] (rows v) and the kernel spectra Dh_f [ns x nr] (rows s):
//   forward (Eq. 2, batch of Eq. 5):  Uh_f[v][b] = sum_r Xh_f[v][r] Dh_f[idx_b][r]
//   adjoint (Eq. 6):                  Gh_f[v][r] = sum_b Rh_f[v][b] conj(Dh_f[idx_b][r])
// The batch gather of kernel rows (the random subset of sources of Eq. 6) happens in the operand
// load: row idx_b of Dh_f is read in place, no gathered copy is made.
//
// With reciprocity (C_r of Eq. 4) the adjoint writes 1/2 (Gh_f + Gh_f^T) directly: since
// Gh_f^T[v][r] = sum_b conj(Dh_f[idx_b][v]) Rh_f[r][b], the symmetric part is one product with
// inner dimension 2 nb, A' = [Rh | conj(Dh_B)^T], B' = [conj(Dh_B) ; Rh^T], evaluated on the upper
// triangle of tiles only and mirrored into the lower triangle through shared memory.
#include <climits>

#include "smdd_fft.cuh"
#include "smdd_internal.h"

namespace smdd {

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gsrc, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(gsrc), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// acc += a * b (complex)
__device__ __forceinline__ void cmac(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// ------------------------------------------------------------------------------------------------
// forward, batches up to 16 and up to 128 rows (scalar products, 4 x 4 outputs per thread):
//   C[f][v][b] = sum_r A[f][v][r] * Dh[f][idx_b][r]
// Such a product is a chain of latencies; the longer chunk (16) through cp.async has fewer of them: 8.4 us at nf 129,
// 32 x 32, batch 8, against 11 us for the packed tiles below.
// CTA: 4 warps, 128 rows v x 16 batch columns, one frequency.  Lane (vg = lane & 7, bg = lane >> 3)
// of warp w owns rows v0 + 32w + vg + 8i and columns b0 + bg + 4j (i, j < 4): a 4 x 4 complex register
// tile.  K (= nr) streams in chunks of 16 through a two-stage cp.async pipeline; every operand load is
// 128-bit (two consecutive k) and the 144-byte row pitch puts the 8 distinct rows of a load in 8
// distinct bank groups.
// ------------------------------------------------------------------------------------------------
constexpr int FW_THREADS = 128, FW_ROWS = 128, FW_NB = 16, FW_KC = 16, FW_LD = FW_KC + 2;
constexpr int FW_STAGE = (FW_ROWS + FW_NB) * FW_LD;   // float2 per stage
constexpr size_t FW_SMEM = 2 * FW_STAGE * sizeof(float2);

template <int F>
__global__ void __launch_bounds__(FW_THREADS, 4) k_cgemm_fwd_small(GemmArgs a) {
    extern __shared__ __align__(16) float2 gsm[];
    const int f = blockIdx.z;
    const int v0 = blockIdx.x * FW_ROWS, b0 = blockIdx.y * FW_NB;
    if (a.nf_active > 0 && f >= a.nf_active) {
        zero_tile<F>(a.C + spec_bin<F>(f, a.sCf), (long long)a.ldb * F, v0, FW_ROWS, b0, FW_NB, a.nv, a.nb);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int vg = lane & 7, bg = lane >> 3;
    const float2 *Af = a.A + spec_bin<F>(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf;

    // kernel row of the batch column this thread stages (one 16-byte chunk per thread per stage)
    const int db = tid >> 3, dpart = tid & 7;
    int drow = -1;
    if (b0 + db < a.nb) {
        drow = a.idx[b0 + db];
        if (drow < 0 || drow >= a.ns) {
            atomicOr(a.status, 1);
            drow = -1;
        }
    }

    auto load_stage = [&](int stage, int k0) {
        float2 *sX = gsm + stage * FW_STAGE;
        float2 *sD = sX + FW_ROWS * FW_LD;
#pragma unroll
        for (int u = 0; u < (FW_ROWS * FW_KC / 2) / FW_THREADS; ++u) {
            const int c = tid + u * FW_THREADS;
            const int row = c >> 3, part = c & 7;
            const int k = k0 + 2 * part, v = v0 + row;
            int bytes = 0;
            const float2 *src = Af;
            if (v < a.nv && k < a.nr) {
                bytes = (k + 1 < a.nr) ? 16 : 8;
                src = Af + (long long)v * a.ldr * F + spec_col<F>(k);
            }
            cp_async16(sX + row * FW_LD + 2 * part, src, bytes);
        }
        {
            const int k = k0 + 2 * dpart;
            int bytes = 0;
            const float2 *src = Df;
            if (drow >= 0 && k < a.nr) {
                bytes = (k + 1 < a.nr) ? 16 : 8;
                src = Df + (long long)drow * a.ldd + k;
            }
            cp_async16(sD + db * FW_LD + 2 * dpart, src, bytes);
        }
        cp_async_commit();
    };

    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    const bool active = v0 + 32 * warp < a.nv;   // warps whose rows all lie past nv skip the products

    const int nk = (a.nr + FW_KC - 1) / FW_KC;
    load_stage(0, 0);
    for (int kc = 0; kc < nk; ++kc) {
        if (kc + 1 < nk) {
            load_stage((kc + 1) & 1, (kc + 1) * FW_KC);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        if (active) {
            const float2 *sX = gsm + (kc & 1) * FW_STAGE + (32 * warp + vg) * FW_LD;
            const float2 *sD = gsm + (kc & 1) * FW_STAGE + FW_ROWS * FW_LD + bg * FW_LD;
#pragma unroll
            for (int kk = 0; kk < FW_KC; kk += 2) {
                float4 x[4], d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4 *>(sX + 8 * i * FW_LD + kk);
#pragma unroll
                for (int j = 0; j < 4; ++j) d[j] = *reinterpret_cast<const float4 *>(sD + 4 * j * FW_LD + kk);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        cmac(acc[i][j], make_float2(x[i].x, x[i].y), make_float2(d[j].x, d[j].y));
                        cmac(acc[i][j], make_float2(x[i].z, x[i].w), make_float2(d[j].z, d[j].w));
                    }
            }
        }
        __syncthreads();
    }

    float2 *Cf = a.C + spec_bin<F>(f, a.sCf);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int v = v0 + 32 * warp + vg + 8 * i;
        if (v >= a.nv) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int b = b0 + bg + 4 * j;
            if (b < a.nb) Cf[(long long)v * a.ldb * F + spec_col<F>(b)] = acc[i][j];
        }
    }
}

// ------------------------------------------------------------------------------------------------
// adjoint: C[f][v][r] = outscale * sum_k A'[v][k] B'[k][r]
//   k < nb :  A' = Rh[f][v][k],            B' = conj(Dh[f][idx_k][r])
//   k >= nb (reciprocity only, k' = k - nb):  A' = conj(Dh[f][idx_k'][v]),  B' = Rh[f][r][k']
// TV x TT tiles with scalar products (4 x 4 outputs per thread, chunks of 16).  32 x 32: finer at triangular and ragged
// edges than the packed 64 x 64 tiles below.  With reciprocity both halves of a chunk are staged at once, one latency: 107
// us against 130 us at nf 513, 201 x 201, batch 16 (1057 and 1118 us at batch 201).  16 x 64: a warp covers 8 rows x 64
// columns, against 16 x 32, so that few rows leave fewer outputs of a warp unused (us, 32 x 32 / 16 x 64, batch 64: 74 / 54 at nf 257,
// 600 columns x 8 rows; 154 / 97 at nf 1025, 300 x 16).
// A warp covers 4*VPN rows x TT columns: lane (vp = lane / RG,
// rg = lane % RG) owns rows v0 + 4*VPN*w + 4vp + {0,1,2,3} and columns r0 + {2rg, 2rg+1, 2rg+TT/2,
// 2rg+TT/2+1}.  Operands are staged by cp.async in their global layouts -- residual-spectrum rows [v][k]
// and kernel-spectrum rows [k][r] -- and conjugated when used; chunks of 16 k per half.  Warps whose
// rows all lie past nv skip the products.
// ------------------------------------------------------------------------------------------------
constexpr int AD_KC = 16, AD_LDR = AD_KC + 2, AD_MAXNB = 1024;

template <int TV_, int TT_, bool RECIP>
struct AdjS {
    static constexpr int TV = TV_, TT = TT_;
    static_assert(!RECIP || TV == TT, "mirrored tiles are square");
    static constexpr int RG = TT / 4;             // lanes along r
    static constexpr int VPN = 32 / RG;           // lane groups along v
    static constexpr int WROWS = 4 * VPN;         // rows per warp
    static constexpr int WARPS = TV / WROWS;
    static constexpr int THREADS = 32 * WARPS;
    static constexpr int RROWS = TV * AD_LDR;     // float2: residual rows of one block
    static constexpr int DROWS = AD_KC * TT;      // float2: kernel rows at one block's columns
    static constexpr size_t SMEM_OPER = (RECIP ? 2 : 1) * (RROWS + DROWS) * sizeof(float2);
    static constexpr size_t SMEM_MIRROR = RECIP ? TT * (TT + 1) * sizeof(float2) : 0;
    static constexpr size_t SMEM = SMEM_OPER > SMEM_MIRROR ? SMEM_OPER : SMEM_MIRROR;
};

// stage rows [c0, c0 + ROWS) x k [k0, k0 + 16) of Rh (row pitch ldb) into s[ROWS][AD_LDR], by NT threads
template <int ROWS, int NT>
__device__ __forceinline__ void stage_rrows(float2 *s, const float2 *Rf, int ldb, int c0, int nc, int k0, int nb, int tid) {
#pragma unroll
    for (int u = 0; u < ROWS * AD_KC / 2 / NT; ++u) {
        const int c = tid + u * NT, row = c >> 3, part = c & 7;
        const int k = k0 + 2 * part;
        int bytes = 0;
        const float2 *src = Rf;
        if (c0 + row < nc && k < nb) {
            bytes = (k + 1 < nb) ? 16 : 8;
            src = Rf + (long long)(c0 + row) * ldb * SPEC_F + spec_col(k);
        }
        cp_async16(s + row * AD_LDR + 2 * part, src, bytes);
    }
}

// stage kernel rows idx[k0 .. k0 + 16) at columns [c0, c0 + TT) into s[16][TT]
template <int TT, int NT>
__device__ __forceinline__ void stage_drows(float2 *s, const float2 *Df, int ldd, const int *sidx, int c0, int nc, int k0,
                                            int nb, int tid) {
    constexpr int PARTS = TT / 2;
#pragma unroll
    for (int u = 0; u < AD_KC * TT / 2 / NT; ++u) {
        const int c = tid + u * NT, kk = c / PARTS, part = c % PARTS;
        const int col = c0 + 2 * part;
        int bytes = 0;
        const float2 *src = Df;
        if (k0 + kk < nb && col < nc) {
            const int srow = sidx[k0 + kk];
            if (srow >= 0) {
                bytes = (col + 1 < nc) ? 16 : 8;
                src = Df + (long long)srow * ldd + col;
            }
        }
        cp_async16(s + kk * TT + 2 * part, src, bytes);
    }
}

// acc += a * conj(b)
__device__ __forceinline__ void cmac_c(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(a.y, b.y, acc.x);
    acc.y = fmaf(a.y, b.x, acc.y);
    acc.y = fmaf(-a.x, b.y, acc.y);
}

template <int TV, int TT, bool RECIP>
__global__ void __launch_bounds__(64, 8) k_cgemm_adj_small(GemmArgs a) {
    using G = AdjS<TV, TT, RECIP>;
    static_assert(G::THREADS == 64, "two warps");
    extern __shared__ __align__(16) float2 gsm[];
    float2 *sRv = gsm;                  // [TV][AD_LDR]  Rh rows of the v block
    float2 *sDr = sRv + G::RROWS;       // [16][TT]      kernel rows at the r block
    float2 *sRr = sDr + G::DROWS;       // [TV][AD_LDR]  Rh rows of the r block (reciprocity)
    float2 *sDv = sRr + G::RROWS;       // [16][TT]      kernel rows at the v block (reciprocity)
    __shared__ int sidx[AD_MAXNB];
    const int f = blockIdx.y;
    int vb, rb;
    if (RECIP) {   // upper-triangular tile enumeration: vb <= rb
        int t = blockIdx.x, row = 0, len = a.tiles_v;
        while (t >= len) { t -= len; ++row; --len; }
        vb = row;
        rb = row + t;
    } else {
        vb = blockIdx.x / a.tiles_r;
        rb = blockIdx.x % a.tiles_r;
    }
    const int v0 = vb * TV, r0 = rb * TT;
    if (a.nf_active > 0 && f >= a.nf_active) {
        const long long row = (long long)a.ldr * SPEC_F;
        zero_tile(a.C + spec_bin(f, a.sCf), row, v0, TV, r0, TT, a.nv, a.nr);
        if (RECIP) zero_tile(a.C + spec_bin(f, a.sCf), row, r0, TT, v0, TV, a.nr, a.nv);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int vp = lane / G::RG, rg = lane % G::RG;
    const int vl = G::WROWS * warp + 4 * vp;     // first local row of the thread
    const bool active = v0 + G::WROWS * warp < a.nv;
    const float2 *Rf = a.A + spec_bin(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf;

    for (int b = tid; b < a.nb; b += G::THREADS) {
        int s = a.idx[b];
        if (s < 0 || s >= a.ns) {
            atomicOr(a.status, 1);
            s = -1;
        }
        sidx[b] = s;
    }
    __syncthreads();

    float2 acc[4][4];   // [row][column: 2rg, 2rg+1, 2rg+TT/2, 2rg+TT/2+1]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);

    for (int k0 = 0; k0 < a.nb; k0 += AD_KC) {
        stage_rrows<TV, G::THREADS>(sRv, Rf, a.ldb, v0, a.nv, k0, a.nb, tid);
        stage_drows<TT, G::THREADS>(sDr, Df, a.ldd, sidx, r0, a.nr, k0, a.nb, tid);
        if (RECIP) {
            stage_rrows<TV, G::THREADS>(sRr, Rf, a.ldb, r0, a.nr, k0, a.nb, tid);
            stage_drows<TT, G::THREADS>(sDv, Df, a.ldd, sidx, v0, a.nv, k0, a.nb, tid);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        const int kn = min(AD_KC, a.nb - k0);
        if (active) {
            // first half: Rh[v][k] * conj(Dh[idx_k][r])
            for (int kk = 0; kk < kn; kk += 2) {   // kn odd: column kn is zero filled
                float4 av[4], b0[2], b1[2];
#pragma unroll
                for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const float4 *>(sRv + (vl + i) * AD_LDR + kk);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    b0[h] = *reinterpret_cast<const float4 *>(sDr + kk * TT + 2 * rg + (TT / 2) * h);
                    b1[h] = *reinterpret_cast<const float4 *>(sDr + (kk + 1) * TT + 2 * rg + (TT / 2) * h);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float2 a0 = make_float2(av[i].x, av[i].y), a1 = make_float2(av[i].z, av[i].w);
                        cmac_c(acc[i][2 * h], a0, make_float2(b0[h].x, b0[h].y));
                        cmac_c(acc[i][2 * h + 1], a0, make_float2(b0[h].z, b0[h].w));
                        cmac_c(acc[i][2 * h], a1, make_float2(b1[h].x, b1[h].y));
                        cmac_c(acc[i][2 * h + 1], a1, make_float2(b1[h].z, b1[h].w));
                    }
            }
            if (RECIP) {
                // second half: conj(Dh[idx_k][v]) * Rh[r][k]  (= the transpose of the first half)
                for (int kk = 0; kk < kn; kk += 2) {
                    float4 d0[2], d1[2], rv[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {   // rows vl + 2h, vl + 2h + 1 at k and k+1
                        d0[h] = *reinterpret_cast<const float4 *>(sDv + kk * TT + vl + 2 * h);
                        d1[h] = *reinterpret_cast<const float4 *>(sDv + (kk + 1) * TT + vl + 2 * h);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int rl = 2 * rg + (j & 1) + (TT / 2) * (j >> 1);
                        rv[j] = *reinterpret_cast<const float4 *>(sRr + rl * AD_LDR + kk);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 dk0 = d0[i >> 1], dk1 = d1[i >> 1];
                        const float2 c0 = (i & 1) ? make_float2(dk0.z, dk0.w) : make_float2(dk0.x, dk0.y);
                        const float2 c1 = (i & 1) ? make_float2(dk1.z, dk1.w) : make_float2(dk1.x, dk1.y);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            cmac_c(acc[i][j], make_float2(rv[j].x, rv[j].y), c0);   // Rh[r][k] conj(Dh[k][v])
                            cmac_c(acc[i][j], make_float2(rv[j].z, rv[j].w), c1);
                        }
                    }
                }
            }
        }
        __syncthreads();
    }

    float2 *Cf = a.C + spec_bin(f, a.sCf);
    const long long crow = (long long)a.ldr * SPEC_F;
    const bool diag = RECIP && (vb == rb);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int vv = vl + i, v = v0 + vv;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int rr = 2 * rg + (TT / 2) * h, r = r0 + rr;
            const float2 x0 = cscale(acc[i][2 * h], a.outscale), x1 = cscale(acc[i][2 * h + 1], a.outscale);
            if (v < a.nv) {
                const bool w0 = r < a.nr && (!diag || v <= r), w1 = r + 1 < a.nr && (!diag || v <= r + 1);
                float2 *dst = Cf + v * crow + spec_col(r);
                if (w0 && w1) *reinterpret_cast<float4 *>(dst) = make_float4(x0.x, x0.y, x1.x, x1.y);
                else {
                    if (w0) dst[0] = x0;
                    if (w1) dst[1] = x1;
                }
            }
            if (RECIP) {   // mirror buffer (r, v); operands are dead after the final barrier
                gsm[rr * (TT + 1) + vv] = x0;
                gsm[(rr + 1) * (TT + 1) + vv] = x1;
            }
        }
    }
    if (RECIP && (diag || !a.no_mirror)) {   // diagonal tiles always mirror (see GemmArgs::no_mirror)
        __syncthreads();
        for (int e = tid; e < TT * TT; e += G::THREADS) {
            const int rr = e / TT, vv = e % TT;
            const int r = r0 + rr, v = v0 + vv;
            if (v < a.nv && r < a.nr && (!diag || v < r)) Cf[r * crow + spec_col(v)] = gsm[rr * (TT + 1) + vv];
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Tile products on the CUDA cores.  A thread owns 8 x 4 complex outputs, the 8 as four pairs of packed FP32 values
// (fma.f32x2: two multiply-adds in one issue slot; the arithmetic rate is that of scalar instructions, but the
// operand loads and duplications then fit in the freed slots): pair p holds i = 2 ti + 2 WTI p and i + 1, so that the
// lanes of a row store 64 contiguous bytes of the output.  Operands lie in shared memory as separate real and
// imaginary planes [k][i] and [k][j]: an LDS.64 of the i operand is a packed pair, the j operand is duplicated
// into pairs in registers (24 cycles of the shared-memory pipe and 64 packed multiply-adds a k and warp; with 4 x 4 outputs the shared-memory pipe, at
// four cycles an LDS.128, would be as busy as the arithmetic).  Chunks of 8 k, double buffered, the next chunk's
// global loads in registers while one is multiplied: one barrier a chunk.
//   FORM 0: c += a b            (forward:  a = model spectra, b = kernel rows)
//   FORM 1: c += conj(a) b      (adjoint:  a = kernel rows, b = residual spectra)
//   FORM 2: c += a conj(b)      (its transpose, for the reciprocity half)
// A warp covers 8 WTI x 4 (32 / WTI) outputs; warps whose outputs all lie outside the matrix skip the products.
// ------------------------------------------------------------------------------------------------
template <int WTI_, int NWI_, int NWJ_, int KC_ = 8>
struct SimtGeom {
    static constexpr int WTI = WTI_, NWI = NWI_, NWJ = NWJ_, KC = KC_;
    static constexpr int WI = 8 * WTI, WJ = 4 * (32 / WTI);      // outputs of a warp
    static constexpr int BI = WI * NWI, BJ = WJ * NWJ;           // outputs of the CTA
    static constexpr int THREADS = 32 * NWI * NWJ;
    // row pitches: 16-byte multiples whose double is 8 mod 32 words, so the transposing stores of 4 k pairs x 8 rows
    // fall on distinct banks (8 x 4 for KC = 16: two to a bank)
    static constexpr int PI = BI + 4, PJ = BJ + 4;
    static constexpr int STAGE = 2 * KC * (PI + PJ);          // floats: Ar, Ai, Br, Bi
    static constexpr size_t SMEM = 2 * STAGE * sizeof(float);
    // LDG.128 units (two complex values) of a chunk per thread
    static constexpr int UI = (BI * KC / 2 + THREADS - 1) / THREADS, UJ = (BJ * KC / 2 + THREADS - 1) / THREADS;
    static constexpr int MINB = (UI > 4 ? 384 : 512) / THREADS;   // resident CTAs: 168 or 128 registers per thread
};

struct SimtAcc {
    f32x2 re[4][4], im[4][4];   // [pair of i][j]
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) re[i][j] = im[i][j] = 0;
    }
};

// one chunk: planes of stage s; ia, jb: the thread's first i and j of the tile
template <class G, int FORM>
__device__ __forceinline__ void simt_chunk(SimtAcc &c, const float *st, int ia, int jb) {
    constexpr int KC = G::KC;
    const float *pa = st + ia, *pb = st + 2 * KC * G::PI + jb;
#pragma unroll
    for (int k = 0; k < KC; ++k) {
        f32x2 ar[4], ai[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            ar[p] = *reinterpret_cast<const f32x2 *>(pa + k * G::PI + 2 * G::WTI * p);
            ai[p] = *reinterpret_cast<const f32x2 *>(pa + (KC + k) * G::PI + 2 * G::WTI * p);
        }
        const float4 b4 = *reinterpret_cast<const float4 *>(pb + k * G::PJ), d4 = *reinterpret_cast<const float4 *>(pb + (KC + k) * G::PJ);
        const float br[4] = {b4.x, b4.y, b4.z, b4.w}, bi[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const f32x2 r = dup2(br[j]), i = dup2(bi[j]), n = dup2(FORM == 1 ? -br[j] : -bi[j]);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                c.re[p][j] = fma2(ar[p], r, c.re[p][j]);
                c.re[p][j] = fma2(ai[p], FORM == 0 ? n : i, c.re[p][j]);
                c.im[p][j] = fma2(ar[p], FORM == 2 ? n : i, c.im[p][j]);
                c.im[p][j] = fma2(ai[p], FORM == 1 ? n : r, c.im[p][j]);
            }
        }
    }
}

// An operand whose rows hold k contiguously (rows of the layout of F bins: row x at base + x ld): unit c of a chunk is
// (row c / (KC / 2), columns k0 + 2 (c % (KC / 2)), + 1); rows past n and columns past nk are zero.
template <int F>
__device__ __forceinline__ float4 krow_load(const float2 *base, long long ld, int x, int n, int k, int nk) {
    if (x >= n || k >= nk) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float2 *p = base + (long long)x * ld + spec_col<F>(k);
    if (k + 1 < nk) return __ldg(reinterpret_cast<const float4 *>(p));
    const float2 v = __ldg(p);
    return make_float4(v.x, v.y, 0.f, 0.f);
}
template <int P, int KC>
__device__ __forceinline__ void krow_store(float *pl, int c, float4 v) {   // pl: real plane; the imaginary one follows
    float *q = pl + 2 * (c % (KC / 2)) * P + c / (KC / 2);
    q[0] = v.x;
    q[P] = v.z;
    q[KC * P] = v.y;
    q[(KC + 1) * P] = v.w;
}
// An operand given by rows k (kernel spectra): unit c is (k = c / (B / 2), columns x0 + 2 (c % (B / 2)), + 1)
__device__ __forceinline__ float4 xrow_load(const float2 *row, int x, int n) {   // row may be null: zero
    if (!row || x >= n) return make_float4(0.f, 0.f, 0.f, 0.f);
    if (x + 1 < n) return __ldg(reinterpret_cast<const float4 *>(row + x));
    const float2 v = __ldg(row + x);
    return make_float4(v.x, v.y, 0.f, 0.f);
}
template <int P, int B, int KC>
__device__ __forceinline__ void xrow_store(float *pl, int c, float4 v) {
    float *q = pl + (c / (B / 2)) * P + 2 * (c % (B / 2));
    *reinterpret_cast<float2 *>(q) = make_float2(v.x, v.z);
    *reinterpret_cast<float2 *>(q + KC * P) = make_float2(v.y, v.w);
}

// ------------------------------------------------------------------------------------------------
// forward: C[f][v][b] = sum_r A[f][v][r] * Dh[f][idx_b][r]   (i = v, j = b, k = r)
// ------------------------------------------------------------------------------------------------
template <class G, int F>
__global__ void __launch_bounds__(G::THREADS, G::MINB) k_cgemm_fwd(GemmArgs a) {
    extern __shared__ __align__(16) float ssm[];
    __shared__ int srow[G::BJ];
    const int f = blockIdx.z, v0 = blockIdx.x * G::BI, b0 = blockIdx.y * G::BJ;
    if (a.nf_active > 0 && f >= a.nf_active) {
        zero_tile<F>(a.C + spec_bin<F>(f, a.sCf), (long long)a.ldb * F, v0, G::BI, b0, G::BJ, a.nv, a.nb);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wi = (warp % G::NWI) * G::WI, wj = (warp / G::NWI) * G::WJ;
    const int ia = wi + 2 * (lane % G::WTI), jb = wj + 4 * (lane / G::WTI);
    const float2 *Af = a.A + spec_bin<F>(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf;
    for (int j = tid; j < G::BJ; j += G::THREADS) {
        int s = -1;
        if (b0 + j < a.nb) {
            s = a.idx[b0 + j];
            if (s < 0 || s >= a.ns) {
                atomicOr(a.status, 1);
                s = -1;
            }
        }
        srow[j] = s;
    }
    __syncthreads();
    const long long arow = (long long)a.ldr * F;
    constexpr int H = G::KC / 2;   // units of a row and chunk
    float4 ra[G::UI], rb[G::UJ];
    auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < G::UI; ++u) {
            const int c = tid + u * G::THREADS;
            if (c < G::BI * H) ra[u] = krow_load<F>(Af, arow, v0 + c / H, a.nv, k0 + 2 * (c % H), a.nr);
        }
#pragma unroll
        for (int u = 0; u < G::UJ; ++u) {
            const int c = tid + u * G::THREADS;
            if (c < G::BJ * H) rb[u] = krow_load<1>(Df, a.ldd, srow[c / H], srow[c / H] < 0 ? INT_MIN : INT_MAX, k0 + 2 * (c % H), a.nr);
        }
    };
    auto store = [&](int s) {
        float *pa = ssm + s * G::STAGE, *pb = pa + 2 * G::KC * G::PI;
#pragma unroll
        for (int u = 0; u < G::UI; ++u)
            if (tid + u * G::THREADS < G::BI * H) krow_store<G::PI, G::KC>(pa, tid + u * G::THREADS, ra[u]);
#pragma unroll
        for (int u = 0; u < G::UJ; ++u)
            if (tid + u * G::THREADS < G::BJ * H) krow_store<G::PJ, G::KC>(pb, tid + u * G::THREADS, rb[u]);
    };
    SimtAcc c;
    c.zero();
    const bool active = v0 + wi < a.nv && b0 + wj < a.nb;
    const int nk = (a.nr + G::KC - 1) / G::KC;
    load(0);
    store(0);
    __syncthreads();
    for (int kc = 0; kc < nk; ++kc) {
        if (kc + 1 < nk) load((kc + 1) * G::KC);
        if (active) simt_chunk<G, 0>(c, ssm + (kc & 1) * G::STAGE, ia, jb);
        if (kc + 1 < nk) store((kc + 1) & 1);
        __syncthreads();
    }
    float2 *Cf = a.C + spec_bin<F>(f, a.sCf);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int v = v0 + ia + 2 * G::WTI * p + e;
            if (v >= a.nv) continue;
#pragma unroll
            for (int j = 0; j < 4; j += 2) {
                const int b = b0 + jb + j;
                const float2 x = e ? make_float2(hi2(c.re[p][j]), hi2(c.im[p][j])) : make_float2(lo2(c.re[p][j]), lo2(c.im[p][j]));
                const float2 y = e ? make_float2(hi2(c.re[p][j + 1]), hi2(c.im[p][j + 1])) : make_float2(lo2(c.re[p][j + 1]), lo2(c.im[p][j + 1]));
                float2 *dst = Cf + (long long)v * a.ldb * F + spec_col<F>(b);
                if (b + 1 < a.nb) *reinterpret_cast<float4 *>(dst) = make_float4(x.x, x.y, y.x, y.y);
                else if (b < a.nb) *dst = x;
            }
        }
}

// ------------------------------------------------------------------------------------------------
// adjoint: C[f][v][r] = outscale * sum_k A'[v][k] B'[k][r]   (i = r, j = v)
//   first half:   Rh[f][v][k] conj(Dh[f][idx_k][r])
//   second half:  conj(Dh[f][idx_k][v]) Rh[f][r][k]      (reciprocity)
// Tiles of 64 x 64 (four warps); with reciprocity the upper-triangular ones, mirrored through shared memory.
// ------------------------------------------------------------------------------------------------
using AdjGeom64 = SimtGeom<4, 2, 2>;
template <class G>
constexpr size_t adj_smem() {   // the operands, or the mirror buffer
    const size_t mirror = G::BI * (G::BI + 1) * sizeof(float2);
    return G::SMEM > mirror ? G::SMEM : mirror;
}

template <class G, bool RECIP>
__global__ void __launch_bounds__(G::THREADS, 512 / G::THREADS) k_cgemm_adj(GemmArgs a) {
    constexpr int TT = G::BI, KC = G::KC, H = KC / 2;
    static_assert(G::BI == G::BJ, "square tiles");
    extern __shared__ __align__(16) float ssm[];
    __shared__ int sidx[AD_MAXNB];
    const int f = blockIdx.y;
    int vb, rb_;
    if (RECIP) {   // upper-triangular tile enumeration: vb <= rb
        int t = blockIdx.x, row = 0, len = a.tiles_v;
        while (t >= len) { t -= len; ++row; --len; }
        vb = row;
        rb_ = row + t;
    } else {
        vb = blockIdx.x / a.tiles_r;
        rb_ = blockIdx.x % a.tiles_r;
    }
    const int v0 = vb * TT, r0 = rb_ * TT;
    const long long crow = (long long)a.ldr * SPEC_F, brow = (long long)a.ldb * SPEC_F;
    float2 *Cf = a.C + spec_bin(f, a.sCf);
    if (a.nf_active > 0 && f >= a.nf_active) {
        zero_tile(Cf, crow, v0, TT, r0, TT, a.nv, a.nr);
        if (RECIP) zero_tile(Cf, crow, r0, TT, v0, TT, a.nr, a.nv);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wi = (warp % G::NWI) * G::WI, wj = (warp / G::NWI) * G::WJ;
    const int ia = wi + 2 * (lane % G::WTI), jb = wj + 4 * (lane / G::WTI);
    const float2 *Rf = a.A + spec_bin(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf;
    for (int b = tid; b < a.nb; b += G::THREADS) {
        int s = a.idx[b];
        if (s < 0 || s >= a.ns) {
            atomicOr(a.status, 1);
            s = -1;
        }
        sidx[b] = s;
    }
    __syncthreads();
    constexpr int NH = RECIP ? 2 : 1;
    float4 ra[G::UI], rb[G::UJ];
    // job = (chunk, half): half 0: i from kernel rows, j from residual rows; half 1: i from residual rows, j from kernel rows
    auto load = [&](int job) {
        const int k0 = (job / NH) * KC, half = job % NH;
#pragma unroll
        for (int u = 0; u < G::UI; ++u) {
            const int c = tid + u * G::THREADS, kk = k0 + c / (TT / 2), x = 2 * (c % (TT / 2));
            const int s = kk < a.nb ? sidx[kk] : -1;
            const float2 *row = s >= 0 ? Df + (long long)s * a.ldd : nullptr;
            const int xr = (half ? r0 : v0) + c / H, nx = half ? a.nr : a.nv;
            const float4 d = xrow_load(row, (half ? v0 : r0) + x, half ? a.nv : a.nr);
            const float4 q = krow_load<SPEC_F>(Rf, brow, xr, nx, k0 + 2 * (c % H), a.nb);
            ra[u] = d;
            rb[u] = q;
        }
    };
    auto store = [&](int job) {
        const int half = job % NH;
        float *pi = ssm + (job & 1) * G::STAGE, *pj = pi + 2 * KC * G::PI;
#pragma unroll
        for (int u = 0; u < G::UI; ++u) {
            const int c = tid + u * G::THREADS;
            xrow_store<G::PI, TT, KC>(half ? pj : pi, c, ra[u]);
            krow_store<G::PJ, KC>(half ? pi : pj, c, rb[u]);
        }
    };
    static_assert(G::UI == G::UJ && G::PI == G::PJ && G::UI * G::THREADS == TT * KC / 2, "both operands are staged alike");
    SimtAcc c;
    c.zero();
    const bool diag = RECIP && (vb == rb_);
    // (the outputs of a diagonal tile below the diagonal are the mirrored ones)
    const bool active = r0 + wi < a.nr && v0 + wj < a.nv && !(diag && wi + G::WI <= wj);
    const int njobs = (a.nb + KC - 1) / KC * NH;
    load(0);
    store(0);
    __syncthreads();
    for (int job = 0; job < njobs; ++job) {
        if (job + 1 < njobs) load(job + 1);
        if (active) {
            if (!RECIP || job % 2 == 0) simt_chunk<G, 1>(c, ssm + (job & 1) * G::STAGE, ia, jb);
            else simt_chunk<G, 2>(c, ssm + (job & 1) * G::STAGE, ia, jb);
        }
        if (job + 1 < njobs) store(job + 1);
        __syncthreads();
    }
    float2 *gsm = reinterpret_cast<float2 *>(ssm);   // mirror buffer (r, v); the operands are dead
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int vv = jb + j, v = v0 + vv;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const int rr = ia + 2 * G::WTI * p, r = r0 + rr;
            const float2 x0 = cscale(make_float2(lo2(c.re[p][j]), lo2(c.im[p][j])), a.outscale);
            const float2 x1 = cscale(make_float2(hi2(c.re[p][j]), hi2(c.im[p][j])), a.outscale);
            if (v < a.nv) {
                const bool w0 = r < a.nr && (!diag || v <= r), w1 = r + 1 < a.nr && (!diag || v <= r + 1);
                float2 *dst = Cf + v * crow + spec_col(r);
                if (w0 && w1) *reinterpret_cast<float4 *>(dst) = make_float4(x0.x, x0.y, x1.x, x1.y);
                else {
                    if (w0) dst[0] = x0;
                    if (w1) dst[1] = x1;
                }
            }
            if (RECIP) {
                gsm[rr * (TT + 1) + vv] = x0;
                gsm[(rr + 1) * (TT + 1) + vv] = x1;
            }
        }
    }
    if (RECIP && (diag || !a.no_mirror)) {   // diagonal tiles always mirror (see GemmArgs::no_mirror)
        __syncthreads();
        for (int e = tid; e < TT * TT; e += G::THREADS) {
            const int rr = e / TT, vv = e % TT;
            const int r = r0 + rr, v = v0 + vv;
            if (v < a.nv && r < a.nr && (!diag || v < r)) Cf[r * crow + spec_col(v)] = gsm[rr * (TT + 1) + vv];
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Few virtual sources (nv <= 8, the matrix-vector regime of a single-virtual-source inversion): the
// products are bound by reading the batch rows of Dh once, so a warp streams one kernel row against
// the nv model rows (forward) or a thread owns one receiver and walks the batch (adjoint).  The operand that every
// kernel row meets again -- the model rows, or the residuals' coefficients -- is staged in shared memory by the CTA or shared
// by two kernel rows of a warp, and several loads of kernel rows are on their way at a time.  (Read from the SPEC_F
// layout for every kernel row, a warp's access touches four half lines: 231 and 222 us at nf 513, 600 x 8, batch 100,
// against 136 and 84 staged.)
// ------------------------------------------------------------------------------------------------
constexpr int GV_THREADS = 256, GV_MAXV = 8;
constexpr int GV_KC = 256;   // columns of a chunk of the model rows (forward)
constexpr int GV_BC = 128;   // batch entries of a chunk of the coefficients (adjoint)

template <int NV>
__device__ __forceinline__ void gemv_reduce(float2 (&acc)[NV]) {   // over the lanes, to lane 0
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            acc[v].x += __shfl_down_sync(0xffffffffu, acc[v].x, o);
            acc[v].y += __shfl_down_sync(0xffffffffu, acc[v].y, o);
        }
}
template <int NV>
__device__ __forceinline__ void gemv_put(const GemmArgs &a, int f, int b, const float2 (&acc)[NV]) {
    float2 *Cf = a.C + spec_bin(f, a.sCf);
#pragma unroll
    for (int v = 0; v < NV; ++v)
        if (v < a.nv) Cf[(long long)v * a.ldb * SPEC_F + spec_col(b)] = make_float2(acc[v].x * a.outscale, acc[v].y * a.outscale);
}

// forward: C[f][v][b] = sum_r A[f][v][r] Dh[f][idx_b][r].  Both operands from global memory, no barrier; a warp takes BW
// neighbouring batch entries at once, which share its loads of the model rows
template <int NV, int BW>
__global__ void __launch_bounds__(GV_THREADS) k_gemv_fwd_direct(GemmArgs a) {
    constexpr int UNROLL = NV == 2 ? 1 : 2;   // (two rows: 9.8 us unrolled against 8.3 at nf 257, 60 columns, batch 64)
    const int f = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = (blockIdx.y * (GV_THREADS / 32) + warp) * BW;
    if (b >= a.nb) return;   // warp-uniform; no barrier in this kernel
    const float2 *Af = a.A + spec_bin(f, a.sAf), *Df = a.Dh + (long long)f * a.sDf;
    const float2 *d[BW];
    bool have[BW];
#pragma unroll
    for (int j = 0; j < BW; ++j) {
        int s = -1;
        if (b + j < a.nb) {
            s = a.idx[b + j];
            if (s < 0 || s >= a.ns) {
                if (lane == 0) atomicOr(a.status, 1);
                s = -1;
            }
        }
        have[j] = s >= 0;
        d[j] = Df + (long long)(s < 0 ? 0 : s) * a.ldd;   // (row 0 for an entry without a source, whose sum is dropped)
    }
    float2 acc[BW][NV];
#pragma unroll
    for (int j = 0; j < BW; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[j][v] = make_float2(0.f, 0.f);
#pragma unroll UNROLL
    for (int r = lane; r < a.nr; r += 32) {
        float2 dv[BW];
#pragma unroll
        for (int j = 0; j < BW; ++j) dv[j] = __ldg(d[j] + r);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (NV <= 2 || v < a.nv) {   // (one or two rows: exactly as many; the loads of a round are issued together)
                const float2 x = __ldg(Af + (long long)v * a.ldr * SPEC_F + spec_col(r));
#pragma unroll
                for (int j = 0; j < BW; ++j) {
                    acc[j][v].x = fmaf(x.x, dv[j].x, fmaf(-x.y, dv[j].y, acc[j][v].x));
                    acc[j][v].y = fmaf(x.x, dv[j].y, fmaf(x.y, dv[j].x, acc[j][v].y));
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < BW; ++j) {
        gemv_reduce<NV>(acc[j]);
        if (!have[j]) {
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[j][v] = make_float2(0.f, 0.f);
        }
        if (lane == 0 && b + j < a.nb) gemv_put<NV>(a, f, b + j, acc[j]);
    }
}

// The model rows staged; 2^split_log2 warps per batch entry, which take the groups of 32 columns in turn (one
// warp in batches of 8 and more; in smaller ones the CTA's warps share the rows)
template <int NV>
__global__ void __launch_bounds__(GV_THREADS, NV == 2 ? 6 : NV == 4 ? 5 : 4) k_gemv_fwd(GemmArgs a, int split_log2) {
    constexpr int WARPS = GV_THREADS / 32, G = GV_KC / 32, ROW = GV_KC / 2;
    constexpr int ST = (NV * ROW + GV_THREADS - 1) / GV_THREADS;   // staged units (two columns) of a thread
    __shared__ float4 rows[2][NV][ROW];
    __shared__ float2 part[WARPS][NV];
    const int f = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wb = WARPS >> split_log2, split = 1 << split_log2, p = warp / wb;
    const int b = blockIdx.y * wb + warp % wb;
    int s = -1;   // a warp past the batch helps to stage
    if (b < a.nb) {
        s = a.idx[b];
        if (s < 0 || s >= a.ns) {
            if (lane == 0) atomicOr(a.status, 1);
            s = -1;
        }
    }
    const float2 *Af = a.A + spec_bin(f, a.sAf);
    const float2 *d = a.Dh + (long long)f * a.sDf + (long long)(s < 0 ? 0 : s) * a.ldd;
    float4 st[ST];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < ST; ++u) {
            const int e = threadIdx.x + u * GV_THREADS, v = e / ROW, c = e % ROW;
            if (v < NV) st[u] = krow_load<SPEC_F>(Af, (long long)a.ldr * SPEC_F, v, a.nv, k0 + 2 * c, a.nr);
        }
    };
    auto put = [&](int buf) {
#pragma unroll
        for (int u = 0; u < ST; ++u) {
            const int e = threadIdx.x + u * GV_THREADS, v = e / ROW, c = e % ROW;
            if (v < NV) rows[buf][v][c] = st[u];
        }
    };
    float2 dv[G];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const int r = k0 + lane + 32 * i;
            dv[i] = s >= 0 && r < a.nr && (i & (split - 1)) == p ? __ldg(d + r) : make_float2(0.f, 0.f);
        }
    };
    float2 acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = make_float2(0.f, 0.f);
    fetch(0);
    load(0);
    put(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < a.nr; k0 += GV_KC, buf ^= 1) {
        const bool more = k0 + GV_KC < a.nr;
        if (more) fetch(k0 + GV_KC);
        if (s >= 0) {
#pragma unroll
            for (int i = 0; i < G; ++i) {
                if (k0 + 32 * i < a.nr && (i & (split - 1)) == p) {   // (columns past nr are zero in both operands)
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        if (v < a.nv) {
                            const float2 x = reinterpret_cast<const float2 *>(rows[buf][v])[lane + 32 * i];
                            acc[v].x = fmaf(x.x, dv[i].x, fmaf(-x.y, dv[i].y, acc[v].x));
                            acc[v].y = fmaf(x.x, dv[i].y, fmaf(x.y, dv[i].x, acc[v].y));
                        }
                    }
                }
            }
        }
        if (more) {
            load(k0 + GV_KC);
            put(buf ^ 1);
            __syncthreads();
        }
    }
    gemv_reduce<NV>(acc);
    if (split > 1) {
        if (lane == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) part[warp][v] = acc[v];
        }
        __syncthreads();
        if (p == 0 && lane == 0)
            for (int q = 1; q < split; ++q)
#pragma unroll
                for (int v = 0; v < NV; ++v) acc[v] = cadd(acc[v], part[warp + q * wb][v]);
    }
    if (b < a.nb && p == 0 && lane == 0) gemv_put<NV>(a, f, b, acc);
}

// adjoint (no reciprocity): C[f][v][r] = outscale * sum_b A[f][v][b] conj(Dh[f][idx_b][r]); one thread
// per receiver r, the batch walked in order (the coefficients are warp-uniform broadcasts)
constexpr int GV_FEW = 8;

template <int NV>
__device__ __forceinline__ void gemv_store(const GemmArgs &a, int f, int r, const float2 (&acc)[NV]) {
    float2 *Cf = a.C + spec_bin(f, a.sCf);
#pragma unroll
    for (int v = 0; v < NV; ++v)
        if (v < a.nv) Cf[(long long)v * a.ldr * SPEC_F + spec_col(r)] = make_float2(acc[v].x * a.outscale, acc[v].y * a.outscale);
}

// batches below GV_FEW, whose chain of latencies bounds them: coefficients from global memory, beside the kernel rows
template <int NV>
__global__ void __launch_bounds__(GV_THREADS) k_gemv_adj_few(GemmArgs a) {
    __shared__ int sidx[GV_FEW];
    const int f = blockIdx.x, r = blockIdx.y * GV_THREADS + threadIdx.x;
    if (threadIdx.x < a.nb) {
        int s = a.idx[threadIdx.x];
        if (s < 0 || s >= a.ns) {
            atomicOr(a.status, 1);
            s = -1;
        }
        sidx[threadIdx.x] = s;
    }
    __syncthreads();
    if (r >= a.nr) return;   // after the only barrier
    const float2 *Af = a.A + spec_bin(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf;
    float2 acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = make_float2(0.f, 0.f);
    for (int b = 0; b < a.nb; ++b) {
        const int s = sidx[b];
        if (s < 0) continue;
        const float2 d = __ldg(Df + (long long)s * a.ldd + r);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (v < a.nv) {
                const float2 c = __ldg(Af + (long long)v * a.ldb * SPEC_F + spec_col(b));
                // c * conj(d)
                acc[v].x = fmaf(c.x, d.x, fmaf(c.y, d.y, acc[v].x));
                acc[v].y = fmaf(c.y, d.x, fmaf(-c.x, d.y, acc[v].y));
            }
        }
    }
    gemv_store<NV>(a, f, r, acc);
}

// larger batches: the coefficients staged, eight kernel rows on their way at a time
template <int NV>
__global__ void __launch_bounds__(GV_THREADS) k_gemv_adj(GemmArgs a) {
    constexpr int UB = 8;
    __shared__ int sidx[GV_BC];
    __shared__ __align__(16) float2 coef[GV_BC][NV];
    const int f = blockIdx.x, r = blockIdx.y * GV_THREADS + threadIdx.x;
    const float2 *Af = a.A + spec_bin(f, a.sAf);
    const float2 *Df = a.Dh + (long long)f * a.sDf + r;
    float2 acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = make_float2(0.f, 0.f);
    for (int b0 = 0; b0 < a.nb; b0 += GV_BC) {
        const int n = min(GV_BC, a.nb - b0);
        if (b0 > 0) __syncthreads();   // the last chunk has been read
        if (threadIdx.x < GV_BC) {
            int s = -1;
            if (threadIdx.x < n) {
                s = a.idx[b0 + threadIdx.x];
                if (s < 0 || s >= a.ns) {
                    atomicOr(a.status, 1);
                    s = -1;
                }
            }
            sidx[threadIdx.x] = s;
        }
        for (int e = threadIdx.x; e < a.nv * GV_BC; e += GV_THREADS) {
            const int v = e / GV_BC, b = e % GV_BC;
            if (b < n) coef[b][v] = __ldg(Af + (long long)v * a.ldb * SPEC_F + spec_col(b0 + b));
        }
        __syncthreads();
        if (r < a.nr) {
#pragma unroll 1
            for (int bb = 0; bb < n; bb += UB) {   // (entries past the batch have no source)
                float2 d[UB];
#pragma unroll
                for (int j = 0; j < UB; ++j) {
                    const int s = sidx[bb + j];
                    d[j] = s >= 0 ? __ldg(Df + (long long)s * a.ldd) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int j = 0; j < UB; ++j) {
                    if (sidx[bb + j] < 0) continue;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        if (v < a.nv) {
                            const float2 c = coef[bb + j][v];
                            // c * conj(d)
                            acc[v].x = fmaf(c.x, d[j].x, fmaf(c.y, d[j].y, acc[v].x));
                            acc[v].y = fmaf(c.y, d[j].x, fmaf(-c.x, d[j].y, acc[v].y));
                        }
                    }
                }
            }
        }
    }
    if (r < a.nr) gemv_store<NV>(a, f, r, acc);
}

bool gemv_supported(int nv) { return nv >= 1 && nv <= GV_MAXV; }

// Which forward kernel (us, direct with one entry a warp / with two / staged; batch 100 unless stated):
//  * rows of at most 128 columns, and one row: direct (nf 257, 60 x 8: 22.3 / 25 / 25; nf 513, 600 x 1: 51 / 50 / 53; nf 1025,
//    180 x 1: 41 / 37 / 42, batch 32: 14.2 / 12.3 / 16.2);
//  * three or four rows, batches of 16 and more: direct, two entries (nf 513, 600 x 3: 107 / 70 / 79; nf 1025, 180 x 3: 84 / 60 / 63);
//  * else staged (nf 1025, 180 x 2: 59 / 57 / 47; 180 x 8: 141 / 154 / 109; nf 513, 600 x 8, batch 1: 16 / 28 / 12).
cudaError_t launch_gemv_fwd(const GemmArgs &a, int nf, cudaStream_t st) {
    if (!gemv_supported(a.nv) || nf < 1) return cudaErrorInvalidValue;
    if (a.nf_active > 0 && a.nf_active < nf) return cudaErrorInvalidValue;   // band limits use the tiled kernels
    constexpr int WARPS = GV_THREADS / 32;
    const bool many = a.nb >= 16;
    if (a.nr <= 128 || a.nv == 1 || (a.nv <= 4 && a.nv > 2 && many)) {
        const int bw = many && ((a.nv == 1 && a.nr <= 256) || (a.nv > 2 && a.nv <= 4)) ? 2 : 1;
        const dim3 grid(nf, (a.nb + WARPS * bw - 1) / (WARPS * bw));
        if (a.nv == 1 && bw == 2) k_gemv_fwd_direct<1, 2><<<grid, GV_THREADS, 0, st>>>(a);
        else if (a.nv == 1) k_gemv_fwd_direct<1, 1><<<grid, GV_THREADS, 0, st>>>(a);
        else if (a.nv == 2) k_gemv_fwd_direct<2, 1><<<grid, GV_THREADS, 0, st>>>(a);
        else if (a.nv <= 4 && bw == 2) k_gemv_fwd_direct<4, 2><<<grid, GV_THREADS, 0, st>>>(a);
        else if (a.nv <= 4) k_gemv_fwd_direct<4, 1><<<grid, GV_THREADS, 0, st>>>(a);
        else k_gemv_fwd_direct<8, 1><<<grid, GV_THREADS, 0, st>>>(a);
        return cudaGetLastError();
    }
    int split = 0;   // (log2)
    while (WARPS >> split > 1 && (WARPS >> (split + 1)) >= a.nb) ++split;
    const int wb = WARPS >> split;
    const dim3 grid(nf, (a.nb + wb - 1) / wb);
    if (a.nv == 2) k_gemv_fwd<2><<<grid, GV_THREADS, 0, st>>>(a, split);
    else if (a.nv <= 4) k_gemv_fwd<4><<<grid, GV_THREADS, 0, st>>>(a, split);
    else k_gemv_fwd<8><<<grid, GV_THREADS, 0, st>>>(a, split);
    return cudaGetLastError();
}

cudaError_t launch_gemv_adj(const GemmArgs &a, int nf, cudaStream_t st) {
    if (!gemv_supported(a.nv) || nf < 1 || a.nb > AD_MAXNB) return cudaErrorInvalidValue;
    if (a.nf_active > 0 && a.nf_active < nf) return cudaErrorInvalidValue;
    const dim3 grid(nf, (a.nr + GV_THREADS - 1) / GV_THREADS);
    auto go = [&](auto kern, auto few) {
        if (a.nb >= GV_FEW) kern<<<grid, GV_THREADS, 0, st>>>(a);
        else few<<<grid, GV_THREADS, 0, st>>>(a);
    };
    if (a.nv == 1) go(k_gemv_adj<1>, k_gemv_adj_few<1>);
    else if (a.nv <= 2) go(k_gemv_adj<2>, k_gemv_adj_few<2>);
    else if (a.nv <= 4) go(k_gemv_adj<4>, k_gemv_adj_few<4>);
    else go(k_gemv_adj<8>, k_gemv_adj_few<8>);
    return cudaGetLastError();
}

// forward tiles
using FwdGeom64 = SimtGeom<4, 2, 2>;    // 64 x 64
using FwdGeom32 = SimtGeom<4, 2, 1>;    // 64 x 32
using FwdGeom32R = SimtGeom<4, 4, 1>;   // 128 x 32
using FwdGeom16 = SimtGeom<8, 2, 1>;    // 128 x 16
static_assert(adj_smem<AdjGeom64>() <= 49152 - AD_MAXNB * 4 && FwdGeom64::SMEM <= 40960 && FwdGeom32::SMEM <= 40960 &&
                  FwdGeom16::SMEM <= 40960 && FW_SMEM <= 49152 && AdjS<32, 32, true>::SMEM <= 49152 - AD_MAXNB * 4 &&
                  AdjS<16, 64, false>::SMEM <= 49152 - AD_MAXNB * 4,
              "no opt-in to more shared memory");

cudaError_t gemm_prepare() { return cudaSuccess; }

template <class G>
static void launch_fwd(const GemmArgs &a, int nf, cudaStream_t st) {
    const dim3 grid((a.nv + G::BI - 1) / G::BI, (a.nb + G::BJ - 1) / G::BJ, nf);
    if (a.plain) k_cgemm_fwd<G, 1><<<grid, G::THREADS, G::SMEM, st>>>(a);
    else k_cgemm_fwd<G, SPEC_F><<<grid, G::THREADS, G::SMEM, st>>>(a);
}

// outputs that tiles of geometry G compute for a product, padding included
template <class G>
static double padded_outputs(const GemmArgs &a) {
    return (double)((a.nv + G::BI - 1) / G::BI * G::BI) * ((a.nb + G::BJ - 1) / G::BJ * G::BJ);
}

// The geometry by the rows nv and the batch nb; us measured at nf 257, 300 columns unless stated (scalar / 128 x 16 /
// 128 x 32 / 64 x 32 / 64 x 64):
//   nb <= 16, nv <= 128: scalar          (100 rows, batch 16: 39.5 / 45.5 / 65 / 65 / 69; 32: 8.4 against 11 at nf 129)
//   nb <= 16, more rows: 128 x 16        (200, 16: 76 / 71 / - / 113 / 124)
//   up to 32 rows:       64 x 64         (24, 24: 40 / 64 / 41 / 41 / 37; 24, 64: 69 / 112 / 45 / 62 / 39)
//   nb <= 32, up to 64:  64 x 32         (48, 32: 65 / 64 / 62 / 43 / 59)
//   nb <= 32, up to 128: 128 x 32        (100 x 100, batch 32: 19.5 against 21.1 for 64 x 32)
//   nb <= 32, more rows: 64 x 32         (301, 32, nf 1025: 439 against 510 for 128 x 32)
//   larger batches: the least padded outputs, weighted by the time per output of the tiles (16 columns 1.3, 32 columns
//   1.1 times that of 64 x 64)           (128, 48: 108 / 98 / 117 / 115 / 108; 256, 80: - / 265 / - / 287 / 320;
//                                         301, 80: - / 363 / - / 336 / 393; 301, 64: - / - / - / 238 / 225)
cudaError_t launch_cgemm_fwd(const GemmArgs &a, int nf, cudaStream_t st) {
    if (a.nb <= 16 && a.nv <= 128) {
        const dim3 grid((a.nv + FW_ROWS - 1) / FW_ROWS, (a.nb + FW_NB - 1) / FW_NB, nf);
        if (a.plain) k_cgemm_fwd_small<1><<<grid, FW_THREADS, FW_SMEM, st>>>(a);
        else k_cgemm_fwd_small<SPEC_F><<<grid, FW_THREADS, FW_SMEM, st>>>(a);
    } else if (a.nb <= 16) {
        launch_fwd<FwdGeom16>(a, nf, st);
    } else if (a.nv <= 32) {
        launch_fwd<FwdGeom64>(a, nf, st);
    } else if (a.nb <= 32) {
        if (a.nv > 64 && a.nv <= 128) launch_fwd<FwdGeom32R>(a, nf, st);
        else launch_fwd<FwdGeom32>(a, nf, st);
    } else {
        const double w16 = 1.3 * padded_outputs<FwdGeom16>(a), w32 = 1.1 * padded_outputs<FwdGeom32>(a), w64 = padded_outputs<FwdGeom64>(a);
        if (w64 <= w32 && w64 <= w16) launch_fwd<FwdGeom64>(a, nf, st);
        else if (w32 <= w16) launch_fwd<FwdGeom32>(a, nf, st);
        else launch_fwd<FwdGeom16>(a, nf, st);
    }
    return cudaGetLastError();
}

// tile = 0, by the sizes (us at nf 257 unless stated):
//  * reciprocity: the packed 64-wide tiles unless their upper triangle has more than 1.2 times the outputs of the scalar
//    32-wide ones (scalar / packed: 201 columns, batch 16, nf 513, 1.43 times: 107 / 130; 210, batch 32, 1.43: 103 / 116;
//    400, batch 16, 1.23: 185 / 187; 128, batch 16, 1.20: 31.0 / 29.7; 192, batch 32, 1.14: 82 / 78; 256, batch 32, 1.11:
//    131 / 118; 512, batch 64, 1.06: 848 / 720);
//  * up to 16 rows and more than 64 columns: the scalar 16 x 64 tiles (scalar 32 x 32 / 16 x 64, batch 64: 17.7 / 16.2 at
//    65 columns x 4 rows, 47 / 34 at 300 x 8, 122 / 81 at 1000 x 16; batch 8: 7.7 / 7.8, 14.3 / 10.3, 26.7 / 18.5);
//  * matrices of one packed tile, and where tiles of 64 would pad the output 1.5 times as much as tiles of 32: the scalar
//    32-wide ones (150 x 65, batch 10, nf 513: 29 against 37; at 150 x 150, 1.44 times, batch 40, the packed ones stay ahead);
//  * else the packed 64-wide ones (scalar 32 / packed 64: 1320 / 974 at nf 1025, 301 x 301, batch 64; 145 / 98 at nf 513,
//    256 x 256, batch 16; 275 / 240 at nf 1025, 237 x 133, batch 27).
// 32 or 64: the scalar 32-wide or the packed 64-wide tiles
bool cgemm_adj_few_rows(int nv, int nr, bool recip) { return !recip && nv <= 16 && nr > 64; }

cudaError_t launch_cgemm_adj(const GemmArgs &a0, bool recip, int nf, cudaStream_t st, int tile) {
    GemmArgs a = a0;
    auto tiles = [](int n, int t) { return (n + t - 1) / t; };
    auto grid = [&](int tv, int tr) {
        a.tiles_v = tiles(a.nv, tv);
        a.tiles_r = tiles(a.nr, tr);
        return dim3(recip ? a.tiles_v * (a.tiles_v + 1) / 2 : a.tiles_v * a.tiles_r, nf);
    };
    if (tile == 0 && cgemm_adj_few_rows(a.nv, a.nr, recip)) {
        using F = AdjS<16, 64, false>;
        const dim3 g = grid(16, 64);
        k_cgemm_adj_small<16, 64, false><<<g, F::THREADS, F::SMEM, st>>>(a);
        return cudaGetLastError();
    }
    bool scalar = tile == 32;
    if (tile == 0 && recip) {
        const double t32 = tiles(a.nv, 32), t64 = tiles(a.nv, 64);
        scalar = 4 * t64 * (t64 + 1) > 1.2 * t32 * (t32 + 1);
    } else if (tile == 0) {
        scalar = (a.nv <= 64 && a.nr <= 64) ||
                 4. * tiles(a.nv, 64) * tiles(a.nr, 64) > 1.5 * tiles(a.nv, 32) * tiles(a.nr, 32);
    }
    if (scalar) {
        using F = AdjS<32, 32, false>;
        using R = AdjS<32, 32, true>;
        const dim3 g = grid(32, 32);
        if (recip) k_cgemm_adj_small<32, 32, true><<<g, R::THREADS, R::SMEM, st>>>(a);
        else k_cgemm_adj_small<32, 32, false><<<g, F::THREADS, F::SMEM, st>>>(a);
    } else {
        using G = AdjGeom64;
        const dim3 g = grid(64, 64);
        if (recip) k_cgemm_adj<G, true><<<g, G::THREADS, adj_smem<G>(), st>>>(a);
        else k_cgemm_adj<G, false><<<g, G::THREADS, adj_smem<G>(), st>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace smdd
