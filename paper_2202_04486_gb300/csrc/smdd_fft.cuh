// FFT building blocks of the MDC trace kernels (sm_103a): real transforms of two traces per thread in packed
// FP32 pairs.
//
// Appendix A evaluates the multi-dimensional convolution as FFT along time -> one complex matrix
// product per frequency -> inverse FFT.  Here every time trace of length nt is zero padded to
// N = nfft = 2M >= 2nt-1 samples (linear, not circular, convolution on [0, nt)) and transformed as a
// real sequence through a complex FFT of length M on z[n] = x[2n] + i x[2n+1]:
//   X[k] = 1/2 (Z[k] + conj Z[M-k]) - i/2 w_N^k (Z[k] - conj Z[M-k]),   k = 0..M,
// and back through the matching pre-processing and an inverse complex FFT of length M.
//
// Two traces per thread.  sm_103a executes add, multiply and fused multiply-add on a pair of FP32 values as
// one instruction (add/mul/fma.f32x2): the arithmetic rate is that of two scalar instructions, the issue slot
// is one.  The trace kernels are bound by issue and by the shared-memory pipe, not by arithmetic, so every
// complex value here is a pair of pairs: (re of trace A, re of trace B), (im of trace A, im of trace B).  Both
// traces share the twiddles, the index arithmetic and one 128-bit shared-memory access per element.
//
// Lanes.  PL = 4 such pairs (8 traces adjacent along the contiguous spectrum axis) are interleaved in the lanes
// of a warp: lane = PL * s + p.  A frequency row of the tile is then one contiguous 64-byte segment over the PL
// lanes of an s, so the edge passes read and write the spectra in global memory directly, without staging a
// tile in shared memory, and the PL lanes share their twiddle loads.
//
// Passes.  M = R_1 R_2 ... R_m (radices 4, 8, 12 or 16, the last one 8).  Forward pass p combines the digit r of
// the time index left over into the frequency digit k_p, in place: the value of (jj, k_1 .. k_p) lies at
// jj + k_p L_p + ... + k_1 L_1 with L_p = M / (R_1 .. R_p).  A pass therefore stores where it loaded, the only
// barriers are the ones between passes, and the inverse runs the same passes backwards through the same
// locations.  The first forward pass takes its inputs from registers and the last inverse pass leaves its
// outputs in registers in the same order and at the same locations, so an inverse FFT, an element-wise epilogue
// and a forward FFT chain without a barrier.  The last forward pass (radix 8) gives a thread the bins u + r S and
// S - u + r S (S = M / 8), i.e. both bins k and M - k of every pair that the real-signal processing combines.
//
// Shared memory: element i of pair p is the 16-byte unit i PL + p.  The k_1 blocks are padded by one element
// and the low bits of jj are mixed (mix()), which makes every 128-bit access of every pass free of bank
// conflicts (8 lanes of a quarter-warp on 8 distinct 16-byte columns; enumerated for every length).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace smdd {

// ------------------------------------------------------------------------------------------------
// complex helpers (float2 = re, im)
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }

// ------------------------------------------------------------------------------------------------
// packed FP32 pairs
// ------------------------------------------------------------------------------------------------
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ f32x2 dup2(float x) { return pk2(x, x); }
__device__ __forceinline__ float lo2(f32x2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(f32x2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return pk2(-lo2(a), -hi2(a)); }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Sum of squares of FP32 values, no less exact than an FP64 sum, without the FP64 unit, which runs at 1/64 of the FP32
// rate here.  Each square is split exactly into p + e (e by a fused multiply-add).  The p are added to a word that starts
// at sigma, a power of two above their sum, so that an addition's rounding error is p - ((hi + p) - hi) exactly (Dekker's
// fast two-sum); these errors and the e are added in the same way to a second word, whose errors go to a third.  Both
// members of a pair at once, 14 packed operations a pair of values, at most SQUARES of a member.  The third word carries
// about 2^-56 of relative error, and total() rounds the sum of the three once to FP64: 2^-53.0 at most, 2^-54.2 rms for 32 random,
// decaying or widely spread values (FP64 additions one by one: up to 2^-49.5, 2^-52 rms; two words with the second
// one summed plainly: 2^-45, and further off with every value).
// The largest |x| of a group of values lies in [2^-44, 2^60), or the group takes the FP64 unit: sigma stays below 2^126,
// and what the e lose below the FP32 range (2^-150 each) below 2^-55 of the group's sum.
struct SumSq {
    static constexpr int SQUARES = 32;
    f32x2 hi, mid, lo = 0;
    float sigma;
    static __device__ __forceinline__ bool in_range(float top) { return top < 0x1p60f && (top >= 0x1p-44f || top == 0.f); }
    // the power of two of a value in range: |x| < 2 pow2(x)
    static __device__ __forceinline__ float pow2(float top) { return __uint_as_float(__float_as_uint(top) & 0x7f800000u); }
    // for values below 2 bound (a power of two, or zero)
    explicit __device__ __forceinline__ SumSq(float bound) : sigma(bound * bound * (4.f * SQUARES)) {
        hi = dup2(sigma);
        mid = dup2(sigma * 0x1p-18f);
    }
    // acc += x, returns the rounding error (|acc| >= |x|)
    static __device__ __forceinline__ f32x2 fast_sum(f32x2 &acc, f32x2 x) {
        const f32x2 t = add2(acc, x), err = sub2(x, sub2(t, acc));
        acc = t;
        return err;
    }
    // a + b, the error to err (Knuth's two-sum)
    static __device__ __forceinline__ float two_sum(float a, float b, float &err) {
        const float t = a + b, z = t - a;
        err = (a - (t - z)) + (b - z);
        return t;
    }
    __device__ __forceinline__ void add(f32x2 x) {
        const f32x2 p = mul2(x, x), e = fma2(x, x, neg2(p));
        const f32x2 e1 = fast_sum(mid, fast_sum(hi, p)), e2 = fast_sum(mid, e);
        lo = add2(lo, add2(e1, e2));
    }
    // the members of each word are added in FP32 with the errors carried down: three conversions and two additions in FP64
    __device__ __forceinline__ double total() const {
        float eh, em, e;
        const float h = two_sum(lo2(hi) - sigma, hi2(hi) - sigma, eh);
        const float m = two_sum(two_sum(lo2(mid) - sigma * 0x1p-18f, hi2(mid) - sigma * 0x1p-18f, em), eh, e);
        return (double)h + ((double)m + (double)((lo2(lo) + hi2(lo)) + (em + e)));
    }
};

// a complex value of two traces, and a twiddle held twice
struct C2 {
    f32x2 re, im;
};
struct W2 {
    f32x2 re, im;
};

__device__ __forceinline__ C2 cadd2(C2 a, C2 b) { return C2{add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 csub2(C2 a, C2 b) { return C2{sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a w (INV: a conj(w))
template <bool INV>
__device__ __forceinline__ C2 ctw2(C2 a, W2 w) {
    const f32x2 n = neg2(w.im);
    return INV ? C2{fma2(a.im, w.im, mul2(a.re, w.re)), fma2(a.re, n, mul2(a.im, w.re))}
               : C2{fma2(a.im, n, mul2(a.re, w.re)), fma2(a.re, w.im, mul2(a.im, w.re))};
}
// a - i b (forward) / a + i b (INV); and the opposite sign
template <bool INV>
__device__ __forceinline__ C2 add_mi(C2 a, C2 b) {
    return INV ? C2{sub2(a.re, b.im), add2(a.im, b.re)} : C2{add2(a.re, b.im), sub2(a.im, b.re)};
}

__device__ __forceinline__ C2 ldsC(const float4 *p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
    return C2{v.x, v.y};
}
__device__ __forceinline__ void stsC(float4 *p, C2 v) { *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(v.re, v.im); }
__device__ __forceinline__ W2 wdup(float2 v) { return W2{dup2(v.x), dup2(v.y)}; }
__device__ __forceinline__ W2 wmul(W2 a, W2 b) {
    return W2{fma2(a.im, neg2(b.im), mul2(a.re, b.re)), fma2(a.re, b.im, mul2(a.im, b.re))};
}
// w e^{-2 pi i r / 16}
template <int r>
__device__ __forceinline__ W2 rot16(W2 w) {
    constexpr float C[8] = {1.f, 0.92387953251128675613f, 0.70710678118654752440f, 0.38268343236508977173f,
                            0.f, -0.38268343236508977173f, -0.70710678118654752440f, -0.92387953251128675613f};
    constexpr float S[8] = {0.f, 0.38268343236508977173f, 0.70710678118654752440f, 0.92387953251128675613f,
                            1.f, 0.92387953251128675613f, 0.70710678118654752440f, 0.38268343236508977173f};
    if constexpr (r == 0) return w;
    else if constexpr (r == 4) return W2{w.im, neg2(w.re)};
    else {
        const f32x2 c = dup2(C[r]), p = dup2(S[r]), n = dup2(-S[r]);
        return W2{fma2(w.im, p, mul2(w.re, c)), fma2(w.re, n, mul2(w.im, c))};
    }
}

// ------------------------------------------------------------------------------------------------
// small DFTs in registers (unnormalised; INV uses the conjugate roots; HALF: the upper half of the inputs is
// zero and not read)
// ------------------------------------------------------------------------------------------------
template <bool INV, bool HALF>
__device__ __forceinline__ void dft4p(C2 &a0, C2 &a1, C2 &a2, C2 &a3) {
    if constexpr (HALF) {
        const C2 x = a0, y = a1;
        a0 = cadd2(x, y);
        a1 = add_mi<INV>(x, y);
        a2 = csub2(x, y);
        a3 = add_mi<!INV>(x, y);
    } else {
        const C2 t0 = cadd2(a0, a2), t1 = csub2(a0, a2), t2 = cadd2(a1, a3), t3 = csub2(a1, a3);
        a0 = cadd2(t0, t2);
        a2 = csub2(t0, t2);
        a1 = add_mi<INV>(t1, t3);
        a3 = add_mi<!INV>(t1, t3);
    }
}

template <bool INV, bool HALF>
__device__ __forceinline__ void dft8p(C2 *a) {
    // even / odd halves: y_k = E_k + w8^k O_k, y_{k+4} = E_k - w8^k O_k
    dft4p<INV, HALF>(a[0], a[2], a[4], a[6]);
    dft4p<INV, HALF>(a[1], a[3], a[5], a[7]);
    const f32x2 h = dup2(0.70710678118654752440f), nh = dup2(-0.70710678118654752440f);
    const C2 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1], o1 = a[3], o2 = a[5], o3 = a[7];
    a[0] = cadd2(e0, o0);
    a[4] = csub2(e0, o0);
    a[2] = add_mi<INV>(e2, o2);
    a[6] = add_mi<!INV>(e2, o2);
    // w8^1 o = h (o.re + o.im, o.im - o.re), w8^3 o = h (o.im - o.re, -(o.re + o.im)) (forward)
    const f32x2 s1 = add2(o1.re, o1.im), d1 = sub2(o1.im, o1.re);
    const f32x2 s3 = add2(o3.re, o3.im), d3 = sub2(o3.im, o3.re);
    if constexpr (!INV) {
        a[1] = C2{fma2(s1, h, e1.re), fma2(d1, h, e1.im)};
        a[5] = C2{fma2(s1, nh, e1.re), fma2(d1, nh, e1.im)};
        a[3] = C2{fma2(d3, h, e3.re), fma2(s3, nh, e3.im)};
        a[7] = C2{fma2(d3, nh, e3.re), fma2(s3, h, e3.im)};
    } else {   // conj(w8) o = h (o.re - o.im, o.re + o.im), conj(w8^3) o = h (-(o.re + o.im), o.re - o.im)
        a[1] = C2{fma2(d1, nh, e1.re), fma2(s1, h, e1.im)};
        a[5] = C2{fma2(d1, h, e1.re), fma2(s1, nh, e1.im)};
        a[3] = C2{fma2(s3, nh, e3.re), fma2(d3, nh, e3.im)};
        a[7] = C2{fma2(s3, h, e3.re), fma2(d3, h, e3.im)};
    }
}

// y + w o and y - w o for a constant w = c - i s (forward; c + i s for INV)
template <bool INV>
__device__ __forceinline__ void comb2(C2 &p, C2 &m, C2 e, C2 o, float c, float s) {
    const f32x2 pc = dup2(c), nc = dup2(-c), ps = dup2(INV ? -s : s), ns = dup2(INV ? s : -s);
    p = C2{fma2(o.re, pc, fma2(o.im, ps, e.re)), fma2(o.im, pc, fma2(o.re, ns, e.im))};
    m = C2{fma2(o.re, nc, fma2(o.im, ns, e.re)), fma2(o.im, nc, fma2(o.re, ps, e.im))};
}

template <bool INV, bool HALF>
__device__ __forceinline__ void dft16p(C2 *a) {
    constexpr float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f;   // cos, sin(pi / 8)
    constexpr float h = 0.70710678118654752440f;
    C2 e[8], o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        e[i] = a[2 * i];
        o[i] = a[2 * i + 1];
    }
    dft8p<INV, HALF>(e);
    dft8p<INV, HALF>(o);
    a[0] = cadd2(e[0], o[0]);
    a[8] = csub2(e[0], o[0]);
    a[4] = add_mi<INV>(e[4], o[4]);
    a[12] = add_mi<!INV>(e[4], o[4]);
    comb2<INV>(a[1], a[9], e[1], o[1], c1, s1);
    comb2<INV>(a[2], a[10], e[2], o[2], h, h);
    comb2<INV>(a[3], a[11], e[3], o[3], s1, c1);
    comb2<INV>(a[5], a[13], e[5], o[5], -s1, c1);
    comb2<INV>(a[6], a[14], e[6], o[6], -h, h);
    comb2<INV>(a[7], a[15], e[7], o[7], -c1, s1);
}

// radix 3: y0 = a0 + a1 + a2, y1/2 = a0 - (a1 + a2)/2 -/+ i (sqrt(3)/2) (a1 - a2) (signs swap for INV)
template <bool INV>
__device__ __forceinline__ void dft3p(C2 &a0, C2 &a1, C2 &a2) {
    const f32x2 mh = dup2(-0.5f), q = dup2(0.86602540378443864676f), nq = dup2(-0.86602540378443864676f);
    const C2 s = cadd2(a1, a2), d = csub2(a1, a2);
    const C2 m = C2{fma2(s.re, mh, a0.re), fma2(s.im, mh, a0.im)};
    a0 = cadd2(a0, s);
    const C2 u = C2{fma2(d.im, q, m.re), fma2(d.re, nq, m.im)}, v = C2{fma2(d.im, nq, m.re), fma2(d.re, q, m.im)};
    a1 = INV ? v : u;
    a2 = INV ? u : v;
}

// radix 12 by the prime-factor map (no twiddles): input n = 4 n1 + 3 n2 mod 12, output k with k1 = k mod 3,
// k2 = k mod 4
template <bool INV>
__device__ __forceinline__ void dft12p(C2 *a) {
    C2 b[4][3];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
        for (int n1 = 0; n1 < 3; ++n1) b[n2][n1] = a[(4 * n1 + 3 * n2) % 12];
        dft3p<INV>(b[n2][0], b[n2][1], b[n2][2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
        dft4p<INV, false>(b[0][k1], b[1][k1], b[2][k1], b[3][k1]);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) a[(4 * k1 + 9 * k2) % 12] = b[k2][k1];
    }
}

template <int R, bool INV, bool HALF>
__device__ __forceinline__ void dftRp(C2 *a) {
    static_assert(R == 4 || R == 8 || R == 12 || R == 16, "radix");
    if constexpr (R == 4) dft4p<INV, HALF>(a[0], a[1], a[2], a[3]);
    else if constexpr (R == 8) dft8p<INV, HALF>(a);
    else if constexpr (R == 12) dft12p<INV>(a);
    else dft16p<INV, HALF>(a);
}

// ------------------------------------------------------------------------------------------------
// plans
// ------------------------------------------------------------------------------------------------
constexpr int FFT_P = 16;   // complex values per thread and trace

__host__ __device__ constexpr int fft_npass(int M) { return M <= 128 ? 2 : M <= 2048 ? 3 : 4; }
__host__ __device__ constexpr int fft_radix(int M, int p) {
    return p == fft_npass(M) - 1 ? 8
         : M == 32 ? 4
         : M == 64 || M == 512 || M == 4096 ? 8
         : M == 1024 ? (p == 0 ? 8 : 16)
         : M == 128 ? 16
         : M == 256 ? (p == 0 ? 8 : 4)
         : M == 1536 ? (p == 0 ? 16 : 12)
         : 16;   // 2048
}
// NS_p = R_1 .. R_{p-1}: frequency digits before pass p (0-based); L_p = M / (R_1 .. R_p)
__host__ __device__ constexpr int fft_span(int M, int p) { return p == 0 ? 1 : fft_span(M, p - 1) * fft_radix(M, p - 1); }
__host__ __device__ constexpr int fft_left(int M, int p) { return M / (fft_span(M, p) * fft_radix(M, p)); }

// Tables (float2).  Passes p >= 1: entry [i][k] (k < NS_p) = w_{NS_p R_p}^{r_i k} for the roots r_i = 1, 2, 3, 4, 8, 12
// below R_p; every other power is one product of two of these (twiddles()).  (Loading every power, in doubled form,
// costs the shared-memory / L1 pipe four cycles per load and warp: 2300 of 9400 such cycles a tile at M = 1024, on the
// busiest pipe of these kernels.)  Then w_N^k for k <= S / 2.
__host__ __device__ constexpr int tw_roots(int R) { return 2 + R / 4; }
__host__ __device__ constexpr int tw_root(int i) { return i < 3 ? i + 1 : 4 * (i - 2); }
__host__ __device__ constexpr int tw_off(int M, int p) {
    int off = 0;
    for (int q = 1; q < p; ++q) off += tw_roots(fft_radix(M, q)) * fft_span(M, q);
    return off;
}
__host__ __device__ constexpr int twn_off(int M) { return tw_off(M, fft_npass(M)); }
__host__ __device__ constexpr int tw_size(int M) { return twn_off(M) + M / 16 + 1; }
// the angle of entry i of the tables, as the fraction num / den of a full turn (w = exp(-2 pi i num / den))
__host__ __device__ inline void tw_angle(int M, int i, int &num, int &den) {
    num = i - twn_off(M);
    den = 2 * M;
    for (int p = 1; p < fft_npass(M); ++p) {
        const int off = tw_off(M, p), NS = fft_span(M, p), R = fft_radix(M, p);
        if (i >= off && i < off + tw_roots(R) * NS) {
            const int root = (i - off) / NS;
            num = tw_root(root) * ((i - off) % NS);
            den = NS * R;
        }
    }
}

// The roots w^{tw_root(i)} of one butterfly, loaded ahead of their use (before the barrier in front of the pass, so
// that the latency of the table loads overlaps it).
template <int R>
struct Roots {
    float2 w[tw_roots(R)];
    template <int NS>
    __device__ __forceinline__ void load(const float2 *__restrict__ tw) {
#pragma unroll
        for (int i = 0; i < tw_roots(R); ++i) w[i] = __ldg(tw + i * NS);
    }
};

// z[r] *= w^r (INV: conj(w)^r), r = 1 .. R - 1
template <int R, bool INV>
__device__ __forceinline__ void twiddles(C2 *z, const Roots<R> &t) {
    const W2 w1 = wdup(t.w[0]), w2 = wdup(t.w[1]), w3 = wdup(t.w[2]);
    z[1] = ctw2<INV>(z[1], w1);
    z[2] = ctw2<INV>(z[2], w2);
    z[3] = ctw2<INV>(z[3], w3);
#pragma unroll
    for (int i = 1; i < R / 4; ++i) {
        const W2 w = wdup(t.w[2 + i]);
        z[4 * i] = ctw2<INV>(z[4 * i], w);
        z[4 * i + 1] = ctw2<INV>(z[4 * i + 1], wmul(w, w1));
        z[4 * i + 2] = ctw2<INV>(z[4 * i + 2], wmul(w, w2));
        z[4 * i + 3] = ctw2<INV>(z[4 * i + 3], wmul(w, w3));
    }
}

// Launch geometry for complex length M: T = M/16 threads per pair of traces, PL pairs interleaved in the lanes,
// G such groups in a CTA (4 for the lengths whose group is at most a warp: with one, the CTA's fixed work -- the
// loss reduction and its atomic above all -- costs a third of the residual step at nt 30 to 128).
template <int M>
struct Team {
    static constexpr int T = M / FFT_P;
    static constexpr int PL = M == 4096 ? 2 : 4;
    static constexpr int GT = PL * T;                    // threads of a group
    static constexpr int G = M <= 128 ? 4 : 1;           // groups in a CTA
    static constexpr int THREADS = GT * G;
    static constexpr int TR = 2 * PL * G;                // traces in a CTA
    static constexpr int R1 = fft_radix(M, 0), L1 = M / R1;
    static constexpr int ELEMS = R1 * (L1 + 1);          // elements of a pair's buffer (padded)
    static constexpr size_t SMEM = (size_t)ELEMS * PL * G * 16;
    // resident CTAs per SM asked of the compiler: 512 threads at 128 registers.  At M = 1536 two CTAs of 384 threads
    // at 80 registers, although they spill: one CTA leaves the SM idle while it waits for its tile (transform alone
    // 1410 -> 1090 us, update 2560 -> 2440 us at nt 1500, 600 x 400); the samples that the update or the residual
    // needs after the inverse transform are then loaded after it (LATE), not held through it.
    static constexpr int MINB = M == 1536 ? 2 : THREADS >= 512 ? 1 : 512 / THREADS;
    static constexpr bool LATE = M == 1536;
};

// Synchronise the threads of a group (a group lies in one warp, or the CTA is one group).
template <int M>
__device__ __forceinline__ void group_sync() {
    static_assert(Team<M>::GT <= 32 || Team<M>::G == 1, "no barrier for several groups of more than a warp");
    if constexpr (Team<M>::GT <= 32) __syncwarp();
    else __syncthreads();
}

// mixing of the low bits of jj (and of the digit of the last pass): lanes whose jj differ by 1 or by 2 fall on
// different 16-byte columns of a quarter-warp's access
template <int PL>
__host__ __device__ __forceinline__ constexpr int mix(int i) {
    return PL == 4 ? (i ^ ((i >> 1) & 1)) : (i ^ ((i >> 2) & 1));
}
// offset of the digits k_1 .. k_p (kk = k_1 + R_1 k_2 + ...)
template <int M>
__device__ __forceinline__ int digit_off(int kk, int p) {
    constexpr int R1 = fft_radix(M, 0), L1 = M / R1;
    if (p == 1) return kk * (L1 + 1);
    int o = (kk % R1) * (L1 + 1);
    kk /= R1;
    for (int q = 1; q < p; ++q) {
        o += (kk % fft_radix(M, q)) * fft_left(M, q);
        kk /= fft_radix(M, q);
    }
    return o;
}
// first-pass butterfly q of thread s: pairs of adjacent jj (one butterfly when R_1 = 16)
template <int M>
__device__ __forceinline__ int first_jj(int s, int q) {
    return Team<M>::R1 == 16 ? s : 2 * s + (q & 1) + 2 * Team<M>::T * (q >> 1);
}

// ------------------------------------------------------------------------------------------------
// passes between registers and shared memory (buf: the group's buffer, offset by the pair)
// ------------------------------------------------------------------------------------------------
// first forward pass: a[q R1 + r] holds z[first_jj(q) + r L1] for r < R1 / 2 (the upper half is the zero
// padding, not read)
template <int M>
__device__ __forceinline__ void fwd_first(C2 (&a)[FFT_P], float4 *buf, int s) {
    constexpr int R = Team<M>::R1, L = Team<M>::L1, PL = Team<M>::PL;
#pragma unroll
    for (int q = 0; q < FFT_P / R; ++q) {
        dftRp<R, false, true>(&a[q * R]);
        float4 *b = buf + mix<PL>(first_jj<M>(s, q)) * PL;
#pragma unroll
        for (int r = 0; r < R; ++r) stsC(b + r * (L + 1) * PL, a[q * R + r]);
    }
}

// last inverse pass: a[q R1 + r] = z[first_jj(q) + r L1], of which the caller uses r < R1 / 2
template <int M>
__device__ __forceinline__ void inv_last(C2 (&a)[FFT_P], const float4 *buf, int s) {
    constexpr int R = Team<M>::R1, L = Team<M>::L1, PL = Team<M>::PL;
#pragma unroll
    for (int q = 0; q < FFT_P / R; ++q) {
        const float4 *b = buf + mix<PL>(first_jj<M>(s, q)) * PL;
#pragma unroll
        for (int r = 0; r < R; ++r) a[q * R + r] = ldsC(b + r * (L + 1) * PL);
        dftRp<R, true, false>(&a[q * R]);
    }
}

// middle pass p, in place (a length whose butterflies do not divide by the threads has a partial last round); the
// barrier before it is inside, behind the loads of the roots
template <int M, bool INV, int p>
__device__ __forceinline__ void mid_pass(float4 *buf, int s, const float2 *__restrict__ tw) {
    constexpr int R = fft_radix(M, p), L = fft_left(M, p), NS = fft_span(M, p), T = Team<M>::T, PL = Team<M>::PL;
    constexpr int NB = M / R, NQ = (NB + T - 1) / T;
    static_assert(T % L == 0 && L % 4 == 0, "every round of a thread has the same jj");
    const int jj = s % L;
    Roots<R> t[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        t[q].template load<NS>(tw + tw_off(M, p) + ((NB % T == 0 || s + T * q < NB) ? s / L + q * (T / L) : 0));
    group_sync<M>();
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        if (NB % T == 0 || s + T * q < NB) {
            const int kk = s / L + q * (T / L);
            float4 *b = buf + (mix<PL>(jj) + digit_off<M>(kk, p)) * PL;
            C2 x[R];
#pragma unroll
            for (int r = 0; r < R; ++r) x[r] = ldsC(b + r * L * PL);
            if constexpr (!INV) {
                twiddles<R, false>(x, t[q]);
                dftRp<R, false, false>(x);
            } else {
                dftRp<R, true, false>(x);
                twiddles<R, true>(x, t[q]);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) stsC(b + r * L * PL, x[r]);
        }
    }
}

template <int M, bool INV, int p>
__device__ __forceinline__ void mid_passes(float4 *buf, int s, const float2 *__restrict__ tw) {
    // forward: p = 1 .. npass - 2; inverse: p = npass - 2 .. 1
    if constexpr (p >= 1 && p <= fft_npass(M) - 2) {
        mid_pass<M, INV, p>(buf, s, tw);
        mid_passes<M, INV, INV ? p - 1 : p + 1>(buf, s, tw);
    }
}

// ------------------------------------------------------------------------------------------------
// edge passes: radix 8 with the real-signal processing
// ------------------------------------------------------------------------------------------------
// Z[k], Z[M-k] (in x, y) from X[k], X[M-k] and w = w_N^k: Z = E + i O, E = X[k] + conj X[M-k],
// O = (X[k] - conj X[M-k]) conj(w); Z[M-k] = conj(E - i O)
__device__ __forceinline__ void real_pre(C2 &x, C2 &y, W2 w) {
    const f32x2 er = add2(x.re, y.re), ei = sub2(x.im, y.im), dr = sub2(x.re, y.re), di = add2(x.im, y.im);
    const f32x2 o_re = fma2(di, w.im, mul2(dr, w.re)), o_im = fma2(dr, neg2(w.im), mul2(di, w.re));
    x = C2{sub2(er, o_im), add2(ei, o_re)};
    y = C2{add2(er, o_im), sub2(o_re, ei)};
}
// X[k], X[M-k] (in x, y) from Z[k], Z[M-k] and w = w_N^k: with e = (Z[k] + conj Z[M-k]) / 2,
// g = w (Z[k] - conj Z[M-k]) / 2: X[k] = e - i g, X[M-k] = conj(e + i g)
__device__ __forceinline__ void real_post(C2 &x, C2 &y, W2 w) {
    const f32x2 hf = dup2(0.5f), nhf = dup2(-0.5f);
    const f32x2 er = add2(x.re, y.re), ei = sub2(x.im, y.im), dr = sub2(x.re, y.re), di = add2(x.im, y.im);
    const f32x2 g_im = fma2(dr, w.im, mul2(di, w.re)), ng_re = fma2(di, w.im, mul2(dr, neg2(w.re)));
    const f32x2 e2 = mul2(er, hf), g2 = mul2(ng_re, hf);
    x = C2{fma2(g_im, hf, e2), fma2(ei, hf, g2)};
    y = C2{fma2(g_im, nhf, e2), fma2(ei, nhf, g2)};
}

// The bins of thread s: A[r] = bin s + r S and B[r] = bin S - s + r S (S/2 + r S for s = 0), r < 8, S = M / 8; for
// s = 0 also bin M (its real part goes to `nyq`).
//
// roots of the edge pass: of the butterflies of A and B, and of the real-signal processing
template <int M>
struct EdgeRoots {
    Roots<8> a, b;
    float2 n;   // w_N^s
    __device__ __forceinline__ void load(const float2 *__restrict__ tw, int s) {
        constexpr int S = M / 8, P = fft_npass(M) - 1;
        n = __ldg(tw + twn_off(M) + s);
        a.template load<S>(tw + tw_off(M, P) + s);
        b.template load<S>(tw + tw_off(M, P) + (s ? S - s : S / 2));
    }
};

// inverse: A, B hold the spectrum; real pre-processing, radix-8 inverse butterflies, twiddles, store
template <int M>
__device__ __forceinline__ void edge_inv(C2 (&A)[8], C2 (&B)[8], f32x2 nyq, float4 *buf, int s, const float2 *__restrict__ tw,
                                         const EdgeRoots<M> &t) {
    constexpr int S = M / 8, PL = Team<M>::PL, P = fft_npass(M) - 1;
    const W2 wn = wdup(t.n);
    if (s != 0) {
        real_pre(A[0], B[7], wn);
        real_pre(A[1], B[6], rot16<1>(wn));
        real_pre(A[2], B[5], rot16<2>(wn));
        real_pre(A[3], B[4], rot16<3>(wn));
        real_pre(A[4], B[3], rot16<4>(wn));
        real_pre(A[5], B[2], rot16<5>(wn));
        real_pre(A[6], B[1], rot16<6>(wn));
        real_pre(A[7], B[0], rot16<7>(wn));
    } else {
        // A: k = r S pairs with M - k = (8 - r) S; k = 0 with bin M (imaginary parts ignored), k = M/2 with itself
        const f32x2 x0 = A[0].re;
        A[0] = C2{add2(x0, nyq), sub2(x0, nyq)};
        real_pre(A[1], A[7], rot16<1>(wn));
        real_pre(A[2], A[6], rot16<2>(wn));
        real_pre(A[3], A[5], rot16<3>(wn));
        A[4] = C2{add2(A[4].re, A[4].re), neg2(add2(A[4].im, A[4].im))};
        // B: k = S/2 + r S pairs with S/2 + (7 - r) S
        const W2 wh = wdup(__ldg(tw + twn_off(M) + S / 2));
        real_pre(B[0], B[7], wh);
        real_pre(B[1], B[6], rot16<1>(wh));
        real_pre(B[2], B[5], rot16<2>(wh));
        real_pre(B[3], B[4], rot16<3>(wh));
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        C2(&z)[8] = h ? B : A;
        const int u = h ? (s ? S - s : S / 2) : s;
        dft8p<true, false>(z);
        twiddles<8, true>(z, h ? t.b : t.a);
        float4 *b = buf + digit_off<M>(u, P) * PL;
#pragma unroll
        for (int r = 0; r < 8; ++r) stsC(b + mix<PL>(r) * PL, z[r]);
    }
}

// forward (the barrier in front of it inside): load, twiddles, radix-8 butterflies, real post-processing; on return A, B hold the spectrum, nyq the
// real part of bin M for s = 0
template <int M>
__device__ __forceinline__ void edge_fwd(C2 (&A)[8], C2 (&B)[8], f32x2 &nyq, const float4 *buf, int s, const float2 *__restrict__ tw) {
    constexpr int S = M / 8, PL = Team<M>::PL, P = fft_npass(M) - 1;
    EdgeRoots<M> t;
    t.load(tw, s);
    group_sync<M>();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        C2(&z)[8] = h ? B : A;
        const int u = h ? (s ? S - s : S / 2) : s;
        const float4 *b = buf + digit_off<M>(u, P) * PL;
#pragma unroll
        for (int r = 0; r < 8; ++r) z[r] = ldsC(b + mix<PL>(r) * PL);
        twiddles<8, false>(z, h ? t.b : t.a);
        dft8p<false, false>(z);
    }
    const W2 wn = wdup(t.n);
    nyq = 0;
    if (s != 0) {
        real_post(A[0], B[7], wn);
        real_post(A[1], B[6], rot16<1>(wn));
        real_post(A[2], B[5], rot16<2>(wn));
        real_post(A[3], B[4], rot16<3>(wn));
        real_post(A[4], B[3], rot16<4>(wn));
        real_post(A[5], B[2], rot16<5>(wn));
        real_post(A[6], B[1], rot16<6>(wn));
        real_post(A[7], B[0], rot16<7>(wn));
    } else {
        nyq = sub2(A[0].re, A[0].im);
        A[0] = C2{add2(A[0].re, A[0].im), 0};
        real_post(A[1], A[7], rot16<1>(wn));
        real_post(A[2], A[6], rot16<2>(wn));
        real_post(A[3], A[5], rot16<3>(wn));
        A[4].im = neg2(A[4].im);
        const W2 wh = wdup(__ldg(tw + twn_off(M) + S / 2));
        real_post(B[0], B[7], wh);
        real_post(B[1], B[6], rot16<1>(wh));
        real_post(B[2], B[5], rot16<2>(wh));
        real_post(B[3], B[4], rot16<3>(wh));
    }
}

}  // namespace smdd
