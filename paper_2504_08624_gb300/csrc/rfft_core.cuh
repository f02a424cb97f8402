// Register-resident transform of ONE real block for overlap-save filtering
// (k_fir_rfft.cu): M = 2N real samples as N complex points, filtered by a
// pointwise product, with no step that pairs mirrored bins.
//
// Arithmetic.  A window w[0..M) is read as the polynomial
// sum_(n < N) (w[n] + i w[n + N]) z^n modulo z^N - i.  Reduced modulo z^M + 1
// a real product of two polynomials of degree < M is their skew-circular
// convolution, and C[z]/(z^N - i) is that ring with z^N written as i; so a
// pointwise product of two transforms here is the skew-circular convolution
// of the two real windows, whose last M - (L - 1) values are the linear one
// (the wrapped part, negated, falls on the first L - 1 values, which
// overlap-save discards anyway).
//
// Tree.  z^S - w splits into (z^(S/2) - r)(z^(S/2) + r), r^2 = w: one
// butterfly u = a + r c, v = a - r c per pair of coefficients, with ONE
// twiddle r per node, whatever the position.  The root's subtree has
// constants; a later pass reads one set per node, shared by every thread of
// the node; positions never enter.  With w = e^(2 pi i h) the children have
// h/2 and h/2 + 1/2, the root h = 1/4; the nodes of a level in storage order
// are the bit-reversed ones: h_e = (h + bitrev(e)) / 2^level.  u takes two
// FMAs per part and v = 2a - u one more (6 for a butterfly of 2 points).
// The inverse of a radix-R subtree is a plain R-point DFT (constants) and
// R - 1 twiddles e^(-2 pi i h j / R) per node.
//
// Pairs.  Samples 2p and 2p + 1 share every twiddle down to the last level,
// so an element holds both (re.x, re.y and im.x, im.y) and every instruction
// is a packed two-lane one: a loaded twiddle serves both lanes.  The last
// level and the filter's product are one step: the product modulo
// z^2 - w of (a + c z) and (ha + hc z) is (ha a + w hc c) + (hc a + ha c) z.
//
// Passes.  Element p = t + T j of thread t first, then blocks of the tree;
// between passes the elements move through shared memory (16-byte words,
// padded one per PE).  A thread writes the words that it itself read in the
// exchange before, so an exchange needs one barrier, over the threads of
// one node.
#pragma once

#include "tfx_common.cuh"

namespace tfx {

// Shape of the N = 2^LOGN point transform: PE elements (2 points each) per
// thread, pass radices 2^RL (over elements), the passes' product N/2.
template <int LOGN>
struct RfShape {
    static constexpr int N = 1 << LOGN, M = 2 * N, NE = N / 2;
    static constexpr int LPE = rfft_log_pe(LOGN), PE = 1 << LPE, T = NE / PE;
    static constexpr int NP = rfft_passes(LOGN);
    static constexpr int rl(int p) { return rfft_radix_log(LOGN, p); }
    static constexpr int radix(int p) { return 1 << rl(p); }
    static constexpr int depth(int p) {  // levels above pass p
        int d = 0;
        for (int q = 0; q < p; ++q) d += rl(q);
        return d;
    }
    static constexpr int span(int p) { return NE >> depth(p); }
    static constexpr int sub(int p) { return span(p) / radix(p); }
    static constexpr int groups(int p) { return PE / radix(p); }  // subtrees per thread (1 but in the last pass)
    // float4 offset of pass p's tables: forward (radix/4 float4 per node),
    // then inverse (radix/2 per node); none for pass 0
    static constexpr int fwd_off(int p) { return rfft_fwd_off(LOGN, p); }
    static constexpr int inv_off(int p) { return rfft_fwd_off(LOGN, p) + (1 << depth(p)) * radix(p) / 4; }
    static constexpr int WORDS = NE + NE / PE;  // shared float4 words of an exchange
};

namespace rf {

#define RF_HD __host__ __device__ __forceinline__

struct Pair {
    float2 re, im;
};

// a * b + c in both lanes, b one value for both
RF_HD float2 fma2(float2 a, float b, float2 c) {
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, make_float2(b, b), c);
#else
    return make_float2(fmaf(a.x, b, c.x), fmaf(a.y, b, c.y));
#endif
}
RF_HD float2 fma2v(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, b, c);
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
RF_HD float2 mul2(float2 a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, make_float2(b, b));
#else
    return make_float2(a.x * b, a.y * b);
#endif
}
RF_HD float2 add2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, b);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}
RF_HD float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
RF_HD float2 sub2(float2 a, float2 b) { return add2(a, neg2(b)); }
RF_HD float2 swap2(float2 a) { return make_float2(a.y, a.x); }

// cos and sin of 2 pi a / 128
RF_HD constexpr float cosq(int a) {
    constexpr double c[33] = {1.0,
                              0.99879545620517239271,
                              0.99518472667219688624,
                              0.98917650996478097345,
                              0.98078528040323044913,
                              0.97003125319454399260,
                              0.95694033573220886494,
                              0.94154406518302077841,
                              0.92387953251128675613,
                              0.90398929312344333159,
                              0.88192126434835502971,
                              0.85772861000027206990,
                              0.83146961230254523708,
                              0.80320753148064490981,
                              0.77301045336273696081,
                              0.74095112535495909118,
                              0.70710678118654752440,
                              0.67155895484701840063,
                              0.63439328416364549822,
                              0.59569930449243334347,
                              0.55557023301960222474,
                              0.51410274419322172659,
                              0.47139673682599764856,
                              0.42755509343028209432,
                              0.38268343236508977173,
                              0.33688985339222005069,
                              0.29028467725446236764,
                              0.24298017990326388995,
                              0.19509032201612826785,
                              0.14673047445536175166,
                              0.09801714032956060199,
                              0.04906767432741801425,
                              0.0};
    a = a < 0 ? -a : a;
    a %= 128;
    if (a > 64) a = 128 - a;
    return (float)(a <= 32 ? c[a] : -c[64 - a]);
}
RF_HD constexpr float sinq(int a) { return cosq(32 - a); }
RF_HD constexpr int brev(int v, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((v >> b) & 1) << (bits - 1 - b);
    return r;
}

// (a, c) -> (a + w c, a - w c)
RF_HD void bf(Pair& a, Pair& c, float wr, float wi) {
    const float2 ur = fma2(c.im, -wi, fma2(c.re, wr, a.re));
    const float2 ui = fma2(c.re, wi, fma2(c.im, wr, a.im));
    c.re = fma2(a.re, 2.f, neg2(ur));
    c.im = fma2(a.im, 2.f, neg2(ui));
    a.re = ur;
    a.im = ui;
}
RF_HD void bf_one(Pair& a, Pair& c) {  // w = 1
    const float2 ur = add2(a.re, c.re), ui = add2(a.im, c.im);
    c.re = sub2(a.re, c.re);
    c.im = sub2(a.im, c.im);
    a.re = ur;
    a.im = ui;
}
RF_HD void bf_mi(Pair& a, Pair& c) {  // w = -i
    const float2 ur = add2(a.re, c.im), ui = sub2(a.im, c.re);
    const float2 vr = sub2(a.re, c.im), vi = add2(a.im, c.re);
    a.re = ur;
    a.im = ui;
    c.re = vr;
    c.im = vi;
}
RF_HD void cmul(Pair& v, float wr, float wi) {
    const float2 r = fma2(v.re, wr, mul2(v.im, -wi));
    v.im = fma2(v.im, wr, mul2(v.re, wi));
    v.re = r;
}

// Forward root subtree (constants): level L, node E.
template <int R, int L = 0, int E = 0, int NV>
RF_HD void fwd_const(Pair (&v)[NV]) {
    if constexpr ((R >> L) > 1) {
        constexpr int H = R >> (L + 1);
        constexpr int a = (1 + 4 * brev(E, L)) * (128 >> (L + 3));
        constexpr float c = cosq(a), s = sinq(a);
#pragma unroll
        for (int q = 0; q < H; ++q) bf(v[E * 2 * H + q], v[E * 2 * H + q + H], c, s);
        if constexpr (E + 1 < (1 << L))
            fwd_const<R, L, E + 1>(v);
        else
            fwd_const<R, L + 1, 0>(v);
    }
}

RF_HD float4 ld4(const float4* p) {
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

// Forward subtree of a node, its twiddles at tp[k * stride] (two per word):
// level 0, level 1, then the even nodes of each level (an odd node's twiddle
// is i times the even one's before it).
template <int R, int OFF, int NV>
RF_HD void fwd_node(Pair (&v)[NV], const float4* __restrict__ tp, int stride) {
    const float4 w01 = ld4(tp);
#pragma unroll
    for (int q = 0; q < R / 2; ++q) bf(v[OFF + q], v[OFF + q + R / 2], w01.x, w01.y);
#pragma unroll
    for (int q = 0; q < R / 4; ++q) bf(v[OFF + q], v[OFF + q + R / 4], w01.z, w01.w);
#pragma unroll
    for (int q = 0; q < R / 4; ++q) bf(v[OFF + R / 2 + q], v[OFF + R / 2 + q + R / 4], -w01.w, w01.z);
#pragma unroll
    for (int nodes = 4; nodes < R; nodes *= 2) {  // level log2(nodes): nodes / 4 words
        const int H = R / (2 * nodes);
#pragma unroll
        for (int k = 0; k < nodes / 4; ++k) {
            const float4 w = ld4(tp + (nodes / 4 + k) * stride);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float wr = e == 0 ? w.x : e == 1 ? -w.y : e == 2 ? w.z : -w.w;
                const float wi = e == 0 ? w.y : e == 1 ? w.x : e == 2 ? w.w : w.z;
#pragma unroll
                for (int q = 0; q < H; ++q)
                    bf(v[OFF + (4 * k + e) * 2 * H + q], v[OFF + (4 * k + e) * 2 * H + q + H], wr, wi);
            }
        }
    }
}

// Plain R-point DFT (e^(-2 pi i jk / R)), bit-reversed slots in, natural out.
template <int R, int OFF, int H = 1, int Q = 0, int NV>
RF_HD void dft(Pair (&v)[NV]) {
    if constexpr (H < R) {
        constexpr int a = (64 / H) * Q;  // 128ths of a turn
        constexpr float c = cosq(a), s = sinq(a);
#pragma unroll
        for (int b = 0; b < R; b += 2 * H) {
            if constexpr (a == 0)
                bf_one(v[OFF + b + Q], v[OFF + b + Q + H]);
            else if constexpr (a == 32)
                bf_mi(v[OFF + b + Q], v[OFF + b + Q + H]);
            else
                bf(v[OFF + b + Q], v[OFF + b + Q + H], c, -s);
        }
        if constexpr (Q + 1 < H)
            dft<R, OFF, H, Q + 1>(v);
        else
            dft<R, OFF, 2 * H, 0>(v);
    }
}

// Inverse twiddles of the root (constants) and of a node (words of two).
template <int R, int J = 1, int NV>
RF_HD void inv_const(Pair (&v)[NV]) {
    if constexpr (J < R) {
        constexpr int a = J * 32 / R;
        constexpr float c = cosq(a), s = sinq(a);
        cmul(v[J], c, -s);
        inv_const<R, J + 1>(v);
    }
}
template <int R, int OFF, int NV>
RF_HD void inv_node(Pair (&v)[NV], const float4* __restrict__ tp, int stride) {
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
        const float4 w = ld4(tp + k * stride);
        if (k > 0) cmul(v[OFF + 2 * k], w.x, w.y);
        cmul(v[OFF + 2 * k + 1], w.z, w.w);
    }
}

template <int LOGN, int P>
RF_HD void forward_pass(Pair (&v)[RfShape<LOGN>::PE], const float4* __restrict__ tw, int t) {
    using F = RfShape<LOGN>;
    constexpr int R = F::radix(P), G = F::groups(P);
    if constexpr (P == 0) {
        static_assert(G == 1 && R <= 32, "root subtree");
        fwd_const<R>(v);
    } else if constexpr (G == 1) {
        fwd_node<R, 0>(v, tw + F::fwd_off(P) + t / F::sub(P), 1 << F::depth(P));
    } else {
        static_assert(F::sub(P) == 1 && (G == 2 || G == 4), "several subtrees per thread: last pass");
        const float4* tp = tw + F::fwd_off(P) + t;
        constexpr int st = 1 << F::depth(P);
        fwd_node<R, 0>(v, tp, st);
        fwd_node<R, R>(v, tp + F::T, st);
        if constexpr (G == 4) {
            fwd_node<R, 2 * R>(v, tp + 2 * F::T, st);
            fwd_node<R, 3 * R>(v, tp + 3 * F::T, st);
        }
    }
}

template <int LOGN, int P>
RF_HD void inverse_pass(Pair (&v)[RfShape<LOGN>::PE], const float4* __restrict__ tw, int t) {
    using F = RfShape<LOGN>;
    constexpr int R = F::radix(P), G = F::groups(P);
    dft<R, 0>(v);
    if constexpr (G >= 2) dft<R, R>(v);
    if constexpr (G >= 4) {
        dft<R, 2 * R>(v);
        dft<R, 3 * R>(v);
    }
    if constexpr (P == 0) {
        inv_const<R>(v);
    } else if constexpr (G == 1) {
        inv_node<R, 0>(v, tw + F::inv_off(P) + t / F::sub(P), 1 << F::depth(P));
    } else {
        const float4* tp = tw + F::inv_off(P) + t;
        constexpr int st = 1 << F::depth(P);
        inv_node<R, 0>(v, tp, st);
        inv_node<R, R>(v, tp + F::T, st);
        if constexpr (G == 4) {
            inv_node<R, 2 * R>(v, tp + 2 * F::T, st);
            inv_node<R, 3 * R>(v, tp + 3 * F::T, st);
        }
    }
}

// Shared-memory word of element j of thread t in pass P: base(t) + off(j).
// Every pattern gives 8 consecutive lanes 8 different 16-byte banks:
// consecutive words, or (last pass) a stride of PE + 1.
template <int LOGN, int P>
RF_HD int word_base(int t) {
    using F = RfShape<LOGN>;
    if constexpr (P == 0) {
        return t + t / F::PE;
    } else if constexpr (F::sub(P) == 1) {
        return (F::PE + 1) * t;
    } else {
        const int n = (t / F::sub(P)) * F::span(P) + t % F::sub(P);
        return n + n / F::PE;
    }
}
template <int LOGN, int P>
RF_HD constexpr int word_off(int j) {
    using F = RfShape<LOGN>;
    const int n = P == 0 ? F::T * j : F::sub(P) * j;
    return F::sub(P) == 1 && P > 0 ? j : n + n / F::PE;
}

template <int LOGN, int P>
RF_HD void put(const Pair (&v)[RfShape<LOGN>::PE], float4* sb, int t) {
    float4* w = sb + word_base<LOGN, P>(t);
#pragma unroll
    for (int j = 0; j < RfShape<LOGN>::PE; ++j)
        w[word_off<LOGN, P>(j)] = make_float4(v[j].re.x, v[j].re.y, v[j].im.x, v[j].im.y);
}
template <int LOGN, int P>
RF_HD void get(Pair (&v)[RfShape<LOGN>::PE], const float4* sb, int t) {
    const float4* r = sb + word_base<LOGN, P>(t);
#pragma unroll
    for (int j = 0; j < RfShape<LOGN>::PE; ++j) {
        const float4 w = r[word_off<LOGN, P>(j)];
        v[j].re = make_float2(w.x, w.y);
        v[j].im = make_float2(w.z, w.w);
    }
}

// The filter's product with the last level folded in.  Per element ha, hc
// (the filter modulo z^2 - w) and q = w hc, scaled by 2/N: three words for
// elements e and e + 1 of thread t at ((3 (e/2) + i) T + t): (ha_e, ha_e+1),
// then (q.re, hc.re, q.im, hc.im) of each.
RF_HD void product_one(Pair& v, float hr, float hi, float4 b) {
    const float2 br = make_float2(b.x, b.y), bi = make_float2(b.z, b.w);
    const float2 sr = swap2(v.re), si = swap2(v.im);
    const float2 r = fma2v(sr, br, fma2v(si, neg2(bi), fma2(v.im, -hi, mul2(v.re, hr))));
    v.im = fma2v(si, br, fma2v(sr, bi, fma2(v.re, hi, mul2(v.im, hr))));
    v.re = r;
}
template <int LOGN>
RF_HD void product(Pair (&v)[RfShape<LOGN>::PE], const float4* __restrict__ H, int t) {
    using F = RfShape<LOGN>;
    const float4* h = H + t;
#pragma unroll
    for (int k = 0; k < F::PE / 2; ++k) {
        const float4 a = ld4(h + (3 * k) * F::T), b0 = ld4(h + (3 * k + 1) * F::T), b1 = ld4(h + (3 * k + 2) * F::T);
        product_one(v[2 * k], a.x, a.y, b0);
        product_one(v[2 * k + 1], a.z, a.w, b1);
    }
}

#ifdef __CUDACC__
// Barrier over the threads that exchange elements between pass p and p + 1:
// one node of pass p, a contiguous run of span(p) / PE threads.
template <int LOGN, int P>
__device__ __forceinline__ void node_sync(int t) {
    using F = RfShape<LOGN>;
    constexpr int G = F::span(P) / F::PE;
    if constexpr (G <= 32)
        __syncwarp();
    else  // named barriers of G threads (the CTA may hold others than the transform's)
        asm volatile("bar.sync %0, %1;" ::"r"(G == F::T ? 1 : 1 + t / G), "n"(G) : "memory");
}

template <int LOGN, int P>
__device__ __forceinline__ void forward_from(Pair (&v)[RfShape<LOGN>::PE], const float4* __restrict__ tw, float4* sb,
                                             int t) {
    forward_pass<LOGN, P>(v, tw, t);
    if constexpr (P + 1 < RfShape<LOGN>::NP) {
        put<LOGN, P>(v, sb, t);
        node_sync<LOGN, P>(t);
        get<LOGN, P + 1>(v, sb, t);
        forward_from<LOGN, P + 1>(v, tw, sb, t);
    }
}
template <int LOGN, int P>
__device__ __forceinline__ void inverse_from(Pair (&v)[RfShape<LOGN>::PE], const float4* __restrict__ tw, float4* sb,
                                             int t) {
    inverse_pass<LOGN, P>(v, tw, t);
    if constexpr (P > 0) {
        put<LOGN, P>(v, sb, t);
        node_sync<LOGN, P - 1>(t);
        get<LOGN, P - 1>(v, sb, t);
        inverse_from<LOGN, P - 1>(v, tw, sb, t);
    }
}
#endif

}  // namespace rf
}  // namespace tfx
