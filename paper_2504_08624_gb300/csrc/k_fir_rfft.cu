// FIR by overlap-save with one real block per transform (rfft_core.cuh): block
// b of a channel reads the window x[bB - J, bB + B) (M = J + B samples, J >=
// L - 1 even, zero outside the signal) and writes y[bB, bB + B); a channel at
// an odd address starts one sample earlier (row_shift).
//
// Against two blocks as real and imaginary parts of one M-point transform
// (k_fir_fft): half the points per CTA for the same M, so that two (M =
// 16384) to eight (M = 4096; 24 at 1024) independent CTAs share an SM and one's loads and
// exchanges run under another's butterflies; two points per packed
// instruction and per 16-byte word; one barrier per exchange; samples loaded
// and stored in pairs; the next window asked into L2 ahead of its CTA.  Bound:
// the L1/shared-memory data pipe (88 % busy at M = 4096, 66 % at 16384:
// exchanges, product table, samples), then the FP32 pipe (58 and 53 %), and
// latency.  Measured, two blocks per transform -> this:
// 64 x 2.88M, 5231 taps 813 -> 513 us (M = 16384); 128 x 4 Mi, 16384 taps
// 4165 (two partitions) -> 2331 us (M = 32768); 12 x 7.94M, 336 taps
// 209 -> 163 us (M = 4096), 2 blocks of 16384 7.5 against 16.7 us; 16384 x 300,
// 65 taps 29.9 -> 24.1 us (M = 1024), 16384 x 1900, 129 taps 66.6 -> 55.6
// (M = 2048; eight elements per thread, three short passes).
// Tried and left: one warp per transform at 2048 points (32 elements per
// thread, one exchange; same time, FP32 latency with 8 warps per SM, and
// slower on small signals: 9.5 against 7.6 us), L1::no_allocate loads (0 to
// 6 % slower), separate real and imaginary planes in the exchange (same), more
// CTAs of fewer registers (their exchanges leave the tables too little L1:
// 2 to 25 % slower), exchanges of four lanes by shuffles (4 %), CTAs that stay
// and take the next window by a bulk copy during the last pass (5 to 10 %:
// its way through shared memory costs more than the latency that it hides).
#include <type_traits>

#include "rfft_core.cuh"

namespace tfx {
namespace {

using namespace rf;

// CTAs per SM: 16 warps of up to 128 registers (8 of up to 255 at n = 14, 24 of
// up to 80 at n = 9 and 10)
__host__ __device__ constexpr int rfft_min_ctas(int n) {
    return n == 9 ? 24 : n == 10 ? 12 : n == 11 ? 8 : n == 12 ? 4 : n == 13 ? 2 : 1;
}

// Window samples s + [0, M) of a row, zero outside [0, N): element j of
// thread t holds samples 2p, 2p + 1 (re) and those N points later (im), p =
// t + T j.  REV: the row holds its samples in reverse time (sample n at row[N
// - 1 - n]).
template <int LOGN, bool REV = false>
__device__ __forceinline__ void load_window(Pair (&v)[RfShape<LOGN>::PE], const float* row, int64_t s, int64_t N,
                                            int t) {
    using F = RfShape<LOGN>;
    if constexpr (REV) {
        const float* e = row + (N - s);  // one past window sample 0
        if (s >= 0 && s + F::M <= N && (reinterpret_cast<uintptr_t>(e) & 7) == 0) {
            const float2* q = reinterpret_cast<const float2*>(e) - 1 - t;
#pragma unroll
            for (int j = 0; j < F::PE; ++j) {
                v[j].re = swap2(__ldg(q - F::T * j));
                v[j].im = swap2(__ldg(q - F::T * j - F::NE));
            }
        } else {
            const int lo = s < 0 ? (int)-s : 0;
            const int hi = N - s < F::M ? (int)(N - s) : F::M;
#pragma unroll
            for (int j = 0; j < F::PE; ++j) {
                const int n = 2 * (t + F::T * j);
                auto at = [&](int o) { return n + o >= lo && n + o < hi ? __ldg(e - 1 - n - o) : 0.f; };
                v[j].re = make_float2(at(0), at(1));
                v[j].im = make_float2(at(F::N), at(F::N + 1));
            }
        }
        return;
    }
    const float* p = row + s + 2 * t;
    if (s >= 0 && s + F::M <= N && (reinterpret_cast<uintptr_t>(row + s) & 7) == 0) {
        const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            v[j].re = __ldg(q + F::T * j);
            v[j].im = __ldg(q + F::T * j + F::NE);
        }
    } else {
        // valid samples: window positions [lo, hi)
        const int lo = s < 0 ? (int)-s : 0;
        const int hi = N - s < F::M ? (int)(N - s) : F::M;
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int n = 2 * (t + F::T * j);
            auto at = [&](int o) { return n + o >= lo && n + o < hi ? __ldg(p + 2 * F::T * j + o) : 0.f; };
            v[j].re = make_float2(at(0), at(1));
            v[j].im = make_float2(at(F::N), at(F::N + 1));
        }
    }
}

// Window positions [J, J + m) are the outputs n0 + [0, m) of a row (REV: in
// reverse time, of a row of N samples).
template <int LOGN, bool REV = false>
__device__ __forceinline__ void store_window(const Pair (&v)[RfShape<LOGN>::PE], float* row, int64_t n0, int J, int m,
                                             int64_t N, int t) {
    using F = RfShape<LOGN>;
    if constexpr (REV) {
        float* e = row + (N - n0 + J) - 2 * t;  // one past window position 2 t
        const int o0 = 2 * t - J;
        const bool vec = (m & 1) == 0 && (reinterpret_cast<uintptr_t>(row + (N - n0)) & 7) == 0;
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int o = o0 + 2 * F::T * j;
            float* q = e - 2 * F::T * j;
            if (vec) {
                if ((unsigned)o < (unsigned)m) reinterpret_cast<float2*>(q)[-1] = swap2(v[j].re);
                if ((unsigned)(o + F::N) < (unsigned)m) reinterpret_cast<float2*>(q)[-1 - F::NE] = swap2(v[j].im);
            } else {
                if ((unsigned)o < (unsigned)m) q[-1] = v[j].re.x;
                if ((unsigned)(o + 1) < (unsigned)m) q[-2] = v[j].re.y;
                if ((unsigned)(o + F::N) < (unsigned)m) q[-1 - F::N] = v[j].im.x;
                if ((unsigned)(o + 1 + F::N) < (unsigned)m) q[-2 - F::N] = v[j].im.y;
            }
        }
        return;
    }
    float* p = row + n0 - J + 2 * t;
    const int o0 = 2 * t - J;
    if ((m & 1) == 0 && (reinterpret_cast<uintptr_t>(row + n0) & 7) == 0) {  // J is even
        float2* q = reinterpret_cast<float2*>(p);
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int o = o0 + 2 * F::T * j;
            if ((unsigned)o < (unsigned)m) q[F::T * j] = v[j].re;
            if ((unsigned)(o + F::N) < (unsigned)m) q[F::T * j + F::NE] = v[j].im;
        }
    } else {
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int o = o0 + 2 * F::T * j;
            if ((unsigned)o < (unsigned)m) p[2 * F::T * j] = v[j].re.x;
            if ((unsigned)(o + 1) < (unsigned)m) p[2 * F::T * j + 1] = v[j].re.y;
            if ((unsigned)(o + F::N) < (unsigned)m) p[2 * F::T * j + F::N] = v[j].im.x;
            if ((unsigned)(o + 1 + F::N) < (unsigned)m) p[2 * F::T * j + 1 + F::N] = v[j].im.y;
        }
    }
}

// Window samples s + [0, M) of a row (on 8 bytes), zero outside [0, N): element j of
// thread t holds samples 2p, 2p + 1 (re) and those N points later (im), p =
// t + T j.  REV: the row holds its samples in reverse time (sample n at row[N
// - 1 - n]).
template <int LOGN, bool REV>
__device__ __forceinline__ void load_row(Pair (&v)[RfShape<LOGN>::PE], const float* row, int64_t s, int64_t N,
                                         int t) {
    using F = RfShape<LOGN>;
    if constexpr (REV) {
        const float* e = row + (N - s);  // one past window sample 0
        if (s >= 0 && s + F::M <= N) {
            const float2* q = reinterpret_cast<const float2*>(e) - 1 - t;
#pragma unroll
            for (int j = 0; j < F::PE; ++j) {
                v[j].re = swap2(__ldg(q - F::T * j));
                v[j].im = swap2(__ldg(q - F::T * j - F::NE));
            }
        } else {
            const int lo = s < 0 ? (int)-s : 0;
            const int hi = N - s < F::M ? (int)(N - s) : F::M;
#pragma unroll
            for (int j = 0; j < F::PE; ++j) {
                const int n = 2 * (t + F::T * j);
                auto at = [&](int o) { return n + o >= lo && n + o < hi ? __ldg(e - 1 - n - o) : 0.f; };
                v[j].re = make_float2(at(0), at(1));
                v[j].im = make_float2(at(F::N), at(F::N + 1));
            }
        }
        return;
    }
    const float* p = row + s + 2 * t;
    if (s >= 0 && s + F::M <= N) {
        const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            v[j].re = __ldg(q + F::T * j);
            v[j].im = __ldg(q + F::T * j + F::NE);
        }
    } else {
        // valid samples: window positions [lo, hi)
        const int lo = s < 0 ? (int)-s : 0;
        const int hi = N - s < F::M ? (int)(N - s) : F::M;
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int n = 2 * (t + F::T * j);
            auto at = [&](int o) { return n + o >= lo && n + o < hi ? __ldg(p + 2 * F::T * j + o) : 0.f; };
            v[j].re = make_float2(at(0), at(1));
            v[j].im = make_float2(at(F::N), at(F::N + 1));
        }
    }
}

// Samples before a row's first by which its blocks start, so that the pairs of
// every window lie on 8 bytes whatever the row's address (block lengths and
// overlaps are even): its samples then move as pairs in all blocks but the
// first and the last.  Moved one by one in every odd row before: 4097 taps,
// 11 x 1,000,003 37.0 -> 34.9 us, a batch of 120 clips 576 -> 548.
// Launches without odd rows keep a form of their own (load_window and
// store_window) except at M = 8192 and below 4096: the compiler's (nvcc 13.0.88)
// order of this one is 2 to 3 % slower at M = 16384 (5231 taps, 64 x 2.88M: 512
// against 523 to 528 us), 0.5 to 1 % at 4096 and 32768, and 5 % faster at 8192
// (2500 taps, 16 x 2.88M: 118.6 against 112.0).  One template with both forms
// as its instantiations: 513 -> 529 us there, 2329 -> 2348 at 32768.
constexpr bool odd_form_only(int n) { return n <= 10 || n == 12; }
// Reversed rows: the input gradient of the spectral training plans (M = 4096, 8192).
constexpr bool reversed_form(int n) { return n == 11 || n == 12; }
template <bool REV>
__device__ __forceinline__ int row_shift(const float* row, int64_t N) {
    return (int)(((reinterpret_cast<uintptr_t>(row) >> 2) + (REV ? (uintptr_t)N : 0)) & 1);
}

// From scalars: a store of the packed result itself keeps both forms of every
// value live beside the branch that stores one by one.  Faster at M = 8192 (2500
// taps, 16 x 2.88M: 117.5 -> 112.0 us), not at the other sizes (4097 taps, 11 x
// 1,000,003 at M = 16384: 35.0 -> 35.8) nor in the batched kernel (548 -> 552).
template <bool SCALARS>
__device__ __forceinline__ void store2(float2* p, float2 v) {
    if constexpr (SCALARS)
        asm volatile("st.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
    else
        *p = v;
}

// Window positions [J, J + m) are the outputs n0 + [0, m) of a row (REV: in
// reverse time, of a row of N samples), the first of them before it if n0 = -1.
template <int LOGN, bool REV, bool SCALARS>
__device__ __forceinline__ void store_row(const Pair (&v)[RfShape<LOGN>::PE], float* row, int64_t n0, int J, int m,
                                          int64_t N, int t) {
    using F = RfShape<LOGN>;
    if constexpr (REV) {
        float* e = row + (N - n0 + J) - 2 * t;  // one past window position 2 t
        const int o0 = 2 * t - J;
        const int lo = n0 < 0 ? 1 : 0;
        const bool vec = (m & 1) == 0 && lo == 0 && (reinterpret_cast<uintptr_t>(row + (N - n0)) & 7) == 0;
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int o = o0 + 2 * F::T * j;
            float* q = e - 2 * F::T * j;
            if (vec) {
                if ((unsigned)o < (unsigned)m) reinterpret_cast<float2*>(q)[-1] = swap2(v[j].re);
                if ((unsigned)(o + F::N) < (unsigned)m) reinterpret_cast<float2*>(q)[-1 - F::NE] = swap2(v[j].im);
            } else {
                const int u = o - lo;
                if ((unsigned)u < (unsigned)(m - lo)) q[-1] = v[j].re.x;
                if ((unsigned)(u + 1) < (unsigned)(m - lo)) q[-2] = v[j].re.y;
                if ((unsigned)(u + F::N) < (unsigned)(m - lo)) q[-1 - F::N] = v[j].im.x;
                if ((unsigned)(u + 1 + F::N) < (unsigned)(m - lo)) q[-2 - F::N] = v[j].im.y;
            }
        }
        return;
    }
    float* p = row + n0 - J + 2 * t;
    const int o0 = 2 * t - J;
    if ((m & 1) == 0 && n0 >= 0 && (reinterpret_cast<uintptr_t>(row + n0) & 7) == 0) {  // J is even
        float2* q = reinterpret_cast<float2*>(p);
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int o = o0 + 2 * F::T * j;
            if ((unsigned)o < (unsigned)m) store2<SCALARS>(q + F::T * j, v[j].re);
            if ((unsigned)(o + F::N) < (unsigned)m) store2<SCALARS>(q + F::T * j + F::NE, v[j].im);
        }
    } else {
        const int lo = n0 < 0 ? 1 : 0;
        m -= lo;
#pragma unroll
        for (int j = 0; j < F::PE; ++j) {
            const int o = o0 - lo + 2 * F::T * j;
            if ((unsigned)o < (unsigned)m) p[2 * F::T * j] = v[j].re.x;
            if ((unsigned)(o + 1) < (unsigned)m) p[2 * F::T * j + 1] = v[j].re.y;
            if ((unsigned)(o + F::N) < (unsigned)m) p[2 * F::T * j + F::N] = v[j].im.x;
            if ((unsigned)(o + 1 + F::N) < (unsigned)m) p[2 * F::T * j + 1 + F::N] = v[j].im.y;
        }
    }
}

// Ask for the window of the block that runs on this SM after this one: the
// CTAs are handed out in order, so about `ahead` blocks on.  Only whole
// windows inside the row, from the 16-byte boundary below their start.
template <int LOGN>
__device__ __forceinline__ void prefetch_window(const float* row, int64_t s, int64_t N) {
    constexpr int M = RfShape<LOGN>::M;
    if (s < 4 || s + M > N) return;
    const uintptr_t p = reinterpret_cast<uintptr_t>(row + s) & ~(uintptr_t)15;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(4 * M) : "memory");
}

// Transform, product and inverse of one block's window.
template <int LOGN>
__device__ __forceinline__ void filter_window(Pair (&v)[RfShape<LOGN>::PE], const float4* H, const float4* tw,
                                              float4* sb, int t) {
    forward_from<LOGN, 0>(v, tw, sb, t);
    product<LOGN>(v, H, t);
    inverse_from<LOGN, RfShape<LOGN>::NP - 1>(v, tw, sb, t);
}

constexpr unsigned SMS = GB300_SMS;

template <int LOGN, bool REV, bool ODD>
__global__ void __launch_bounds__(RfShape<LOGN>::T, rfft_min_ctas(LOGN)) k_fir_rfft(RfftArgs a) {
    extern __shared__ float4 sb4[];
    const int t = threadIdx.x;
    const unsigned nbpc = (unsigned)a.nbpc;
    const unsigned c = blockIdx.x / nbpc, r = blockIdx.x - c * nbpc;
    int64_t n0 = (int64_t)r * a.B;
    if constexpr (ODD) {
        n0 -= row_shift<REV>(a.x + c * a.ldx, a.N);
        if (n0 >= a.N) return;  // (an even row among odd ones: its last block may be empty)
    }
    Pair v[RfShape<LOGN>::PE];
    after_previous();
    if constexpr (ODD)
        load_row<LOGN, REV>(v, a.x + c * a.ldx, n0 - a.J, a.N, t);
    else
        load_window<LOGN, REV>(v, a.x + c * a.ldx, n0 - a.J, a.N, t);
    const unsigned kn = blockIdx.x + SMS * rfft_min_ctas(LOGN);
    if (t == 0 && kn < (unsigned)a.nb) {
        const unsigned cn = kn / nbpc, rn = kn - cn * nbpc;
        const int64_t sn = (int64_t)rn * a.B - a.J;
        prefetch_window<LOGN>(a.x + cn * a.ldx, REV ? a.N - sn - RfShape<LOGN>::M : sn, a.N);
    }
    filter_window<LOGN>(v, a.H, a.tw, sb4, t);
    const int m = a.N - n0 < a.B ? (int)(a.N - n0) : a.B;
    if constexpr (ODD)
        store_row<LOGN, REV, LOGN == 12>(v, a.y + c * a.ldy, n0, a.J, m, a.N, t);
    else
        store_window<LOGN, REV>(v, a.y + c * a.ldy, n0, a.J, m, a.N, t);
}

// The same over many clips in one launch: CTA k takes block k - prefix[u] of
// its clip u = unit_of[k], with the clip's own product table.
template <int LOGN>
__global__ void __launch_bounds__(RfShape<LOGN>::T, rfft_min_ctas(LOGN))
    k_fir_rfft_batched(const BatchFft* __restrict__ units, const int64_t* __restrict__ prefix,
                       const int32_t* __restrict__ unit_of, BatchBases bases, const float4* __restrict__ tw) {
    extern __shared__ float4 sb4[];
    const int t = threadIdx.x;
    const int u = __ldg(unit_of + blockIdx.x);
    const BatchFft d = units[u];
    const unsigned nbpc = (unsigned)d.nbpc, k = (unsigned)(blockIdx.x - prefix[u]);
    const unsigned c = k / nbpc, r = k - c * nbpc;
    const float* x = bases.ptr(d.x_sel) + d.x_off;
    const int J = RfShape<LOGN>::M - d.B;
    const float* row = x + c * d.N;
    const int64_t n0 = (int64_t)r * d.B - row_shift<false>(row, d.N);
    if (n0 >= d.N) return;
    Pair v[RfShape<LOGN>::PE];
    load_row<LOGN, false>(v, row, n0 - J, d.N, t);
    const unsigned kn = k + SMS * rfft_min_ctas(LOGN);  // (of this clip only)
    if (t == 0 && kn < (unsigned)d.nb) {
        const unsigned cn = kn / nbpc, rn = kn - cn * nbpc;
        prefetch_window<LOGN>(x + cn * d.N, (int64_t)rn * d.B - J, d.N);
    }
    filter_window<LOGN>(v, d.H, tw, sb4, t);
    store_row<LOGN, false, false>(v, bases.ptr(d.y_sel) + d.y_off + c * d.N, n0, J,
                                  d.N - n0 < d.B ? (int)(d.N - n0) : d.B, d.N, t);
}

// The product table of a filter from its FP32 taps on the device (coefficient
// updates without a host round trip): the filter's own forward transform of
// the taps is ha and hc of every element, q = w hc in FP64 from the plan's
// roots.  Every CTA does the whole transform and writes two elements of each
// thread: FP64 is what the last step costs (2 FMAs per clock and SM).  An
// update of 129 / 1025 / 4097 / 12000 / 16384 taps with the roots from
// sincospi in one CTA 24.3 / 27.6 / 51.8 / 105 / 109 us, so 4.0 / 4.7 / 6.6 /
// 8.9 / 8.9 us (taps rounded once by k_update_fir_taps, over several CTAs).
template <int LOGN>
__global__ void __launch_bounds__(RfShape<LOGN>::T, 1)
    k_fir_rfft_table(const float* __restrict__ taps, int L, const float4* __restrict__ tw,
                     const double2* __restrict__ roots, float4* __restrict__ H) {
    using F = RfShape<LOGN>;
    extern __shared__ float4 sb4[];
    const int t = threadIdx.x;
    Pair v[F::PE];
    auto at = [&](int n) { return n < L ? __ldg(taps + n) : 0.f; };
#pragma unroll
    for (int j = 0; j < F::PE; ++j) {
        const int n = 2 * (t + F::T * j);
        v[j].re = make_float2(at(n), at(n + 1));
        v[j].im = make_float2(at(n + F::N), at(n + F::N + 1));
    }
    forward_from<LOGN, 0>(v, tw, sb4, t);
    constexpr float sc = 2.0f / F::N;
#pragma unroll
    for (int e = 0; e < F::PE; ++e) {
        if (e / 2 != (int)blockIdx.x) continue;
        // w of element 4k + i is w, -w, iw, -iw of element 4k
        const double2 w4 = __ldg(roots + (F::PE * t + e) / 4);
        const double c = e % 4 == 0 ? w4.x : e % 4 == 1 ? -w4.x : e % 4 == 2 ? -w4.y : w4.y;
        const double s = e % 4 == 0 ? w4.y : e % 4 == 1 ? -w4.y : e % 4 == 2 ? w4.x : -w4.x;
        const float hcr = v[e].re.y * sc, hci = v[e].im.y * sc;
        float4* w = H + (3 * (e / 2)) * F::T + t;
        reinterpret_cast<float2*>(w)[e % 2] = make_float2(v[e].re.x * sc, v[e].im.x * sc);
        w[(1 + e % 2) * F::T] = make_float4((float)(c * hcr - s * hci), hcr, (float)(c * hci + s * hcr), hci);
    }
}

template <int LOGN>
constexpr size_t smem_bytes() {
    return RfShape<LOGN>::WORDS * sizeof(float4);
}

template <typename F>
cudaError_t by_size(int n, F f) {
    switch (n) {
        case 9: return f(std::integral_constant<int, 9>());
        case 10: return f(std::integral_constant<int, 10>());
        case 11: return f(std::integral_constant<int, 11>());
        case 12: return f(std::integral_constant<int, 12>());
        case 13: return f(std::integral_constant<int, 13>());
        case 14: return f(std::integral_constant<int, 14>());
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_fir_rfft(int n, const RfftArgs& args, cudaStream_t s) {
    RfftArgs a = args;
    if (a.C <= 0 || a.N <= 0) return cudaSuccess;
    // blocks per row: of one sample more where a row's blocks may start early
    const int64_t first = (int64_t)(reinterpret_cast<uintptr_t>(a.x) >> 2) + (a.rev ? a.N : 0);
    const bool odd = (first & 1) != 0 || (a.C > 1 && (a.ldx & 1) != 0);
    a.nbpc = (a.N + (odd ? 1 : 0) + a.B - 1) / a.B;
    a.nb = a.C * a.nbpc;
    if (a.nb > INT32_MAX) return cudaErrorInvalidValue;
    return by_size(n, [&](auto k) {
        constexpr int LN = decltype(k)::value;
        // more than one wave: set up while the kernel before ends (8 x 5.29M, 355
        // taps, one call after another: 81.0 -> 78.5 us; 11 x 1.0M, 4097 taps
        // 39.0 -> 37.0); a few blocks are paced by the host, whose part of such
        // a launch is about 1 us longer
        auto launch = [&](auto kernel) {
            if (!a.rev && a.nb > SMS * rfft_min_ctas(LN))
                return launch_serial(kernel, (unsigned)a.nb, RfShape<LN>::T, smem_bytes<LN>(), s, a);
            kernel<<<(unsigned)a.nb, RfShape<LN>::T, smem_bytes<LN>(), s>>>(a);
            return cudaGetLastError();
        };
        constexpr bool E = odd_form_only(LN);
        if constexpr (reversed_form(LN))
            if (a.rev) return launch(odd ? k_fir_rfft<LN, true, true> : k_fir_rfft<LN, true, E>);
        if (a.rev) return cudaErrorInvalidValue;
        return launch(odd ? k_fir_rfft<LN, false, true> : k_fir_rfft<LN, false, E>);
    });
}

cudaError_t launch_fir_rfft_batched(int n, const BatchFft* units, const int64_t* prefix, const int32_t* unit_of,
                                    int64_t ctas, BatchBases bases, const float4* tw, cudaStream_t s) {
    if (ctas <= 0) return cudaSuccess;
    return by_size(n, [&](auto k) {
        constexpr int LN = decltype(k)::value;
        k_fir_rfft_batched<LN>
            <<<(unsigned)ctas, RfShape<LN>::T, smem_bytes<LN>(), s>>>(units, prefix, unit_of, bases, tw);
        return cudaGetLastError();
    });
}

cudaError_t launch_fir_rfft_table(int n, const float* taps, int L, const float4* tw, const double2* roots, float4* H,
                                  cudaStream_t s) {
    return by_size(n, [&](auto k) {
        constexpr int LN = decltype(k)::value;
        k_fir_rfft_table<LN>
            <<<RfShape<LN>::PE / 2, RfShape<LN>::T, smem_bytes<LN>(), s>>>(taps, L, tw, roots, H);
        return cudaGetLastError();
    });
}

cudaError_t prepare_fir_rfft(int n) {
    return by_size(n, [&](auto k) {
        constexpr int LN = decltype(k)::value;
        constexpr int smem = (int)smem_bytes<LN>();
        constexpr bool E = odd_form_only(LN);
        cudaError_t e = cudaSuccess;
        auto set = [&](auto kernel) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        };
        set(k_fir_rfft<LN, false, true>);
        set(k_fir_rfft<LN, false, E>);
        if constexpr (reversed_form(LN)) {
            set(k_fir_rfft<LN, true, true>);
            set(k_fir_rfft<LN, true, E>);
        }
        set(k_fir_rfft_batched<LN>);
        set(k_fir_rfft_table<LN>);
        return e;
    });
}

}  // namespace tfx
