// Direct FIR of 1 to 64 taps, y[n] = sum_k h[k] x[n - k] (x zero before the
// signal): independent tiles, a register-blocked sliding window.
//
// Bound: the phases of a tile (load, sums, store) and the FP32 pipe, 43 %
// busy (1 FMA per tap and sample; 33 taps cost 7 us of it on 6 x 1.44M
// samples, whose bytes take 10 us of HBM).  A tile is 2048 outputs of one
// channel, 16 consecutive ones per thread: one 16-byte window word and one
// 16-byte tap word from shared memory per 64 FMAs.  Tiles start on 16-byte
// boundaries of the row (whatever its address), so samples always move in as
// 16-byte words; outputs pass through the same shared buffer to leave in
// order.  Measured, the scan kernel's tiles (k_unit, which wait for their
// predecessor's published input tail and take the taps 16 at a time) -> this:
// 6 x 1,440,007 samples, 33 taps 81 -> 18 us, 63 taps 25 us; 12 x 7.94M, 33
// taps 170 us (0.67 of HBM).  256 threads per tile 19.2 us; packed two-lane
// products 20.4 us (the odd taps' pairs cost register moves).
#include "tfx_common.cuh"

namespace tfx {
namespace {

constexpr int DT = 128, DR = 16, DTILE = DT * DR, DHALO = 64;
constexpr int DWORDS = (DTILE + DHALO) / 4;

// Shared position of sample i: four floats of padding per 16, so that the
// 8 lanes of a 16-byte phase, 16 samples apart, touch 8 different banks.
__device__ __forceinline__ int dpad(int i) { return i + ((i >> 4) << 2); }

// Four samples n..n+3 of a row, zero outside [0, N); p is 16-byte aligned.
__device__ __forceinline__ float4 load4(const float* p, int64_t n, int64_t N) {
    if (n >= 0 && n + 4 <= N) return __ldg(reinterpret_cast<const float4*>(p));
    auto at = [&](int o) { return n + o >= 0 && n + o < N ? __ldg(p + o) : 0.f; };
    return make_float4(at(0), at(1), at(2), at(3));
}

__global__ void __launch_bounds__(DT, 10) k_fir_direct(FirDirectArgs a) {
    __shared__ __align__(16) float sm[(DTILE + DHALO) / 4 * 5];
    __shared__ __align__(16) float taps[DHALO];
    const int t = threadIdx.x;
    const unsigned c = blockIdx.x / (unsigned)a.nt, k = blockIdx.x - c * (unsigned)a.nt;
    const float* x = a.x + c * a.ldx;
    float* y = a.y + c * a.ldy;
    // first output of the tile: a multiple of DTILE less the row's offset
    // from a 16-byte boundary
    const int64_t n0 = (int64_t)k * DTILE - (int64_t)((reinterpret_cast<uintptr_t>(x) >> 2) & 3);
    if (n0 >= a.N) return;
    if (t < DHALO) taps[t] = t < a.L ? __ldg(a.taps + t) : 0.f;
    const float* xw = x + n0 - DHALO + 4 * t;
    float* st = sm + dpad(4 * t);  // (4 DT samples on: 5 DT floats on)
    const bool inner = n0 >= DHALO && n0 + DTILE <= a.N;
    if (inner) {
        float4 v[DWORDS / DT + 1];
#pragma unroll
        for (int j = 0; j <= DWORDS / DT; ++j)
            if (t + DT * j < DWORDS) v[j] = __ldg(reinterpret_cast<const float4*>(xw) + DT * j);
#pragma unroll
        for (int j = 0; j <= DWORDS / DT; ++j)
            if (t + DT * j < DWORDS) *reinterpret_cast<float4*>(st + 5 * DT * j) = v[j];
    } else {
#pragma unroll 1
        for (int j = 0; j <= DWORDS / DT; ++j)
            if (t + DT * j < DWORDS)
                *reinterpret_cast<float4*>(st + 5 * DT * j) =
                    load4(xw + 4 * DT * j, n0 - DHALO + 4 * (t + DT * j), a.N);
    }
    __syncthreads();

    // w[i]: x at the thread's first output - 64 + i.  Output i takes tap k
    // from w[64 + i - k]; every index is constant, and each four taps need
    // four older samples (the newest ones are dead by then).
    const float* wp = sm + dpad(DR * t);
    float w[DHALO + DR], acc[DR];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(wp + 80 + 4 * q);
        w[64 + 4 * q] = v.x, w[65 + 4 * q] = v.y, w[66 + 4 * q] = v.z, w[67 + 4 * q] = v.w;
    }
#pragma unroll
    for (int i = 0; i < DR; ++i) acc[i] = 0.f;
#pragma unroll
    for (int k = 0; k < DHALO; k += 4) {
        if (k < a.L) {
            const int o = DHALO - 4 - k;
            const float4 v = *reinterpret_cast<const float4*>(wp + o + 4 * (o / 16));
            w[o] = v.x, w[o + 1] = v.y, w[o + 2] = v.z, w[o + 3] = v.w;
            const float4 h = *reinterpret_cast<const float4*>(taps + k);
#pragma unroll
            for (int i = 0; i < DR; ++i) {
                acc[i] = fmaf(h.x, w[64 + i - k], acc[i]);
                acc[i] = fmaf(h.y, w[63 + i - k], acc[i]);
                acc[i] = fmaf(h.z, w[62 + i - k], acc[i]);
                acc[i] = fmaf(h.w, w[61 + i - k], acc[i]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(sm + dpad(DR * t) + 4 * q) =
            make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
    __syncthreads();
    const float* ld = sm + dpad(4 * t);
    float* yw = y + n0 + 4 * t;
    if (inner && (reinterpret_cast<uintptr_t>(yw) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < DTILE / 4 / DT; ++j)
            reinterpret_cast<float4*>(yw)[DT * j] = *reinterpret_cast<const float4*>(ld + 5 * DT * j);
    } else {
        // one sample per lane and store: consecutive lanes, consecutive samples
#pragma unroll 4
        for (int i = t; i < DTILE; i += DT) {
            const int64_t n = n0 + i;
            if (n >= 0 && n < a.N) y[n] = sm[dpad(i & ~3) + (i & 3)];
        }
    }
}

}  // namespace

cudaError_t launch_fir_direct(FirDirectArgs a, cudaStream_t s) {
    if (a.C <= 0 || a.N <= 0) return cudaSuccess;
    if (a.L < 1 || a.L > DHALO) return cudaErrorInvalidValue;
    a.nt = (a.N + 3 + DTILE - 1) / DTILE;  // (a row may begin up to 3 samples into its first tile)
    if (a.C * a.nt > INT32_MAX) return cudaErrorInvalidValue;
    k_fir_direct<<<(unsigned)(a.C * a.nt), DT, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace tfx
