// SOS cascade with FP64 carries (poles of radius > 0.999) in phases: no tile
// waits for another.
//
// Per section the recursion's state at every tile start is needed before the
// tile's outputs.  The look-back kernel (k_sos_warp) hands it from tile to
// tile inside one launch, a serial chain of about one memory round trip per
// 32 tiles (88 of them on 2.88M samples: 130 of 178 us).  Here every section
// takes a launch that only forms the tiles' end states from zero
// (k_sos_phase<false>), a launch that scans them along each channel in FP64
// (k_carry_scan), and the next launch starts from the true states; the last
// one writes the outputs.  Each launch reads the signal again (S + 1 reads,
// one write) and redoes the sections before its own, which costs less than
// the chain while S is small.  One section on 8 x 2.88M samples: 175 -> 53 us
// (12 bytes a sample against HBM would take 41), two 263 -> 103.  A launch
// after the first is let in while the scan before it runs: its samples are
// loaded and its first section passed from zero by then (58 -> 53 us, 68 ->
// 61.3 with the host's launches).
// Bound: memory latency with four CTAs per SM (64 registers; three 60 us,
// without the next tile's prefetch 59), then FP64, whose pipe does 2 FMAs per
// clock and SM (66 -> 38 us for the last launch when the scan over a tile's
// warps moved from it, one per warp, to the first launch, one per tile).
//
// Arithmetic: per lane and 32-sample chunk as k_sos_warp (FP32 recursions
// from zero, FP32 warp scan of the chunk end states, chunk start states
// summed in FP64 and rounded once), the carries between warps and tiles by
// FP64 powers of the chunk transfer.  A CTA's tile is 8 warps x 1024 samples;
// samples move through shared memory so that lanes read consecutive words.
#include "tfx_common.cuh"

namespace tfx {
namespace {

constexpr int PT = T_CHUNK, PW = 8, PTILE = PW * 32 * PT;  // 8192 samples per CTA
constexpr int PCTAS = 4;           // CTAs per SM
constexpr int PROW = PT + 4;                               // padded shared row of a lane (floats)

struct PhaseArgs {
    UnitArgs a;
    double2* carry;   // [S][C][ntile]: tile end states from zero, then (scanned) tile start states
    double2* before;  // [S][C][ntile][PW]: the state that a tile's warps before each one leave, from zero
    int64_t ntile;
    int stop;        // first launches: the section whose end states are wanted
};

// 1024 samples of a row from n0 into / out of the warp's shared rows.
__device__ __forceinline__ void warp_in(float* sm, const float* p, int64_t n0, int64_t N, int lane) {
    if (n0 + 32 * PT <= N && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
        const float4* q = reinterpret_cast<const float4*>(p) + lane;
        float4 v[PT / 4];
#pragma unroll
        for (int i = 0; i < PT / 4; ++i) v[i] = q[32 * i];
#pragma unroll
        for (int i = 0; i < PT / 4; ++i) {
            const int n = 4 * (lane + 32 * i);
            *reinterpret_cast<float4*>(sm + (n / PT) * PROW + n % PT) = v[i];
        }
    } else {
#pragma unroll 8
        for (int i = 0; i < PT; ++i) {
            const int n = lane + 32 * i;
            sm[(n / PT) * PROW + n % PT] = n0 + n < N ? p[n] : 0.f;
        }
    }
}
__device__ __forceinline__ void warp_out(const float* sm, float* p, int64_t n0, int64_t N, int lane) {
    if (n0 + 32 * PT <= N && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
        float4* q = reinterpret_cast<float4*>(p) + lane;
#pragma unroll
        for (int i = 0; i < PT / 4; ++i) {
            const int n = 4 * (lane + 32 * i);
            q[32 * i] = *reinterpret_cast<const float4*>(sm + (n / PT) * PROW + n % PT);
        }
    } else {
#pragma unroll 8
        for (int i = 0; i < PT; ++i) {
            const int n = lane + 32 * i;
            if (n0 + n < N) p[n] = sm[(n / PT) * PROW + n % PT];
        }
    }
}

// m v + d
__device__ __forceinline__ double2 mva2d(double4 m, double2 v, double2 d) {
    return make_double2(fma(m.x, v.x, fma(m.y, v.y, d.x)), fma(m.z, v.x, fma(m.w, v.y, d.y)));
}

template <bool FINAL>
__global__ void __launch_bounds__(32 * PW, PCTAS) k_sos_phase(PhaseArgs g) {
    __shared__ __align__(16) float rows[PW][32 * PROW];
    __shared__ float2 ends[PW];
    const UnitArgs& a = g.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned nt = (unsigned)g.ntile;
    const unsigned b = FINAL ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    // the last launch walks the tiles backwards: the ones read last are still in L2
    const unsigned c = b / nt, k = b - c * nt;
    const int64_t n0 = (int64_t)k * PTILE + warp * 32 * PT;
    float* sm = rows[warp];
    warp_in(sm, a.x + c * a.ldx + n0, n0, a.N, lane);
    // ask for the tile that runs on this SM next (the CTAs start in order)
    constexpr unsigned AHEAD = GB300_SMS * PCTAS;
    if (threadIdx.x == 0 && blockIdx.x + AHEAD < gridDim.x) {
        const unsigned bn = FINAL ? b - AHEAD : b + AHEAD, cn = bn / nt, kn = bn - cn * nt;
        if ((int64_t)(kn + 1) * PTILE <= a.N) {
            const uintptr_t q =
                (reinterpret_cast<uintptr_t>(a.x + cn * a.ldx + (int64_t)kn * PTILE) + 15) & ~(uintptr_t)15;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q), "r"(4 * PTILE - 16) : "memory");
        }
    }
    __syncwarp();
    float u[PT];
#pragma unroll
    for (int i = 0; i < PT / 4; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(sm + lane * PROW + 4 * i);
        u[4 * i] = v.x, u[4 * i + 1] = v.y, u[4 * i + 2] = v.z, u[4 * i + 3] = v.w;
    }
    const int S = a.k.S, last = FINAL ? S : g.stop;
    bool waited = false;  // the carries of the launches before this one are there
    float2 st = make_float2(0.f, 0.f);
    float pa1 = 0.f, pa2 = 0.f;
    for (int s = 0; s <= last; ++s) {
        const bool fix = s > 0, run = s < S;
        float b0 = 0.f, c1 = 0.f, c2 = 0.f, a1 = 0.f, a2 = 0.f;
        if (run) {
            const float* cf = a.k.coef + 8 * s;
            b0 = cf[0], c1 = cf[1], c2 = cf[2], a1 = cf[3], a2 = cf[4];
        }
        // section s - 1's response to its true start state, then section s from zero
        float w1 = 0.f, w2 = 0.f, h1 = 0.f, h2 = 0.f;
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            float v = u[t];
            if (fix) {
                const float h = t == 0 ? st.x : t == 1 ? fmaf(-pa1, h1, st.y) : fmaf(-pa1, h1, -pa2 * h2);
                h2 = h1;
                h1 = h;
                v += h;
            }
            if (run) {
                u[t] = fmaf(b0, v, w1);
                const float n1 = fmaf(c1, v, fmaf(-a1, w1, w2));
                w2 = fmaf(c2, v, -a2 * w1);
                w1 = n1;
            } else {
                u[t] = v;
            }
        }
        if (!run) break;
        const float4* P = a.k.pw + (size_t)s * PW_LEN;
        const double4* P64 = a.k.pw64 + (size_t)s * PW_LEN;
        float2 v = make_float2(w1, w2);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float4 Pd = P[d];
            const float ox = __shfl_up_sync(0xffffffffu, v.x, d), oy = __shfl_up_sync(0xffffffffu, v.y, d);
            if (lane >= d) {
                const float2 t2 = mv2(Pd, make_float2(ox, oy));
                v.x += t2.x;
                v.y += t2.y;
            }
        }
        const float px = __shfl_up_sync(0xffffffffu, v.x, 1), py = __shfl_up_sync(0xffffffffu, v.y, 1);
        const int64_t tile = ((int64_t)s * a.C + c) * g.ntile + k;
        if (!waited) after_previous();
        waited = true;
        if (!FINAL && s == last) {
            // the warps' end states scanned over the CTA (warp 0, FP64): what
            // the warps before each one leave behind, and the tile's end state
            if (lane == 31) ends[warp] = v;
            let_next();
            __syncthreads();
            if (warp > 0) return;
            double2 d = make_double2(0.0, 0.0);
            if (lane < PW) d = make_double2((double)ends[lane].x, (double)ends[lane].y);
#pragma unroll
            for (int o = 1; o < PW; o <<= 1) {
                const double ox = __shfl_up_sync(0xffffffffu, d.x, o), oy = __shfl_up_sync(0xffffffffu, d.y, o);
                if (lane >= o) d = mva2d(P64[32 * o], make_double2(ox, oy), d);
            }
            const double ox = __shfl_up_sync(0xffffffffu, d.x, 1), oy = __shfl_up_sync(0xffffffffu, d.y, 1);
            if (lane < PW) g.before[tile * PW + lane] = lane > 0 ? make_double2(ox, oy) : make_double2(0.0, 0.0);
            if (lane == PW - 1) g.carry[tile] = d;
            return;
        }
        // true start states: the tile's, carried over the warps before this
        // one, then over the lanes before this one
        const double2 d = mva2d(P64[32 * warp], g.carry[tile], g.before[tile * PW + warp]);
        const double2 t2 =
            mva2d(P64[lane], d, lane > 0 ? make_double2((double)px, (double)py) : make_double2(0.0, 0.0));
        st = make_float2((float)t2.x, (float)t2.y);
        pa1 = a1;
        pa2 = a2;
    }
    if constexpr (FINAL) {
#pragma unroll
        for (int i = 0; i < PT / 4; ++i)
            *reinterpret_cast<float4*>(sm + lane * PROW + 4 * i) =
                make_float4(u[4 * i], u[4 * i + 1], u[4 * i + 2], u[4 * i + 3]);
        __syncwarp();
        warp_out(sm, a.y + c * a.ldy + n0, n0, a.N, lane);
    }
}

// Tile start states from the tiles' end states from zero, in place: e_k ->
// sum_(m < k) T^(k - 1 - m) e_m, T the transfer of a whole tile.  One CTA per
// channel: each thread a run of tiles, the runs joined by a scan whose
// matrices T^(run 2^d) one warp squares, before the wait: the launch before
// lets this one in as its CTAs end, and the tables are older than the first,
// ordinary launch of the sequence.  FP64 bounds it (a warp's matrix product
// takes its SM 128 cycles): 17.4 -> 15.5 us on 1 x 3.1M samples, 55.5 -> 53.4
// on 8 x 2.88M, 74.1 -> 65.7 on 64 x 100,000 with three sections against
// powers formed after the wait, two squarings more and 128 threads always.  Threads by the tiles
// (scan_threads): 64 x 100,000 22.1 us with 128, 21.0 with 32; 1 x 8M 27.9 with
// 128, 30.2 with 64, 34.1 with 32, 28.2 with 256.  Let in at the start of the
// launch before instead: 14.8 on 1 x 3.1M, but 80 on 64 x 100,000.  A warp with
// its runs in registers: 19.1 and 83.
constexpr int CT = 128;
__global__ void __launch_bounds__(CT) k_carry_scan(double2* __restrict__ carry, int64_t ntile,
                                                   const double4* __restrict__ P64) {
    __shared__ double4 pw[6];        // T^(run 2^d)
    __shared__ double2 wend[CT / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    let_next();
    double2* e = carry + (int64_t)blockIdx.x * ntile;
    const double4 T = P64[PTILE / PT];
    const int nthr = blockDim.x;
    const int64_t run = (ntile + nthr - 1) / nthr, k0 = t * run, k1 = k0 + run < ntile ? k0 + run : ntile;
    if (warp == 0) {
        double4 Tr = make_double4(1.0, 0.0, 0.0, 1.0), q = T;
        for (int64_t b = run; b > 0; b >>= 1) {
            if (b & 1) Tr = mm2d(Tr, q);
            if (b > 1) q = mm2d(q, q);
        }
        for (int d = 0; d < 6; ++d) {
            if (lane == 0) pw[d] = Tr;
            if (d < 5) Tr = mm2d(Tr, Tr);
        }
    }
    after_previous();
    double2 v = make_double2(0.0, 0.0);
    for (int64_t k = k0; k < k1; ++k) v = mva2d(T, v, e[k]);
    __syncthreads();
    auto scan = [&](int lanes, int d0) {
        for (int d = 0; (1 << d) < lanes; ++d) {
            const int o = 1 << d;
            const double ox = __shfl_up_sync(0xffffffffu, v.x, o), oy = __shfl_up_sync(0xffffffffu, v.y, o);
            if (lane >= o) v = mva2d(pw[d0 + d], make_double2(ox, oy), v);
        }
    };
    scan(32, 0);
    if (lane == 31) wend[warp] = v;
    // exclusive within the warp
    double2 s = make_double2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
    if (lane == 0) s = make_double2(0.0, 0.0);
    __syncthreads();
    // the state at the warp's first run, carried to this lane's
    if (warp > 0) {
        double2 w = make_double2(0.0, 0.0);
        for (int m = 0; m < warp; ++m) w = mva2d(pw[5], w, wend[m]);
        for (int d = 0; d < 5; ++d) {  // T^(run lane) w
            const double2 x = mva2d(pw[d], w, make_double2(0.0, 0.0));
            if (lane >> d & 1) w = x;
        }
        s.x += w.x;
        s.y += w.y;
    }
    for (int64_t k = k0; k < k1; ++k) {
        const double2 x = e[k];
        e[k] = s;
        s = mva2d(T, s, x);
    }
}

}  // namespace

// Threads of k_carry_scan: one per tile, from a warp to CT.
static unsigned scan_threads(int64_t ntile) { return ntile <= 32 ? 32 : ntile <= 64 ? 64 : CT; }

int sos_phase_launches(int S) { return 2 * S + 1; }

size_t sos_phase_scratch(int S, int64_t C, int64_t N) {
    return (size_t)S * (size_t)C * (size_t)((N + PTILE - 1) / PTILE) * (PW + 1) * sizeof(double2);
}

cudaError_t launch_sos_phases(const UnitArgs& a, void* scratch, cudaStream_t s) {
    PhaseArgs g{};
    g.a = a;
    g.carry = static_cast<double2*>(scratch);
    g.ntile = (a.N + PTILE - 1) / PTILE;
    g.before = g.carry + (int64_t)a.k.S * a.C * g.ntile;
    if (a.C <= 0 || g.ntile <= 0) return cudaSuccess;
    if (a.C * g.ntile > INT32_MAX || !a.k.pw64) return cudaErrorInvalidValue;
    const unsigned ctas = (unsigned)(a.C * g.ntile);
    for (int k = 0; k < a.k.S; ++k) {
        g.stop = k;
        cudaError_t e = cudaSuccess;
        if (k == 0) {
            k_sos_phase<false><<<ctas, 32 * PW, 0, s>>>(g);
            e = cudaGetLastError();
        } else {
            e = launch_serial(k_sos_phase<false>, ctas, 32 * PW, 0, s, g);
        }
        if (e == cudaSuccess)
            e = launch_serial(k_carry_scan, (unsigned)a.C, scan_threads(g.ntile), 0, s,
                              g.carry + (int64_t)k * a.C * g.ntile, g.ntile,
                              a.k.pw64 + (size_t)k * PW_LEN);
        if (e != cudaSuccess) return e;
    }
    return launch_serial(k_sos_phase<true>, ctas, 32 * PW, 0, s, g);
}

}  // namespace tfx
