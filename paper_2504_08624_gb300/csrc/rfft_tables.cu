// Host tables of the real-block transform (rfft_core.cuh): the nodes'
// twiddles and a filter's product constants, in FP64, rounded once.  What
// depends on the size alone is formed once per process (0.8 MB for all six
// sizes): its sines and cosines were 159 of the 185 us of tables that a plan of
// 4096-sample blocks takes (host time), and a batch creates a plan per clip (500
// clips of an FIR each: 126 -> 48 ms).
#include <cmath>
#include <complex>
#include <mutex>
#include <vector>

#include "plan_internal.cuh"

namespace tfx {
namespace {

int brev(int v, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((v >> b) & 1) << (bits - 1 - b);
    return r;
}

// e^(2 pi i num / den), the fraction reduced to one turn in integers first
std::complex<double> turn(int64_t num, int64_t den) {
    const double a = 2.0 * M_PI * (double)(num % den) / (double)den;
    return {std::cos(a), std::sin(a)};
}

// h of node b at depth d is (1/4 + bitrev_d(b)) / 2^d = node_num(b, d) / 2^(d + 2)
int64_t node_num(int b, int d) { return 1 + 4 * (int64_t)brev(b, d); }

// Of a size: the device's twiddles, and the square root r of every node's
// constant (node b of depth d at 2^d - 1 + b) and the last nodes' constants w.
struct Size {
    std::once_flag once;
    std::vector<float4> tables;
    std::vector<std::complex<double>> roots, last;
};
std::vector<float4> form_tables(int n);

const Size& size_of(int n) {
    static Size sizes[RF_MAX_N - RF_MIN_N + 1];
    Size& s = sizes[n - RF_MIN_N];
    std::call_once(s.once, [&] {
        s.tables = form_tables(n);
        for (int d = 0; d < n - 1; ++d)
            for (int b = 0; b < (1 << d); ++b) s.roots.push_back(turn(node_num(b, d), (int64_t)1 << (d + 3)));
        for (int b = 0; b < (1 << (n - 1)); ++b) s.last.push_back(turn(node_num(b, n - 1), (int64_t)1 << (n + 1)));
    });
    return s;
}

std::vector<float4> form_tables(int n) {
    std::vector<float4> out((size_t)rfft_table_words(n));
    const int PE = 1 << rfft_log_pe(n);
    int d = rfft_radix_log(n, 0);
    for (int p = 1; p < rfft_passes(n); ++p) {
        const int rl = rfft_radix_log(n, p), R = 1 << rl, K = 1 << d, G = PE / R, T = K / G;
        float2* fwd = reinterpret_cast<float2*>(out.data() + rfft_fwd_off(n, p));
        float2* inv = fwd + (size_t)K * R / 2;
        for (int b = 0; b < K; ++b) {
            // row position: several subtrees per thread (last pass) are
            // stored group by group, so that a warp reads consecutive words
            const size_t at = G == 1 ? (size_t)b : (size_t)(b % G) * T + b / G;
            auto put = [&](float2* tab, int k, std::complex<double> w) {
                tab[2 * ((size_t)(k / 2) * K + at) + k % 2] = make_float2((float)w.real(), (float)w.imag());
            };
            // node e of level l of the subtree: depth d + l, index b 2^l + e;
            // its twiddle is the square root, h / 2
            for (int l = 0; l < rl; ++l)
                for (int e = 0; e < (1 << l); e += 2)
                    put(fwd, l == 0 ? 0 : (1 << (l - 1)) + e / 2,
                        turn(node_num((b << l) + e, d + l), (int64_t)1 << (d + l + 3)));
            for (int j = 0; j < R; ++j)
                put(inv, j, std::conj(turn(node_num(b, d) * j, (int64_t)1 << (d + 2 + rl))));
        }
        d += rl;
    }
    return out;
}

}  // namespace

const std::vector<float4>& rfft_tables(int n) { return size_of(n).tables; }

std::vector<double2> rfft_roots(int n, int turns, int step) {
    const int D = n - 1;
    std::vector<double2> out(((size_t)1 << D) / step);
    for (size_t k = 0; k < out.size(); ++k) {
        const std::complex<double> w =
            turns == 1 ? size_of(n).last[k * step] : turn(node_num((int)k * step, D), (int64_t)turns << (D + 2));
        out[k] = make_double2(w.real(), w.imag());
    }
    return out;
}

namespace {

// The taps modulo the last nodes z^2 - w: two coefficients per element.
std::vector<std::complex<double>> filter_pairs(int n, const double* taps, int L) {
    const int N = 1 << n, D = n - 1;
    std::vector<std::complex<double>> v(N);
    for (int k = 0; k < N; ++k) v[k] = {k < L ? taps[k] : 0.0, k + N < L ? taps[k + N] : 0.0};
    const std::vector<std::complex<double>>& roots = size_of(n).roots;
    for (int d = 0; d < D; ++d) {
        const int S = N >> d;
        for (int b = 0; b < (1 << d); ++b) {
            const std::complex<double> r = roots[(size_t)((1 << d) - 1 + b)];
            std::complex<double>* u = v.data() + (size_t)b * S;
            for (int k = 0; k < S / 2; ++k) {
                const std::complex<double> a = u[k], c = r * u[k + S / 2];
                u[k] = a + c;
                u[k + S / 2] = a - c;
            }
        }
    }
    return v;
}

}  // namespace

void rfft_filter_pairs(int n, const double* taps, int L, float4* out) {
    const auto v = filter_pairs(n, taps, L);
    for (size_t p = 0; p < v.size() / 2; ++p)
        out[p] = make_float4((float)v[2 * p].real(), (float)v[2 * p].imag(), (float)v[2 * p + 1].real(),
                             (float)v[2 * p + 1].imag());
}

void rfft_filter_table(int n, const double* taps, int L, float4* out) {
    const int N = 1 << n, PE = 1 << rfft_log_pe(n), T = N / 2 / PE;
    const auto v = filter_pairs(n, taps, L);
    const std::vector<std::complex<double>>& last = size_of(n).last;
    const double sc = 2.0 / N;
    for (int p = 0; p < N / 2; ++p) {
        const std::complex<double> ha = v[2 * p] * sc, hc = v[2 * p + 1] * sc;
        const std::complex<double> q = last[(size_t)p] * hc;
        const int t = p / PE, e = p % PE;
        float4* w = out + (size_t)(3 * (e / 2)) * T + t;
        reinterpret_cast<float2*>(w)[e % 2] = make_float2((float)ha.real(), (float)ha.imag());
        w[(size_t)(1 + e % 2) * T] =
            make_float4((float)q.real(), (float)hc.real(), (float)q.imag(), (float)hc.imag());
    }
}

}  // namespace tfx
