// NormalFloat code book (Sec. 2.2) built on the host in fp64 and uploaded to constant memory,
// plus host-only helpers of the C ABI (storage formula, sizes, status strings).
#pragma once

#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <utility>

#include "common.cuh"

namespace lq {

namespace detail {

// Gaussian quantile by Newton's method on Phi(x) - p, started from a closed-form guess.
inline double gauss_quantile(double p) {
    if (p == 0.5) return 0.0;
    const bool upper = p > 0.5;
    const double pp = upper ? 1.0 - p : p;                 // lower tail probability
    const double t = std::sqrt(-2.0 * std::log(pp));
    double x = -(t - (2.30753 + 0.27061 * t) / (1.0 + t * (0.99229 + 0.04481 * t)));  // rough start
    const double inv_sqrt_2pi = 0.3989422804014326779;
    for (int it = 0; it < 60; ++it) {
        const double cdf = 0.5 * std::erfc(-x / std::sqrt(2.0));
        const double pdf = inv_sqrt_2pi * std::exp(-0.5 * x * x);
        const double step = (cdf - pp) / pdf;
        x -= step;
        if (std::fabs(step) < 1e-17 * std::fmax(1.0, std::fabs(x))) break;
    }
    return upper ? -x : x;
}

struct HostTables {
    float codebook[4][256];
    float threshold[4][256];
    BinEntry bins[kMaxBins + 1];              // 8-bit codes
    int nbins;
    float2 curve[3][kCurveCoefs + 1];
    // Bin count for `n - 1` thresholds: the candidate with the largest distance between any threshold and any
    // bin edge among those with at most one threshold per bin.
    double best_bins(int t, int n, int* nb_out) const {
        const int lo = (n <= 16) ? 48 : 1000, hi = (n <= 16) ? 96 : kMaxBins;
        int best_nb = 0;
        double best_clear = -1.0;
        for (int nb = lo; nb <= hi; ++nb) {
            double clear = 1e9;
            bool ok = true;
            int prev_bin = -1;
            for (int i = 0; i + 1 < n && ok; ++i) {
                const double pos = (static_cast<double>(threshold[t][i]) + 1.0) * 0.5 * nb;
                const int b = static_cast<int>(std::floor(pos));
                if (b == prev_bin) ok = false;
                prev_bin = b;
                const double d = std::fmin(pos - std::floor(pos), std::ceil(pos) - pos) * 2.0 / nb;
                clear = std::fmin(clear, d);
            }
            if (ok && clear > best_clear) { best_clear = clear; best_nb = nb; }
        }
        *nb_out = best_nb;
        return best_clear;
    }
    void build_bins() {
        constexpr int t = 3, n = 256;
        best_bins(t, n, &nbins);
        for (int k = 0; k <= kMaxBins; ++k) { bins[k].thr = INFINITY; bins[k].base = n - 1; }
        int below = 0;
        for (int k = 0; k < nbins; ++k) {
            bins[k].base = below;
            bins[k].thr = INFINITY;
            while (below + 1 < n) {
                const double pos = (static_cast<double>(threshold[t][below]) + 1.0) * 0.5 * nbins;
                if (static_cast<int>(std::floor(pos)) != k) break;
                bins[k].thr = threshold[t][below];
                ++below;
            }
        }
    }
    // Coefficients of P(x) = E(|x|) + x O(|x|), P(T_k) = k at the thresholds (3-bit codes: and P(1) = 7.55), by Gaussian
    // elimination with row pivoting; 2^b0 and half of the "close to a threshold" range are added to the constant term.
    void build_curve(int b0) {
        const int t = bits_index(b0), n = 1 << b0;
        const int ne = curve_even(b0), no = curve_odd(b0), m = ne + no;
        double A[kCurveCoefs][kCurveCoefs + 1];
        for (int i = 0; i < m; ++i) {
            const double x = i + 1 < n ? 0.5 * (static_cast<double>(codebook[t][i]) + static_cast<double>(codebook[t][i + 1])) : 1.0;
            const double y = std::fabs(x);
            double p = 1.0;
            for (int j = 0; j < ne; ++j, p *= y) A[i][j] = p;
            p = x;
            for (int j = 0; j < no; ++j, p *= y) A[i][ne + j] = p;
            A[i][m] = i + 1 < n ? i + 1.0 : 7.55;
        }
        for (int c = 0; c < m; ++c) {
            int pv = c;
            for (int r = c + 1; r < m; ++r) if (std::fabs(A[r][c]) > std::fabs(A[pv][c])) pv = r;
            for (int k = 0; k <= m; ++k) std::swap(A[c][k], A[pv][k]);
            for (int r = 0; r < m; ++r) {
                if (r == c) continue;
                const double f = A[r][c] / A[c][c];
                for (int k = c; k <= m; ++k) A[r][k] -= f * A[c][k];
            }
        }
        for (int j = 0; j < m; ++j) {
            double v = A[j][m] / A[j][j];
            if (j == 0) v += n + std::ldexp(0.5 * curve_limit(b0), b0 - 23);
            curve[t][j] = make_float2(static_cast<float>(v), static_cast<float>(v));
        }
        for (int j = m; j <= kCurveCoefs; ++j) curve[t][j] = make_float2(0.0f, 0.0f);
    }
    // What the encoder takes from the curve, evaluated as the kernel does: every float within 32768 of its neighbours around each threshold,
    // and every 61st float of [2^-24, 1 + 4 ulp] with both signs.  Smallest distance between a threshold and a float whose fraction does
    // not call it close to one; -2 if such a float gets a wrong code.
    double curve_clearance(int b0) const {
        const int t = bits_index(b0), n = 1 << b0, ne = curve_even(b0), no = curve_odd(b0);
        double least = 1.0;
        bool right = true;
        auto check = [&](uint32_t bits_of_x) {
            float x;
            std::memcpy(&x, &bits_of_x, 4);
            const float y = std::fabs(x);
            float e = curve[t][ne - 1].x, o = curve[t][ne + no - 1].x;
            for (int i = ne - 2; i >= 0; --i) e = std::fmaf(e, y, curve[t][i].x);
            for (int i = no - 2; i >= 0; --i) o = std::fmaf(o, y, curve[t][ne + i].x);
            const float p = std::fmaf(x, o, e);
            uint32_t bits;
            std::memcpy(&bits, &p, 4);
            if ((bits & ((1u << (23 - b0)) - 1u)) < curve_limit(b0)) return;
            int below = 0;
            while (below + 1 < n && x > threshold[t][below]) ++below;
            right = right && static_cast<int>((bits >> (23 - b0)) & (n - 1)) == below;
            for (int k = below > 0 ? below - 1 : 0; k <= below && k + 1 < n; ++k)
                least = std::fmin(least, std::fabs(static_cast<double>(x) - 0.5 * (static_cast<double>(codebook[t][k]) + static_cast<double>(codebook[t][k + 1]))));
        };
        constexpr uint32_t kSign = 0x80000000u, kOne = 0x3F800000u + 4u;      // 1 + 4 ulp
        check(0u);
        check(kSign);
        for (uint32_t x = 0x33800000u; x <= kOne; x += 61) { check(x); check(x | kSign); }
        for (int k = 0; k + 1 < n; ++k) {
            uint32_t at;
            std::memcpy(&at, &threshold[t][k], 4);
            for (uint32_t x = at - 32768u; x != at + 32768u; ++x)
                if ((x & ~kSign) <= kOne) check(x);
        }
        return right ? least : -2.0;
    }
    HostTables() {
        const int bits[4] = {2, 3, 4, 8};
        const double delta = 0.5 * (1.0 / 30.0 + 1.0 / 32.0);
        for (int t = 0; t < 4; ++t) {
            const int b = bits[t], n = 1 << b, half = n >> 1;
            double q[256];
            // upper side first: probabilities 1/2 + (1/2 - delta) i / 2^(b-1), i = 1 .. 2^(b-1)
            for (int i = 1; i <= half; ++i)
                q[half - 1 + i] = gauss_quantile(0.5 + (0.5 - delta) * static_cast<double>(i) / half);
            q[half - 1] = 0.0;                              // probability exactly 1/2
            // lower side: delta + (1/2 - delta) i / (2^(b-1) - 1), i = 0 .. 2^(b-1) - 2
            for (int i = 0; i + 1 < half; ++i)
                q[i] = gauss_quantile(delta + (0.5 - delta) * static_cast<double>(i) / (half - 1));
            const double top = q[n - 1];
            for (int i = 0; i < 256; ++i) { codebook[t][i] = 0.0f; threshold[t][i] = INFINITY; }
            for (int i = 0; i < n; ++i) codebook[t][i] = static_cast<float>(q[i] / top);
            for (int i = 0; i + 1 < n; ++i) {
                const double mid = 0.5 * (static_cast<double>(codebook[t][i]) + static_cast<double>(codebook[t][i + 1]));
                float th = static_cast<float>(mid);
                if (static_cast<double>(th) > mid) th = std::nextafterf(th, -INFINITY);
                threshold[t][i] = th;                       // largest fp32 <= midpoint
            }
        }
        build_bins();
        for (int b0 = 2; b0 <= 4; ++b0) build_curve(b0);
    }
};

inline const HostTables& host_tables() {
    static const HostTables t;
    return t;
}

}  // namespace detail

const float* host_codebook(int b0) { return detail::host_tables().codebook[bits_index(b0)]; }

int ensure_tables() {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return LQLORA_ERR_CUDA; }
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return LQLORA_OK;
    const detail::HostTables& t = detail::host_tables();
    if (cudaMemcpyToSymbol(c_codebook, t.codebook, sizeof(t.codebook)) != cudaSuccess ||
        cudaMemcpyToSymbol(c_threshold, t.threshold, sizeof(t.threshold)) != cudaSuccess ||
        cudaMemcpyToSymbol(g_codebook8, t.codebook[3], sizeof(t.codebook[3])) != cudaSuccess ||
        cudaMemcpyToSymbol(c_curve, t.curve, sizeof(t.curve)) != cudaSuccess ||
        cudaMemcpyToSymbol(g_bins, t.bins, sizeof(t.bins)) != cudaSuccess ||
        cudaMemcpyToSymbol(c_nbins, &t.nbins, sizeof(t.nbins)) != cudaSuccess) {
        cudaGetLastError();
        return LQLORA_ERR_CUDA;
    }
    done[dev] = true;
    return LQLORA_OK;
}

static std::atomic<int64_t> g_launches{0};
void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

}  // namespace lq

extern "C" {

double lqlora_storage_bits_per_param(const lqlora_config* cfg) {
    if (lq::check_config(cfg) != LQLORA_OK) return -1.0;
    const int b2 = cfg->b2 < 0 ? -cfg->b2 : cfg->b2;
    return static_cast<double>(cfg->b0) + static_cast<double>(cfg->b1) / cfg->B0 +
           static_cast<double>(b2) / (static_cast<double>(cfg->B0) * cfg->B1);
}

int lqlora_packed_sizes(int64_t N, int64_t K, const lqlora_config* cfg, size_t* code_bytes,
                        size_t* scale_bytes, size_t* scale2_bytes, size_t* encode_workspace_bytes) {
    int rc = lq::check_config(cfg);
    if (rc != LQLORA_OK) return rc;
    rc = lq::check_shape(N, K, cfg);
    if (rc != LQLORA_OK) return rc;
    const int64_t Np = (N + lq::kTileRows - 1) / lq::kTileRows * lq::kTileRows;
    const int64_t nblk = N * K / cfg->B0;
    const int64_t ngrp = (nblk + cfg->B1 - 1) / cfg->B1;
    if (code_bytes) *code_bytes = static_cast<size_t>(Np) * K * cfg->b0 / 8;
    // scale codes: a bit stream of b1 bits each (eight codes take b1 bytes); second-level scales: 4 or 2 bytes each
    if (scale_bytes) *scale_bytes = (cfg->b1 == 8) ? static_cast<size_t>(nblk) : static_cast<size_t>((nblk + 7) / 8) * cfg->b1;
    if (scale2_bytes) *scale2_bytes = static_cast<size_t>(ngrp) * (cfg->b2 == lq::kB2Fp32 ? 4 : 2);
    // encoder scratch: the block absmax values, plus byte codes and fp32 scales before packing
    if (encode_workspace_bytes)
        *encode_workspace_bytes = (static_cast<size_t>(nblk) * sizeof(float) + 255) / 256 * 256 +
                                  (lq::packed_scales(cfg) ? (static_cast<size_t>(nblk) + 255) / 256 * 256 + static_cast<size_t>(ngrp) * 4 : 0);
    return LQLORA_OK;
}

int lqlora_nf_codebook(int b0, float* out_host) {
    if (!out_host) return LQLORA_ERR_NULL_POINTER;
    if (!(b0 == 2 || b0 == 3 || b0 == 4 || b0 == 8)) return LQLORA_ERR_INVALID_CONFIG;
    const float* cb = lq::host_codebook(b0);
    for (int i = 0; i < (1 << b0); ++i) out_host[i] = cb[i];
    return LQLORA_OK;
}

double lqlora_encode_search_clearance(int b0) {
    if (!(b0 == 2 || b0 == 3 || b0 == 4 || b0 == 8)) return -1.0;
    int nb = 0;
    return lq::detail::host_tables().best_bins(lq::bits_index(b0), 1 << b0, &nb);
}

double lqlora_encode_curve_clearance(int b0) {
    if (!(b0 == 2 || b0 == 3 || b0 == 4)) return -1.0;
    return lq::detail::host_tables().curve_clearance(b0);
}

int64_t lqlora_launch_count(void) { return lq::g_launches.load(std::memory_order_relaxed); }

const char* lqlora_status_string(int status) {
    switch (status) {
        case LQLORA_OK: return "ok";
        case LQLORA_ERR_INVALID_CONFIG: return "invalid quantization configuration";
        case LQLORA_ERR_INVALID_SHAPE: return "invalid shape";
        case LQLORA_ERR_NULL_POINTER: return "null pointer";
        case LQLORA_ERR_MISALIGNED: return "pointer not 16-byte aligned";
        case LQLORA_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case LQLORA_ERR_CUDA: return "CUDA error";
        case LQLORA_ERR_TIMEOUT: return "device-side wait timed out";
        case LQLORA_ERR_UNSUPPORTED: return "unsupported arguments";
        default: return "unknown status";
    }
}

}  // extern "C"
