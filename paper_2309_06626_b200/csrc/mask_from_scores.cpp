// Algorithm 1, getMask, for one layer on the host: average pooling of the score map, then the
// floor(sparsity * P + 1/2) positions with the smallest pooled score (ties in raster order) are dropped.
//
// What bounds it.  Window sums are fp64 sums in raster order of the window, so the additions of one window are
// a serial chain of 4 clocks each; only windows are independent.  Window by window, a 224 x 224 score cost 40 us at
// any output resolution (50 176 chained additions), ranking 12 544 positions with nth_element on (score,
// position) pairs another 100 us.  Here a score row is walked once and added to all its windows' sums, so the
// chains of neighbouring windows overlap in the core's out-of-order window, and the ranking is one histogram over
// the score's range: only the positions in the bucket that holds the threshold are ordered.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <new>
#include <utility>
#include <vector>

#include "asx.h"

namespace {

// sum[j] += row[j * RW], row[j * RW + 1], ... in this order, for `n` windows (RW = 0: width `rw`).  Four windows at a
// time, four independent chains in registers, in scalar code: a vector of windows would have to be gathered at
// stride RW, and what the compiler (or four-by-four transposes by hand) makes of that is slower (45 us, 11-19 us
// against 13-16 us for the whole 224 x 224 score).
template <int RW>
__attribute__((optimize("no-tree-vectorize", "no-tree-slp-vectorize")))
void add_row(double* __restrict__ sum, const float* __restrict__ row, int n, int rw)
{
    const size_t width = RW ? RW : rw;
    int j = 0;
    for (; j + 4 <= n; j += 4) {
        const float *w0 = row + j * width, *w1 = w0 + width, *w2 = w1 + width, *w3 = w2 + width;
        double a0 = sum[j], a1 = sum[j + 1], a2 = sum[j + 2], a3 = sum[j + 3];
        for (size_t b = 0; b < width; ++b) {
            a0 += (double)w0[b];
            a1 += (double)w1[b];
            a2 += (double)w2[b];
            a3 += (double)w3[b];
        }
        sum[j] = a0; sum[j + 1] = a1; sum[j + 2] = a2; sum[j + 3] = a3;
    }
    for (; j < n; ++j) {
        double a = sum[j];
        for (size_t b = 0; b < width; ++b) a += (double)row[j * width + b];
        sum[j] = a;
    }
}

void pool(const float* score, int W0, int Ho, int Wo, int rh, int rw, double* out)
{
    const double area = (double)((int64_t)rh * rw);
    for (int i = 0; i < Ho; ++i) {
        double* sum = out + (size_t)i * Wo;
        for (int j = 0; j < Wo; ++j) sum[j] = 0.0;
        for (int a = 0; a < rh; ++a) {
            const float* row = score + ((size_t)i * rh + a) * W0;
            switch (rw) {                             // ratios of the usual networks, with the inner loop unrolled
                case 2: add_row<2>(sum, row, Wo, rw); break;
                case 4: add_row<4>(sum, row, Wo, rw); break;
                case 8: add_row<8>(sum, row, Wo, rw); break;
                case 16: add_row<16>(sum, row, Wo, rw); break;
                default: add_row<0>(sum, row, Wo, rw); break;
            }
        }
        for (int j = 0; j < Wo; ++j) sum[j] /= area;
    }
}

constexpr int BUCKETS = 2048;

// mask[p] = 0 for the n_drop entries with the smallest (value, p), 0 < n_drop < P; the rest of `mask` is 1 on entry.
void drop_smallest(const double* v, int64_t P, int64_t n_drop, uint8_t* mask)
{
    // extremes in eight lanes, which the compiler turns into vectors; a NaN makes its sum one
    double lo8[8], hi8[8], nan8[8];
    for (int l = 0; l < 8; ++l) { lo8[l] = hi8[l] = v[0]; nan8[l] = 0.0; }
    int64_t q = 0;
    for (; q + 8 <= P; q += 8)
        for (int l = 0; l < 8; ++l) {
            const double x = v[q + l];
            lo8[l] = x < lo8[l] ? x : lo8[l];
            hi8[l] = x > hi8[l] ? x : hi8[l];
            nan8[l] += x;
        }
    for (; q < P; ++q) {
        lo8[0] = v[q] < lo8[0] ? v[q] : lo8[0];
        hi8[0] = v[q] > hi8[0] ? v[q] : hi8[0];
        nan8[0] += v[q];
    }
    double lo = lo8[0], hi = hi8[0], sum = 0.0;
    for (int l = 0; l < 8; ++l) {
        lo = lo8[l] < lo ? lo8[l] : lo;
        hi = hi8[l] > hi ? hi8[l] : hi;
        sum += nan8[l];
    }
    const bool ordered = std::isfinite(sum);          // no NaN and no infinity among the values
    // Monotone map of a value to a bucket: subtraction, product with a positive number and truncation all keep the order.
    const double scale = (double)BUCKETS / (hi - lo);
    std::vector<std::pair<double, int64_t>> tied;     // candidates for the last drops
    int64_t below = 0;
    if (ordered && std::isfinite(hi - lo) && std::isfinite(scale) && scale > 0.0) {
        std::unique_ptr<uint16_t[]> bucket(new uint16_t[(size_t)P]);
        uint16_t* const at = bucket.get();
        uint32_t count[2][BUCKETS] = {{0}};           // two tables: neighbours in one bucket do not wait for each other's store
        for (int64_t p = 0; p < P; ++p) {
            const int b = (int)((v[p] - lo) * scale);
            at[p] = (uint16_t)(b < BUCKETS ? b : BUCKETS - 1);
        }
        for (int64_t p = 0; p + 1 < P; p += 2) {
            ++count[0][at[p]];
            ++count[1][at[p + 1]];
        }
        if (P & 1) ++count[0][at[P - 1]];
        int cut = 0;
        auto in_bucket = [&](int b) { return (int64_t)count[0][b] + count[1][b]; };
        while (below + in_bucket(cut) < n_drop) below += in_bucket(cut++);
        tied.reserve((size_t)in_bucket(cut));
        const uint16_t c16 = (uint16_t)cut;
        for (int64_t p = 0; p < P; ++p) mask[p] = at[p] >= c16;
        for (int64_t p = 0; p < P; ++p)
            if (at[p] == c16) tied.emplace_back(v[p], p);
    } else {                                          // all values alike, infinities or NaN: order all positions
        tied.reserve((size_t)P);
        for (int64_t p = 0; p < P; ++p) tied.emplace_back(v[p], p);
    }
    const int64_t more = n_drop - below;
    if (more < (int64_t)tied.size()) std::nth_element(tied.begin(), tied.begin() + (more - 1), tied.end());
    for (int64_t k = 0; k < more; ++k) mask[tied[(size_t)k].second] = 0;
}

}  // namespace

extern "C" asx_status asx_mask_from_scores(const float* score, int H0, int W0, int Ho, int Wo, double sparsity,
                                           uint8_t* mask_out)
{
    if (score == nullptr || mask_out == nullptr || H0 < 1 || W0 < 1 || Ho < 1 || Wo < 1 || Ho > H0 || Wo > W0 ||
        !(sparsity >= 0.0 && sparsity <= 1.0) || (int64_t)Ho * Wo >= (1ll << 31))
        return ASX_ERR_INVALID_ARG;
    const int rh = H0 / Ho, rw = W0 / Wo;                 // ratio = input_res // layer.res
    const int64_t P = (int64_t)Ho * Wo;
    int64_t n_drop = (int64_t)std::floor(sparsity * (double)P + 0.5);
    if (n_drop > P) n_drop = P;
    std::memset(mask_out, n_drop < P ? 1 : 0, (size_t)P);
    if (n_drop == 0 || n_drop == P) return ASX_OK;        // nothing to rank
    try {
        std::unique_ptr<double[]> pooled(new double[(size_t)P]);
        pool(score, W0, Ho, Wo, rh, rw, pooled.get());
        drop_smallest(pooled.get(), P, n_drop, mask_out);
    } catch (const std::bad_alloc&) {
        return ASX_ERR_OOM;
    }
    return ASX_OK;
}
