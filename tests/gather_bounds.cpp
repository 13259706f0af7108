// Host-side check of the gather kernel's planner and addressing, without a GPU
// (run by tests/test_gather_bounds.py).  For a list of layer shapes and seeded
// random ones it restates the kernel's rules and checks, against the plan:
//  - the shared-memory layout: operands, stages, records and barriers disjoint,
//    inside 227 KB, aligned for bulk copies; descriptor fields in range;
//  - every word a producer loads lies inside the input or the filters, and the
//    masked granules of a pixel and a filter multiply to the direct sum of the
//    convolution there;
//  - every tile and output channel is taken by exactly one CTA;
//  - chunks take at most 1024 products each.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_1908_11263_gb300/csrc/internal.h"

using namespace qnn;

static int fails = 0;
#define CHECK(cond)                                                     \
    do {                                                                \
        if (!(cond)) {                                                  \
            if (fails < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
            ++fails;                                                    \
        }                                                               \
    } while (0)

// The 16 bytes of a granule at offset p of `t`, bytes [lo, hi) valid: the aligned
// words that overlap them, the rest zero.
static void granule(const std::vector<uint8_t> &t, long long p, int lo, int hi, uint8_t (&out)[16])
{
    for (int b = 0; b < 16; ++b) out[b] = 0;
    if (hi <= lo) return;
    const int sh = static_cast<int>(((p % 4) + 4) % 4);
    const long long a = p - sh, end = static_cast<long long>(t.size());
    uint8_t q[20] = {};
    for (int k = 0; k < 5; ++k) {
        if (!(4 * k + 4 > lo + sh && 4 * k < hi + sh)) continue;
        CHECK(a + 4 * k >= 0);
        for (int b = 0; b < 4; ++b) {
            if (a + 4 * k + 4 <= end) {
                q[4 * k + b] = t[a + 4 * k + b];
            } else if (a + 4 * k + b < end) {
                q[4 * k + b] = t[a + 4 * k + b];
            }
        }
    }
    for (int b = lo; b < hi; ++b) out[b] = q[b + sh];
}

static void check(const ConvShape &s, int w_rows, std::mt19937 &rng)
{
    const int sms = 152;
    const bool prepared = w_rows > 0;
    const GatherPlan p = plan_conv_gather(s, w_rows, sms);
    std::printf("%dx%dx%dx%d->%d k%dx%d s%d,%d p%d,%d w_rows%d: ok=%d", s.n, s.h, s.w, s.c, s.m, s.kh, s.kw, s.sh, s.sw,
                s.ph, s.pw, w_rows, p.ok);
    if (!p.ok) {
        std::printf("\n");
        return;
    }
    std::printf(" %s %s %s ncols=%d stages=%d w_slots=%d grid=%d\n", p.flat ? "flat" : "im2col",
                p.aligned ? "aligned" : "bytes", p.resident ? "resident" : "streamed", p.ncols, p.stages, p.w_slots, p.grid);
    // K axis: the granules are the filter's values, each tap's or kernel row's rounded up
    CHECK(p.gran_row * 16 >= s.kw * s.c && (p.gran_row - 1) * 16 < s.kw * s.c);
    CHECK(p.flat ? p.taps == s.kh * s.kw && p.cgr * 16 == s.c : p.taps == 1 && p.cgr == p.gran_row * s.kh);
    CHECK(p.nxs * 4 >= p.cgr && (p.nxs - 1) * 4 < p.cgr);
    CHECK(p.chunk_stages >= 1 && p.chunk_stages * p.taps * 64 <= 1024);
    if (prepared) CHECK(s.c % 16 == 0 && p.taps * p.cgr * 16 == s.kh * s.kw * s.c);
    // layout: filters, pixel stages, barriers; descriptor fields
    const uint32_t x_bytes = 8 * p.plane_x;
    CHECK(p.ncols % 64 == 0 && p.ncols >= 64 && p.ncols <= 256 && p.stages >= 2 && p.stages <= 8);
    CHECK(p.plane_x >= static_cast<uint32_t>(p.npos) * 16 && p.plane_x % 32 == 16 && p.plane_x / 16 < (1 << 14));
    CHECK(p.npos <= (p.flat ? 8 * 64 : p.ncols) && (p.flat || p.aligned || p.ncols <= 128) && (p.flat || p.ncols <= 192));
    CHECK(p.stage_bytes % 16 == 0 && p.off_x % 128 == 0 && p.item_w % 16 == 0 && p.item_w == 8 * p.plane_w);
    CHECK(p.plane_w >= static_cast<uint32_t>(p.w_rows) * 16 && p.plane_w % 16 == 0);
    const long long items = 1ll * p.nxs * p.taps;
    if (p.resident) {
        CHECK(p.stage_bytes >= x_bytes && p.off_x >= items * p.item_w && p.parts >= 1 && p.parts <= 4);
    } else if (prepared) {
        CHECK(p.stage_bytes >= x_bytes && p.w_slots >= 2 && p.w_slots <= 9 && (!p.unrolled || (p.w_slots == 9 && p.taps == 9)) && p.off_x >= p.w_slots * p.item_w);
    } else {
        CHECK(p.stage_bytes >= x_bytes + p.item_w);
    }
    CHECK(p.off_bar >= p.off_x + p.stages * p.stage_bytes && p.off_bar % 8 == 0);
    CHECK(p.smem_bytes <= 232448 && p.smem_bytes >= p.off_bar + 1440 + 256 * 16);
    // the MMA reads 128 filter rows of every plane, laid out or not
    const long long last_w = p.resident ? items : prepared ? p.w_slots : 0;
    if (last_w) CHECK((last_w - 1) * p.item_w + 7ll * p.plane_w + 128 * 16 <= p.smem_bytes);
    else CHECK(p.item_w >= 7 * p.plane_w + 128 * 16);
    // tiles, and two accumulators at least
    CHECK(p.grid == p.mstep * p.n_ntiles && p.grid <= sms && p.mstep <= p.mtiles && p.n_ntiles * p.w_rows >= s.m);
    CHECK(1ll * p.mtiles * p.ncols >= p.npix && (p.mtiles - 1ll) * p.ncols < p.npix && 512 / p.ncols >= 2);
    const int hp = s.h + s.ph;
    CHECK(p.npix == (p.flat ? 1ll * s.n * hp * p.wp : 1ll * s.n * s.oh * s.ow));

    // sampled accumulators, the granules against the direct sum
    std::vector<uint8_t> x(static_cast<size_t>(s.n) * s.h * s.w * s.c), w(static_cast<size_t>(s.m) * s.kh * s.kw * s.c);
    for (auto &v : x) v = static_cast<uint8_t>(rng());
    for (auto &v : w) v = static_cast<uint8_t>(rng());
    const int kwc = s.kw * s.c, row_c = s.w * s.c;
    const long long npix = 1ll * s.n * s.oh * s.ow;
    for (int t = 0; t < 24; ++t) {
        const long long pix = t == 0 ? 0 : t == 1 ? npix - 1 : static_cast<long long>(rng() % npix);
        const int o = t == 1 ? s.m - 1 : static_cast<int>(rng() % s.m);
        const int img = static_cast<int>(pix / (s.oh * s.ow)), rem = static_cast<int>(pix % (s.oh * s.ow));
        const int oy = rem / s.ow, ox = rem % s.ow, iy = oy * s.sh - s.ph, ix = ox * s.sw - s.pw;
        const long long base = (1ll * img * s.h + iy) * row_c + 1ll * ix * s.c;
        long long got = 0, want = 0;
        for (int tap = 0; tap < p.taps; ++tap) {
            // flat: the staged position this tap reads, within the tile's window
            const int ti = tap / s.kw, tj = tap % s.kw;
            const long long q = (1ll * img * hp + oy) * p.wp + ox, pos = q + ti * p.wp + tj;
            bool pos_ok = false;
            long long pos_at = 0;
            if (p.flat) {
                CHECK(q < p.npix && q % p.ncols + ti * p.wp + tj < p.npos);
                const int b = static_cast<int>(pos / (hp * p.wp)), pr = static_cast<int>(pos % (hp * p.wp));
                const int r = pr / p.wp, c = pr % p.wp;
                pos_ok = b < s.n && r >= s.ph && c >= s.pw;
                pos_at = ((1ll * b * s.h + r - s.ph) * s.w + c - s.pw) * s.c;
            }
            for (int g = 0; g < p.cgr; ++g) {
                uint8_t xa[16], wa[16];
                if (p.flat) {
                    if (pos_ok) CHECK(pos_at >= 0 && pos_at + 16 * (g + 1) <= static_cast<long long>(x.size()));
                    granule(x, pos_at + 16 * g, 0, pos_ok ? 16 : 0, xa);
                    granule(w, (1ll * o * p.taps + tap) * s.c + 16 * g, 0, 16, wa);
                } else {
                    const int i = g / p.gran_row, r = (g % p.gran_row) * 16;
                    const bool row_ok = iy + i >= 0 && iy + i < s.h;
                    if (p.aligned) {
                        const int j = r / s.c;
                        const bool ok = row_ok && ix + j >= 0 && ix + j < s.w;
                        const long long at = base + 1ll * i * row_c + r;
                        if (ok) CHECK(at % 16 == 0 && at >= 0 && at + 16 <= static_cast<long long>(x.size()));
                        granule(x, at, 0, ok ? 16 : 0, xa);
                        CHECK((1ll * o * s.kh + i) * kwc + r + 16 <= static_cast<long long>(w.size()));
                    } else {
                        const int lo = std::min(16, std::max(0, -ix * s.c - r));
                        const int hi = row_ok && r < kwc ? std::max(0, std::min(16, (s.w - ix) * s.c - r)) : 0;
                        granule(x, base + 1ll * i * row_c + r, lo, hi, xa);
                    }
                    granule(w, (1ll * o * s.kh + i) * kwc + r, 0, std::min(16, kwc - r), wa);
                }
                // staged x - 128, and 128 * sum(w) put back
                for (int b = 0; b < 16; ++b)
                    got += (static_cast<int>(xa[b]) - 128) * static_cast<int8_t>(wa[b]) + 128 * static_cast<int8_t>(wa[b]);
            }
        }
        for (int i = 0; i < s.kh; ++i)
            for (int j = 0; j < s.kw; ++j)
                for (int c = 0; c < s.c; ++c)
                    if (iy + i >= 0 && iy + i < s.h && ix + j >= 0 && ix + j < s.w)
                        want += static_cast<int>(x[((1ll * img * s.h + iy + i) * s.w + ix + j) * s.c + c]) *
                                static_cast<int8_t>(w[((1ll * o * s.kh + i) * s.kw + j) * s.c + c]);
        CHECK(got == want);
    }
    // flat: the walk over a block of columns (the epilogue's) meets every output pixel once, in order
    if (p.flat && p.npix < 20000) {
        long long next = 0;
        for (int p0 = 0; p0 < p.mtiles * p.ncols; p0 += 16) {
            int b = p0 / (hp * p.wp), pr = p0 % (hp * p.wp), r = pr / p.wp, c = pr % p.wp;
            long long at = (1ll * b * s.oh + r) * s.ow + c;
            for (int k = 0; k < 16; ++k) {
                if (c < s.ow && r < s.oh && b < s.n) {
                    CHECK(at == next);
                    ++next;
                }
                ++at;
                if (++c == p.wp) {
                    c = 0;
                    at -= p.wp - s.ow;
                    if (++r == hp) {
                        r = 0;
                        ++b;
                        at -= 1ll * (hp - s.oh) * s.ow;
                    }
                }
            }
        }
        CHECK(next == npix);
    }
}

static ConvShape shape(int n, int h, int w, int c, int m, int kh, int kw, int sh, int sw, int ph, int pw)
{
    ConvShape s{};
    s.n = n; s.h = h; s.w = w; s.c = c; s.m = m; s.kh = kh; s.kw = kw;
    s.sh = sh; s.sw = sw; s.ph = ph; s.pw = pw; s.bits = 8;
    s.oh = (h + 2 * ph - kh) / sh + 1;
    s.ow = (w + 2 * pw - kw) / sw + 1;
    return s;
}

int main()
{
    std::mt19937 rng(1908);
    const ConvShape fixed[] = {
        shape(64, 56, 56, 64, 128, 3, 3, 2, 2, 1, 1), shape(37, 33, 45, 20, 44, 3, 3, 1, 1, 1, 1),
        shape(64, 28, 28, 128, 128, 3, 3, 1, 1, 1, 1), shape(64, 14, 14, 256, 256, 3, 3, 1, 1, 1, 1),
        shape(64, 14, 14, 256, 512, 1, 1, 1, 1, 0, 0), shape(1, 5, 7, 3, 10, 5, 5, 2, 2, 2, 2),
        shape(1, 1, 1, 1, 1, 1, 1, 1, 1, 0, 0),        shape(2, 9, 9, 17, 33, 3, 3, 3, 2, 5, 4),
        shape(1, 4, 4, 512, 520, 3, 3, 2, 2, 1, 1),    shape(3, 8, 8, 48, 16, 3, 3, 1, 1, 1, 1),
    };
    for (const ConvShape &s : fixed)
        for (int w_rows : {0, 128}) check(s, w_rows, rng);
    auto in = [&](int lo, int hi) { return lo + static_cast<int>(rng() % (hi - lo + 1)); };
    for (int k = 0; k < 300; ++k) {
        const int kh = in(1, 7), kw = in(1, 7), ph = in(0, 3), pw = in(0, 3);
        const int h = std::max(in(1, 30), kh - 2 * ph), w = std::max(in(1, 30), kw - 2 * pw);
        const int c = in(0, 2) ? in(1, 80) : 16 * in(1, 20);
        const ConvShape s = shape(in(1, 6), std::max(1, h), std::max(1, w), c, in(1, 200), kh, kw,
                                  k % 2 ? 1 : in(1, 3), k % 2 ? 1 : in(1, 3), ph, pw);
        const int rows[] = {0, 128, 0, 64, 16, 32};
        check(s, rows[k % 6], rng);
    }
    std::printf("fails=%d\n", fails);
    return fails != 0;
}
