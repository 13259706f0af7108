// Host-side model of the gather kernel's loads, outputs and chunks as they are in
// conv_gather.cuh, without a GPU (run by tests/test_gather_loads.py).  Against the
// planner's plans for listed and seeded random layers:
//  - Gran<false>::load: five aligned words only where all lie inside the tensor, else
//    single bytes, each of them inside; the bytes it returns;
//  - produce_x, produce_flat and fetch_w: every load of every tile and stage;
//  - output_pixel: every column of every tile, each output pixel once;
//  - make_chunks: with sums of |w| no chunk of any filter passes 2^24, and the
//    accumulators in flight fit TMEM.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_1908_11263_gb300/csrc/internal.h"

using namespace qnn;

static int fails = 0;
static long long whole = 0, single = 0, chunks_seen = 0, many_chunks = 0;
#define CHECK(cond)                                                     \
    do {                                                                \
        if (!(cond)) {                                                  \
            if (fails < 20) std::printf("FAIL line %d: %s\n", __LINE__, #cond); \
            ++fails;                                                    \
        }                                                               \
    } while (0)

// Gran<false>::load and get at offset p of a tensor: bytes [lo, hi) of the 16 there.
static void load_bytes(const std::vector<uint8_t> &t, long long p, int lo, int hi, uint8_t (&out)[16])
{
    const long long size = static_cast<long long>(t.size());
    const int sh = static_cast<int>(((p % 4) + 4) % 4);
    const long long a = p - sh;
    uint8_t q[20] = {};
    if (hi > lo && a >= 0 && a + 20 <= size) {
        ++whole;
        for (int k = 0; k < 5; ++k) {
            CHECK((a + 4 * k) % 4 == 0 && a + 4 * k >= 0 && a + 4 * k + 4 <= size);
            for (int b = 0; b < 4; ++b) q[4 * k + b] = t[static_cast<size_t>(a + 4 * k + b)];
        }
    } else if (hi > lo) {
        ++single;
        for (int b = 0; b < 20; ++b)
            if (b >= lo + sh && b < hi + sh) {
                CHECK(a + b >= 0 && a + b < size);
                if (a + b >= 0 && a + b < size) q[b] = t[static_cast<size_t>(a + b)];
            }
    }
    for (int b = 0; b < 16; ++b) out[b] = b >= lo && b < hi ? q[b + sh] : 0;
}

// An aligned granule (16 bytes in one load).
static void load_whole(long long p, long long size)
{
    CHECK(p % 16 == 0 && p >= 0 && p + 16 <= size);
}

static void check_loads(const ConvShape &s, const GatherPlan &p, std::mt19937 &rng)
{
    std::vector<uint8_t> x(static_cast<size_t>(s.n) * s.h * s.w * s.c), w(static_cast<size_t>(s.m) * s.kh * s.kw * s.c);
    for (auto &v : x) v = static_cast<uint8_t>(rng());
    for (auto &v : w) v = static_cast<uint8_t>(rng());
    const long long xbytes = static_cast<long long>(x.size()), row_c = 1ll * s.w * s.c;
    const int kwc = s.kw * s.c, gr = p.gran_row;
    // filters on the caller's layout: every granule of every filter
    if (p.w_rows == 128 && !p.flat)
        for (int o = 0; o < s.m; ++o)
            for (int g = 0; g < p.cgr; ++g) {
                const int i = g / gr, r = g % gr * 16;
                const long long at = (1ll * o * s.kh + i) * kwc + r;
                if (p.aligned) {
                    load_whole(at, static_cast<long long>(w.size()));
                } else {
                    uint8_t v[16];
                    load_bytes(w, at, 0, std::min(16, kwc - r), v);
                    for (int b = 0; b < std::min(16, kwc - r); ++b) CHECK(v[b] == w[static_cast<size_t>(at + b)]);
                }
            }
    // pixels: every column of every tile (sampled for large layers), every granule
    const long long cols = 1ll * p.mtiles * p.ncols, step = std::max(1ll, cols / 3000);
    for (long long col = 0; col < cols; col += step) {
        if (p.flat) {
            // positions of the tile's window that this column's taps reach
            const int per = (s.h + s.ph) * p.wp;
            const long long img = col / per, rem = col % per, r = rem / p.wp, c = rem % p.wp;
            const bool ok = img < s.n && r >= s.ph && c >= s.pw;
            if (!ok) continue;
            const long long at = ((img * s.h + r - s.ph) * s.w + c - s.pw) * s.c;
            for (int g = 0; g < p.cgr; ++g) load_whole(at + 16ll * g, xbytes);
            continue;
        }
        const long long img = col / (1ll * s.oh * s.ow), rem = col % (1ll * s.oh * s.ow);
        const bool real = col < p.npix;
        const int iy = real ? static_cast<int>(rem / s.ow) * s.sh - s.ph : -32768;
        const int ix = static_cast<int>(rem % s.ow) * s.sw - s.pw;
        const long long base = (img * s.h + iy) * row_c + 1ll * ix * s.c;
        for (int g = 0; g < p.nxs * 4; ++g) {
            const bool in = g < p.cgr;
            const int i = g / gr, r = g % gr * 16;
            const bool row_ok = in && iy + i >= 0 && iy + i < s.h;
            if (p.aligned) {
                const int j = r / s.c;
                if (row_ok && ix + j >= 0 && ix + j < s.w) load_whole(base + i * row_c + r, xbytes);
                continue;
            }
            const int lo = std::min(16, std::max(0, -ix * s.c - r));
            const int hi = row_ok && r < kwc ? std::max(0, std::min(16, (s.w - ix) * s.c - r)) : 0;
            uint8_t v[16];
            load_bytes(x, base + i * row_c + r, lo, hi, v);
            for (int b = lo; b < hi; ++b) CHECK(v[b] == x[static_cast<size_t>(base + i * row_c + r + b)]);
        }
    }
}

static void check_outputs(const ConvShape &s, const GatherPlan &p)
{
    const long long npix = 1ll * s.n * s.oh * s.ow;
    std::vector<uint8_t> met(static_cast<size_t>(npix), 0);
    for (long long q = 0; q < 1ll * p.mtiles * p.ncols; ++q) {
        long long pix = -1;
        if (!p.flat) {
            pix = q < p.npix ? q : -1;
        } else {
            const int per = (s.h + s.ph) * p.wp;
            const long long img = q / per, rem = q % per, r = rem / p.wp, c = rem % p.wp;
            if (c < s.ow && r < s.oh && img < s.n) pix = (img * s.oh + r) * s.ow + c;
        }
        if (pix < 0) continue;
        CHECK(pix < npix);
        if (pix < npix) ++met[static_cast<size_t>(pix)];
    }
    for (uint8_t v : met) CHECK(v == 1);
}

// make_chunks on sums of |w| by filter and stage (flat plans with at most 16 stages).
static void check_chunks(const ConvShape &s, const GatherPlan &p, std::mt19937 &rng)
{
    const int kChunkAbs = 1 << 17;
    const bool carried = p.flat && p.nxs <= 16;
    for (int kind = 0; kind < 3; ++kind) {
        // ordinary, extreme and sparse filters: a stage's sum is at most 128 per product
        std::vector<std::vector<int>> abs(static_cast<size_t>(p.w_rows), std::vector<int>(static_cast<size_t>(p.nxs)));
        std::vector<int> most(static_cast<size_t>(p.nxs), 0);
        for (auto &f : abs)
            for (int st = 0; st < p.nxs; ++st) {
                const int products = std::min(4, p.cgr - 4 * st) * 16 * p.taps;
                const int mean = kind == 0 ? 64 : kind == 1 ? 128 : static_cast<int>(rng() % 8);
                f[static_cast<size_t>(st)] = products * mean;
                CHECK(f[static_cast<size_t>(st)] <= kChunkAbs);
                most[static_cast<size_t>(st)] = std::max(most[static_cast<size_t>(st)], f[static_cast<size_t>(st)]);
            }
        uint32_t ends = 0;
        int every = p.chunk_stages, n = (p.nxs + p.chunk_stages - 1) / p.chunk_stages;
        if (carried) {
            every = 0;
            n = 1;
            int sum = 0;
            for (int st = 0; st < p.nxs; ++st) {
                const int v = most[static_cast<size_t>(st)];
                if (st && sum + v > kChunkAbs) {
                    ends |= 1u << (st - 1);
                    ++n;
                    sum = 0;
                }
                sum += v;
            }
        }
        auto end = [&](int st) {
            return st == p.nxs - 1 || (st < 32 && every == 0 ? (ends >> st) & 1u : every != 0 && (st + 1) % every == 0);
        };
        int count = 0;
        std::vector<long long> sum(static_cast<size_t>(p.w_rows), 0);
        for (int st = 0; st < p.nxs; ++st) {
            for (size_t f = 0; f < abs.size(); ++f) {
                sum[f] += abs[f][static_cast<size_t>(st)];
                CHECK(128 * sum[f] <= 1 << 24);
            }
            if (end(st)) {
                ++count;
                std::fill(sum.begin(), sum.end(), 0);
            }
        }
        CHECK(count == n);
        const int fit = 512 / p.ncols;
        const int regions = n <= fit ? n : 1, groups = n <= fit ? std::min(4, fit / n) : std::min(4, fit - 1);
        CHECK(groups >= 1 && (groups * regions + (n > fit ? 1 : 0)) * p.ncols <= 512);
        chunks_seen += n;
        many_chunks += n > fit;
    }
    (void)s;
}

static void check(const ConvShape &s, int w_rows, std::mt19937 &rng)
{
    const GatherPlan p = plan_conv_gather(s, w_rows, 152);
    if (!p.ok) return;
    std::printf(" %s %s %s\n", p.flat ? "flat" : "im2col", p.aligned ? "aligned" : "bytes", p.resident ? "resident" : "streamed");
    check_loads(s, p, rng);
    if (1ll * p.mtiles * p.ncols < 400000) check_outputs(s, p);
    check_chunks(s, p, rng);
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
    std::mt19937 rng(20);
    const ConvShape fixed[] = {
        shape(2, 33, 45, 20, 44, 3, 3, 1, 1, 1, 1),   shape(3, 28, 28, 128, 128, 3, 3, 1, 1, 1, 1),
        shape(1, 14, 14, 512, 256, 3, 3, 1, 1, 1, 1), shape(2, 14, 14, 256, 512, 1, 1, 1, 1, 0, 0),
        shape(1, 5, 7, 3, 10, 5, 5, 2, 2, 2, 2),      shape(1, 1, 1, 21, 1, 1, 1, 1, 1, 0, 0),
        shape(1, 5, 3, 21, 300, 1, 1, 1, 1, 3, 0),    shape(2, 9, 9, 17, 33, 3, 3, 3, 2, 5, 4),
        shape(1, 1, 1, 1, 1, 1, 1, 1, 1, 0, 0),       shape(1, 1, 3, 2, 5, 1, 3, 1, 1, 0, 1),
        shape(1, 8, 8, 1600, 16, 3, 3, 1, 1, 1, 1),   shape(1, 40, 17, 31, 9, 7, 3, 2, 1, 3, 1),
    };
    for (const ConvShape &s : fixed)
        for (int w_rows : {0, 16, 128}) check(s, w_rows, rng);
    auto in = [&](int lo, int hi) { return lo + static_cast<int>(rng() % (hi - lo + 1)); };
    for (int k = 0; k < 300; ++k) {
        const int kh = in(1, 7), kw = in(1, 7), ph = in(0, 3), pw = in(0, 3);
        const int h = std::max(in(1, 30), kh - 2 * ph), w = std::max(in(1, 30), kw - 2 * pw);
        const int c = in(0, 2) ? in(1, 60) : 16 * in(1, 20);
        const ConvShape s = shape(in(1, 4), std::max(1, h), std::max(1, w), c, in(1, 150), kh, kw, k % 2 ? 1 : in(1, 3),
                                  k % 2 ? 1 : in(1, 3), ph, pw);
        const int rows[] = {0, 128, 0, 64, 16, 32};
        check(s, rows[k % 6], rng);
    }
    std::printf("words %d bytes %d chunks %d many %d\n", whole > 0, single > 0, chunks_seen > 0, many_chunks > 0);
    std::printf("fails=%d\n", fails);
    return fails != 0;
}
