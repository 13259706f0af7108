// Host-side check of the window kernel's stacked images (plan_conv_win with a
// period, and plan_conv_win_batch): for seeded random layers, over every tile of
// the batch,
//   - the rows the loader copies are consecutive, inside the tensor and fit a raw stage;
//   - every window row an output row needs is either the input row it stands for,
//     at its place in the raw stage, or padding;
//   - every output row of every image belongs to exactly one tile row, and its 2x2
//     windows stay within one image and start on an even tile row when pooled;
//   - the prepared image is the one of the plan without stacked images.
// The kernel's row arithmetic is restated here, with its 32-bit and 64-bit reciprocals.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "../paper_1908_11263_gb300/csrc/internal.h"

using namespace qnn;

static int fails = 0, plans = 0, chosen = 0;
#define CHECK(c, ...)                                  \
    do {                                               \
        if (!(c) && ++fails < 50) {                    \
            std::printf("FAIL %s: ", #c);              \
            std::printf(__VA_ARGS__);                  \
            std::printf("\n");                         \
        }                                              \
    } while (0)

static int div64(long long n, unsigned d)
{
    if (d <= 1) return static_cast<int>(n);
    const unsigned long long m = (~0ull / d) + 1ull;
    return static_cast<int>((static_cast<unsigned __int128>(static_cast<unsigned long long>(n)) * m) >> 64);
}

static void check(ConvShape s)
{
    const WinPlan base = plan_conv_win(s), best = plan_conv_win_batch(s);
    CHECK(base.ok == best.ok, "accepts the same layers");
    if (!base.ok) return;
    CHECK(best.period == 0 || best.total_tiles < base.total_tiles, "stacked images save tiles");
    chosen += best.period != 0;
    int period = s.h + s.ph;
    if (s.pool) period += period & 1;
    CHECK(best.period == 0 || best.period == period, "period %d", best.period);
    if (s.oh > period || period < 2 || period > 4096) {
        CHECK(best.period == 0, "not stacked");
        return;
    }
    const WinPlan p = plan_conv_win(s, false, period);
    if (!p.ok) return;
    ++plans;
    CHECK(p.period == period && p.smem_bytes <= 232448u, "plan");
    if (p.s == base.s)
        CHECK(p.b_bytes == base.b_bytes && p.tail_bytes == base.tail_bytes && p.img_bytes == base.img_bytes &&
                  p.off_mtab - p.off_rec == base.off_mtab - base.off_rec &&
                  p.off_pre - p.off_rec == base.off_pre - base.off_rec &&
                  p.off_tap - p.off_rec == base.off_tap - base.off_rec && p.nt == base.nt,
              "prepared image");
    const uint32_t m32 = static_cast<uint32_t>(((1ull << 32) + period - 1) / period);
    std::vector<int> made(static_cast<size_t>(s.n) * s.oh, 0);
    CHECK(p.total_tiles == p.tiles_per_img, "one tall image");
    for (int ty = 0; ty < p.tiles_y; ++ty) {
        const int img = div64(ty * 16, static_cast<unsigned>(period)), oy0 = ty * 16 - img * period;
        CHECK(img == ty * 16 / period && img < s.n, "first image of tile %d", ty);
        auto row_of = [&](int r, int &q, int &row) {
            q = static_cast<int>((static_cast<uint64_t>(static_cast<uint32_t>(oy0 + r)) * m32) >> 32);
            row = oy0 + r - q * period;
            CHECK(q == (oy0 + r) / period, "row %d of tile %d", r, ty);
        };
        auto before = [&](int r) {
            int q, row;
            row_of(r, q, row);
            if (q >= s.n - img) return (s.n - img) * s.h;
            return q * s.h + std::min(s.h, std::max(0, row - s.ph));
        };
        const int b0 = before(0), rows = before(p.wh) - b0;
        CHECK(rows >= 0 && static_cast<long long>(rows) * p.raw_row_bytes <= p.raw_bytes, "raw stage of tile %d", ty);
        CHECK(img * s.h + b0 >= 0 && img * s.h + b0 + rows <= s.n * s.h, "copied rows of tile %d", ty);
        for (int r = 0; r < 16; ++r) {
            int q, oy;
            row_of(r, q, oy);
            if (q >= s.n - img || oy >= s.oh) continue;
            ++made[static_cast<size_t>(img + q) * s.oh + oy];
            if (s.pool) CHECK((r & 1) == (oy & 1), "pool window of tile %d", ty);
            for (int i = 0; i < s.kh; ++i) {  // what output row oy needs: input row oy - ph + i of its image
                int wq, wrow;
                row_of(r + i, wq, wrow);
                const int iy = wrow - s.ph, want = oy - s.ph + i;
                const bool real = iy >= 0 && iy < s.h && wq < s.n - img, inside = want >= 0 && want < s.h;
                CHECK(real == inside, "window row %d of tile %d", r + i, ty);
                if (!real) continue;
                const int raw = wq * s.h + iy - b0;
                CHECK(raw >= 0 && raw < rows && img * s.h + b0 + raw == (img + q) * s.h + want, "raw row of tile %d", ty);
            }
        }
    }
    for (size_t k = 0; k < made.size(); ++k) CHECK(made[k] == 1, "output row %zu made %d times", k, made[k]);
}

int main()
{
    unsigned long long rng = 0x57ACCEDull;
    auto next = [&](int lo, int hi) {
        rng = rng * 6364136223846793005ull + 1442695040888963407ull;
        return lo + static_cast<int>((rng >> 33) % static_cast<unsigned long long>(hi - lo + 1));
    };
    for (int k = 0; k < 600; ++k) {
        static const int kBits[6] = {8, 8, 8, 4, 2, 1};
        ConvShape s{};
        s.bits = kBits[next(0, 5)];
        s.c = s.bits == 8 ? (next(0, 3) == 0 ? 3 : 8 * next(1, 8)) : 32 * next(1, 2);
        s.m = 8 * next(1, 16);
        s.kh = next(1, 7);
        s.kw = next(1, 5);
        s.ph = next(0, s.kh);  // (one more than any output row can use)
        s.pw = s.kw / 2;
        s.h = next(std::max(1, s.kh - 2 * s.ph), k % 8 == 0 ? 300 : 40);
        s.w = 16 * next(1, 4);
        s.n = next(1, 500);
        s.sh = s.sw = 1;
        s.oh = s.h + 2 * s.ph - s.kh + 1;
        s.ow = s.w + 2 * s.pw - s.kw + 1;
        s.pool = s.bits != 1 && s.oh > 1 && s.ow > 1 && next(0, 1);
        s.thr = (s.bits == 4 || s.bits == 2) && !s.pool && next(0, 1);
        check(s);
    }
    std::printf("plans=%d chosen=%d fails=%d\n", plans, chosen, fails);
    return fails || plans < 200 || chosen < 50;
}
