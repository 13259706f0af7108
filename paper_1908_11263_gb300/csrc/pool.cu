// Max-pooling on packed NHWC activations (Sec. IV-A; split over output pixels as
// in Sec. IV-B).  One thread produces 16 output bytes (pixels of whole 16-byte
// vectors: 128-bit loads and a field-wise vmax at any Q) or one output byte (any
// layout).  No padding, floor output size.
#include <cstdint>
#include <type_traits>

#include "conv_common.cuh"
#include "device.cuh"
#include "internal.h"

namespace qnn {
namespace {

// One thread produces one 16-byte vector of an output pixel (pixels whose bytes
// are whole 16-byte vectors).  Bound by HBM; the index takes three
// multiplications (64-bit divisions by run-time sizes took longer than the
// loads), and the four loads of the 2 x 2 window go out together.
// INT-2 2048 x 16 x 16 x 64: 2.6 us (6.9).  Outputs of 2^31 vectors and more have a
// 64-bit index and divisions: 2049 x 1024 x 1024 x 16, 1 x 1, takes 15.0 ms, 314 byte by byte.
//
// Other windows: their row unrolled (by the compiler) up to one wave of blocks (64
// images of 56 x 56 x 64, 3 x 3 stride 2, INT-8: 5.4 us, 6.0 rolled), rolled beyond it, where the registers of
// the unrolled form halve the warps in flight (64 of 256 x 256 x 64: 65.9 us, 87.2).
enum PoolForm { kTwo = 0, kUnrolled = 1, kRolled = 2 };

template <int BITS, int FORM, class Index>
__global__ void __launch_bounds__(256) maxpool_vec_kernel(Index total, int h, int w, int vec_per_pix, int k, int s,
                                                          int oh, int ow, FastDiv fd_vec, FastDiv fd_ow, FastDiv fd_oh,
                                                          const uint4 *x, uint4 *y)
{
    pdl_wait();
    pdl_trigger();
    const Index gid = static_cast<Index>(blockIdx.x) * 256 + threadIdx.x;
    if (gid >= total) return;
    int b, oy, ox, v;
    if constexpr (sizeof(Index) == 8) {
        const Index pix = gid / vec_per_pix, row = pix / ow;
        v = static_cast<int>(gid - pix * vec_per_pix);
        ox = static_cast<int>(pix - row * ow);
        b = static_cast<int>(row / oh);
        oy = static_cast<int>(row - static_cast<Index>(b) * oh);
    } else {
        const int pix = fdiv(static_cast<int>(gid), fd_vec), row = fdiv(pix, fd_ow);
        v = static_cast<int>(gid) - pix * vec_per_pix;
        ox = pix - row * ow;
        b = fdiv(row, fd_oh);
        oy = row - b * oh;
    }
    const uint4 *src = x + ((static_cast<long long>(b) * h + oy * s) * w + ox * s) * vec_per_pix + v;
    uint4 best = make_uint4(0, 0, 0, 0);
    auto take = [&](const uint4 &t) {
        best.x = max_fields<BITS>(best.x, t.x);
        best.y = max_fields<BITS>(best.y, t.y);
        best.z = max_fields<BITS>(best.z, t.z);
        best.w = max_fields<BITS>(best.w, t.w);
    };
    if (FORM == kTwo) {
        const uint4 *low = src + static_cast<long long>(w) * vec_per_pix;
        const uint4 t0 = src[0], t1 = src[vec_per_pix], t2 = low[0], t3 = low[vec_per_pix];
        take(t0);
        take(t1);
        take(t2);
        take(t3);
    } else if (FORM == kUnrolled) {
        for (int i = 0; i < k; ++i)
            for (int j = 0; j < k; ++j) take(src[(static_cast<long long>(i) * w + j) * vec_per_pix]);
    } else {
        for (int i = 0; i < k; ++i)
#pragma unroll 1
            for (int j = 0; j < k; ++j) take(src[(static_cast<long long>(i) * w + j) * vec_per_pix]);
    }
    y[gid] = best;
}

template <int BITS>
__global__ void __launch_bounds__(256) maxpool_byte_kernel(int n, int h, int w, int c, int k, int s, int oh, int ow,
                                                           const uint8_t *x, uint8_t *y)
{
    const int bytes_per_pix = c * BITS / 8;
    const long long total = static_cast<long long>(n) * oh * ow * bytes_per_pix;
    const long long gid = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (gid >= total) return;
    const int byte = static_cast<int>(gid % bytes_per_pix);
    const long long pix = gid / bytes_per_pix;
    const int ox = static_cast<int>(pix % ow);
    const int oy = static_cast<int>((pix / ow) % oh);
    const int b = static_cast<int>(pix / (static_cast<long long>(ow) * oh));
    constexpr int per = 8 / BITS;
    constexpr int mask = (1 << BITS) - 1;
    int best[per];
#pragma unroll
    for (int f = 0; f < per; ++f) best[f] = 0;
    for (int i = 0; i < k; ++i)
        for (int j = 0; j < k; ++j) {
            const long long src = ((static_cast<long long>(b) * h + oy * s + i) * w + ox * s + j) * bytes_per_pix + byte;
            const int t = x[src];
#pragma unroll
            for (int f = 0; f < per; ++f) best[f] = max(best[f], (t >> (f * BITS)) & mask);
        }
    int out = 0;
#pragma unroll
    for (int f = 0; f < per; ++f) out |= best[f] << (f * BITS);
    y[gid] = static_cast<uint8_t>(out);
}

}  // namespace

cudaError_t launch_maxpool(int n, int h, int w, int c, int k, int s, int bits, const uint8_t *x, uint8_t *y,
                           cudaStream_t st)
{
    const int oh = (h - k) / s + 1, ow = (w - k) / s + 1;
    const long long pix = static_cast<long long>(n) * oh * ow;
    if (pix == 0) return cudaSuccess;
    const int bytes_per_pix = c * bits / 8;
    const bool vec = bytes_per_pix % 16 == 0 && (reinterpret_cast<uintptr_t>(x) % 16) == 0 &&
                     (reinterpret_cast<uintptr_t>(y) % 16) == 0;
    if (vec) {
        const int vpp = bytes_per_pix / 16;
        const long long total = pix * vpp;
        const FastDiv fv = make_fastdiv(static_cast<uint32_t>(vpp)), fw = make_fastdiv(static_cast<uint32_t>(ow)),
                      fh = make_fastdiv(static_cast<uint32_t>(oh));
        const uint4 *xv = reinterpret_cast<const uint4 *>(x);
        uint4 *yv = reinterpret_cast<uint4 *>(y);
        auto go = [&](auto kern) {
            return launch_pdl(kern, static_cast<unsigned>((total + 255) / 256), 256, 0, st, total, h, w, vpp, k, s, oh, ow,
                              fv, fw, fh, xv, yv);
        };
        auto pick = [&](auto bits_const) {
            constexpr int B = decltype(bits_const)::value;
            if (total >= (1ll << 31)) return go(maxpool_vec_kernel<B, kRolled, long long>);
            if (k == 2) return go(maxpool_vec_kernel<B, kTwo, unsigned>);
            return total <= 2048ll * device_sm_count() ? go(maxpool_vec_kernel<B, kUnrolled, unsigned>)
                                                       : go(maxpool_vec_kernel<B, kRolled, unsigned>);
        };
        return bits == 8   ? pick(std::integral_constant<int, 8>())
               : bits == 4 ? pick(std::integral_constant<int, 4>())
                           : pick(std::integral_constant<int, 2>());
    } else {
        const long long total = pix * (c * bits / 8);
        const unsigned grid = static_cast<unsigned>((total + 255) / 256);
        if (bits == 8) maxpool_byte_kernel<8><<<grid, 256, 0, st>>>(n, h, w, c, k, s, oh, ow, x, y);
        else if (bits == 4) maxpool_byte_kernel<4><<<grid, 256, 0, st>>>(n, h, w, c, k, s, oh, ow, x, y);
        else maxpool_byte_kernel<2><<<grid, 256, 0, st>>>(n, h, w, c, k, s, oh, ow, x, y);
    }
    return cudaGetLastError();
}

}  // namespace qnn
