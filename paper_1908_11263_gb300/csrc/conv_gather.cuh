// Quantized INT-8 HWC convolution on the sm_103a tensor cores with the output
// channels along the MMA's rows and output pixels along its columns: the
// gather kernel.  It serves INT-8 layers that the window kernel's plan does not
// take: more than 128 filters, many channels, any stride, padding, channel count
// and alignment, except where the general kernel or the CUDA cores are faster
// (general_beats_gather, direct_beats_gather).
//
// What it computes (Sec. III-B, Eq. 6; Sec. III-A): for every output pixel p
// and channel o,
//   acc = dot(W(o), im2col(p))                       exact integer, int32
//   y   = clip(floor(((acc + bias_o) * kappa_o + lambda_o) / 2^shift_o), 0, 255)
//
// Why channels are rows.  The accumulator then has a channel per TMEM lane, so
// a lane of the epilogue keeps its channel's constants in registers; with
// pixels in the lanes every value needs its channel's constants broadcast from
// shared memory, which the tensor cores' operand reads keep busy (measured on
// such a form of this kernel: 4,000 to 4,600 cycles for 128 x 128 outputs).
// An M = 128, N = 256, K = 16 MMA reads 12 KB of operands in its 128 cycles,
// two of N = 128 read 16 KB, the shared-memory bandwidth itself.  N is any
// multiple of 64 up to 256, chosen so that the tiles fill the SMs evenly.
//
// Granules.  The K axis moves in granules of 16 values: what one 16-byte load
// brings, and one MMA consumes.  A stage holds four granules of every pixel.
//
// Pixel operand, im2col (kIm2col): columns are output pixels of the whole
// batch in memory order, K is kh kernel rows of kw * c contiguous input bytes
// (each rounded up to whole granules), at any stride.  With c a multiple of
// 16 a granule lies inside one input pixel and its load is aligned; otherwise
// it is put together from the words it overlaps and masked to the bytes
// inside the image.
//
// Pixel operand, flat window (kFlat, stride 1): the input is read as one
// sequence of positions, every image row preceded by pad_w zero positions and
// every image by pad_h zero rows.  Tap (i, j) of the output at position q is
// the input at q + i * wp + j (wp = w + pad_w): what lies past a row's or an
// image's end is the next one's padding.  A stage holds the positions of a
// tile and its halo for 64 channels once, and each tap is the same operand
// started i * wp + j positions on (Eq. 7: neighbouring output pixels read
// neighbouring input pixels), so a value is loaded and converted once instead
// of kh * kw times.  Of the columns, only those of the positions past ow and
// oh are wasted (1 - w h / ((w + pad) (h + pad)): 7 % at 28 x 28, pad 1).
//
// Exactness: activations are staged as x - 128 and filters as themselves, both
// exact in fp16.  The accumulator starts at 0 and a chunk's sum of |product|
// is at most 2^24, so every partial sum is an integer that fp32 holds exactly
// and every product a multiple of the accumulator's last place.  Any 1,024
// products fit a chunk; prepared layers carry each filter's sum of |w| per
// stage, which allows longer chunks.  The chunks of a tile stay in TMEM and
// are added as int32 in the epilogue.
//
// Filter operand: kept in shared memory for all of a CTA's tiles when it fits
// (every CTA keeps one block of 128 channels), else brought in per stage and
// tap.  kWConvert: converted from the caller's packed filters by the producers
// (no workspace; the compression constants are derived here as well); kWCopy:
// bulk copies of the fp16 filters that conv_tc_prep_kernel laid out.
//
// Measured per launch (was: general tensor-core kernel for the first three, CUDA
// cores for the others): 28 x 28 x 128 -> 128 3 x 3, batch 64: 16.8 us (49.5);
// 14 x 14 x 256 -> 256 3 x 3: 16.4 us (48.0); 14 x 14 x 256 -> 512 1 x 1: 12.6 us
// (30.7); 56 x 56 x 64 -> 128 3 x 3 stride 2: 20.2 us (1,637); 33 x 45 x 20 -> 44
// 3 x 3, batch 37: 17.0 us (70; 25.4 with a branch per word of an unaligned
// granule; 18.2 on new buffers in each call).  The flat-window layers are bound by
// the MMA warp's issue (an item of four N = 192 MMAs takes 550 cycles, 384 without
// any wait); im2col layers by the latency of the producers' global loads.
//
// Warp roles (one persistent CTA per SM, 18 warps):
//   warps 0-7    producers: global memory -> registers -> staged fp16
//   warps 8-15   epilogue: two per TMEM lane quarter, each on half the columns
//   warp 16      MMA issue
//   warp 17      bulk copies of the filters (kWCopy)
#pragma once

#include <mutex>

#include "conv_common.cuh"
#include "device.cuh"
#include "internal.h"

namespace qnn {
namespace gather {

constexpr int kProdWarps = 8, kEpiWarps = 8;
constexpr int kEpiWarp0 = 8, kMmaWarp = 16, kLoadWarp = 17;
constexpr int kWarps = 18;
constexpr int kThreads = kWarps * 32;
constexpr int kRowsW = 128;          // output channels per tile (MMA M)
constexpr int kSlabGran = 4;         // granules (MMA k-steps) per stage
constexpr int kMaxStages = 8, kMaxW = 9, kMaxSlots = 4;
constexpr int kChunkGranules = 64;   // 64 * 16 products of at most 2^14: 2^24
constexpr int kChunkAbs = 1 << 17;   // 128 * sum |w| <= 2^24
constexpr int kTabled = 256;         // granules whose place is tabulated
constexpr int kMaxAbs = 16;          // stages whose sums of |w| a prepared layer carries
constexpr int kMaxIter = 8;          // pixels per producer thread and stage
constexpr uint32_t kSmemLimit = 232448;  // 227 KB opt-in dynamic shared memory per block
// Planes: 8 K-values of every row, 16 bytes per row.  Where producers write
// them the plane stride is an odd number of 16-byte units: the eight lanes of
// a store phase (two rows by four granules) meet eight different bank groups.
constexpr uint32_t kPlaneW = kRowsW * 16 + 16;
constexpr uint32_t kItemW = 2 * kSlabGran * kPlaneW;
enum { kIm2col = 0, kFlat = 1 };
enum { kWConvert = 0, kWCopy = 1 };

struct Args {
    const uint8_t *x;
    uint8_t *y;
    const uint8_t *w;       // packed filters (kWConvert)
    const int32_t *bias;
    const int16_t *kappa;
    const int32_t *lambda;
    const uint8_t *shifts;
    int shift;
    const uint8_t *wpack;   // kWCopy: fp16 filters [n-tile][K / 8][w_rows][8]
    const int4 *chan;       // kWCopy: [2][n-tiles * w_rows] records
    uint32_t preload;       // kWCopy: what the records subtract from the sums for the general kernel's pre-loads
    const int32_t *wabs;    // kWCopy: sums of |w| [filter][kMaxAbs], or null
    int h, w_, c, m, kh, kw, sh, sw, ph, pw, oh, ow;
    int row_c;              // input bytes per image row (w * c)
    int kwc;                // kw * c
    uint32_t xbytes, wbytes;
    int npix;               // columns in all (im2col: output pixels; flat: positions)
    int images;
    int ncols, mtiles, n_ntiles, mstep;  // columns per tile; tiles; channel blocks; CTAs per channel block
    int npos;               // staged positions (im2col: ncols)
    int wp;                 // flat: positions per row
    int taps, cgr, nxs;     // taps per stage; granules per tap; stages per tile
    int chunk_stages;       // stages per chunk where no sums of |w| are carried
    int stages, w_slots, resident, w_rows, parts;
    int unrolled;           // flat, 3 x 3, nine filter slots
    uint32_t plane_x, stage_bytes, plane_w, item_w, off_x, off_rec, off_bar;
    FastDiv fd_gr;          // granules per kernel row
    FastDiv fd_c;           // channels
    FastDiv fd_pix, fd_row; // columns per image, per row of it
    int *status;
};

struct Shared {
    uint64_t x_full[kMaxStages], x_empty[kMaxStages];
    uint64_t w_full[kMaxW], w_empty[kMaxW];
    uint64_t acc_full[kMaxSlots], acc_empty[kMaxSlots];
    uint64_t done;
    uint32_t tmem;
    int abs_max[kMaxAbs];
    int sums[2][kRowsW];    // per filter: positive part, negative part
    int4 gran[kTabled];     // im2col: kernel row, first byte in it, kernel column, input offset of a granule
};

// One 16-byte granule as loaded: whole (aligned kernels) or the five words it
// overlaps with its position in them and its valid bytes.
template <bool ALIGNED>
struct Gran;

template <>
struct Gran<true> {
    uint4 v;
    __device__ __forceinline__ void zero() { v = make_uint4(0, 0, 0, 0); }
    __device__ __forceinline__ uint4 get() const { return v; }
};

template <>
struct Gran<false> {
    uint32_t q[5];
    uint32_t meta;  // bit shift | first valid byte << 8 | end of the valid bytes << 16
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int k = 0; k < 5; ++k) q[k] = 0;
        meta = 0;
    }
    // bytes [lo, hi) of the 16 at p (any alignment) of the tensor [begin, end): the
    // five aligned words around them, read whole where all lie inside the tensor,
    // else only what overlaps the bytes (one branch, taken at the tensor's ends)
    __device__ __forceinline__ void load(const uint8_t *p, int lo, int hi, const uint8_t *begin, const uint8_t *end)
    {
        const uint32_t sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p) & 3u);
        const uint8_t *a = p - sh;
        meta = (sh * 8u) | static_cast<uint32_t>(lo) << 8 | static_cast<uint32_t>(max(lo, hi)) << 16;
        if (hi > lo && a >= begin && a + 20 <= end) {
            const uint32_t *q4 = reinterpret_cast<const uint32_t *>(a);
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k] = q4[k];
            return;
        }
        const int b0 = lo + static_cast<int>(sh), b1 = hi + static_cast<int>(sh);
#pragma unroll
        for (int k = 0; k < 5; ++k) q[k] = 0;
        if (hi > lo) {
#pragma unroll
            for (int b = 0; b < 20; ++b)
                if (b >= b0 && b < b1) q[b / 4] |= static_cast<uint32_t>(a[b]) << (8 * (b % 4));
        }
    }
    __device__ __forceinline__ uint4 get() const
    {
        const uint32_t sh = meta & 0xFFu;
        const int lo = static_cast<int>((meta >> 8) & 0xFFu), hi = static_cast<int>(meta >> 16);
        uint32_t r[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) r[k] = __funnelshift_r(q[k], q[k + 1], sh);
        if (lo == 0 && hi == 16) return make_uint4(r[0], r[1], r[2], r[3]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // keep bytes [lo, hi) of the granule: byte b of word k is byte 4k + b
            const int l = min(max(lo - 4 * k, 0), 4), e = min(max(hi - 4 * k, 0), 4);
            const uint32_t below_e = e == 4 ? 0xFFFFFFFFu : (1u << (8 * e)) - 1u;
            const uint32_t below_l = l == 4 ? 0xFFFFFFFFu : (1u << (8 * l)) - 1u;
            r[k] &= below_e & ~below_l;
        }
        return make_uint4(r[0], r[1], r[2], r[3]);
    }
};

// Two planes of one row: 16 values as fp16 (flip 0x80808080: signed bytes as
// themselves, 0: unsigned ones minus 128).
__device__ __forceinline__ void store_gran(uint32_t addr, uint32_t plane, uint4 v, uint32_t flip)
{
    sts128(addr, cvt_u8x8(make_uint2(v.x ^ flip, v.y ^ flip)));
    sts128(addr + plane, cvt_u8x8(make_uint2(v.z ^ flip, v.w ^ flip)));
}

// ---------------------------------------------------------------- producers (warps 0-7): filters

// Granule g of filter o (zeros past the kernel row's end and past m).
template <bool ALIGNED>
__device__ __forceinline__ void fetch_w(const Args &a, int o, int g, Gran<ALIGNED> &v)
{
    if (g >= a.cgr || o >= a.m) {
        v.zero();
        return;
    }
    const int i = fdiv(g, a.fd_gr), r = (g - i * static_cast<int>(a.fd_gr.d)) * 16;
    const uint8_t *p = a.w + static_cast<uint32_t>((o * a.kh + i) * a.kwc + r);
    if constexpr (ALIGNED) v.v = *reinterpret_cast<const uint4 *>(p);
    else v.load(p, 0, min(16, a.kwc - r), a.w, a.w + a.wbytes);
}

// Sums of the positive and the negative weights of a granule.
__device__ __forceinline__ void add_sums(uint4 t, int &all, int &neg)
{
    const uint32_t wd[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        all = __dp4a(static_cast<int>(wd[k]), 0x01010101, all);
        // prmt with a sign-replicating selector: 0xFF in every negative byte
        neg = __dp4a(static_cast<int>(wd[k] & prmt(wd[k], 0u, 0xBA98u)), 0x01010101, neg);
    }
}

// The four lanes of a row add up and one of them adds to the row's sums.
__device__ __forceinline__ void put_sums(Shared *sh, int row, int all, int neg)
{
#pragma unroll
    for (int d = 1; d < 4; d <<= 1) {
        all += __shfl_xor_sync(0xffffffffu, all, d);
        neg += __shfl_xor_sync(0xffffffffu, neg, d);
    }
    if ((threadIdx.x & 3) == 0) {
        atomicAdd(&sh->sums[0][row], all - neg);
        atomicAdd(&sh->sums[1][row], neg);
    }
}

// The packed filters of channel block nt, once, stage by stage: the MMA warp
// starts on the first part while the rest is converted.  A thread keeps its
// two rows, so that their sums stay in registers.
template <bool ALIGNED>
__device__ __forceinline__ void convert_filters(const Args &a, uint8_t *smem, Shared *sh, int nt)
{
    constexpr int kBatch = ALIGNED ? 4 : 2;  // stages whose loads go out together (two rows each)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3, pr = lane >> 2;
    const int per_part = (a.nxs + a.parts - 1) / a.parts;
    const uint32_t dst0 = smem_addr(smem) + 2 * q * kPlaneW + (warp * 8 + pr) * 16;
    const int o = nt * kRowsW + warp * 8 + pr;
    // rows with channels (the others' operand is not read for any output)
    const bool two = nt * kRowsW + 64 + warp * 8 < a.m, one = nt * kRowsW + warp * 8 < a.m;
    int all[2] = {0, 0}, neg[2] = {0, 0};
    for (int part = 0; part < a.parts; ++part) {
        const int s1 = min(a.nxs, (part + 1) * per_part);
        for (int s = part * per_part; one && s < s1; s += kBatch) {
            Gran<ALIGNED> v[kBatch][2];
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (s + b < s1 && (h == 0 || two))
                        fetch_w<ALIGNED>(a, o + h * 64, (s + b) * kSlabGran + q, v[b][h]);
                    else
                        v[b][h].zero();
                }
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (s + b < s1 && (h == 0 || two)) {
                        const uint4 t = v[b][h].get();
                        store_gran(dst0 + (s + b) * kItemW + h * 1024, kPlaneW, t, 0x80808080u);
                        add_sums(t, all[h], neg[h]);
                    }
        }
        if (part == a.parts - 1) {
            put_sums(sh, warp * 8 + pr, all[0], neg[0]);
            put_sums(sh, 64 + warp * 8 + pr, all[1], neg[1]);
        }
        fence_proxy_async_smem();
        mbar_arrive(&sh->w_full[part]);
    }
}

// kWConvert without room for the whole filters: every stage's filter operand,
// behind the stage's pixels (warps 4-7).  The sums come from the first tile.
template <bool ALIGNED>
__device__ __forceinline__ void produce_w(const Args &a, uint8_t *smem, Shared *sh, int mt0, int nt)
{
    constexpr int kIter = kRowsW / 32;  // rows per thread
    const int warp = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31, q = lane & 3;
    const int row0 = warp * 8 + (lane >> 2);
    const uint32_t dst0 = smem_addr(smem + a.off_x) + (a.stage_bytes - kItemW) + 2 * q * kPlaneW + row0 * 16;
    int stage = 0;
    uint32_t ph = 0;
    int all[kIter] = {}, neg[kIter] = {};
    for (int mt = mt0; mt < a.mtiles; mt += a.mstep) {
        for (int s = 0; s < a.nxs; ++s) {
            Gran<ALIGNED> v[kIter];
#pragma unroll
            for (int it = 0; it < kIter; ++it)
                fetch_w<ALIGNED>(a, nt * kRowsW + row0 + it * 32, s * kSlabGran + q, v[it]);
            if (!mbar_wait_warp(&sh->x_empty[stage], ph ^ 1u, a.status)) return;
            const uint32_t dst = dst0 + stage * a.stage_bytes;
#pragma unroll
            for (int it = 0; it < kIter; ++it) {
                const uint4 t = v[it].get();
                store_gran(dst + it * 512, kPlaneW, t, 0x80808080u);
                if (mt == mt0) add_sums(t, all[it], neg[it]);
            }
            fence_proxy_async_smem();
            mbar_arrive(&sh->x_full[stage]);
            if (++stage == a.stages) {
                stage = 0;
                ph ^= 1u;
            }
        }
        if (mt == mt0) {
#pragma unroll
            for (int it = 0; it < kIter; ++it) put_sums(sh, row0 + it * 32, all[it], neg[it]);
            mbar_arrive(&sh->w_full[0]);  // the records may be made
        }
    }
}

// ---------------------------------------------------------------- producers: pixels, im2col

// The pixels of a producer thread (columns row0 + it * 32 of a tile): offset of
// the window's origin in the input (modulo 2^32; inputs are smaller than that)
// and its row and column there.
struct Pixels {
    uint32_t base[kMaxIter];
    int16_t iy[kMaxIter], ix[kMaxIter];
};

template <int ITER>
__device__ __forceinline__ void decode_pixels(const Args &a, int mtile, int row0, Pixels &px)
{
#pragma unroll
    for (int it = 0; it < ITER; ++it) {
        const int col = row0 + it * 32, p = mtile * a.ncols + col;
        const int img = fdiv(p, a.fd_pix);
        const int rem = p - img * static_cast<int>(a.fd_pix.d);
        const int oy = fdiv(rem, a.fd_row), ox = rem - oy * a.ow;
        const int iy = oy * a.sh - a.ph, ix = ox * a.sw - a.pw;
        // past the last pixel: outside the image
        px.iy[it] = static_cast<int16_t>(p < a.npix && col < a.ncols ? iy : INT16_MIN);
        px.ix[it] = static_cast<int16_t>(ix);
        px.base[it] = (static_cast<uint32_t>(img * a.h + iy) * static_cast<uint32_t>(a.row_c)) +
                      static_cast<uint32_t>(ix) * static_cast<uint32_t>(a.c);
    }
}

// Where granule g lies: kernel row i, byte r of it, kernel column j (aligned
// kernels), offset from the window's origin.
__device__ __forceinline__ int4 gran_place(const Args &a, int g)
{
    const int i = fdiv(g, a.fd_gr), r = (g - i * static_cast<int>(a.fd_gr.d)) * 16;
    return make_int4(i, r, fdiv(r, a.fd_c), i * a.row_c + r);
}

// Granule g of the thread's pixels.
template <bool ALIGNED, int ITER>
__device__ __forceinline__ void fetch_x(const Args &a, const Shared *sh, const Pixels &px, int g,
                                        Gran<ALIGNED> (&v)[ITER])
{
    const bool in = g < a.cgr;
    const int4 place = a.cgr <= kTabled ? sh->gran[min(g, kTabled - 1)] : gran_place(a, g);
    const int i = place.x, r = place.y;
    const uint32_t off = static_cast<uint32_t>(place.w);
    if constexpr (ALIGNED) {
        const int j = place.z;
#pragma unroll
        for (int it = 0; it < ITER; ++it) {
            const bool ok = in && static_cast<unsigned>(px.iy[it] + i) < static_cast<unsigned>(a.h) &&
                            static_cast<unsigned>(px.ix[it] + j) < static_cast<unsigned>(a.w_);
            v[it].zero();
            if (ok) v[it].v = *reinterpret_cast<const uint4 *>(a.x + (px.base[it] + off));
        }
    } else {
#pragma unroll
        for (int it = 0; it < ITER; ++it) {
            // bytes of the kernel row inside the image: [-ix * c, (w - ix) * c), cut to the granule
            const bool row_ok = in && static_cast<unsigned>(px.iy[it] + i) < static_cast<unsigned>(a.h);
            const int lo = min(16, max(0, -px.ix[it] * a.c - r));
            // (what lies past the kernel row's end meets zero filter values)
            const int hi = row_ok && r < a.kwc ? max(0, min(16, (a.w_ - px.ix[it]) * a.c - r)) : 0;
            // (the offset of byte lo is a true one; the granule's own start may lie before the input)
            v[it].load(a.x + static_cast<uint32_t>(px.base[it] + off + static_cast<uint32_t>(lo)) - lo, lo, hi, a.x,
                       a.x + a.xbytes);
        }
    }
}

// Stages s0, s0 + step, ... of the CTA's sequence (tile by tile) by four warps:
// a column of a tile is taken by four lanes, a granule each.  The loads of the
// next stage are in flight while a stage is converted and stored.
template <bool ALIGNED, int ITER>
__device__ __forceinline__ void produce_x(const Args &a, uint8_t *smem, Shared *sh, int mt0, int s0, int step)
{
    const int warp = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31, q = lane & 3;
    const int row0 = warp * 8 + (lane >> 2);
    const uint32_t dst0 = smem_addr(smem + a.off_x) + 2 * q * a.plane_x + row0 * 16;
    int mt = mt0, s = s0, stage = s0 % a.stages;
    uint32_t ph = static_cast<uint32_t>(s0 / a.stages) & 1u;
    // to the stage's tile; true when that is another one
    auto settle = [&]() {
        bool moved = false;
        while (s >= a.nxs) {
            s -= a.nxs;
            mt += a.mstep;
            moved = true;
        }
        return moved;
    };
    settle();
    if (mt >= a.mtiles) return;
    Pixels px;
    decode_pixels<ITER>(a, mt, row0, px);
    Gran<ALIGNED> va[ITER], vb[ITER];
    fetch_x<ALIGNED, ITER>(a, sh, px, s * kSlabGran + q, va);
    auto turn = [&](Gran<ALIGNED>(&use)[ITER], Gran<ALIGNED>(&load)[ITER]) {
        s += step;
        const bool moved = settle();
        const bool more = mt < a.mtiles;
        if (more) {
            if (moved) decode_pixels<ITER>(a, mt, row0, px);
            fetch_x<ALIGNED, ITER>(a, sh, px, s * kSlabGran + q, load);
        }
        if (!mbar_wait_warp(&sh->x_empty[stage], ph ^ 1u, a.status)) return false;
        const uint32_t dst = dst0 + stage * a.stage_bytes;
#pragma unroll
        for (int it = 0; it < ITER; ++it)
            if (row0 + it * 32 < a.ncols) store_gran(dst + it * 512, a.plane_x, use[it].get(), 0u);
        fence_proxy_async_smem();
        mbar_arrive(&sh->x_full[stage]);
        stage += step;
        if (stage >= a.stages) {
            stage -= a.stages;
            ph ^= 1u;
        }
        return more;
    };
    while (turn(va, vb) && turn(vb, va)) {
    }
}

// ---------------------------------------------------------------- producers: pixels, flat window

// All eight warps on every stage: a position is taken by four lanes, a granule
// each; 64 channels of the tile's positions and their halo.
__device__ __forceinline__ void produce_flat(const Args &a, uint8_t *smem, Shared *sh, int mt0)
{
    constexpr uint32_t kOutside = 0xFFFFFFFFu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3;
    const int row0 = warp * 8 + (lane >> 2);
    const uint32_t dst0 = smem_addr(smem + a.off_x) + 2 * q * a.plane_x + row0 * 16;
    int stage = 0;
    uint32_t ph = 0;
    uint32_t base[kMaxIter];
    uint4 v[kMaxIter];
    auto decode = [&](int mt) {
#pragma unroll
        for (int it = 0; it < kMaxIter; ++it) {
            const int idx = row0 + it * 64, p = mt * a.ncols + idx;
            const int img = fdiv(p, a.fd_pix);
            const int rem = p - img * static_cast<int>(a.fd_pix.d);
            const int r = fdiv(rem, a.fd_row), c = rem - r * a.wp;
            const bool ok = idx < a.npos && img < a.images && r >= a.ph && c >= a.pw;
            base[it] = ok ? static_cast<uint32_t>(img * a.h + r - a.ph) * static_cast<uint32_t>(a.row_c) +
                                static_cast<uint32_t>(c - a.pw) * static_cast<uint32_t>(a.c)
                          : kOutside;
        }
    };
    auto fetch = [&](int s) {
        const int g = s * kSlabGran + q;
#pragma unroll
        for (int it = 0; it < kMaxIter; ++it) {
            v[it] = make_uint4(0, 0, 0, 0);
            if (base[it] != kOutside && g < a.cgr)
                v[it] = *reinterpret_cast<const uint4 *>(a.x + (base[it] + static_cast<uint32_t>(g) * 16u));
        }
    };
    if (mt0 >= a.mtiles) return;
    decode(mt0);
    fetch(0);
    for (int mt = mt0; mt < a.mtiles; mt += a.mstep) {
        for (int s = 0; s < a.nxs; ++s) {
            if (!mbar_wait_warp(&sh->x_empty[stage], ph ^ 1u, a.status)) return;
            const uint32_t dst = dst0 + stage * a.stage_bytes;
#pragma unroll
            for (int it = 0; it < kMaxIter; ++it)
                if (row0 + it * 64 < a.npos) store_gran(dst + it * 1024, a.plane_x, v[it], 0u);
            fence_proxy_async_smem();
            mbar_arrive(&sh->x_full[stage]);
            if (++stage == a.stages) {
                stage = 0;
                ph ^= 1u;
            }
            // the next stage's loads travel while the MMAs of this one run
            if (s + 1 < a.nxs) {
                fetch(s + 1);
            } else if (mt + a.mstep < a.mtiles) {
                decode(mt + a.mstep);
                fetch(0);
            }
        }
    }
}

// ---------------------------------------------------------------- filter copies (warp 17, kWCopy)

__device__ __forceinline__ void copy_filters(const Args &a, uint8_t *smem, Shared *sh, int mt0, int nt)
{
    const uint32_t gran_bytes = static_cast<uint32_t>(a.w_rows) * 32u;
    const uint8_t *src0 = a.wpack + static_cast<size_t>(nt) * a.taps * a.cgr * gran_bytes;
    if (a.resident) {  // all of them, once, in parts
        const int per_part = (a.nxs * a.taps + a.parts - 1) / a.parts;
        if ((threadIdx.x & 31) == 0) {
            for (int part = 0; part < a.parts; ++part) {
                uint32_t total = 0;
                const int i0 = part * per_part, i1 = min(a.nxs * a.taps, i0 + per_part);
                for (int i = i0; i < i1; ++i)
                    total += static_cast<uint32_t>(min(kSlabGran, a.cgr - i / a.taps * kSlabGran)) * gran_bytes;
                mbar_arrive_expect_tx(&sh->w_full[part], total);
                for (int i = i0; i < i1; ++i) {
                    const int s = i / a.taps, tap = i - s * a.taps;
                    bulk_g2s(smem + i * a.item_w, src0 + static_cast<size_t>(tap * a.cgr + s * kSlabGran) * gran_bytes,
                             static_cast<uint32_t>(min(kSlabGran, a.cgr - s * kSlabGran)) * gran_bytes,
                             &sh->w_full[part]);
                }
            }
        }
        __syncwarp();
        for (int part = 0; part < a.parts; ++part) mbar_wait_warp(&sh->w_full[part], 0, a.status);
        return;
    }
    int slot = 0, issued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int mt = mt0; mt < a.mtiles && ok; mt += a.mstep) {
        for (int s = 0; s < a.nxs && ok; ++s) {
            const uint32_t bytes = static_cast<uint32_t>(min(kSlabGran, a.cgr - s * kSlabGran)) * gran_bytes;
            for (int tap = 0; tap < a.taps; ++tap) {
                if (!mbar_wait_warp(&sh->w_empty[slot], ph ^ 1u, a.status)) {
                    ok = false;
                    break;
                }
                if ((threadIdx.x & 31) == 0) {
                    mbar_arrive_expect_tx(&sh->w_full[slot], bytes);
                    bulk_g2s(smem + slot * a.item_w, src0 + static_cast<size_t>(tap * a.cgr + s * kSlabGran) * gran_bytes,
                             bytes, &sh->w_full[slot]);
                }
                __syncwarp();
                ++issued;
                if (++slot == a.w_slots) {
                    slot = 0;
                    ph ^= 1u;
                }
            }
        }
    }
    // every copy lands before the block exits
    for (int k = 0; k < a.w_slots && k < issued; ++k) {
        if (--slot < 0) {
            slot = a.w_slots - 1;
            ph ^= 1u;
        }
        mbar_wait_warp(&sh->w_full[slot], ph, a.status);
    }
}

// ---------------------------------------------------------------- chunks and accumulators

// The chunks of a tile and where they stand in TMEM.
struct Chunks {
    uint32_t ends;   // bit s: a chunk ends with stage s (stages below 32)
    int every;       // stages per chunk past that
    int n;           // chunks
    int regions;     // accumulators handed over together: all chunks of a tile, or 1 with running sums
    int groups;      // hand-overs in flight
    int per_tile;    // hand-overs per tile
    __device__ __forceinline__ bool end(int s, int nxs) const
    {
        return s == nxs - 1 || (s < 32 && every == 0 ? (ends >> s) & 1u : every != 0 && (s + 1) % every == 0);
    }
};

__device__ __forceinline__ void chunk_sync() { asm volatile("bar.sync 2, %0;" ::"n"((kEpiWarps + 1) * 32) : "memory"); }

// Epilogue and MMA warps: from the filters' sums of |w| (the largest of each
// stage over the CTA's filters) where the layer carries them, else by the bound
// that holds for all filters.
template <int WSRC>
__device__ __forceinline__ Chunks make_chunks(const Args &a, Shared *sh, int nt)
{
    Chunks c;
    c.ends = 0;
    c.every = a.chunk_stages;
    c.n = (a.nxs + a.chunk_stages - 1) / a.chunk_stages;
    if (WSRC == kWCopy && a.wabs) {
        const int et = static_cast<int>(threadIdx.x) - kEpiWarp0 * 32;
        const int o = nt * a.w_rows + (et & (kRowsW - 1));
        if (et < kEpiWarps * 32 && (et & (kRowsW - 1)) < a.w_rows)
            for (int s = et / kRowsW; s < a.nxs; s += kEpiWarps * 32 / kRowsW)
                atomicMax(&sh->abs_max[s], a.wabs[static_cast<size_t>(o) * kMaxAbs + s]);
        chunk_sync();
        c.every = 0;
        c.n = 1;
        int sum = 0;
        for (int s = 0; s < a.nxs; ++s) {
            const int v = sh->abs_max[s];
            if (s && sum + v > kChunkAbs) {
                c.ends |= 1u << (s - 1);
                ++c.n;
                sum = 0;
            }
            sum += v;
        }
    }
    const int fit = 512 / a.ncols;  // accumulators that fit in TMEM
    if (c.n <= fit) {
        c.regions = c.n;
        c.groups = min(kMaxSlots, fit / c.n);
        c.per_tile = 1;
    } else {  // one at a time, running sums in the last
        c.regions = 1;
        c.groups = min(kMaxSlots, fit - 1);
        c.per_tile = c.n;
    }
    return c;
}

// ---------------------------------------------------------------- MMA issue (warp 16)

// A value every lane has alike, told to the compiler (uniform registers: the
// MMA's operands then need no moves).
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

__device__ __forceinline__ uint64_t desc_of(uint32_t lo, uint32_t hi)
{
    return (static_cast<uint64_t>(hi) << 32) | lo;
}

// Descriptors of a K-major operand without its start address, as two words.
struct DescWords {
    uint32_t lo, hi;
};

__device__ __forceinline__ DescWords desc_words(uint32_t plane)
{
    const uint64_t t = smem_desc(0, plane, 128);
    return {static_cast<uint32_t>(t), static_cast<uint32_t>(t >> 32)};
}

// The MMAs of one item: one tap of one stage, `steps` granules.  `between` runs
// between the last two of four (see below); its result is returned.
template <class F>
__device__ __forceinline__ bool issue_item(uint32_t d, uint32_t wlo, uint32_t whi, uint32_t xlo, uint32_t xhi,
                                           uint32_t idesc, uint32_t step_w, uint32_t step_x, int steps, uint32_t acc,
                                           F between)
{
    bool ok;
    if (steps == kSlabGran) {
        mma_f16_ss_warp_nc(d, desc_of(wlo, whi), desc_of(xlo, xhi), idesc, acc);
        mma_f16_ss_warp_nc(d, desc_of(wlo + step_w, whi), desc_of(xlo + step_x, xhi), idesc, 1u);
        mma_f16_ss_warp_nc(d, desc_of(wlo + 2 * step_w, whi), desc_of(xlo + 2 * step_x, xhi), idesc, 1u);
        ok = between();
        mma_f16_ss_warp_nc(d, desc_of(wlo + 3 * step_w, whi), desc_of(xlo + 3 * step_x, xhi), idesc, 1u);
    } else {
        for (int k = 0; k < steps; ++k, wlo += step_w, xlo += step_x) {
            mma_f16_ss_warp_nc(d, desc_of(wlo, whi), desc_of(xlo, xhi), idesc, acc);
            acc = 1u;
        }
        ok = between();
    }
    return ok;
}

// The next item's barrier is awaited between the MMAs of this one: a wait
// takes 100 to 200 cycles even when its phase is complete, and the tensor cores
// queue only a few MMAs.
template <int XMODE, int WSRC>
__device__ __forceinline__ void mma_role(const Args &a, uint8_t *smem, Shared *sh, uint32_t tmem0, int mt0,
                                         const Chunks &ck0)
{
    const uint32_t tmem = uniform(tmem0);
    Chunks ck;
    ck.ends = uniform(ck0.ends);
    ck.every = static_cast<int>(uniform(static_cast<uint32_t>(ck0.every)));
    ck.regions = static_cast<int>(uniform(static_cast<uint32_t>(ck0.regions)));
    ck.groups = static_cast<int>(uniform(static_cast<uint32_t>(ck0.groups)));
    const uint32_t idesc = idesc_f16_f32(kRowsW, static_cast<uint32_t>(a.ncols));
    const DescWords wt = desc_words(a.plane_w), xt = desc_words(a.plane_x);
    const uint32_t x16 = xt.lo + (smem_addr(smem + a.off_x) >> 4), w16 = wt.lo + (smem_addr(smem) >> 4);
    const uint32_t step_x = 2 * (a.plane_x >> 4), step_w = 2 * (a.plane_w >> 4), item16 = a.item_w >> 4;
    const uint32_t stage16 = a.stage_bytes >> 4;
    const bool own_w = WSRC == kWCopy || a.resident;  // filters apart from the pixel stages
    const bool ring_w = own_w && !a.resident;
    const int tiles = (a.mtiles - mt0 + a.mstep - 1) / a.mstep;
    const int nxs = a.nxs, last_steps = a.cgr - (nxs - 1) * kSlabGran;
    int stage = 0, wi = 0, group = 0;
    uint32_t x_ph = 0, w_ph = 0, g_ph = 0;
    int stages_left = tiles * nxs;  // stages still to come
    bool ok = mbar_wait_warp(&sh->x_full[0], 0, a.status);
    if (ring_w && ok) ok = mbar_wait_warp(&sh->w_full[0], 0, a.status);
    const int per_part = (nxs * (XMODE == kFlat ? a.taps : 1) + a.parts - 1) / a.parts;
    int part = 0, part_left = 0;  // resident filters: parts still arriving (first tile)
    for (int tile = 0; tile < tiles && ok; ++tile) {
        int region = 0;
        uint32_t acc = 0;  // 0: the next MMA starts a chunk
        uint32_t wres = w16;  // resident filters: the item's
        for (int s = 0; s < nxs && ok; ++s) {
            // (never awaited ahead: with all accumulators in one hand-over it comes after this tile's last MMA)
            if (acc == 0 && region == 0 && !mbar_wait_warp(&sh->acc_empty[group], g_ph ^ 1u, a.status)) {
                ok = false;
                break;
            }
            const uint32_t d = tmem + (group * ck.regions + region) * a.ncols;
            uint32_t xlo = x16 + stage * stage16;
            const int steps = s == nxs - 1 ? last_steps : kSlabGran;
            const int this_stage = stage;
            --stages_left;
            if (++stage == a.stages) {
                stage = 0;
                x_ph ^= 1u;
            }
            auto next_stage = [&]() {
                return stages_left == 0 || mbar_wait_warp(&sh->x_full[stage], x_ph, a.status);
            };
            if (XMODE == kFlat && a.unrolled) {
                // 3 x 3 with a ring slot per tap: the slots, barriers and offsets of a kernel
                // row's taps are constants apart (in the general loop below the scalar work
                // between two items took 270 cycles)
                const bool last = stages_left == 0;
                uint32_t wlo = w16, full = smem_addr(&sh->w_full[0]), drained = smem_addr(&sh->w_empty[0]);
#pragma unroll 1
                for (int ti = 0; ti < 3; ++ti) {
#pragma unroll
                    for (int tj = 0; tj < 3; ++tj) {
                        tc_fence_after();
                        ok &= issue_item(d, wlo + tj * item16, wt.hi, xlo + tj, xt.hi, idesc, step_w, step_x, steps, acc,
                                         [&]() {
                                             if (tj < 2) return mbar_wait_warp_at(full + 8 * (tj + 1), w_ph, a.status);
                                             if (ti < 2) return mbar_wait_warp_at(full + 24, w_ph, a.status);
                                             return last || mbar_wait_warp_at(full - 48, w_ph ^ 1u, a.status);
                                         });
                        mma_commit_warp_at(drained + 8 * tj);
                        acc = 1u;
                    }
                    wlo += 3 * item16;
                    xlo += a.wp;
                    full += 24;
                    drained += 24;
                }
                w_ph ^= 1u;
                mma_commit_warp(&sh->x_empty[this_stage]);
                if (!ok) break;
                ok = next_stage();
            } else if (XMODE == kFlat) {
                int left = a.taps;
                for (int ti = 0; ti < a.kh && ok; ++ti, xlo += a.wp) {
                    for (int tj = 0; tj < a.kw && ok; ++tj) {
                        --left;
                        if (ring_w) {
                            const uint32_t wlo = w16 + wi * item16;
                            uint64_t *const used = &sh->w_empty[wi];
                            if (++wi == a.w_slots) {
                                wi = 0;
                                w_ph ^= 1u;
                            }
                            tc_fence_after();
                            ok = issue_item(d, wlo, wt.hi, xlo + tj, xt.hi, idesc, step_w, step_x, steps, acc, [&]() {
                                return (left == 0 && stages_left == 0) ||
                                       mbar_wait_warp(&sh->w_full[wi], w_ph, a.status);
                            });
                            mma_commit_warp(used);
                        } else {
                            if (tile == 0 && part_left-- == 0) {
                                ok = mbar_wait_warp(&sh->w_full[part++], 0, a.status);
                                part_left = per_part - 1;
                                if (!ok) break;
                            }
                            tc_fence_after();
                            issue_item(d, wres, wt.hi, xlo + tj, xt.hi, idesc, step_w, step_x, steps, acc,
                                       []() { return true; });
                            wres += item16;
                        }
                        acc = 1u;
                    }
                }
                if (!ok) break;
                mma_commit_warp(&sh->x_empty[this_stage]);
                ok = next_stage();
            } else if (own_w) {
                uint32_t wlo = wres;
                uint64_t *used = nullptr;
                if (ring_w) {
                    wlo = w16 + wi * item16;
                    used = &sh->w_empty[wi];
                    if (++wi == a.w_slots) {
                        wi = 0;
                        w_ph ^= 1u;
                    }
                } else if (tile == 0 && part_left-- == 0) {
                    ok = mbar_wait_warp(&sh->w_full[part++], 0, a.status);
                    part_left = per_part - 1;
                    if (!ok) break;
                }
                tc_fence_after();
                ok = issue_item(d, wlo, wt.hi, xlo, xt.hi, idesc, step_w, step_x, steps, acc, [&]() {
                    return next_stage() && (!ring_w || stages_left == 0 ||
                                            mbar_wait_warp(&sh->w_full[wi], w_ph, a.status));
                });
                if (ring_w) mma_commit_warp(used);
                mma_commit_warp(&sh->x_empty[this_stage]);
                wres += item16;
                acc = 1u;
            } else {
                const uint32_t wlo = wt.lo + (xlo - xt.lo) + ((a.stage_bytes - a.item_w) >> 4);
                tc_fence_after();
                ok = issue_item(d, wlo, wt.hi, xlo, xt.hi, idesc, step_w, step_x, steps, acc, next_stage);
                mma_commit_warp(&sh->x_empty[this_stage]);
                acc = 1u;
            }
            if (ck.end(s, nxs)) {
                acc = 0;
                if (++region == ck.regions || s == nxs - 1) {
                    region = 0;
                    mma_commit_warp(&sh->acc_full[group]);
                    if (++group == ck.groups) {
                        group = 0;
                        g_ph ^= 1u;
                    }
                }
            }
        }
    }
    // every issued MMA completes before TMEM is released
    mma_commit_warp(&sh->done);
    mbar_wait_warp(&sh->done, 0, a.status);
}

// ---------------------------------------------------------------- epilogue (warps 8-15)

// The compression record of the lane's channel (as conv_tc_prep_kernel's, with
// acc + bias = s + beta for the integer sum s of the chunks).
template <int WSRC>
__device__ __forceinline__ bool channel_record(const Args &a, Shared *sh, int nt, int row, bool has, int4 &r0, int4 &r1)
{
    const int o = nt * a.w_rows + row;
    if (WSRC == kWCopy) {
        if (has) {
            r0 = a.chan[o];
            r1 = a.chan[a.n_ntiles * a.w_rows + o];
            // (the records are modulo 2^32: lam2 = beta * kappa + lambda)
            r0.x = static_cast<int32_t>(static_cast<uint32_t>(r0.x) + a.preload * static_cast<uint32_t>(r0.y));
            r1.x = static_cast<int32_t>(static_cast<uint32_t>(r1.x) + a.preload);
        }
        return true;
    }
    // the filters' sums are complete
    if (!mbar_wait_warp(&sh->w_full[a.resident ? a.parts - 1 : 0], 0, a.status)) return false;
    if (!has) return true;
    const int32_t b = a.bias ? a.bias[o] : 0;
    const int pos = sh->sums[0][row], ng = sh->sums[1][row];
    const uint32_t beta = static_cast<uint32_t>(b) + 128u * static_cast<uint32_t>(pos + ng);
    const int32_t kap = a.kappa[o], lam = a.lambda[o], shf = a.shifts ? a.shifts[o] : a.shift;
    // every accumulator of this channel lies in [255 * neg, 255 * pos]
    const long long u0 = 255ll * ng + b, u1 = 255ll * pos + b;
    const bool direct = in_i32(u0 * kap + lam) && in_i32(u1 * kap + lam);
    long long ulo = 0, uhi = 0;
    const bool clamp = !direct && saturation_bounds(kap, lam, shf, 255, &ulo, &uhi);
    const int mode = direct ? kModeDirect : clamp ? kModeClamp : kModeWide;
    r0 = make_int4(static_cast<int32_t>(beta * static_cast<uint32_t>(kap) + static_cast<uint32_t>(lam)), kap, shf, mode);
    r1 = make_int4(static_cast<int32_t>(beta), static_cast<int32_t>(ulo), static_cast<int32_t>(uhi), lam);
    return true;
}

// 32 columns of the sums, from the hand-over's regions.
__device__ __forceinline__ void load_sums(uint32_t addr, int regions, uint32_t stride, int (&v)[32])
{
    uint32_t t[32];
    tmem_ld16(addr, *reinterpret_cast<uint32_t(*)[16]>(t));
    tmem_ld16(addr + 16, *reinterpret_cast<uint32_t(*)[16]>(t + 16));
    tmem_wait_ld();
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        asm volatile("" : "+r"(t[k]));  // uses stay after the wait
        v[k] = acc_to_int(t[k], k);
    }
#pragma unroll 1
    for (int r = 1; r < regions; ++r) {
        tmem_ld16(addr + r * stride, *reinterpret_cast<uint32_t(*)[16]>(t));
        tmem_ld16(addr + r * stride + 16, *reinterpret_cast<uint32_t(*)[16]>(t + 16));
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            asm volatile("" : "+r"(t[k]));
            v[k] += acc_to_int(t[k], k);
        }
    }
}

// Output pixel of column p of the whole layer, or -1.
template <int XMODE>
__device__ __forceinline__ int output_pixel(const Args &a, int p)
{
    if (XMODE == kIm2col) return p < a.npix ? p : -1;
    // position -> output pixel; positions past the row's or the image's outputs have none
    const int img = fdiv(p, a.fd_pix);
    const int rem = p - img * static_cast<int>(a.fd_pix.d);
    const int r = fdiv(rem, a.fd_row), c = rem - r * a.wp;
    return c < a.ow && r < a.oh && img < a.images ? (img * a.oh + r) * a.ow + c : -1;
}

// Lane = output channel, 32 columns = output pixels at a time; four lanes
// exchange bytes so that a store holds four channels of a pixel and a warp's
// store four pixels' 32 consecutive bytes.
template <int XMODE, int WSRC>
__device__ __forceinline__ void epilogue_role(const Args &a, Shared *sh, uint32_t tmem, int mt0, int nt)
{
    const Chunks ck = make_chunks<WSRC>(a, sh, nt);
    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int quarter = warp & 3, half = (warp - kEpiWarp0) >> 2;
    const int cw = a.ncols / 2, col0 = half * cw;
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + col0;
    const int row = quarter * 32 + lane;
    const bool has = row < a.w_rows && nt * a.w_rows + row < a.m;
    const bool any = __any_sync(0xffffffffu, has);  // warps past the last channel only hand buffers back
    const uint32_t sel1 = lane & 1 ? 0x3715u : 0x6240u, sel2 = lane & 2 ? 0x3276u : 0x5410u;
    const int ch0 = nt * a.w_rows + quarter * 32 + (lane & ~3);  // first of the four channels the lane stores
    const int nch = max(0, min(4, min(a.m, (nt + 1) * a.w_rows) - ch0));
    const bool words = (a.m & 3) == 0;  // whole aligned words (blocks of filters are multiples of four)
    uint8_t *const ych = a.y + ch0;
    // The lane's constants.  Filters converted stage by stage have their sums once
    // the first tile's last stage is staged, and that may wait for this warp to
    // hand accumulators back: those constants are made when they are first used.
    int4 r0 = make_int4(0, 0, 0, kModeDirect), r1 = make_int4(0, 0, 0, 0);
    bool ready = WSRC == kWCopy || a.resident;
    if (ready && !channel_record<WSRC>(a, sh, nt, row, has, r0, r1)) return;
    const uint32_t sums_addr = lane_addr + ck.groups * a.ncols;  // running sums (per_tile > 1)
    int group = 0;
    uint32_t ph = 0;
    for (int mt = mt0; mt < a.mtiles; mt += a.mstep) {
        for (int hand = 0; hand < ck.per_tile; ++hand) {
            if (!mbar_wait_warp(&sh->acc_full[group], ph, a.status)) return;
            tc_fence_after();
            if (!ready && hand == ck.per_tile - 1) {
                ready = true;
                if (!channel_record<WSRC>(a, sh, nt, row, has, r0, r1)) return;
            }
            const bool direct = __all_sync(0xffffffffu, r0.w == kModeDirect);
            const uint32_t lam2 = static_cast<uint32_t>(r0.x), kap = static_cast<uint32_t>(r0.y);
            const uint32_t shift = static_cast<uint32_t>(r0.z);
            const uint32_t src = lane_addr + group * ck.regions * a.ncols;
#pragma unroll 1
            for (int b0 = 0; any && b0 < cw; b0 += 32) {
                int v[32];
                load_sums(src + b0, ck.regions, a.ncols, v);
                if (ck.per_tile > 1) {
                    uint32_t t[16];
                    if (hand > 0) {
#pragma unroll
                        for (int h = 0; h < 32; h += 16) {
                            tmem_ld16(sums_addr + b0 + h, t);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 16; ++k) v[h + k] += static_cast<int>(t[k]);
                        }
                    }
                    if (hand < ck.per_tile - 1) {
#pragma unroll
                        for (int h = 0; h < 32; h += 16) {
#pragma unroll
                            for (int k = 0; k < 16; ++k) t[k] = static_cast<uint32_t>(v[h + k]);
                            tmem_st16(sums_addr + b0 + h, t);
                        }
                        tmem_wait_st();
                        continue;
                    }
                }
                if (direct) {
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        v[k] = static_cast<int32_t>(static_cast<uint32_t>(v[k]) * kap + lam2) >> shift;
                } else {
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        v[k] = r0.w == kModeDirect
                                   ? static_cast<int32_t>(static_cast<uint32_t>(v[k]) * kap + lam2) >> shift
                                   : static_cast<int>(compress_slow(static_cast<uint32_t>(v[k]), r0, r1, 255u));
                }
                const int p0 = mt * a.ncols + col0 + b0;  // the block's first column
                const int mine = XMODE == kFlat ? output_pixel<XMODE>(a, p0 + lane) : 0;
                // Lane i of four has words of four pixels' bytes of its channel; afterwards
                // it has pixel i's bytes of the four channels.  All eight words go through
                // each step together: one at a time, with its store, took 160 cycles each.
                uint32_t w[8];
#pragma unroll
                for (int g = 0; g < 8; ++g)
                    w[g] = pack2_sat<8>(v[4 * g + 1], v[4 * g], pack2_sat<8>(v[4 * g + 3], v[4 * g + 2], 0u));
#pragma unroll
                for (int g = 0; g < 8; ++g) w[g] = prmt(w[g], __shfl_xor_sync(0xffffffffu, w[g], 1), sel1);
#pragma unroll
                for (int g = 0; g < 8; ++g) w[g] = prmt(w[g], __shfl_xor_sync(0xffffffffu, w[g], 2), sel2);
                int pix[8];
#pragma unroll
                for (int g = 0; g < 8; ++g)
                    pix[g] = XMODE == kFlat ? __shfl_sync(0xffffffffu, mine, 4 * g + (lane & 3))
                                            : output_pixel<XMODE>(a, p0 + 4 * g + (lane & 3));
                if (words) {
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        if (pix[g] >= 0 && nch > 0)
                            *reinterpret_cast<uint32_t *>(ych + static_cast<long long>(pix[g]) * a.m) = w[g];
                } else {
#pragma unroll 1
                    for (int b = 0; b < nch; ++b) {
#pragma unroll
                        for (int g = 0; g < 8; ++g)
                            if (pix[g] >= 0)
                                ych[static_cast<long long>(pix[g]) * a.m + b] = static_cast<uint8_t>(w[g] >> (8 * b));
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->acc_empty[group]);
            if (++group == ck.groups) {
                group = 0;
                ph ^= 1u;
            }
        }
    }
}

// ---------------------------------------------------------------- the kernel

template <bool ALIGNED, int XMODE, int WSRC>
__global__ void __launch_bounds__(kThreads, 1) conv_gather_kernel(const Args a)
{
    extern __shared__ __align__(128) uint8_t smem[];
    Shared *sh = reinterpret_cast<Shared *>(smem + a.off_bar);
    const int warp = threadIdx.x >> 5;
    if (warp == kMmaWarp) {
        if ((threadIdx.x & 31) == 0) {
            // pixel stages: four warps each (im2col), all eight (flat window; converted filters behind the pixels)
            const int x_count = XMODE == kFlat || (WSRC == kWConvert && !a.resident) ? 256 : 128;
            // filters: one copy, or the converting threads (per part; the sums of streamed filters)
            const int w_count = WSRC == kWCopy ? 1 : a.resident ? 256 : 128;
            for (int s = 0; s < kMaxStages; ++s) {
                mbar_init(&sh->x_full[s], x_count);
                mbar_init(&sh->x_empty[s], 1);
            }
            for (int s = 0; s < kMaxW; ++s) {
                mbar_init(&sh->w_full[s], w_count);
                mbar_init(&sh->w_empty[s], 1);
            }
            for (int s = 0; s < kMaxSlots; ++s) {
                mbar_init(&sh->acc_full[s], 1);
                mbar_init(&sh->acc_empty[s], kEpiWarps);
            }
            mbar_init(&sh->done, 1);
            fence_mbar_init();
        }
        __syncwarp();
        tmem_alloc(&sh->tmem, 512);
        tmem_relinquish();
    } else if (warp < kProdWarps) {
        if (threadIdx.x < kMaxAbs) sh->abs_max[threadIdx.x] = 0;
        sh->sums[threadIdx.x / kRowsW][threadIdx.x % kRowsW] = 0;
    } else if (XMODE == kIm2col && warp < kEpiWarp0 + kEpiWarps) {
        const int g = static_cast<int>(threadIdx.x) - kEpiWarp0 * 32;  // kTabled threads
        if (g < a.cgr) sh->gran[g] = gran_place(a, g);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem;
    // everything the previous kernel in the stream wrote is visible from here on
    pdl_wait();

    // the grid is a multiple of the channel blocks: a CTA keeps one block
    const int nt = static_cast<int>(blockIdx.x) % a.n_ntiles, mt0 = static_cast<int>(blockIdx.x) / a.n_ntiles;
    if (warp < kProdWarps) {
        const int group = warp >> 2;
        if constexpr (XMODE == kFlat) {
            produce_flat(a, smem, sh, mt0);
        } else {
            bool pixels = true;
            int s0 = group, step = 2;
            if constexpr (WSRC == kWConvert) {
                if (a.resident) {
                    convert_filters<ALIGNED>(a, smem, sh, nt);
                } else {
                    pixels = group == 0;
                    s0 = 0;
                    step = 1;
                    if (!pixels) produce_w<ALIGNED>(a, smem, sh, mt0, nt);
                }
            }
            if (pixels) {
                if (a.ncols <= 64) produce_x<ALIGNED, 2>(a, smem, sh, mt0, s0, step);
                else if (a.ncols <= 128) produce_x<ALIGNED, 4>(a, smem, sh, mt0, s0, step);
                else produce_x<ALIGNED, 6>(a, smem, sh, mt0, s0, step);
            }
        }
    } else if (warp < kEpiWarp0 + kEpiWarps) {
        epilogue_role<XMODE, WSRC>(a, sh, tmem, mt0, nt);
    } else if (warp == kMmaWarp) {
        const Chunks ck = make_chunks<WSRC>(a, sh, nt);
        // the next kernel in the stream may launch now; it waits for this one before it
        // touches memory
        pdl_trigger();
        mma_role<XMODE, WSRC>(a, smem, sh, tmem, mt0, ck);
    } else if (WSRC == kWCopy) {
        copy_filters(a, smem, sh, mt0, nt);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace gather
}  // namespace qnn
