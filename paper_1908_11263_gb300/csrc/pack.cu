// Sub-byte packing and unpacking (Sec. IV-A, "Sub-byte Extensions"): Q-bit
// values stored 8/Q per byte, element e at bits [(e mod (8/Q)) * Q, +Q) of byte
// e / (8/Q).
//
// Bound by HBM.  A thread moves groups of 16 values: 16 unpacked bytes on one
// side, 2 Q packed ones on the other, kGroups of them a block apart so that all
// their loads are in flight at once.  Measured at 16.8 M INT-2 values packed and
// 8.4 M unpacked: 2.4 and 2.5 us (one byte per thread: 9.5 and 5.7).
#include <algorithm>
#include <cstdint>

#include "device.cuh"
#include "internal.h"

namespace qnn {
namespace {

constexpr int kThreads = 256, kGroups = 4;

template <int BITS>
struct PackedGroup;  // 16 values
template <>
struct PackedGroup<8> {
    using type = uint4;
};
template <>
struct PackedGroup<4> {
    using type = uint2;
};
template <>
struct PackedGroup<2> {
    using type = uint32_t;
};

// The low Q bits of four bytes, packed (2 or 1 bytes).
__device__ __forceinline__ uint32_t pack4_int4(uint32_t w)
{
    w &= 0x0F0F0F0Fu;
    w |= w >> 4;  // bytes 0 and 2: a pair each
    return (w & 0xFFu) | ((w >> 8) & 0xFF00u);
}

__device__ __forceinline__ uint32_t pack4_int2(uint32_t w)
{
    // the four fields meet in the top byte, 2 bits apart; what else the product
    // has stays below bit 24 (3 * (2^22 + 2^20 + 2^18 + 2^14 + 2^12 + 2^6) < 2^24)
    return ((w & 0x03030303u) * 0x01041040u) >> 24;
}

__device__ __forceinline__ uint4 pack16(uint4 v, uint4 *) { return v; }
__device__ __forceinline__ uint2 pack16(uint4 v, uint2 *)
{
    return make_uint2(pack4_int4(v.x) | pack4_int4(v.y) << 16, pack4_int4(v.z) | pack4_int4(v.w) << 16);
}
__device__ __forceinline__ uint32_t pack16(uint4 v, uint32_t *)
{
    return pack4_int2(v.x) | pack4_int2(v.y) << 8 | pack4_int2(v.z) << 16 | pack4_int2(v.w) << 24;
}

// One word of eight nibbles, or one byte of four crumbs, as bytes.
__device__ __forceinline__ uint2 unpack8_int4(uint32_t w, bool is_signed)
{
    uint32_t lo = w & 0x0F0F0F0Fu, hi = (w >> 4) & 0x0F0F0F0Fu;
    if (is_signed) {  // bit 3 into bits 4-7
        lo |= (lo & 0x08080808u) * 0x1Eu;
        hi |= (hi & 0x08080808u) * 0x1Eu;
    }
    return make_uint2(__byte_perm(lo, hi, 0x5140), __byte_perm(lo, hi, 0x7362));
}

__device__ __forceinline__ uint32_t unpack4_int2(uint32_t b, bool is_signed)
{
    uint32_t t = (b | b << 12) & 0x000F000Fu;
    t = (t | t << 6) & 0x03030303u;
    return is_signed ? t | (t & 0x02020202u) * 0x7Eu : t;  // bit 1 into bits 2-7
}

__device__ __forceinline__ uint4 unpack16(uint4 v, bool) { return v; }
__device__ __forceinline__ uint4 unpack16(uint2 v, bool is_signed)
{
    const uint2 a = unpack8_int4(v.x, is_signed), b = unpack8_int4(v.y, is_signed);
    return make_uint4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ uint4 unpack16(uint32_t v, bool is_signed)
{
    return make_uint4(unpack4_int2(v & 0xFFu, is_signed), unpack4_int2((v >> 8) & 0xFFu, is_signed),
                      unpack4_int2((v >> 16) & 0xFFu, is_signed), unpack4_int2(v >> 24, is_signed));
}

// Packed byte i: of the bytes past the last whole group, and every byte of
// tensors that are not aligned for groups.
template <int BITS>
__device__ __forceinline__ void pack_byte(const int8_t *src, uint8_t *dst, long long i)
{
    constexpr int per = 8 / BITS;
    int out = 0;
#pragma unroll
    for (int f = 0; f < per; ++f) out |= (src[i * per + f] & ((1 << BITS) - 1)) << (f * BITS);
    dst[i] = static_cast<uint8_t>(out);
}

template <int BITS>
__device__ __forceinline__ void unpack_byte(const uint8_t *src, int8_t *dst, long long i, int is_signed)
{
    constexpr int per = 8 / BITS;
    const int byte = src[i];
#pragma unroll
    for (int f = 0; f < per; ++f) {
        int v = (byte >> (f * BITS)) & ((1 << BITS) - 1);
        if (is_signed && v >= (1 << (BITS - 1))) v -= (1 << BITS);
        dst[i * per + f] = static_cast<int8_t>(v);
    }
}

// Bytes of a tensor that is not aligned for groups: every thread strides over them.
template <int BITS>
__global__ void __launch_bounds__(kThreads) pack_bytes_kernel(const int8_t *src, uint8_t *dst, long long nbytes)
{
    pdl_wait();
    pdl_trigger();
    const long long step = static_cast<long long>(gridDim.x) * kThreads;
#pragma unroll 1  // (unrolled, every thread divides to learn its number of turns: 1.4 us per wave of blocks)
    for (long long i = static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x; i < nbytes; i += step)
        pack_byte<BITS>(src, dst, i);
}

template <int BITS>
__global__ void __launch_bounds__(kThreads) unpack_bytes_kernel(const uint8_t *src, int8_t *dst, long long nbytes,
                                                                int is_signed)
{
    pdl_wait();
    pdl_trigger();
    const long long step = static_cast<long long>(gridDim.x) * kThreads;
#pragma unroll 1
    for (long long i = static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x; i < nbytes; i += step)
        unpack_byte<BITS>(src, dst, i, is_signed);
}

// groups of 16 values, then packed bytes [2 * Q * groups, nbytes)
template <int BITS>
__global__ void __launch_bounds__(kThreads) pack_kernel(const int8_t *src, uint8_t *dst, long long groups,
                                                        long long nbytes)
{
    using P = typename PackedGroup<BITS>::type;
    pdl_wait();
    pdl_trigger();
    const long long g0 = static_cast<long long>(blockIdx.x) * (kThreads * kGroups) + threadIdx.x;
    uint4 v[kGroups];
#pragma unroll
    for (int k = 0; k < kGroups; ++k)
        if (g0 + k * kThreads < groups) v[k] = reinterpret_cast<const uint4 *>(src)[g0 + k * kThreads];
#pragma unroll
    for (int k = 0; k < kGroups; ++k)
        if (g0 + k * kThreads < groups)
            reinterpret_cast<P *>(dst)[g0 + k * kThreads] = pack16(v[k], static_cast<P *>(nullptr));
    // (fewer than a group's bytes)
    const long long i = groups * 2 * BITS + static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x;
    if (i < nbytes) pack_byte<BITS>(src, dst, i);
}

template <int BITS>
__global__ void __launch_bounds__(kThreads) unpack_kernel(const uint8_t *src, int8_t *dst, long long groups,
                                                          long long nbytes, int is_signed)
{
    using P = typename PackedGroup<BITS>::type;
    pdl_wait();
    pdl_trigger();
    const long long g0 = static_cast<long long>(blockIdx.x) * (kThreads * kGroups) + threadIdx.x;
    P v[kGroups];
#pragma unroll
    for (int k = 0; k < kGroups; ++k)
        if (g0 + k * kThreads < groups) v[k] = reinterpret_cast<const P *>(src)[g0 + k * kThreads];
#pragma unroll
    for (int k = 0; k < kGroups; ++k)
        if (g0 + k * kThreads < groups) reinterpret_cast<uint4 *>(dst)[g0 + k * kThreads] = unpack16(v[k], is_signed != 0);
    // (fewer than a group's bytes)
    const long long i = groups * 2 * BITS + static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x;
    if (i < nbytes) unpack_byte<BITS>(src, dst, i, is_signed);
}

bool aligned(const void *p, int bytes) { return reinterpret_cast<uintptr_t>(p) % bytes == 0; }

unsigned group_blocks(long long groups)
{
    return static_cast<unsigned>((groups + kThreads * kGroups - 1) / (kThreads * kGroups));
}

// One wave of blocks at most: 16.8 M INT-2 values packed from an odd address take
// 5.8 us, 9.9 with a block for every 256 bytes.
unsigned byte_blocks(long long nbytes)
{
    return static_cast<unsigned>(
        std::min((nbytes + kThreads - 1) / kThreads, 2048ll / kThreads * device_sm_count()));
}

}  // namespace

cudaError_t launch_pack(const int8_t *src, uint8_t *dst, long long count, int bits, cudaStream_t st)
{
    const long long nbytes = count * bits / 8;
    if (nbytes == 0) return cudaSuccess;
    // whole groups where both sides are aligned for them
    const long long groups = aligned(src, 16) && aligned(dst, 2 * bits) ? count / 16 : 0;
    if (groups == 0) {
        auto go = [&](auto kern) { return launch_pdl(kern, byte_blocks(nbytes), kThreads, 0, st, src, dst, nbytes); };
        return bits == 8 ? go(pack_bytes_kernel<8>) : bits == 4 ? go(pack_bytes_kernel<4>) : go(pack_bytes_kernel<2>);
    }
    auto go = [&](auto kern) { return launch_pdl(kern, group_blocks(groups), kThreads, 0, st, src, dst, groups, nbytes); };
    return bits == 8 ? go(pack_kernel<8>) : bits == 4 ? go(pack_kernel<4>) : go(pack_kernel<2>);
}

cudaError_t launch_unpack(const uint8_t *src, int8_t *dst, long long count, int bits, int is_signed, cudaStream_t st)
{
    const long long nbytes = count * bits / 8;
    if (nbytes == 0) return cudaSuccess;
    const long long groups = aligned(src, 2 * bits) && aligned(dst, 16) ? count / 16 : 0;
    if (groups == 0) {
        auto go = [&](auto kern) {
            return launch_pdl(kern, byte_blocks(nbytes), kThreads, 0, st, src, dst, nbytes, is_signed);
        };
        return bits == 8   ? go(unpack_bytes_kernel<8>)
               : bits == 4 ? go(unpack_bytes_kernel<4>)
                           : go(unpack_bytes_kernel<2>);
    }
    auto go = [&](auto kern) {
        return launch_pdl(kern, group_blocks(groups), kThreads, 0, st, src, dst, groups, nbytes, is_signed);
    };
    return bits == 8 ? go(unpack_kernel<8>) : bits == 4 ? go(unpack_kernel<4>) : go(unpack_kernel<2>);
}

}  // namespace qnn
