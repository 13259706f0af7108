// Host side of the gather kernel (conv_gather.cuh): the planner and the launches.
#include <algorithm>

#include "conv_gather.cuh"

namespace qnn {

namespace {

uint32_t round_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }
long long ceil_to(long long v, long long a) { return (v + a - 1) / a; }

}  // namespace

GatherPlan plan_conv_gather(const ConvShape &s, int w_rows, int sms)
{
    using namespace gather;
    GatherPlan p{};
    p.ok = false;
    const bool prepared = w_rows > 0;
    if (s.bits != 8 || s.thr || s.pool || s.oh <= 0 || s.ow <= 0 || s.n < 0) return p;
    // rows and columns, padding included, in 16 bits; offsets in the input and the filters in 32
    if (s.h + 2ll * s.ph > 32767 || s.w + 2ll * s.pw > 32767 || s.kh > 16384) return p;
    if (static_cast<long long>(s.n) * s.h * s.w * s.c > INT32_MAX) return p;
    if (static_cast<long long>(s.m) * s.kh * s.kw * s.c > INT32_MAX) return p;
    p.aligned = s.c % 16 == 0;
    if (prepared && !p.aligned) return p;  // (the prepared layout pads each tap to 16 channels)
    p.w_rows = prepared ? w_rows : kRowsW;
    p.n_ntiles = (s.m + p.w_rows - 1) / p.w_rows;
    if (p.n_ntiles > sms) return p;
    const long long kwc = static_cast<long long>(s.kw) * s.c;
    const long long gr = ceil_to(kwc, 16);
    p.gran_row = static_cast<int>(gr);
    if (gr * s.kh > (1 << 20)) return p;
    const int ngran = static_cast<int>(gr * s.kh), taps = s.kh * s.kw;
    const uint32_t tail = sizeof(Shared);
    long long best = -1;
    for (int mode : {kFlat, kIm2col}) {
        const bool flat = mode == kFlat;
        // the flat window needs stride 1, the fp16 filters by tap and 64-channel stages of at most 1,024 products
        if (flat && (!prepared || taps == 1 || taps > kChunkGranules / kSlabGran || s.sh != 1 || s.sw != 1 ||
                     s.ph >= s.kh || s.pw >= s.kw))
            continue;
        GatherPlan q = p;
        q.flat = flat;
        q.taps = flat ? taps : 1;
        q.cgr = flat ? s.c / 16 : ngran;
        q.nxs = (q.cgr + kSlabGran - 1) / kSlabGran;
        q.chunk_stages = std::max(1, kChunkGranules / kSlabGran / q.taps);
        q.wp = s.w + s.pw;
        const long long cols = flat ? static_cast<long long>(s.n) * (s.h + s.ph) * q.wp
                                    : static_cast<long long>(s.n) * s.oh * s.ow;
        if (cols > INT32_MAX - 4096) continue;
        q.npix = static_cast<int>(cols);
        // unaligned granules take six registers each: at most four columns per producer thread
        for (int ncols : {256, 192, 128, 64}) {
            if (!flat && ncols > (p.aligned ? 192 : 128)) continue;
            q.ncols = ncols;
            q.npos = flat ? ncols + (s.kh - 1) * q.wp + s.kw - 1 : ncols;
            if (q.npos > kMaxIter * 64) continue;
            q.plane_x = static_cast<uint32_t>(flat ? (q.npos + 6) / 8 * 8 + 1 : ncols + 1) * 16;
            const uint32_t x_bytes = 2 * kSlabGran * q.plane_x;
            q.plane_w = prepared ? static_cast<uint32_t>(w_rows) * 16 : kPlaneW;
            q.item_w = 2 * kSlabGran * q.plane_w;
            const long long items = static_cast<long long>(q.nxs) * q.taps;
            uint32_t w_area = 0;
            q.resident = items * q.item_w + 3ll * x_bytes + tail + 256 <= kSmemLimit;
            q.stages = 0;
            q.w_slots = 0;
            q.unrolled = 0;
            if (q.resident) {
                w_area = round_up(static_cast<uint32_t>(items) * q.item_w, 128);
                q.stage_bytes = x_bytes;
                q.stages = static_cast<int>(std::min<uint32_t>(kMaxStages, (kSmemLimit - tail - w_area) / x_bytes));
            } else if (!prepared) {
                q.stage_bytes = x_bytes + q.item_w;
                q.stages = static_cast<int>(std::min<uint32_t>(kMaxStages, (kSmemLimit - tail) / q.stage_bytes));
            } else {
                q.stage_bytes = x_bytes;
                // a flat stage lasts all taps: two or three of them, the rest for the filters
                // (a slot for each tap of a 3 x 3 kernel, where they fit)
                q.unrolled = flat && s.kh == 3 && s.kw == 3 && tail + 2 * x_bytes + 9 * q.item_w + 128 <= kSmemLimit;
                if (q.unrolled) {
                    q.stages = 2;
                    q.w_slots = 9;
                }
                for (int st = flat ? 3 : 5; st >= 2 && !q.unrolled; --st) {
                    if (tail + st * x_bytes + 2 * q.item_w > kSmemLimit) continue;
                    const int slots = static_cast<int>(
                        std::min<uint32_t>(8, (kSmemLimit - tail - st * x_bytes) / q.item_w));
                    if (std::min(slots, flat ? 4 : st) > std::min(q.w_slots, flat ? 4 : q.stages)) {
                        q.stages = st;
                        q.w_slots = slots;
                    }
                }
                w_area = round_up(static_cast<uint32_t>(q.w_slots) * q.item_w, 128);
            }
            if (q.stages < 2) continue;
            q.mtiles = static_cast<int>(ceil_to(cols, ncols));
            q.mstep = std::max(1, std::min(sms / q.n_ntiles, q.mtiles));
            // Tiles per CTA, times the cycles of a tile: per MMA the larger of its own
            // (ncols / 2, at least 48) and those of the shared-memory traffic (operands
            // read, pixels and filters written; 128 bytes per cycle), and about 600 for
            // the first stage and the hand-overs
            const long long traffic = 4096 + 32 * ncols + (flat ? 32ll * q.npos / q.taps : 32ll * ncols) +
                                      (q.resident ? 0 : 4096);
            const long long mma = std::max({48ll, ncols / 2ll, traffic / 128});
            const long long cost = ceil_to(q.mtiles, q.mstep) * (static_cast<long long>(q.taps) * q.cgr * mma + 600);
            if (best >= 0 && cost >= best) continue;
            best = cost;
            q.parts = static_cast<int>(std::min<long long>(4, items));
            q.off_x = w_area;
            q.off_bar = w_area + q.stages * q.stage_bytes;
            // more than half of an SM's shared memory, so that one CTA takes each SM
            q.smem_bytes = std::max<uint32_t>(q.off_bar + tail, 120u * 1024u);
            q.grid = q.mstep * q.n_ntiles;
            q.ok = true;
            p = q;
        }
        if (p.ok) break;
    }
    return p;
}

// The CUDA-core kernel has no pipeline to fill: a few loads per output, and few
// outputs, are done there before the gather kernel's first tile is.  Both times in
// microseconds as measured over 370 random small layers (each within 8 % of the
// CUDA-core kernel's, 15 % of the gather kernel's); of those no choice is more than
// 18 % slower than the other kernel.  50 images of 60 x 29 x 3 -> 23, 1 x 1: 8.7 us
// on CUDA cores, 22.0 here; 36 of 10 x 58 x 1 -> 11, 3 x 3: 6.6 and 10.3; 12 of 41 x 5 x 4
// -> 13, 3 x 4 stride 2: 11.2 and 5.5.
bool direct_beats_gather(const GatherPlan &p, const ConvShape &s, int sms)
{
    const bool words = s.c % 4 == 0;  // four channels per load
    const long long taps = static_cast<long long>(s.kh) * s.kw, loads = taps * (words ? s.c / 4 : s.c);
    if (loads > 20) return false;
    const double waves = static_cast<double>(s.n) * s.oh * s.ow * ((s.m + 7) / 8) / (1024.0 * sms);
    const double filled = loads * std::min(s.m, 8) / 8.0;  // a thread's outputs, of eight
    const double direct = words ? 2.45 + 0.32 * taps + 0.45 * filled + waves * (2.7 + 0.31 * filled)
                                : 2.50 + 0.20 * taps + 0.14 * filled + waves * (3.2 + 0.10 * filled);
    const double rounds = static_cast<double>((p.mtiles + p.mstep - 1) / p.mstep);
    const double gather = 4.5 + 0.9 * rounds * p.nxs + 1.4 * (rounds * p.ncols / 64 - 1);
    return direct < gather;
}

// The general kernel takes layers with prepared filters in less time where the
// gather kernel runs im2col (a kernel of more than 16 taps) and 64 channels of
// filters per step are streamed there, and where few filters stay resident there.
// Times in microseconds as measured over 670 random layers (within 10 % each);
// choosing by them leaves 22 us of the 493 that the gather kernel loses on 49 of the
// layers.  25 images of 6 x 6 x 256 -> 16, 5 x 5: 68.0 us here, 47.0 there; 64 of 32 x
// 32 x 64 -> 64, 7 x 7: 112.7 and 92.3; 15 of 7 x 7 x 256 -> 16, 3 x 3: 14.9 and 12.8; 14 of
// 14 x 14 x 192 -> 280, 5 x 5: 53.2 and 56.6.  In one-shot calls the general kernel starts
// beside the preparation, the gather kernel after it (2.1 us): 44 of 14 x 14 x 80 -> 8,
// 3 x 3, take 12.1 us there and 15.4 here; 327 us lost on 365 layers become 11.
bool general_beats_gather(const GatherPlan &p, const TcPlan &t, int sms, bool one_shot)
{
    if (t.b_resident && t.nt > 32) return false;
    const double rounds = static_cast<double>((p.mtiles + p.mstep - 1) / p.mstep), ksteps = static_cast<double>(p.taps) * p.cgr;
    double gather;
    if (p.flat) {
        gather = p.ncols <= 128   ? 3.1 + rounds * (3.1 + 0.060 * ksteps)
                 : p.ncols == 192 ? 5.4 + rounds * (2.4 + 0.063 * ksteps)
                                  : 4.7 + rounds * (2.7 + 0.084 * ksteps);
    } else {
        gather = p.ncols <= 64    ? 1.9 + rounds * (1.7 + 0.155 * ksteps)
                 : p.ncols <= 128 ? 4.5 + rounds * (1.2 + 0.160 * ksteps)
                                  : 5.5 + rounds * (1.0 + (p.resident ? 0.145 : 0.179) * ksteps);
    }
    const double tiles = static_cast<double>((t.total_tiles + sms - 1) / sms);
    double general;
    if (t.b_resident) {
        general = 4.0 + tiles * (1.5 + 0.034 * t.mmas_per_tile + 0.6 * t.nslab);
    } else {
        const double mma = t.cs == 64 ? (t.nt == 128 ? 0.133 : 0.110) : t.cs == 32 ? 0.19 : 0.36;
        general = 5.9 + tiles * (1.7 + mma * t.mmas_per_tile);
    }
    return general < gather + (one_shot ? 2.1 : 0.0);
}

namespace {

using namespace gather;

template <bool ALIGNED, int XMODE, int WSRC>
cudaError_t launch_one(const Args &a, const GatherPlan &p, cudaStream_t st)
{
    // the opt-in shared-memory limit is raised once per device, outside any stream capture
    static std::mutex mu;
    static bool raised[64] = {};
    auto kern = conv_gather_kernel<ALIGNED, XMODE, WSRC>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        if (!raised[dev]) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
            if (e != cudaSuccess) return e;
            raised[dev] = true;
        }
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(p.grid));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = p.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

Args gather_args(const GatherPlan &p, const ConvShape &s)
{
    Args a{};
    a.h = s.h; a.w_ = s.w; a.c = s.c; a.m = s.m; a.kh = s.kh; a.kw = s.kw;
    a.sh = s.sh; a.sw = s.sw; a.ph = s.ph; a.pw = s.pw; a.oh = s.oh; a.ow = s.ow;
    a.row_c = s.w * s.c;
    a.kwc = s.kw * s.c;
    a.xbytes = static_cast<uint32_t>(s.n) * s.h * s.w * s.c;
    a.wbytes = static_cast<uint32_t>(s.m) * s.kh * s.kw * s.c;
    a.npix = p.npix;
    a.images = s.n;
    a.ncols = p.ncols;
    a.mtiles = p.mtiles;
    a.n_ntiles = p.n_ntiles;
    a.mstep = p.mstep;
    a.npos = p.npos;
    a.wp = p.wp;
    a.taps = p.taps;
    a.cgr = p.cgr;
    a.nxs = p.nxs;
    a.chunk_stages = p.chunk_stages;
    a.stages = p.stages;
    a.w_slots = p.w_slots;
    a.resident = p.resident;
    a.w_rows = p.w_rows;
    a.parts = p.parts;
    a.unrolled = p.unrolled;
    a.plane_x = p.plane_x;
    a.stage_bytes = p.stage_bytes;
    a.plane_w = p.plane_w;
    a.item_w = p.item_w;
    a.off_x = p.off_x;
    a.off_bar = p.off_bar;
    a.fd_gr = make_fastdiv(static_cast<uint32_t>(p.gran_row));
    a.fd_c = make_fastdiv(static_cast<uint32_t>(s.c));
    a.fd_pix = make_fastdiv(static_cast<uint32_t>(p.flat ? (s.h + s.ph) * p.wp : s.oh * s.ow));
    a.fd_row = make_fastdiv(static_cast<uint32_t>(p.flat ? p.wp : s.ow));
    a.status = device_status_ptr();
    return a;
}

}  // namespace

cudaError_t launch_conv_gather(const GatherPlan &p, const ConvShape &s, const ConvParams &c, cudaStream_t st)
{
    if (s.n == 0) return cudaSuccess;
    Args a = gather_args(p, s);
    if (!a.status) return cudaErrorInvalidSymbol;
    a.x = c.x;
    a.y = c.y;
    a.w = c.w;
    a.bias = c.bias;
    a.kappa = c.kappa;
    a.lambda = c.lambda;
    a.shifts = c.shifts;
    a.shift = c.shift;
    return p.aligned ? launch_one<true, kIm2col, kWConvert>(a, p, st) : launch_one<false, kIm2col, kWConvert>(a, p, st);
}

cudaError_t launch_conv_gather_prepared(const GatherPlan &p, const TcPlan &prep, const ConvShape &s, const uint8_t *x,
                                        uint8_t *y, const void *workspace, cudaStream_t st)
{
    if (s.n == 0) return cudaSuccess;
    Args a = gather_args(p, s);
    if (!a.status) return cudaErrorInvalidSymbol;
    a.x = x;
    a.y = y;
    a.wpack = static_cast<const uint8_t *>(workspace);
    a.chan = reinterpret_cast<const int4 *>(a.wpack + conv_tc_chan_offset(prep));
    a.preload = static_cast<uint32_t>(prep.nchunks) * kMagic;
    // the sums of |w| stand behind the records (by 64-channel group: the flat window's stages)
    a.wabs = p.flat && p.nxs <= kMaxAbs ? reinterpret_cast<const int32_t *>(a.chan + 2 * p.n_ntiles * p.w_rows) : nullptr;
    return p.flat ? launch_one<true, kFlat, kWCopy>(a, p, st) : launch_one<true, kIm2col, kWCopy>(a, p, st);
}

}  // namespace qnn
