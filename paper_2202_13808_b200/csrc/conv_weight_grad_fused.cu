// Conv2d weight gradient straight from the compressed cache (Eq. 4-5, retained term), bf16, filters of up to 3 x 3:
//   dW[j,c,u,v] = sum_{n,y,x} dY[n,j,y,x] * R(a-hat)[n,c, y*stride+u-pad, x*stride+v-pad]
//
// No dense copy of the input exists in global memory.  A CTA owns 128 output channels j and a block of input channels, walks
// over bands of image rows (or whole small images), and for every band its producer warps
//   * inflate the band's piece of R(a-hat) into shared memory: a lane owns two pixels and builds the 16 bytes of their eight
//     channels from eight mask words (the same for a half-warp), reading the retained values with predicated loads that are
//     contiguous over the warp, so that 16-byte stores write zeros and values alike,
//   * copy the band of dY into shared memory as it is (cp.async; 8 pixels of a channel are 16 bytes, 8 channels a core matrix),
// while one thread feeds the previous band to tcgen05.mma.  dY is the K-major operand: core matrix (8-pixel group of the band) *
// (channels / 8) + channel / 8, without swizzle.  X lies pixel-major: 8 channels (16 bytes) of consecutive pixels of one image
// row follow one another,
//   address = row * row_pitch + (channel / 8) * group_pitch + pixel * 16 + (channel % 8) * 2,
// which is the canonical MN-major layout without swizzle.  In it
//   * the horizontal tap offset v is a start address 16 * v bytes further on (no shifted copies: with the 128-byte swizzle
//     or with pixels innermost an offset of one pixel could not be expressed),
//   * the filter rows u are extra columns of the product: row_pitch = (channels / 8) * group_pitch, so the column groups
//     behind the block's last one are the next image row, and N = R * channels in one instruction,
//   * rows need no common multiple: the two 8-pixel halves of a K = 16 step may lie in different rows (the descriptor's
//     K stride says how far apart they are).
// Stride 2 keeps the even and the odd padded columns in separate planes.  The reduction is split over the CTAs; every split
// stores its accumulator as it comes out of tensor memory and a second kernel adds the splits in order.
//
// Bound by filling the stages: some 400 warp instructions per 64 pixels x 8 channels of X, everything included (13.7 M for 64 -> 64 on
// 56 x 56), at four warps a scheduler, which wait for the values' trip through L2 and for shared memory (issue slots 40 % busy); both lanes'
// pixels of a pair share one mask lookup, the mask words are requested a task ahead and the loads of a warp's first task are under way before it
// waits for the stage, so that one trip to memory per band is exposed.  The taps of a K step share the dY operand in the collector.  16
// producer warps: 20 (80 registers) are up to 8 % slower.  64 images, gamma 0.8, graph replay, a whole call / filling by itself / the product by
// itself / launches, epilogue and reduction (by handing over stages that were not filled, and by leaving all MMAs but one out): 3 x 3
// 64 -> 64 on 56 x 56 36.1 / 21.4 / 13.1 / 10.7 us (525 MMAs of 128 x 96 x 16 at 49 cycles, the full rate; half of their rows are unused),
// 256 -> 256 on 14 x 14 34.0 / 15.5 / 9.2 / 15.2, 512 -> 512 on 7 x 7 53.9 / 25.4 / 9.0 / 24.8, 128 -> 128 on 28 x 28 33.3 / 17.1 / 9.0 / 13.0, stride 2
// 128 -> 128 on 56 x 56 53.2 / 37.8 / 7.7 / 14.9.  Where it came from, over rotating inputs: dense copies of conv_weight_grad_tc.cu (decompression,
// shifted or gathered copies, GEMM on 64-pixel rows) -> dY transposed through registers -> dY copied as it lies, before the reduction had
// forms: 64 -> 64 on 56 x 56 59 -> 50 -> 37 us, 28 x 28 131 -> 39 -> 36, 14 x 14 125 -> 45 -> 43, 7 x 7 334 -> 86 -> 81, stride 2 on 56 x 56
// 213 -> 59 -> 55; 1 x 1 of stride 2 256 -> 512 on 56 x 56 292 -> 129 -> 117.
#include <cstring>
#include <type_traits>

#include "weight_grad_common.cuh"

namespace dropit {

namespace {

constexpr int kProdWarps = 16;                       // four per lane quarter of the accumulator in the epilogue
constexpr int kThreads = 32 * (kProdWarps + 1);      // producer warps, then the MMA warp
constexpr int kMaxStages = 4;
constexpr int kMaxPairs = 64;                        // K = 16 steps of a band
constexpr size_t kSmemBudget = 222 * 1024;

struct FusedConvParams {
    int B, Ca, H, W, Cz, Ho, Wo;                     // flat (1x1, stride 1): H = Ho = 1, W = Wo = pixels of the plane
    int R, S, stride, pad;
    int cb, mt;                                      // channels per block (multiple of 16), rows of dY kept per band (64 or 128)
    int flat;
    int yb, ni;                                      // output rows per band; images per band (> 1 only for whole images)
    int xb;                                          // flat: pixels per band
    int cores;                                       // 8-pixel groups per output row
    int gp;                                          // pixels per channel group and row of X (one plane)
    int planes;                                      // column parities kept (1 or 2)
    int row_step, x_rows;                            // X rows per output row; X rows of one image in a band
    int in_step;                                     // input rows per X row
    // the X side of a band: segments of consecutive input pixels (a whole image's rows, or one row where every other row is
    // skipped), cut into slots of 64 pixels, in the order [channel group][image][segment][slot]
    int segs, seg_pixels, seg_slots, slots;          // segments of an image, pixels and slots of a segment, slots of the band
    uint32_t seg_magic, segs_magic, ni_magic;        // slot / seg_slots = (slot * seg_magic) >> 20 and so on
    uint32_t w_magic;                                // pixel / W
    uint32_t cores_magic, yb_magic, step_magic;      // core / cores, row / yb, dY task / dY steps
    uint32_t s_magic;                                // tap / S
    int x_bytes, dy_bytes, stages;                   // per pipeline stage
    int vec;                                         // pixels per copy of dY that the row length allows: 8, 4, 2, 1
    int dy_warp0, dy_idle, dy_extra;                 // see next_dy: first warp without a task of X in the last round, their number, their share
    int bands, bands_total, bands_per_split, splits; // bands per image (or per group of images); over the batch; per CTA
    int tiles_c, tiles_j;
    int ncols, chunks;                               // accumulator columns R * S * cb; 32-column chunks
    uint32_t tmem_cols;
    uint32_t k;
    const uint16_t *dy, *values;                     // for mend_nonfinite
    const uint32_t *mask, *offsets;
    uint2 pairs[kMaxPairs];                          // low descriptor words of a band's K = 16 steps, relative to the stage: dY, X
};

struct FusedConvCtl {
    uint64_t full[kMaxStages], empty[kMaxStages], accum;
    uint32_t tmem_base;
    int abort_flag;
    alignas(16) uint2 home[kProdWarps][2];   // per producer warp: where the slots of its task go
    uint2 meta[kProdWarps][32];  // ... [word of a task][channel] (mask bits, position of their first value)
};

// x / d for x * d < 2^20, with magic = 2^20 / d + 1
__host__ __device__ __forceinline__ uint32_t magic_of(uint32_t d) { return (1u << 20) / d + 1u; }
__host__ __device__ __forceinline__ uint32_t quotient(uint32_t x, uint32_t magic) { return (x * magic) >> 20; }

// Shared-memory matrix descriptor without swizzle.  Low word: start address and the distance between the two core matrices of a
// K = 16 step; high word: the distance between groups of eight rows (dY) or columns (X), and the descriptor version.
__host__ __device__ __forceinline__ uint32_t desc_low(uint32_t addr, uint32_t k_stride) { return (addr >> 4) | ((k_stride >> 4) << 16); }
__device__ __forceinline__ uint64_t desc_of(uint32_t low, uint32_t high) { return (uint64_t)low | ((uint64_t)high << 32); }
__device__ __forceinline__ uint32_t desc_high(uint32_t mn_stride) { return (mn_stride >> 4) | (1u << 14); }

__device__ __forceinline__ void sts_zero16(uint32_t addr) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
}

// Asynchronous copy of `bytes` (0 or BYTES) to shared memory, zeros for the rest.
template <int BYTES>
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const uint16_t* src, uint32_t bytes) {
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// *p if `bit` is not zero, else 0; a predicated load, not a branch.
__device__ __forceinline__ uint32_t ldg_u16_if(const uint16_t* p, uint32_t bit) {
    uint32_t v;
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u32 %0, 0;\n\t@p ld.global.nc.u16 %0, [%1];\n\t}"
        : "=r"(v) : "l"(p), "r"(bit));
    return v;
}

// The values of two neighbouring elements of a 32-element word of the mask, bits bit0 and bit0 + 1; pos = position of the
// word's first value.
__device__ __forceinline__ void load_two(const uint16_t* __restrict__ values, uint32_t word, uint32_t pos, uint32_t bit0, uint32_t& v0,
                                         uint32_t& v1) {
    const uint32_t b = word >> bit0;
    const uint16_t* src = values + (pos + __popc(word & ((1u << bit0) - 1u)));
    v0 = ldg_u16_if(src, b & 1u);
    v1 = ldg_u16_if(src + (b & 1u), b & 2u);
}

struct Place {
    uint32_t group, img, seg, pixel;     // pixel: of the slot's first element inside the segment
};
__device__ __forceinline__ Place place_of(const FusedConvParams& p, uint32_t index, int groups) {
    Place r;
    const uint32_t a = quotient(index, p.seg_magic), b = quotient(a, p.segs_magic);
    r.pixel = (index - a * p.seg_slots) * 64;
    r.seg = a - b * p.segs;
    r.group = quotient(b, p.ni_magic);
    r.img = b - r.group * p.ni;
    return r;
}

// Channels of a task of dY: half as many where its loads would otherwise take the registers that the prefetched values need.
__host__ __device__ constexpr int dy_task_channels(int vec) { return vec <= 2 ? 32 : 64; }

// VEC: pixels per copy of dY that the row length allows (8: rows are whole aligned 16-byte groups; 4; 2; 1: rows that start anywhere,
// through registers)
template <int VEC>
__global__ void __launch_bounds__(kThreads, 1)
conv_wg_fused_kernel(const uint16_t* __restrict__ dy, const uint16_t* __restrict__ values, const uint32_t* __restrict__ mask,
                     const uint32_t* __restrict__ offsets, const __grid_constant__ FusedConvParams p, float* __restrict__ partial,
                     int32_t* dev_status, uint32_t wait_limit) {
    extern __shared__ __align__(128) uint8_t csm[];
    constexpr int kChannels = dy_task_channels(VEC);
    const int warp = __shfl_sync(kFullMask, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform
    const int stage_bytes = p.x_bytes + p.dy_bytes;
    const uint32_t smem0 = ptx::smem_u32(csm);
    FusedConvCtl* ctl = reinterpret_cast<FusedConvCtl*>(csm + (size_t)p.stages * stage_bytes);
    const int tile = blockIdx.x, split = blockIdx.y;
    const int c0 = (tile % p.tiles_c) * p.cb, j0 = (tile / p.tiles_c) * kBM;
    const int band0 = split * p.bands_per_split;
    const int nb = min(p.bands_total, band0 + p.bands_per_split) - band0;     // >= 1

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            ptx::mbar_init(&ctl->full[s], kProdWarps);
            ptx::mbar_init(&ctl->empty[s], 1);
        }
        ptx::mbar_init(&ctl->accum, 1);
        ctl->abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (warp == kProdWarps) {
        ptx::tmem_alloc(&ctl->tmem_base, p.tmem_cols);
        ptx::tmem_relinquish();
    }
    const uint32_t row_pitch = (uint32_t)(p.cb / 8) * p.gp * 16, core_pitch = (uint32_t)p.mt * 16;
    // padding columns, and the rows of dY behind a band's last one, are read but never written: zero
    for (int i = threadIdx.x; i < p.stages * stage_bytes / 16; i += kThreads) sts_zero16(smem0 + i * 16);
    const int total_cores = p.ni * p.yb * p.cores, pairs = (total_cores + 1) / 2;
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    volatile int* abort_flag = &ctl->abort_flag;
    ptx::grid_dependency_wait();

    if (warp < kProdWarps) {
        // ---------------- producers ----------------
        const uint32_t nwords = (uint32_t)(((int64_t)p.B * p.Ca * p.H * p.W + 31) / 32);
        const uint32_t plane_elems = (uint32_t)p.H * p.W, plane_pitch = (uint32_t)p.x_bytes / p.planes;
        const int groups = p.cb / 8, x_tasks = (p.slots + 1) / 2;
        const int dy_steps = (total_cores + 3) / 4, dy_tasks = dy_steps * (p.mt / kChannels);
        const size_t dy_plane = (size_t)p.Ho * p.Wo;
        [[maybe_unused]] const size_t dy_total = dy_plane * p.Cz * p.B;
        const int dy_rank = (warp + kProdWarps - p.dy_warp0) % kProdWarps;
        // the warps without a task of X in the last round take the first dy_extra tasks of dY, all warps share the others
        const int dy_first = dy_rank < p.dy_idle && p.dy_extra > 0 ? dy_rank : p.dy_extra + dy_rank;
        auto next_dy = [&](int t) {
            if (t >= p.dy_extra) return t + kProdWarps;
            return t + p.dy_idle < p.dy_extra ? t + p.dy_idle : p.dy_extra + dy_rank;
        };
        const int slot = lane >> 3, sub = lane & 7;
        uint2* meta = ctl->meta[warp];
        uint2* home = ctl->home[warp];
        const uint32_t bit0 = (2u * lane) & 31u;       // the lane's first pixel in its 32-pixel word
        int n0 = (band0 / p.bands) * p.ni, piece = band0 % p.bands;      // image and piece of the image
        // ---- X: a task is two slots, a slot 64 consecutive pixels of 8 channels.  The mask bits of its four 32-pixel words per
        // channel and the position of their first value (lane = (channel sub, word slot)) are requested a task ahead, across bands
        struct Bits { uint4 chunk; uint32_t next, first, at, lead, len; };
        auto request = [&](uint32_t index, int n_first, int piece_of) {
            const int yi0 = piece_of * p.yb * p.stride - p.pad, kx0 = p.flat ? piece_of * p.xb : 0;
            const int run_end = p.flat ? min(p.W, kx0 + p.xb) : (int)plane_elems;   // no pixel of the plane from here on
            Bits r;
            r.chunk = make_uint4(0, 0, 0, 0);
            r.next = r.first = r.at = r.lead = r.len = 0;
            if (index >= 2u * p.slots) return r;
            Place at = place_of(p, index >> 1, groups);
            at.pixel += (index & 1u) * 32;
            const int row = yi0 + (int)at.seg * p.in_step;                     // first input row of the segment
            const int px = (p.flat ? kx0 : row * p.W) + (int)at.pixel;
            const int c = c0 + (int)at.group * 8 + sub;
            int lo = max(px, 0), hi = min(min(px + 32, run_end), px + p.seg_pixels - (int)at.pixel);
            if (n_first + (int)at.img < p.B && c < p.Ca && lo < hi) {
                r.at = ((uint32_t)(n_first + at.img) * p.Ca + c) * plane_elems + lo;   // flat index of the slot's first element
                r.lead = lo - px;
                r.len = hi - lo;
                const uint32_t ch = r.at >> 7, w1 = (r.at >> 5) + 1;
                r.first = __ldg(offsets + ch);
                if (w1 < nwords) r.next = __ldg(mask + w1);
                if (ch * 4 + 3 < nwords) {
                    r.chunk = __ldg(reinterpret_cast<const uint4*>(mask) + ch);
                } else {                             // the tensor's last chunk may be short
                    r.chunk.x = __ldg(mask + ch * 4);
                    if (ch * 4 + 1 < nwords) r.chunk.y = __ldg(mask + ch * 4 + 1);
                    if (ch * 4 + 2 < nwords) r.chunk.z = __ldg(mask + ch * 4 + 2);
                }
            }
            return r;
        };
        auto record = [&](const Bits& r) {
            const uint32_t in = (r.at >> 5) & 3u, sh = r.at & 31u;
            uint32_t m = r.chunk.x, pos = r.first;
            if (in > 0) { pos += __popc(m); m = r.chunk.y; }
            if (in > 1) { pos += __popc(m); m = r.chunk.z; }
            if (in > 2) { pos += __popc(m); m = r.chunk.w; }
            pos += __popc(m & ((1u << sh) - 1u));
            uint32_t bits = __funnelshift_r(m, r.next, sh);
            if (r.len < 32) bits &= (1u << r.len) - 1u;
            if (pos + __popc(bits) > p.k) bits = 0;   // a table that does not match the mask must not read past the values
            return make_uint2(bits << r.lead, pos);
        };
        Bits ahead = request(warp * 4 + slot, n0, piece);
        for (int i = 0; i < nb; ++i) {
            const int s = i % p.stages;
            const int y0 = p.flat ? 0 : piece * p.yb, k0 = p.flat ? piece * p.xb : 0;
            const bool turn = piece + 1 == p.bands;                        // the next band opens another image
            const int next_n = turn ? n0 + p.ni : n0, next_piece = turn ? 0 : piece + 1;
            const uint32_t xbuf = smem0 + s * stage_bytes, ybuf = xbuf + p.x_bytes;
            // ---- dY: a task is four 8-pixel groups of 64 or 32 channels; a lane copies one group of the channels sub, sub + 8, ...
            struct DyPlace { int core, row, xc, jset; bool live; };
            auto dy_place = [&](int t) {
                DyPlace r;
                r.jset = (int)quotient(t, p.step_magic);
                r.core = (t - r.jset * dy_steps) * 4 + slot;
                r.live = r.core < total_cores;
                r.row = (int)quotient(r.core, p.cores_magic);
                r.xc = r.core - r.row * p.cores;
                return r;
            };
            // the first channel's source and the pixels that exist there (not positive: none); where it goes
            auto dy_source = [&](const DyPlace& at, int& nv) {
                const int img = (int)quotient(at.row, p.yb_magic), y = y0 + at.row - img * p.yb, x = k0 + at.xc * 8;
                nv = n0 + img < p.B && y < p.Ho ? min(8, p.Wo - x) : 0;
                return dy + ((size_t)(n0 + img) * p.Cz + j0 + at.jset * kChannels + sub) * dy_plane + (size_t)y * p.Wo + x;
            };
            auto dy_target = [&](const DyPlace& at) { return ybuf + at.core * core_pitch + (at.jset * kChannels + sub) * 16; };
            [[maybe_unused]] auto copy_dy = [&](int t) {
                const DyPlace at = dy_place(t);
                if (!at.live) return;
                int nv;
                const uint16_t* src = dy_source(at, nv);
                size_t step = 8 * dy_plane;
                if (nv <= 0) { src = dy; step = 0; }                       // zeros, from a valid address
                uint32_t dst = dy_target(at);
                const int left = p.Cz - (j0 + at.jset * kChannels + sub);
#pragma unroll
                for (int g = 0; g < kChannels / 8; ++g) {
                    if (g * 8 < left) {
#pragma unroll
                        for (int h = 0; h < 8; h += VEC) cp_async_zfill<VEC * 2>(dst + h * 2, src + (h < nv ? h : 0), h < nv ? VEC * 2 : 0);
                    }
                    dst += 128;
                    src += step;
                }
            };
            // Rows that are not 8-byte aligned (copied 4 bytes at a time, asynchronously, 256 -> 256 on 14 x 14 took 57 us instead of 43) go through registers: the aligned words around the piece, shifted by half a word for odd
            // starts.  The loads of the warp's first task are issued before it waits for the stage and works on X.
            [[maybe_unused]] auto load_dy = [&](int t, uint32_t (&w)[kChannels / 8][4]) {
                const DyPlace at = dy_place(t);
                int nv;
                const uint16_t* src = dy_source(at, nv);
                if (!at.live) nv = 0;
                const int left = p.Cz - (j0 + at.jset * kChannels + sub);
#pragma unroll
                for (int g = 0; g < kChannels / 8; ++g) {
                    w[g][0] = w[g][1] = w[g][2] = w[g][3] = 0;
                    if constexpr (VEC == 2) {
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            if (2 * h < nv && g * 8 < left) w[g][h] = __ldg(reinterpret_cast<const uint32_t*>(src) + h);
                    } else if (nv > 0 && g * 8 < left) {
                        const size_t at0 = (size_t)(src - dy);
                        const uint32_t odd = (uint32_t)at0 & 1u;
                        const uint32_t* words = reinterpret_cast<const uint32_t*>(dy) + (at0 >> 1);
                        uint32_t raw[5];
#pragma unroll
                        for (int h = 0; h < 5; ++h) {
                            raw[h] = 0;
                            if (2 * h < nv + (int)odd) {     // the tensor's last element may have no right neighbour
                                if (((at0 >> 1) + h) * 2 + 1 < dy_total) raw[h] = __ldg(words + h);
                                else raw[h] = __ldg(reinterpret_cast<const uint16_t*>(words + h));
                            }
                        }
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            w[g][h] = odd ? __funnelshift_r(raw[h], raw[h + 1], 16) : raw[h];
                            if (2 * h + 1 >= nv) w[g][h] &= 2 * h < nv ? 0xFFFFu : 0u;   // pixels of the next row
                        }
                    }
                    src += 8 * dy_plane;
                }
            };
            [[maybe_unused]] auto store_dy = [&](int t, const uint32_t (&w)[kChannels / 8][4]) {
                const DyPlace at = dy_place(t);
                if (!at.live) return;
                const uint32_t dst = dy_target(at);
#pragma unroll
                for (int g = 0; g < kChannels / 8; ++g)
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst + g * 128), "r"(w[g][0]), "r"(w[g][1]), "r"(w[g][2]),
                                 "r"(w[g][3]) : "memory");
            };
            // The retained values of a task are loaded into registers (a slot at a time: the lane gets the 8 channels of its two
            // pixels), then stored; for the warp's first task of the band the loads are on their way before it waits for the stage.
            uint4 x4[4];
            auto load_x = [&](int t) {
                meta[lane] = record(ahead);
                if (lane < 2) {
                    const uint32_t index = t * 2 + lane;
                    const Place at = place_of(p, index, groups);
                    home[lane] = make_uint2(xbuf + (at.img * p.x_rows + at.seg) * row_pitch + at.group * p.gp * 16,
                                            index < (uint32_t)p.slots ? at.pixel : (uint32_t)p.seg_pixels);
                }
                const bool more = t + kProdWarps < x_tasks;
                if (more || i + 1 < nb)
                    ahead = request((more ? t + kProdWarps : warp) * 4 + slot, more ? n0 : next_n, more ? piece : next_piece);
                __syncwarp();
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t v[2][8];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const uint4 m = reinterpret_cast<const uint4*>(meta)[(q * 2 + (lane >> 4)) * 4 + h];
                        load_two(values, m.x, m.y, bit0, v[0][2 * h], v[1][2 * h]);
                        load_two(values, m.z, m.w, bit0, v[0][2 * h + 1], v[1][2 * h + 1]);
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        x4[2 * q + e] = make_uint4(v[e][0] | (v[e][1] << 16), v[e][2] | (v[e][3] << 16), v[e][4] | (v[e][5] << 16),
                                                   v[e][6] | (v[e][7] << 16));
                }
            };
            auto store_x = [&]() {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint2 at = home[q >> 1];       // where the slot's first pixel is: segment's address, pixel of the segment
                    const uint32_t rel = at.y + 2 * lane + (q & 1);
                    bool keep = rel < (uint32_t)p.seg_pixels;
                    uint32_t x = rel, to = at.x;
                    if (!p.flat) {
                        const uint32_t row = quotient(rel, p.w_magic);
                        x = rel - row * p.W + p.pad;
                        to += row * row_pitch;
                        if (p.stride == 2) {             // even and odd columns in separate planes
                            if (x & 1u) {
                                keep = keep && p.planes == 2;
                                to += plane_pitch;
                            }
                            x >>= 1;
                        }
                    }
                    if (keep)
                        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(to + x * 16), "r"(x4[q].x), "r"(x4[q].y),
                                     "r"(x4[q].z), "r"(x4[q].w) : "memory");
                }
                __syncwarp();                            // the records may be overwritten
            };
            [[maybe_unused]] uint32_t w[kChannels / 8][4];
            if (warp < x_tasks) load_x(warp);
            if constexpr (VEC <= 2)
                if (dy_first < dy_tasks) load_dy(dy_first, w);
            if (i >= p.stages) {
                const bool ok = ptx::mbar_wait_warp(&ctl->empty[s], ((i / p.stages) - 1) & 1, wait_limit);
                if (!ok) *abort_flag = 1;
            }
            if (__any_sync(kFullMask, *abort_flag != 0)) break;
            if constexpr (VEC > 2)
                for (int t = dy_first; t < dy_tasks; t = next_dy(t)) copy_dy(t);
            if (warp < x_tasks) store_x();
            for (int t = warp + kProdWarps; t < x_tasks; t += kProdWarps) {
                load_x(t);
                store_x();
            }
            if constexpr (VEC > 2) {
                asm volatile("cp.async.wait_all;" ::: "memory");
            } else {
                for (int t = dy_first; t < dy_tasks; t = next_dy(t)) {
                    if (t != dy_first) load_dy(t, w);
                    store_dy(t, w);
                }
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&ctl->full[s]);
            n0 = next_n;
            piece = next_piece;
        }
        ptx::launch_dependents();
        // ---------------- epilogue: the accumulator leaves in the order it has in tensor memory ----------------
        bool ok = ptx::mbar_wait_warp(&ctl->accum, 0, wait_limit);
        if (!ok || *abort_flag) {
            *abort_flag = 1;
        } else {
            ptx::tc_fence_after();
            const int quarter = warp & 3;
            if (j0 + 32 * quarter < p.Cz) {
                float4* plane = reinterpret_cast<float4*>(partial) + ((size_t)split * gridDim.x + tile) * p.chunks * 8 * kBM;
                for (int ch = warp >> 2; ch < p.chunks; ch += kProdWarps / 4) {
                    uint32_t r[32];
                    ptx::tmem_ld_32x32(tmem_base + ((uint32_t)(32 * quarter) << 16) + ch * 32, r);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int e4 = 0; e4 < 8; ++e4)
                        __stcg(plane + (size_t)(ch * 8 + e4) * kBM + 32 * quarter + lane,
                               make_float4(__uint_as_float(r[4 * e4]), __uint_as_float(r[4 * e4 + 1]), __uint_as_float(r[4 * e4 + 2]),
                                           __uint_as_float(r[4 * e4 + 3])));
                }
            }
        }
    } else {
        // ---------------- MMA issuer (the whole warp runs the loop, one thread issues) ----------------
        const uint32_t leader = ptx::elect_one();
        const uint32_t n_inst = (uint32_t)(p.R * p.cb);
        const uint32_t idesc = ptx::make_idesc_bf16(kBM, (int)n_inst, false, true);
        const uint32_t high_a = desc_high(128), high_b = desc_high(p.gp * 16);
        const uint32_t plane_pitch = (uint32_t)p.x_bytes / p.planes;
        // where a horizontal tap's columns start, in descriptor units
        const uint32_t shift1 = (p.stride == 2 ? plane_pitch : 16u) >> 4, shift2 = (p.stride == 2 ? 16u : 32u) >> 4;
        for (int i = 0; i < nb; ++i) {
            const int s = i % p.stages;
            if (!__all_sync(kFullMask, !*abort_flag && ptx::mbar_wait_spin(&ctl->full[s], (i / p.stages) & 1, wait_limit))) {
                *abort_flag = 1;
                break;
            }
            ptx::tc_fence_after();
            const uint32_t stage = (smem0 + s * stage_bytes) >> 4;
            // The horizontal taps of a K step share its dY operand, which is read from shared memory once: the MMAs would
            // otherwise take all of its bandwidth (128 x 96 x 16: 7 KB per 48 cycles).
            using ptx::CollectA;
            const auto steps = [&](auto taps) {
                constexpr int S = decltype(taps)::value;
#pragma unroll 2
                for (int q = 0; q < pairs; ++q) {
                    const uint64_t ad = desc_of(p.pairs[q].x + stage, high_a);
                    const uint32_t b_low = p.pairs[q].y + stage, acc = (i > 0 || q > 0) ? 1u : 0u;
                    ptx::umma_bf16_elected<S == 1 ? CollectA::kDiscard : CollectA::kFill>(tmem_base, ad, desc_of(b_low, high_b), idesc, acc, leader);
                    if constexpr (S > 1)
                        ptx::umma_bf16_elected<S == 2 ? CollectA::kLastUse : CollectA::kUse>(tmem_base + n_inst, ad, desc_of(b_low + shift1, high_b),
                                                                                             idesc, acc, leader);
                    if constexpr (S > 2)
                        ptx::umma_bf16_elected<CollectA::kLastUse>(tmem_base + 2 * n_inst, ad, desc_of(b_low + shift2, high_b), idesc, acc, leader);
                }
            };
            if (p.S == 1) steps(std::integral_constant<int, 1>{});
            else if (p.S == 2) steps(std::integral_constant<int, 2>{});
            else steps(std::integral_constant<int, 3>{});
            if (leader) ptx::umma_commit(&ctl->empty[s]);
            __syncwarp();
        }
        if (leader) ptx::umma_commit(&ctl->accum);      // also after an abort: it then tells when the MMAs in flight are done
        __syncwarp();
        ptx::mbar_wait_warp(&ctl->accum, 0, kWaitLimit);   // no MMA may be in flight when tensor memory is freed
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kProdWarps) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, p.tmem_cols);
    }
    if (*abort_flag && threadIdx.x == 0 && dev_status) atomicExch(dev_status, (int)DROPIT_ERR_TIMEOUT);
}

// Number of retained elements in front of flat index e; `kept`: whether e is one of them.
__device__ __forceinline__ uint32_t retained_before(const uint32_t* __restrict__ mask, const uint32_t* __restrict__ offsets, uint32_t e,
                                                    bool& kept) {
    const uint32_t w = e >> 5, bit = 1u << (e & 31u), word = __ldg(mask + w);
    uint32_t pos = __ldg(offsets + (e >> 7)) + __popc(word & (bit - 1u));
#pragma unroll
    for (uint32_t i = 1; i < 4; ++i)
        if ((w & 3u) >= i) pos += __popc(__ldg(mask + (w - i)));
    kept = (word & bit) != 0;
    return pos;
}

constexpr int kRedWarps = 8;

// Where the sums of a block of the reduction go, and its output: 32 rows of dW from j0 on, TAPS taps from tap0 on of four channels from c on
// (CHANNELS, 1 x 1 filters: 4 * TAPS channels).
template <int FORM_TAPS, bool CHANNELS>
struct RedBlock {
    static constexpr int kTaps = CHANNELS ? 1 : FORM_TAPS, kChannels = CHANNELS ? 4 * FORM_TAPS : 4;
    static constexpr int kRowFloats = kTaps * kChannels, kPitch = kRowFloats + 1;      // a row of the sums, [channel][tap]
    int c, j0, tap0;
    __device__ __forceinline__ void store(const FusedConvParams& p, const float* sums, float* __restrict__ dw, int accumulate) const {
        const int taps = p.R * p.S;
        for (int i = threadIdx.x; i < 32 * kRowFloats; i += 32 * kRedWarps) {
            const int row = i / kRowFloats, e = i - row * kRowFloats, ch = e / kTaps;
            if (j0 + row < p.Cz && c + ch < p.Ca) {
                float* d = dw + ((size_t)(j0 + row) * p.Ca + c + ch) * taps + tap0 + (e - ch * kTaps);
                const float v = sums[row * kPitch + e];
                *d = accumulate ? *d + v : v;
            }
        }
    }
};

// The channels c .. c + chs - 1 (chs < 32) that hold an infinity or a NaN, a bit each.  Called by the whole block; a warp takes an image's
// channels, whose values follow one another in the cache, in one go (lane i: the values in front of channel c + i).
__device__ __forceinline__ uint32_t nonfinite_channels(const FusedConvParams& p, int c, int chs, uint32_t* found) {
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const uint32_t plane = (uint32_t)p.H * p.W, total = (uint32_t)p.B * p.Ca * plane;
    if (threadIdx.x == 0) *found = 0;
    __syncthreads();
    for (int n = g; n < p.B; n += kRedWarps) {
        const uint32_t e = ((uint32_t)n * p.Ca + c + min(lane, chs)) * plane;
        bool kept;
        const uint32_t at = e < total ? min(retained_before(p.mask, p.offsets, e, kept), p.k) : p.k;
        const uint32_t first = __shfl_sync(kFullMask, at, 0), last = __shfl_sync(kFullMask, at, chs);
        bool odd = false;
        for (uint32_t i = first + lane; i < last; i += 32) odd |= (__ldg(p.values + i) & 0x7F80u) == 0x7F80u;
        if (!__any_sync(kFullMask, odd)) continue;
        for (int ch = 0; ch < chs; ++ch) {
            const uint32_t from = __shfl_sync(kFullMask, at, ch), to = __shfl_sync(kFullMask, at, ch + 1);
            odd = false;
            for (uint32_t i = from + lane; i < to; i += 32) odd |= (__ldg(p.values + i) & 0x7F80u) == 0x7F80u;
            if (odd) atomicOr(found, 1u << ch);
        }
    }
    __syncthreads();
    return *found;
}

// The sums in `out` ([row][channel][tap]) that are not finite, of the channels that hold an infinity or a NaN: added up again term by term.
// The K steps cover whole 8-pixel groups; behind a row's last output and behind the band's last group dY is zero there, but X may be a
// pixel that the tap does not see, and zero times infinity is NaN.
// A thread looks up what its pixel of dY meets at each tap, a round of 256 pixels ahead; then a warp goes over the 256 pixels with four rows of
// dY, whose loads are contiguous.  A channel is searched once for all of its taps.  64 images, gamma 0.8, nothing odd / one infinity in
// X / one NaN in dY: 256 -> 256 on 14 x 14 34 / 297 / 40 us (with the taps one after the other, each searching, and a lane per row of dY,
// whose loads are 32 sectors: 1369 / 359; the same in nine times as many blocks, one per tap: 222 / 98); 512 -> 512 on 7 x 7 54 / 114 / 60
// (481 / 300; 138 / 144); 64 -> 64 on 56 x 56, one tap per block either way, 36 / 2390 / 94 (2330 / 151).
// What bounds it: two barriers and the trips to L2 in every round, on the few SMs that have such a channel.
// Called by the whole block, whose sums it stores: it is not part of the kernel's own code, whose registers it would take, and nothing of that is
// kept across the call.
template <int TAPS>
struct MendShared {
    uint32_t x[kRedWarps][TAPS][32];       // bf16 in the upper half; bit 0: retained
    size_t from[kRedWarps * 32];           // the pixel in the first row of dY
    uint32_t found;
};
template <typename Block>
__device__ __noinline__ void mend_nonfinite(const FusedConvParams& p, const Block blk, float* out, MendShared<Block::kTaps>& sh,
                                            float* __restrict__ dw, int accumulate) {
    constexpr int TAPS = Block::kTaps, kRows = 32 / kRedWarps;
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, c = blk.c;
    const uint32_t dy_plane = (uint32_t)p.Ho * p.Wo, pixels = (uint32_t)p.B * dy_plane;
    const int j = min(blk.j0 + g * kRows, p.Cz - 1), more = p.Cz - 1 - j;       // (behind the last row: not used)
    for (uint32_t todo = nonfinite_channels(p, c, min(Block::kChannels, p.Ca - c), &sh.found); todo; todo &= todo - 1u) {
        const int ch = __ffs(todo) - 1;
        float acc[kRows][TAPS];
#pragma unroll
        for (int r = 0; r < kRows; ++r)
#pragma unroll
            for (int t = 0; t < TAPS; ++t) acc[r][t] = 0.f;
        uint32_t met[TAPS];                                 // looked up one round ahead
        size_t at_dy;
        auto look_up = [&](uint32_t q0) {
            const uint32_t q = min(q0 + threadIdx.x, pixels - 1u), n = q / dy_plane, at = q - n * dy_plane;
            const int y = (int)(at / p.Wo) * p.stride - p.pad, x = (int)(at % p.Wo) * p.stride - p.pad;
            int u = blk.tap0 / p.S, v = blk.tap0 - u * p.S;
            at_dy = (size_t)n * p.Cz * dy_plane + at;
#pragma unroll
            for (int t = 0; t < TAPS; ++t) {
                const int iy = y + u, ix = x + v;
                const bool in = q0 + threadIdx.x < pixels && iy >= 0 && iy < p.H && ix >= 0 && ix < p.W;
                bool kept;
                const uint32_t pos = retained_before(p.mask, p.offsets, in ? ((n * p.Ca + c + ch) * p.H + iy) * p.W + ix : 0u, kept);
                const uint32_t value = __ldg(p.values + min(pos, p.k - 1u));
                met[t] = in && kept && pos < p.k ? value << 16 | 1u : 0u;
                if (++v == p.S) { v = 0; ++u; }
            }
        };
        look_up(0);
        for (uint32_t q0 = 0; q0 < pixels; q0 += 32 * kRedWarps) {
            __syncthreads();                                // the pixels before these are done with
            sh.from[threadIdx.x] = at_dy;
#pragma unroll
            for (int t = 0; t < TAPS; ++t) sh.x[g][t][lane] = met[t];
            __syncthreads();
            if (q0 + 32 * kRedWarps < pixels) look_up(q0 + 32 * kRedWarps);
#pragma unroll(TAPS == 1 ? 2 : 4)
            for (int w = 0; w < kRedWarps; ++w) {
                const uint16_t* src = p.dy + sh.from[w * 32 + lane] + (size_t)j * dy_plane;
                float d[kRows];
#pragma unroll
                for (int r = 0; r < kRows; ++r) d[r] = __uint_as_float((uint32_t)__ldg(src + (size_t)min(r, more) * dy_plane) << 16);
#pragma unroll
                for (int t = 0; t < TAPS; ++t) {
                    const uint32_t xv = sh.x[w][t][lane];
                    if (xv & 1u) {
#pragma unroll
                        for (int r = 0; r < kRows; ++r) acc[r][t] = fmaf(d[r], __uint_as_float(xv & 0xFFFF0000u), acc[r][t]);
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r)
#pragma unroll
            for (int t = 0; t < TAPS; ++t) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[r][t] += __shfl_xor_sync(kFullMask, acc[r][t], o);
                float* sum = out + (g * kRows + r) * Block::kPitch + ch * TAPS + t;
                if (lane == 0 && !isfinite(*sum)) *sum = acc[r][t];
            }
    }
    __syncthreads();
    blk.store(p, out, dw, accumulate);
}

// dw[j,c,u,v] (=|+=) sum over splits, in split order within a warp's share and then over the warps.  A block takes 32 rows, four
// channels and TAPS of the filter's taps (CHANNELS, 1 x 1 filters: TAPS times four channels); its eight warps share out the splits.
// Sums that are not finite are looked at again (mend_nonfinite).
// All taps of a channel in one block write whole stretches of dW (144 bytes of a row of 3 x 3 filters, where one tap wrote 4 bytes in
// every 36), keep nine loads per thread in flight and are a ninth of the blocks.  256 -> 256 on 14 x 14, 64 images, against one tap per block:
// 4.9 sectors a store request instead of 32, 130 k sectors written to L2 instead of 885 k, 2.5 M warp instructions instead of 10.9 M; per call
// 43.3 -> 35.0 us, 512 -> 512 on 7 x 7 82.2 -> 57.6, stride 2 256 -> 256 on 28 x 28 64.3 -> 56.1 (with the divisions behind the loads 33.8, 53.5, 53.6).
template <int TAPS, bool CHANNELS = false>
__global__ void __launch_bounds__(32 * kRedWarps, TAPS == 1 ? 5 : (TAPS < 9 ? 4 : 2))
conv_fused_reduce_kernel(const float4* __restrict__ partial, const __grid_constant__ FusedConvParams p, float* __restrict__ dw, int accumulate) {
    using Block = RedBlock<TAPS, CHANNELS>;
    constexpr int kPitch = Block::kPitch;
    __shared__ float4 sums[kRedWarps][TAPS][32];
    __shared__ float out[32 * kPitch];                  // [row][channel][tap]
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    // Blocks: (32 rows, groups of channels and sets of taps, block of channels).  The columns of the partial tiles are in the order [v][u][channel]:
    // with one tap per block, or none but channels, blockIdx.y counts them as they lie.  What else the block's number says is worked out behind
    // the loads: with the divisions in front of them calls of 8 images took 14.7 instead of 13.6 us (64 -> 64 on 56 x 56), 13.1 / 11.8 (40 -> 72
    // on 23 x 23), 32.7 / 28.7 (512 -> 512 on 7 x 7).
    const int groups = p.cb / Block::kChannels, j0 = 32 * blockIdx.x, quarter = blockIdx.x % (kBM / 32);
    const int tile = (int)(blockIdx.x / (kBM / 32)) * p.tiles_c + blockIdx.z, c0 = blockIdx.z * p.cb;
    const int tap_set = TAPS == 3 ? (int)blockIdx.y / groups : 0;      // (nine taps are all there are)
    int group = (int)blockIdx.y - tap_set * groups;
    const uint32_t first = CHANNELS ? group * TAPS : group;
    ptx::grid_dependency_wait();                        // the partial tiles come from the kernel before this one
    // Groups behind the last channel; one tap per block has to divide to tell, and does so later.
    if (TAPS > 1 && c0 + group * Block::kChannels >= p.Ca) return;
    const size_t plane = (size_t)p.tiles_c * p.tiles_j * p.chunks * 8 * kBM;
    const float4* src = partial + ((size_t)tile * p.chunks * 8 + first) * kBM + 32 * quarter + lane;
    uint32_t at[TAPS];
#pragma unroll
    for (int t = 0; t < TAPS; ++t) {
        if constexpr (TAPS == 9) at[t] = (uint32_t)(t % 3 * 3 + t / 3) * groups * kBM;
        else if constexpr (TAPS == 3) {
            const uint32_t tap = tap_set * TAPS + t, u = quotient(tap, p.s_magic), v = tap - u * p.S;
            at[t] = (v * p.R + u) * groups * kBM;
        } else at[t] = (uint32_t)t * kBM;
    }
    constexpr int kTapFloats = CHANNELS ? 4 : 1, kChFloats = CHANNELS ? 1 : TAPS;      // how far apart in a row of `out`
    float4 acc[TAPS];
#pragma unroll
    for (int t = 0; t < TAPS; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    int s = g;
    // Splits whose loads are in flight: as many as fit the registers; the 16 channels' form hardly ever has more than two for a warp
    constexpr int kDeep = TAPS == 1 ? 4 : (TAPS == 3 ? 2 : 1);
    if constexpr (kDeep > 1) {
        for (; s + (kDeep - 1) * kRedWarps < p.splits; s += kDeep * kRedWarps) {
            float4 x[kDeep][TAPS];
#pragma unroll
            for (int w = 0; w < kDeep; ++w)
#pragma unroll
                for (int t = 0; t < TAPS; ++t) x[w][t] = __ldcg(src + (size_t)(s + w * kRedWarps) * plane + at[t]);
#pragma unroll
            for (int w = 0; w < kDeep; ++w)
#pragma unroll
                for (int t = 0; t < TAPS; ++t) { acc[t].x += x[w][t].x; acc[t].y += x[w][t].y; acc[t].z += x[w][t].z; acc[t].w += x[w][t].w; }
        }
    }
    for (; s < p.splits; s += kRedWarps) {
        float4 x[TAPS];
#pragma unroll
        for (int t = 0; t < TAPS; ++t) x[t] = __ldcg(src + (size_t)s * plane + at[t]);
#pragma unroll
        for (int t = 0; t < TAPS; ++t) { acc[t].x += x[t].x; acc[t].y += x[t].y; acc[t].z += x[t].z; acc[t].w += x[t].w; }
    }
#pragma unroll
    for (int t = 0; t < TAPS; ++t) sums[g][t][lane] = acc[t];
    int tap0 = tap_set * TAPS;
    if constexpr (TAPS == 1) {
        const int column = group / groups, v = column / p.R;
        group -= column * groups;
        tap0 = (column - v * p.R) * p.S + v;
    }
    const int c = c0 + group * Block::kChannels;
    if (TAPS == 1 && c >= p.Ca) return;
    __syncthreads();
    bool odd = false;
    for (int i = threadIdx.x; i < 32 * TAPS; i += 32 * kRedWarps) {
        const int t = i >> 5, row = i & 31;
        float4 a = sums[0][t][row];
#pragma unroll
        for (int w = 1; w < kRedWarps; ++w) {
            const float4 o = sums[w][t][row];
            a.x += o.x; a.y += o.y; a.z += o.z; a.w += o.w;
        }
        float* o = out + row * kPitch + t * kTapFloats;
        o[0] = a.x; o[kChFloats] = a.y; o[2 * kChFloats] = a.z; o[3 * kChFloats] = a.w;
        odd |= !isfinite(a.x * 0.f + a.y * 0.f + a.z * 0.f + a.w * 0.f) && j0 + row < p.Cz;   // one of the four is not finite
    }
    const Block blk = {c, j0, tap0};
    if (__syncthreads_or(odd)) {
        using Mend = MendShared<Block::kTaps>;
        static_assert(sizeof(Mend) <= sizeof(sums), "");
        mend_nonfinite(p, blk, out, reinterpret_cast<Mend&>(sums), dw, accumulate);      // (the sums have been read)
        return;
    }
    blk.store(p, out, dw, accumulate);
}

size_t stage_bytes_of(FusedConvParams& p) {
    const size_t row_pitch = (size_t)(p.cb / 8) * p.gp * 16;
    // With an odd number of 8-pixel groups the last K = 16 step reads one more K row than the band has: zeros in dY,
    // pixels or zeros in X (mend_nonfinite mends what infinities make of that).  With 64 channels of dY per band the instruction's rows 64..127 are the next 8-pixel group
    // (their results are not used).
    const int odd = (p.ni * p.yb * p.cores) & 1;
    const size_t x = (size_t)(p.ni * p.x_rows + odd * p.row_step) * row_pitch * p.planes;
    const size_t y = (size_t)(p.ni * p.yb * p.cores + odd + (p.mt == 64 ? 1 : 0)) * p.mt * 16;
    p.x_bytes = (int)align_up(x, 128 * p.planes);
    p.dy_bytes = (int)align_up(y, 128);
    return (size_t)p.x_bytes + p.dy_bytes;
}

bool make_fused_conv_plan(FusedConvParams& p, int B, int Ca, int H, int W, int Cz, int R, int S, int stride, int pad, int64_t k) {
    p = FusedConvParams{};
    if (R > 3 || S > 3 || stride > 2 || pad > 2 || B < 1) return false;
    p.B = B; p.Ca = Ca; p.Cz = Cz; p.R = R; p.S = S; p.stride = stride; p.pad = pad; p.k = (uint32_t)k;
    p.H = H; p.W = W;
    p.Ho = (H + 2 * pad - R) / stride + 1;
    p.Wo = (W + 2 * pad - S) / stride + 1;
    p.flat = R == 1 && S == 1 && stride == 1 && pad == 0;
    if (p.flat) { p.W = p.Wo = H * W; p.H = p.Ho = 1; }
    const int cb_max = (256 / R < 512 / (R * S) ? 256 / R : 512 / (R * S)) / 16 * 16;   // N <= 256 columns, 512 of tensor memory
    const int blocks = (Ca + cb_max - 1) / cb_max;
    p.cb = (int)align_up((size_t)(Ca + blocks - 1) / blocks, 16);
    p.mt = Cz > 64 ? 128 : 64;
    p.planes = stride == 2 && S > 1 ? 2 : 1;
    p.row_step = R == 1 ? 1 : stride;
    p.in_step = R == 1 ? stride : 1;
    p.tiles_c = (Ca + p.cb - 1) / p.cb;
    p.tiles_j = (Cz + kBM - 1) / kBM;
    p.stages = 2;
    p.vec = p.Wo % 8 == 0 ? 8 : (p.Wo % 4 == 0 ? 4 : (p.Wo % 2 == 0 ? 2 : 1));
    // What a task of dY costs, in tasks of X; fitted: with half of it or twice as much the bands chosen are up to a quarter slower
    // where rows are odd, and 5 to 10 % where they are even.
    const float dy_cost = p.vec >= 4 ? 0.2f : (p.vec == 2 ? 0.3f : 0.6f);
    const int64_t tiles = (int64_t)p.tiles_c * p.tiles_j;
    if (tiles > 65535) return false;
    // 1 x 1 filters of stride 2: every block of 128 outputs inflates X again, for a single tap and in slots of 64 pixels that a short
    // row fills by less than half (0.84 us per million elements of all slots).  From some size on the dense copies, made once, are ahead, if
    // there are channels enough for their GEMM: batch 64, 1024 -> 2048 on 14 x 14 (470 M elements) 401 against 358 us, 512 -> 2048 on
    // 28 x 28 411 / 346; batch 128 760 / 614 and 841 / 625.  Not so below (batch 64, 512 -> 1024 on 28 x 28, 235 M: 197 / 209), with fewer channels
    // (batch 128, 256 -> 1024 on 28 x 28 197 / 262) or on longer rows (batch 64, 512 -> 1280 on 40 x 40 350 / 527).
    if (R == 1 && S == 1 && stride == 2 && W <= 32 && Ca >= 512 && (int64_t)p.tiles_j * B * Ca * p.Ho * 64 >= 240000000) return false;
    if (!p.flat) {
        p.cores = (p.Wo + 7) / 8;
        // columns an 8-pixel group of any tap can reach, at the plane's resolution
        const int reach = p.cores * 8 + (S - 1) / stride + 1, padded = ((W + 7) / 8 * 8 + pad + stride - 1) / stride + 1;
        p.gp = reach > padded ? reach : padded;
    }
    // An image in `pieces` equal bands (pieces == 1: `ni` images in one band); returns what the slowest CTA takes, in units
    // of a producer task, or -1 if such a band does not fit.  A band costs half a task on top of its rounds of tasks
    // (handing the stage over, waiting for the product of the band before last).
    auto set_band = [&](int pieces, int ni) -> float {
        p.ni = ni;
        if (p.flat) {
            p.xb = (int)align_up((size_t)(p.W + pieces - 1) / pieces, pieces > 1 ? 32 : 16);
            p.cores = p.xb / 8;
            p.gp = p.xb + 1;
            p.yb = 1;
            p.bands = (p.W + p.xb - 1) / p.xb;
        } else {
            p.yb = (p.Ho + pieces - 1) / pieces;
            p.bands = (p.Ho + p.yb - 1) / p.yb;
        }
        p.x_rows = (p.yb - 1) * p.row_step + R;
        if (p.ni * p.yb * p.cores > 2 * kMaxPairs || stage_bytes_of(p) * p.stages + sizeof(FusedConvCtl) + 128 > kSmemBudget) return -1.f;
        p.bands_total = (B + ni - 1) / ni * p.bands;
        p.segs = p.in_step > 1 ? p.x_rows : 1;
        p.seg_pixels = p.flat ? p.xb : (p.in_step > 1 ? W : p.x_rows * W);
        p.seg_slots = (p.seg_pixels + 63) / 64;
        p.slots = p.seg_slots * p.segs * p.ni * (p.cb / 8);
        int splits = (int)(sm_count() / tiles);
        if (splits < 1) splits = 1;
        if (splits > p.bands_total) splits = p.bands_total;
        p.bands_per_split = (p.bands_total + splits - 1) / splits;
        p.splits = (p.bands_total + p.bands_per_split - 1) / p.bands_per_split;
        const int x_tasks = (p.slots + 1) / 2, dy_tasks = (p.ni * p.yb * p.cores + 3) / 4 * (p.mt / dy_task_channels(p.vec));
        p.dy_warp0 = x_tasks % kProdWarps;
        p.dy_idle = p.dy_warp0 ? kProdWarps - p.dy_warp0 : 0;
        p.dy_extra = p.dy_idle * (int)(1.f / dy_cost);
        const int shared = dy_tasks > p.dy_extra ? dy_tasks - p.dy_extra : 0;
        return p.bands_per_split * (0.5f + (float)((x_tasks + kProdWarps - 1) / kProdWarps) + (float)((shared + kProdWarps - 1) / kProdWarps) * dy_cost);
    };
    int best_pieces = 0, best_ni = 0;
    float best = 0.f;
    // (no more than 64 pieces are tried: a plane of more than 128 rows that fits shared memory only row by row is refused)
    const int most_pieces = p.flat ? (p.W + 31) / 32 : p.Ho;
    for (int pieces = 1; pieces <= most_pieces && pieces <= 64; ++pieces) {
        if (!p.flat && pieces > 1 && (p.Ho + pieces - 1) / pieces == (p.Ho + pieces - 2) / (pieces - 1)) continue;
        for (int ni = 1; ni <= (pieces == 1 ? B : 1); ++ni) {
            const float cost = set_band(pieces, ni);
            if (cost < 0.f) break;
            if (best_ni == 0 || cost < best) { best = cost; best_pieces = pieces; best_ni = ni; }
        }
    }
    if (best_ni == 0) return false;
    set_band(best_pieces, best_ni);
    const int cores_total = p.ni * p.yb * p.cores;
    p.seg_magic = magic_of((uint32_t)p.seg_slots);
    p.segs_magic = magic_of((uint32_t)p.segs);
    p.ni_magic = magic_of((uint32_t)p.ni);
    p.w_magic = magic_of((uint32_t)W);
    p.s_magic = magic_of((uint32_t)S);
    p.cores_magic = magic_of((uint32_t)p.cores);
    p.yb_magic = magic_of((uint32_t)p.yb);
    p.step_magic = magic_of((uint32_t)((cores_total + 3) / 4));
    // what the division by multiplication and the table of K steps can take
    const int64_t most = p.slots + 2 * kProdWarps + 2;
    if (cores_total > 2 * kMaxPairs || most * p.seg_slots >= (1 << 20) || most * p.segs >= (1 << 20) || most * p.ni >= (1 << 20) ||
        (int64_t)cores_total * p.cores >= (1 << 20) || (!p.flat && (int64_t)(p.seg_pixels + 64) * W >= (1 << 20)))
        return false;
    p.ncols = R * S * p.cb;
    p.chunks = (p.ncols + 31) / 32;
    p.tmem_cols = 32;
    while ((int)p.tmem_cols < p.chunks * 32) p.tmem_cols *= 2;
    if (p.tmem_cols > 512) return false;
    {
        const uint32_t row_pitch = (uint32_t)(p.cb / 8) * p.gp * 16, core_pitch = (uint32_t)p.mt * 16;
        for (int i = 0; i < (cores_total + 1) / 2; ++i) {
            uint32_t a[2], b[2];
            for (int h = 0; h < 2; ++h) {
                const int core = 2 * i + h, row = core / p.cores, xc = core % p.cores;
                // the group behind the last row counts as a row of the last image
                const int img = row / p.yb < p.ni ? row / p.yb : p.ni - 1, y = row - img * p.yb;
                a[h] = p.x_bytes + core * core_pitch;
                b[h] = (img * p.x_rows + y * p.row_step) * row_pitch + xc * 128;
            }
            p.pairs[i] = make_uint2(desc_low(a[0], a[1] - a[0]), desc_low(b[0], b[1] - b[0]));
        }
    }
    return true;
}

// The plan of the last shape that this thread asked for: the search over bands costs half a microsecond, and a layer is
// planned twice per call (workspace query and launch).
bool cached_fused_conv_plan(FusedConvParams& p, int B, int Ca, int H, int W, int Cz, int R, int S, int stride, int pad, int64_t k) {
    struct Last {
        int key[10];
        bool ok;
        FusedConvParams p;
    };
    static thread_local Last last = {};
    const int key[10] = {B, Ca, H, W, Cz, R, S, stride, pad, sm_count()};
    if (std::memcmp(key, last.key, sizeof(key)) != 0) {
        last.ok = make_fused_conv_plan(last.p, B, Ca, H, W, Cz, R, S, stride, pad, 0);
        std::memcpy(last.key, key, sizeof(key));
    }
    if (!last.ok) return false;
    p = last.p;
    p.k = (uint32_t)k;
    return true;
}

}  // namespace

// 0 when this kernel does not take the shape.
size_t conv_fused_workspace_bytes(int B, int Ca, int H, int W, int Cz, int R, int S, int stride, int pad) {
    FusedConvParams p;
    if (!cached_fused_conv_plan(p, B, Ca, H, W, Cz, R, S, stride, pad, 0)) return 0;
    return (size_t)p.splits * p.tiles_c * p.tiles_j * p.chunks * 32 * kBM * 4;
}

// Caller has validated pointers, sizes and alignment, and B >= 1, k >= 1; bitmask caches only.
dropit_status conv_fused_run(const void* dy, const void* values, const void* mask, const uint32_t* offsets, int B, int Ca, int H,
                             int W, int Cz, int R, int S, int stride, int pad, int64_t k, float* dw, int accumulate,
                             void* workspace, size_t workspace_bytes, int32_t* dev_status, cudaStream_t stream) {
    FusedConvParams p;
    if (!cached_fused_conv_plan(p, B, Ca, H, W, Cz, R, S, stride, pad, k)) return DROPIT_ERR_UNSUPPORTED;
    const int tiles = p.tiles_c * p.tiles_j;
    if (workspace_bytes < (size_t)p.splits * tiles * p.chunks * 32 * kBM * 4) return DROPIT_ERR_WORKSPACE;
    const int vec = p.vec == 8 ? 3 : p.vec / 2;
    auto kern = vec == 3 ? conv_wg_fused_kernel<8> : (vec == 2 ? conv_wg_fused_kernel<4> : (vec == 1 ? conv_wg_fused_kernel<2> : conv_wg_fused_kernel<1>));
    static PerDeviceOnce attr[4];
    PerDeviceOnce& once = attr[vec];
    if (once.needed()) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess)
            return DROPIT_ERR_CUDA;
        once.mark();
    }
    float* partial = reinterpret_cast<float*>(workspace);
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles, (unsigned)p.splits);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)p.stages * (p.x_bytes + p.dy_bytes) + sizeof(FusedConvCtl);
    cfg.stream = stream;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<const uint16_t*>(dy), reinterpret_cast<const uint16_t*>(values),
                           reinterpret_cast<const uint32_t*>(mask), offsets, p, partial, dev_status,
                           spin_limit(kWaitLimit)) != cudaSuccess) {
        (void)cudaGetLastError();
        return DROPIT_ERR_CUDA;
    }
    dropit_status st = check_launch();
    if (st != DROPIT_OK) return st;
    const int quarters = ((Cz < kBM ? Cz : kBM) + 31) / 32, sets = R * S, blocks = tiles * quarters * (p.cb / 4);
    // As many taps (channels) per block as leave two blocks per SM.  One / three / nine taps (blocks with nine): 64 -> 64 on 56 x 56 (32)
    // 35.9 / 36.6 / 38.2 us, 8 images of 40 -> 72 on 23 x 23 (36) 12.3 / 12.8 / 15.1, stride 2 128 -> 128 on 56 x 56 (144) 55.2 / 53.5 / 54.7, 8 images
    // of 64 -> 320 on 13 x 13 (176) 14.6 / 11.9 / 12.5, 256 -> 256 on 14 x 14 (576) 40.2 / 34.2 / 33.9, 8 images of 512 -> 512 on 7 x 7 (2112)
    // 48.3 / 32.9 / 29.1.
    const int least = 2 * sm_count();
    const int per = sets == 1 ? (blocks / 4 >= least ? 4 : 1)
                              : (sets == 9 && blocks >= least ? 9 : (sets % 3 == 0 && blocks * (sets / 3) >= least ? 3 : 1));
    auto reduce = per == 9 ? conv_fused_reduce_kernel<9> : (per == 4 ? conv_fused_reduce_kernel<4, true>
                                                                     : (per == 3 ? conv_fused_reduce_kernel<3> : conv_fused_reduce_kernel<1>));
    cfg.gridDim = dim3((unsigned)((Cz + 31) / 32), (unsigned)(per == 4 ? p.cb / 16 : p.cb / 4 * (sets / per)), (unsigned)p.tiles_c);
    cfg.blockDim = dim3(32 * kRedWarps);
    cfg.dynamicSmemBytes = 0;
    p.dy = reinterpret_cast<const uint16_t*>(dy);
    p.values = reinterpret_cast<const uint16_t*>(values);
    p.mask = reinterpret_cast<const uint32_t*>(mask);
    p.offsets = offsets;
    if (cudaLaunchKernelEx(&cfg, reduce, reinterpret_cast<const float4*>(partial), p, dw, accumulate) != cudaSuccess) {
        (void)cudaGetLastError();
        return DROPIT_ERR_CUDA;
    }
    return check_launch();
}

}  // namespace dropit
