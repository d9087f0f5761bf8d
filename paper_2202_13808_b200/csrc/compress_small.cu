// Min-k selection + packing of a small tensor by ONE thread-block cluster (Sec. 3.3 "Min-K Elements",
// Sec. 3.2 a-hat = {a_Xr, X_r}).
//
// A tensor of up to 2^19 elements fits the shared memory of 16 SMs, so it is read from global memory once and the whole
// selection runs between CTAs that can write into each other's shared memory and meet at the hardware's cluster barrier,
// instead of at a grid barrier through L2 or between launches.
//   1. every warp brings one super-block (1024 elements) into shared memory;
//   2. each CTA counts the upper 15 bits of the keys in 2^15 16-bit counters (a bf16 key has no more bits);
//   3. the threshold is found digit by digit: 8 bits, then 7 (fp32: then 8 and 8 more over the keys that still match).
//      A round is: each CTA writes its row of 128 or 256 counts into every CTA of the cluster, one cluster barrier, and
//      every CTA finds the same digit from the same rows.  The rows of the CTAs in front of it also give a CTA its
//      exclusive prefix of keys above and at the threshold, so the ordered compaction needs no further exchange.
//      fp32, up to 1024 keys that match in their upper 15 bits: their lower halves are sent round once instead, and every CTA
//      finds both lower digits from that list;
//   4. element i is retained iff key_i > T, or key_i == T and fewer than q equal keys precede it.  A lane owns 32
//      consecutive elements, i.e. one mask word; the retained values are moved to the front of the super-block in
//      shared memory and leave coalesced.
// Nothing is sampled and no scratch in global memory is used: any distribution of values takes the same path.  Equal keys
// make the counting atomics collide; zeros are counted in registers because ReLU outputs are half zeros.  Other values that fill more
// than half of an fp32 tensor of 300 Ki elements and more are slower here than with the histogram launches (2^19 elements, half of them equal
// 31.6 against 27.2 us, all 39.7 against 26.1; none 21.2 against 26.0).  Counting the commonest key of a sample in registers, not zero,
// brought these to 26 us and cost all other calls 0.6 to 1 us.
// Bound by latency: barriers, the trips between CTAs (about 1 us a digit round) and the shared-memory counting.  Measured per
// call (graph replay, gamma 0.9): bf16 8 Ki / 48 Ki / 196 Ki / 512 Ki elements 5.8 / 6.3 / 8.0 / 11.9 us, where the grid-wide
// kernel's full histogram takes 60 us at any of these sizes; fp32 9.3 / 9.9 / 12.0 / 17.5 us (9.8 / 10.9 / 13.9 / 20.3 without the list and
// the programmatic launch, which takes 0.7 us off every call behind a kernel that leaves SMs free), where the three
// histogram launches and the compaction take 27 us at 600 Ki.  (Counting through a branch per element, only by the warps
// that own a super-block, and a third barrier per round: 8.0 / 8.9 / 10.3 / 12.8 and 14.2 / 16.9 / 20.7 us.)  At 2^19 bf16
// elements (11.9 us) the sampled grid-wide kernel (13.2 us) is about to overtake: two super-blocks per warp measured 17.4 us at
// 800 Ki against its 16.1, so there the line lies.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace dropit {

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCtas = 16;
constexpr int kSb = 1024;                                // elements of a super-block, one per warp
constexpr int kSbPerCta = 8;                             // super-blocks a CTA is given before the cluster grows
constexpr uint32_t kTopBins = 1u << 15;
constexpr int kRowBins = 256;                            // counts of one CTA in one digit round
constexpr size_t kHistBytes = (size_t)kTopBins * 2;
constexpr size_t kGatherBytes = (size_t)2 * kMaxCtas * kRowBins * 4;
// Most keys that are ranked from a list, a word each.  Keys that lie side by side are found by a few warps, one key after the other: 1000 /
// 2000 / 4090 of them take 13.6 / 15.7 / 20.3 us at 196 Ki elements, where the two digit rounds take 14.4 / 14.5 / 15.5, and 11.0 / 12.3 / 15.1 at
// 48 Ki (11.3 / 11.3 / 12.3).  Scattered ones are ahead up to 3000.
constexpr uint32_t kListCap = 1024;
static_assert(kListCap <= kMaxCtas * kRowBins, "a gather buffer holds the list");

struct SmallShared {
    uint32_t row[kRowBins];        // this CTA's counts of the current digit
    uint2 warp_tot[kWarps];
    uint32_t digit, cum;           // the digit found, keys above it
    uint32_t before_gt, before_eq; // in the CTAs in front of this one: keys above / at the digit
    uint32_t at;                   // keys at the digit, over the cluster
    uint32_t listed, list_before;  // keys this CTA has put on the list; on the list in front of its own: keys above | at T << 16
};

template <typename Tr> struct SmallCfg {
    static constexpr int kSlotBytes = kSb * Tr::kElemBytes;
    static constexpr int kVecs = kSlotBytes / 16;                        // 16-byte vectors of a super-block
    static constexpr int kOwnVecs = kVecs / 32;                          // ... of a lane's 32 elements: 4 or 8
    static constexpr size_t kDataBytes = (size_t)kWarps * kSlotBytes;
    static constexpr size_t kSmemBytes = kDataBytes + kHistBytes + kGatherBytes + sizeof(SmallShared);
};
static_assert(kWarps * kSb < (1 << 16), "a 16-bit counter must hold every element of a CTA");
static_assert(kSmallMaxElems == (int64_t)kWarps * kMaxCtas * kSb, "one super-block per warp");

__device__ __forceinline__ uint32_t cluster_nctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t warp_inclusive_scan(uint32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFullMask, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// [addr] += v if `on`; a predicated instruction, not a branch (a branch around every count tripled the counting passes).
__device__ __forceinline__ void red_shared_if(uint32_t addr, uint32_t v, bool on) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.shared.add.u32 [%0], %1;\n\t}" ::"r"(addr), "r"(v), "r"(on ? 1u : 0u) : "memory");
}

// One digit round: sh.row[0 .. nb) holds this CTA's counts.  Finds the digit in which the descending running count
// over the cluster reaches k_rem, subtracts from k_rem the keys above it and brings run_gt / run_eq (keys above / at the
// digits fixed so far, in the CTAs in front of this one) up to date.
// `rows`: gather buffer of the current digit round, [CTA][kRowBins] (two alternate: a CTA that is ahead by one round writes the other one).
__device__ __forceinline__ uint32_t digit_round(SmallShared& sh, const uint32_t* rows, int nb, uint32_t rank, uint32_t ctas,
                                                uint32_t& k_rem, uint32_t& run_gt, uint32_t& run_eq, bool first) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    __syncthreads();   // the row is complete
    if (first) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every CTA of the cluster is running
    const uint32_t mine = ptx::smem_u32(rows) + rank * (kRowBins * 4);
    for (uint32_t i = t; i < ctas * nb; i += kThreads) {
        const uint32_t dest = i / nb, b = i % nb;    // nb is 128 or 256
        ptx::st_cluster_u32(ptx::map_shared_to_cta(mine + b * 4, dest), sh.row[b]);
    }
    ptx::cluster_sync_all();
    // thread t < nb looks at bin nb - 1 - t: a prefix over the threads is a count from the top, over the cluster (h) and over
    // the CTAs in front of this one (f)
    const int bin = nb - 1 - t;
    uint32_t h = 0, f = 0, h_inc = 0, f_inc = 0;
    if (t < nb) {
        for (uint32_t r = 0; r < ctas; ++r) {
            const uint32_t v = rows[r * kRowBins + bin];
            h += v;
            if (r < rank) f += v;
        }
        h_inc = h;
        f_inc = f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t yh = __shfl_up_sync(kFullMask, h_inc, o), yf = __shfl_up_sync(kFullMask, f_inc, o);
            if (lane >= o) { h_inc += yh; f_inc += yf; }
        }
        if (lane == 31) sh.warp_tot[warp] = make_uint2(h_inc, f_inc);
    }
    __syncthreads();
    if (t < nb) {
        uint32_t cum = h_inc - h, before = f_inc - f;
#pragma unroll
        for (int w = 0; w < kRowBins / 32 - 1; ++w) {
            if (w < warp) {
                const uint2 v = sh.warp_tot[w];
                cum += v.x;
                before += v.y;
            }
        }
        if (cum < k_rem && k_rem <= cum + h) {
            sh.digit = (uint32_t)bin;
            sh.cum = cum;
            sh.before_gt = before;
            sh.before_eq = f;
            sh.at = h;
        }
    }
    __syncthreads();
    k_rem -= sh.cum;
    run_gt += sh.before_gt;
    run_eq = sh.before_eq;
    return sh.digit;       // (the next round's first barrier comes before anything here is written again)
}

// One digit of the keys on a list of `m` entries, found by every warp for itself from the counts of its 256 values in sh.row: the
// largest one with k_rem entries at or above it; k_rem loses those above it.
__device__ __forceinline__ uint32_t list_digit(const SmallShared& sh, int lane, uint32_t& k_rem) {
    constexpr int kPer = kRowBins / 32;          // values per lane
    static_assert(kPer == 8, "");
    const uint4 a = reinterpret_cast<const uint4*>(sh.row)[lane * 2], b = reinterpret_cast<const uint4*>(sh.row)[lane * 2 + 1];
    uint32_t ge = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(kFullMask, ge, o);
        if (lane + o < 32) ge += y;
    }
    const int owner = 31 - __clz(__ballot_sync(kFullMask, ge >= k_rem));      // (lane 0 holds all entries that still match: at least k_rem)
    const uint32_t behind = __shfl_sync(kFullMask, ge, (owner + 1) & 31);
    k_rem -= owner < 31 ? behind : 0u;
    const uint32_t c = sh.row[owner * kPer + (lane & 7)];
    ge = c;
#pragma unroll
    for (int o = 1; o < kPer; o <<= 1) {
        const uint32_t y = __shfl_down_sync(kFullMask, ge, o, kPer);
        if ((lane & 7) + o < kPer) ge += y;
    }
    const int bin = 31 - __clz(__ballot_sync(kFullMask, ge >= k_rem) & 0xFFu);
    k_rem -= __shfl_sync(kFullMask, ge - c, bin);
    return (uint32_t)(owner * kPer + bin);
}

template <typename Tr, bool INDEX32>
__global__ void __launch_bounds__(kThreads, 1)
small_compress_kernel(const uint4* __restrict__ x, uint32_t n, uint32_t k, uint32_t sb_per_cta,
                      typename Tr::elem_t* __restrict__ values, uint32_t* __restrict__ mask, int32_t* __restrict__ indices,
                      uint32_t* __restrict__ offsets) {
    using elem_t = typename Tr::elem_t;
    using Cfg = SmallCfg<Tr>;
    constexpr int ES = Tr::kElemBytes, G = Tr::kVecElems, OV = Cfg::kOwnVecs;
    constexpr bool kF32 = ES == 4;
    extern __shared__ __align__(16) unsigned char ssm[];
    uint32_t* hist = reinterpret_cast<uint32_t*>(ssm + Cfg::kDataBytes);          // two 16-bit counters per word
    uint32_t* gather = reinterpret_cast<uint32_t*>(ssm + Cfg::kDataBytes + kHistBytes);
    SmallShared& sh = *reinterpret_cast<SmallShared*>(ssm + Cfg::kDataBytes + kHistBytes + kGatherBytes);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t rank = ptx::cluster_ctarank(), ctas = cluster_nctarank();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");          // waited for in the first digit round

    const uint32_t sb = rank * sb_per_cta + warp;
    const bool active = (uint32_t)warp < sb_per_cta && (uint64_t)sb * kSb < n;     // the warp has a super-block
    const uint32_t data = ptx::smem_u32(ssm) + warp * Cfg::kSlotBytes;
    const uint32_t nvec_full = n / G;

    ptx::grid_dependency_wait();      // launched programmatically: the input may come from the kernel before this one
    if (active) {
#pragma unroll
        for (int j = 0; j < OV; ++j) {
            const uint32_t vi = sb * Cfg::kVecs + j * 32 + lane;
            const uint32_t dst = data + (j * 32 + lane) * 16;
            if (vi == nvec_full && (n % G) != 0) {           // ragged last vector of the tensor: assembled by hand
                const elem_t* xe = reinterpret_cast<const elem_t*>(x) + (size_t)vi * G;
                uint32_t w[4] = {0, 0, 0, 0};
                for (uint32_t e = 0; e < n % G; ++e) {
                    if constexpr (kF32) w[e] = xe[e];
                    else w[e >> 1] |= (uint32_t)xe[e] << ((e & 1) * 16);
                }
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                             : "memory");
            } else {
                const bool in = vi < nvec_full;               // vectors past the end are zero-filled by the copy itself
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(x + (in ? vi : 0)), "r"(in ? 16u : 0u)
                             : "memory");
            }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (t == 0) sh.listed = sh.list_before = 0;
    for (uint32_t i = t; i < kHistBytes / 16; i += kThreads) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // ---- counts of the upper 15 key bits ----
    // visit(key, exists) for every element of the CTA's super-blocks (zero padding does not exist), in any order: all threads
    // share the 16-byte vectors, also when only some warps own a super-block
    const uint32_t cta_vecs = min(sb_per_cta, (n + kSb - 1) / kSb - min((n + kSb - 1) / kSb, rank * sb_per_cta)) * Cfg::kVecs;
    const uint32_t cta_first = rank * sb_per_cta * kSb, data0 = ptx::smem_u32(ssm);
    auto for_each_key = [&](auto visit) {
        for (uint32_t v = t; v < cta_vecs; v += kThreads) {
            uint32_t w[4];
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                         : "r"(data0 + v * 16) : "memory");
            const uint32_t e0 = cta_first + v * G;
#pragma unroll
            for (int e = 0; e < G; ++e) {
                uint32_t key;
                if constexpr (kF32) key = w[e] & 0x7FFFFFFFu;
                else key = ((e & 1) ? (w[e >> 1] >> 16) : w[e >> 1]) & 0x7FFFu;
                visit(key, e0 + e < n);
            }
        }
    };
    {
        uint32_t zeros = 0;
        const uint32_t hist_addr = ptx::smem_u32(hist);
        for_each_key([&](uint32_t key, bool exists) {
            const uint32_t top = kF32 ? key >> 16 : key;
            zeros += top == 0 && exists ? 1u : 0u;
            red_shared_if(hist_addr + (top >> 1) * 4, 1u << ((top & 1u) * 16), top != 0 && exists);
        });
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) zeros += __shfl_xor_sync(kFullMask, zeros, o);
        if (lane == 0 && zeros) atomicAdd(&hist[0], zeros);
    }
    __syncthreads();

    // ---- digit 1: sums of 128 neighbouring counters (four threads each; the reads are rotated against bank conflicts) ----
    uint32_t k_rem = k;
    {
        const uint4* own = reinterpret_cast<const uint4*>(hist + t * 16);
        uint32_t sum = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint4 v = own[j ^ ((t >> 1) & 3)];
            sum += (v.x & 0xFFFFu) + (v.x >> 16) + (v.y & 0xFFFFu) + (v.y >> 16) + (v.z & 0xFFFFu) + (v.z >> 16) +
                   (v.w & 0xFFFFu) + (v.w >> 16);
        }
        sum += __shfl_xor_sync(kFullMask, sum, 1);
        sum += __shfl_xor_sync(kFullMask, sum, 2);
        if ((t & 3) == 0) sh.row[t >> 2] = sum;
    }
    uint32_t run_gt = 0, run_eq = 0;   // keys above / at T in front of this CTA
    const uint32_t d1 = digit_round(sh, gather, 256, rank, ctas, k_rem, run_gt, run_eq, true);
    // ---- digit 2: the 128 counters behind that sum ----
    if (t < 128) {
        const uint32_t w = hist[d1 * 64 + (t >> 1)];
        sh.row[t] = (t & 1) ? w >> 16 : w & 0xFFFFu;
    }
    uint32_t T = d1 * 128 + digit_round(sh, gather + kMaxCtas * kRowBins, 128, rank, ctas, k_rem, run_gt, run_eq, false);
    if constexpr (kF32) {
        // ---- digits 3 and 4: the lower 16 bits, over the keys whose upper bits match ----
        const uint32_t row_addr = ptx::smem_u32(sh.row);
        const uint32_t m = sh.at;
        if (m <= kListCap) {
            // Few keys match (some 300 of 196 Ki normal ones): their lower halves go on a list that every CTA holds, this CTA's
            // behind those of the CTAs in front of it, and every CTA finds both digits on its own.  One trip through the cluster
            // and one pass over the elements instead of two.  They are collected first and sent by all threads: sent by the thread
            // that finds a key, to one CTA after the other, 300 of 196 Ki took 13.0 us instead of 12.3, 1000 of 512 Ki 20.1 instead of 18.3.
            const uint32_t front = run_eq;
            // (this CTA has read the second round's rows, the cluster the first round's; a CTA on its own finds its keys where the list is)
            uint32_t* found = gather + (ctas > 1 ? kMaxCtas * kRowBins : 0);
            for_each_key([&](uint32_t key, bool exists) {
                if (exists && (key >> 16) == T) found[atomicAdd(&sh.listed, 1u)] = key & 0xFFFFu;
            });
            if (ctas > 1) {
                __syncthreads();
                const uint32_t own = sh.listed;
                const uint32_t to = ptx::map_shared_to_cta(ptx::smem_u32(gather + front), (uint32_t)warp & (ctas - 1u));    // (a power of two)
                for (uint32_t i = (uint32_t)warp / ctas * 32 + lane; i < own; i += kThreads / ctas) ptx::st_cluster_u32(to + i * 4, found[i]);
            }
            if (t < kRowBins) sh.row[t] = 0;
            ptx::cluster_sync_all();
            for (uint32_t i = t; i < m; i += kThreads) red_shared_if(row_addr + (gather[i] >> 8) * 4, 1u, true);
            __syncthreads();
            const uint32_t d3 = list_digit(sh, lane, k_rem);
            __syncthreads();
            if (t < kRowBins) sh.row[t] = 0;
            __syncthreads();
            for (uint32_t i = t; i < m; i += kThreads) red_shared_if(row_addr + (gather[i] & 0xFFu) * 4, 1u, (gather[i] >> 8) == d3);
            __syncthreads();
            const uint32_t low = d3 << 8 | list_digit(sh, lane, k_rem);
            uint32_t before = 0;
            for (uint32_t i = t; i < front; i += kThreads) before += (gather[i] > low ? 1u : 0u) | (gather[i] == low ? 1u << 16 : 0u);
            before = __reduce_add_sync(kFullMask, before);
            if (lane == 0 && before) atomicAdd(&sh.list_before, before);
            __syncthreads();
            run_gt += sh.list_before & 0xFFFFu;
            run_eq = sh.list_before >> 16;
            T = T << 16 | low;
        } else {
#pragma unroll 1
            for (int shift = 8; shift >= 0; shift -= 8) {
                if (t < kRowBins) sh.row[t] = 0;
                __syncthreads();
                for_each_key([&](uint32_t key, bool exists) {
                    red_shared_if(row_addr + ((key >> shift) & 0xFFu) * 4, 1u, exists && (key >> (shift + 8)) == T);
                });
                T = (T << 8) | digit_round(sh, gather + (shift == 8 ? 0 : kMaxCtas * kRowBins), 256, rank, ctas, k_rem, run_gt,
                                           run_eq, false);
            }
        }
    }
    const uint32_t q = k_rem;          // ties at T that are retained, lowest flat indices first
    ptx::launch_dependents();

    // ---- ordered compaction ----
    // the lane's 32 elements of a super-block, its vectors in an order rotated by the lane (a quarter-warp reads eight
    // different 16-byte columns): w[4 * j ..] is the lane's vector j ^ rot
    const uint32_t rot = kF32 ? (uint32_t)lane & 7u : ((uint32_t)lane >> 1) & 3u;
    uint32_t g32 = 0, e32 = 0;
    if (active) {
#pragma unroll
        for (int j = 0; j < OV; ++j) {
            uint32_t w[4];
            const uint32_t v = (uint32_t)j ^ rot;
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                         : "r"(data + (lane * OV + v) * 16) : "memory");
            uint32_t g = 0, eq = 0;
#pragma unroll
            for (int e = 0; e < G; ++e) {
                uint32_t key;
                if constexpr (kF32) key = w[e] & 0x7FFFFFFFu;
                else key = ((e & 1) ? (w[e >> 1] >> 16) : w[e >> 1]) & 0x7FFFu;
                g |= (key > T ? 1u : 0u) << e;
                eq |= (key == T ? 1u : 0u) << e;
            }
            g32 |= g << (v * G);
            e32 |= eq << (v * G);
        }
        const uint32_t first = sb * kSb + lane * 32;            // zero padding must not tie with T = 0
        if (first + 32 > n) e32 &= first < n ? (1u << (n - first)) - 1u : 0u;
    }
    const uint32_t cnt = __popc(g32) | (__popc(e32) << 16);      // a CTA has fewer than 2^16 elements: packed sums do not overflow
    const uint32_t inc = warp_inclusive_scan(cnt, lane);
    const uint32_t excl = inc - cnt, tot = __shfl_sync(kFullMask, inc, 31);
    if (lane == 0) sh.warp_tot[warp].x = tot;
    __syncthreads();
    if (!active) return;
    {
        const uint32_t other = sh.warp_tot[lane].x;
        const uint32_t before = warp_inclusive_scan(other, lane) - other;
        const uint32_t mine = __shfl_sync(kFullMask, before, warp);
        run_gt += mine & 0xFFFFu;
        run_eq += mine >> 16;
    }
    const uint32_t eq_before = run_eq + (excl >> 16), ne = __popc(e32);
    const uint32_t room = eq_before < q ? q - eq_before : 0u;
    uint32_t ke = e32;
    if (room < ne) {                           // the quota ends inside this lane's ties: the first `room` of them stay
        uint32_t m = e32;
        ke = 0;
        for (uint32_t r = 0; r < room; ++r) {
            ke |= m & (0u - m);
            m &= m - 1;
        }
    }
    const uint32_t keep = g32 | ke;
    const uint32_t base = run_gt + min(run_eq, q);                                         // retained before the super-block
    const uint32_t kept = run_gt + (tot & 0xFFFFu) + min(run_eq + (tot >> 16), q) - base;  // ... in it
    const uint32_t pos = run_gt + (excl & 0xFFFFu) + min(eq_before, q);                    // ... before the lane's elements
    const uint32_t word = sb * 32 + lane, nwords = (n + 31) / 32;
    if (word < nwords) {
        if ((lane & 3) == 0) offsets[word >> 2] = pos;
        if constexpr (!INDEX32) mask[word] = keep;
    }
    // move the retained values to the front of the super-block: read everything, then write
    const uint32_t idx_stage = ptx::smem_u32(hist) + warp * (kSb * 2);   // INDEX32: positions inside the super-block
    uint32_t w[4 * OV];
#pragma unroll
    for (int j = 0; j < OV; ++j)
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[4 * j]), "=r"(w[4 * j + 1]), "=r"(w[4 * j + 2]), "=r"(w[4 * j + 3])
                     : "r"(data + (lane * OV + ((uint32_t)j ^ rot)) * 16) : "memory");
    __syncwarp();
#pragma unroll
    for (int j = 0; j < OV; ++j) {
        const uint32_t e_first = ((uint32_t)j ^ rot) * G;
        uint32_t p = pos - base + __popc(keep & ((1u << e_first) - 1u));
        const uint32_t bits = keep >> e_first;
#pragma unroll
        for (int e = 0; e < G; ++e) {
            if ((bits >> e) & 1u) {
                if constexpr (kF32) {
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(data + p * 4), "r"(w[4 * j + e]) : "memory");
                } else {
                    const uint32_t v = (e & 1) ? w[4 * j + e / 2] >> 16 : w[4 * j + e / 2];
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(data + p * 2), "r"(v) : "memory");
                }
                if constexpr (INDEX32)
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(idx_stage + p * 2), "r"(lane * 32 + e_first + e) : "memory");
                ++p;
            }
        }
    }
    __syncwarp();
    for (uint32_t i = lane; i < kept; i += 32) {
        uint32_t v;
        if constexpr (kF32) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(data + i * 4) : "memory");
        else asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(data + i * 2) : "memory");
        values[base + i] = (elem_t)v;
        if constexpr (INDEX32) {
            asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(idx_stage + i * 2) : "memory");
            indices[base + i] = (int32_t)(sb * kSb + v);
        }
    }
}

// Largest cluster of this kernel that fits the current device (16 needs the opt-in to non-portable sizes), 0 if none.
template <typename Tr, bool INDEX32>
int max_cluster() {
    static std::atomic<int> cached[64];      // value + 1; 0 = not looked up yet
    const int dev = current_device();
    if (dev < 0 || dev >= 64) return 0;
    int c = cached[dev].load(std::memory_order_acquire);
    if (c == 0) {
        auto kern = small_compress_kernel<Tr, INDEX32>;
        c = 1;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SmallCfg<Tr>::kSmemBytes) == cudaSuccess &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            for (int size = kMaxCtas; size >= 8 && c == 1; size /= 2) {
                cudaLaunchAttribute attr[1];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = (unsigned)size;
                attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)size);
                cfg.blockDim = dim3(kThreads);
                cfg.dynamicSmemBytes = SmallCfg<Tr>::kSmemBytes;
                cfg.attrs = attr;
                cfg.numAttrs = 1;
                int fit = 0;
                if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) == cudaSuccess && fit > 0) c = size + 1;
            }
        }
        (void)cudaGetLastError();
        cached[dev].store(c, std::memory_order_release);
    }
    return c - 1;
}

template <typename Tr, bool INDEX32>
bool launch_small(const void* x, int64_t n, int64_t k, void* values, void* meta, uint32_t* offsets, cudaStream_t stream,
                  dropit_status* status) {
    using Cfg = SmallCfg<Tr>;
    const int limit = max_cluster<Tr, INDEX32>();
    const int64_t sbs = (n + kSb - 1) / kSb;
    if (limit == 0 || sbs > (int64_t)limit * kWarps) return false;
    // 8 super-blocks per CTA until the cluster is full: at 48 Ki elements 4 / 8 / 16 measure 7.0 / 6.8 / 7.5 us
    int ctas = 1;
    while (ctas < limit && sbs > (int64_t)ctas * kSbPerCta) ctas *= 2;
    const int64_t per = (sbs + ctas - 1) / ctas;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    // programmatic: the cluster may be set up while the kernel before it drains; it waits before it reads anything
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg::kSmemBytes;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, small_compress_kernel<Tr, INDEX32>, reinterpret_cast<const uint4*>(x), (uint32_t)n, (uint32_t)k,
                           (uint32_t)per, reinterpret_cast<typename Tr::elem_t*>(values),
                           INDEX32 ? (uint32_t*)nullptr : reinterpret_cast<uint32_t*>(meta),
                           INDEX32 ? reinterpret_cast<int32_t*>(meta) : (int32_t*)nullptr, offsets) != cudaSuccess) {
        (void)cudaGetLastError();
        *status = DROPIT_ERR_CUDA;
        return true;
    }
    *status = check_launch();
    return true;
}

}  // namespace

// Takes the call if the tensor is small enough for one cluster of this device; 0 < k <= n.  Returns false otherwise.
bool small_compress(const void* x, int64_t n, int64_t k, dropit_dtype dtype, bool index32, void* values, void* meta,
                    uint32_t* offsets, cudaStream_t stream, dropit_status* status) {
    if (n > kSmallMaxElems) return false;
    if (dtype == DROPIT_BF16)
        return index32 ? launch_small<Bf16Traits, true>(x, n, k, values, meta, offsets, stream, status)
                       : launch_small<Bf16Traits, false>(x, n, k, values, meta, offsets, stream, status);
    return index32 ? launch_small<F32Traits, true>(x, n, k, values, meta, offsets, stream, status)
                   : launch_small<F32Traits, false>(x, n, k, values, meta, offsets, stream, status);
}

}  // namespace dropit
