// prefill_mma.cu -- tree-masked prefill attention on tcgen05 (bf16 or e4m3 KV,
// head_dim 128).
//
// Every token of every chunk is a query (paper Sec. 3.1: after a join the new
// text is prefilled against the whole tree), so the pass is a dense
// contraction.  The work queue holds pairs of 128-row tiles of one chunk and
// kv head over one list of pages (position k: items 2k and 2k + 1, the second
// without rows when there is no second tile).  One persistent CTA per SM runs
// a pair against blocks of 128 keys (8 pages), so that a staged block serves
// 256 rows:
//
//   warps 0-3   tile A: softmax (thread r owns row r, TMEM lane r), the next
//               pair's Q rows, then the row's (m, l) and O
//   warps 4-7   tile B: the same
//   warp 8      producer: TMA of K, then V, of each block into a ring.  bf16:
//               a 4 KB box per page, one lane each, laid out so that the MMA
//               reads 8 pages anywhere in the pool as one operand (a 2 KB box
//               per page and column block took permuted pages from 495 to 595
//               us on the join; one 32 KB box for consecutive pages is level).
//               e4m3: one 16 KB box when the block's 8 pages are consecutive,
//               else a box per 4 pages or per page
//   warp 9      MMA issuer: S_t = Q_t K^T (M 128, N 128, both operands in
//               shared memory) and O_t += P_t V (P in TMEM) for t = A, B in
//               turn (two issuers let the tiles fall into step, both in their
//               softmax or both waiting: join prefill 555 -> 727 us)
//   warp 10     scheduler: pulls pairs and stages their records
//   warps 12-15 with e4m3 KV: widen each staged block to f16
//
// TMEM, 512 columns: O_A, O_B at 0 and 128, S_A, S_B at 256 and 384.  P (bf16,
// f16 with e4m3 KV) goes over the first 64 columns of its S in two halves,
// each announced by itself, so that PV of the first 64 keys runs while the
// second half is exponentiated.  The issuer sends PV_t(i), then S_t(i + 1): the
// tensor core executes one thread's MMAs in order, so the S of the next block
// needs no wait before it overwrites the P it follows, and the commit of
// S_t(i + 1) also says that PV_t(i) is done (what a rescale of O waits for).
// While a tile's softmax runs, the tensor core works for the other.
//
// Why this shape: with 64-key blocks and two S buffers a tile (the pair tile
// of the decode kernel) S is held by its shared-memory reads (128 x 16 of Q
// and 64 x 16 of K per 128 x 64 x 16 product: 48 cycles against 32 of
// arithmetic) and every wait, mask test and TMEM round trip is paid per 64
// keys.  128-key blocks balance the two (64 and 64 cycles) and halve the
// rest; they want 128 scores a thread in registers, so the warps of a pair
// take registers from the others (setmaxnreg; the shares sum to no more than
// the launch holds).
//
// Measured (32 q / 8 kv heads, attention kernel): join, 1024 queries over 41k
// keys, 486 us of 348 us of arithmetic at 1.95 PFLOP/s, where the decode
// kernel's pair tile took 583 us; with e4m3 KV 654 us (whole paths) against 970;
// fork, 16 x 64 queries over 2112 keys, a pass of 39 us without a merge against 59
// with one.  A pair of blocks takes about 3400 cycles against 2048 of tensor work: a tile's
// chain is 300 cycles to read S, 400 for the maxima, 1100 for the
// exponentials, then 768 of its own PV half and S.  Tried and slower: an issuer
// per tile (both tiles fall into step, 555 -> 727 us), the first half
// exponentiated before the maxima are known (553 -> 584 us), two threads a row
// (705 us).  With e4m3 KV the chain is about 4500 cycles, as the widening warps
// share the schedulers and the shared memory with the softmax; 8 widening
// warps (832 us), or widening over the raw bytes in a ring of 5 slots (932
// us), are slower than a ring of 4 raw and 3 widened slots.
//
// Every wait is bounded (%globaltimer); on expiry the error is recorded, the
// copies in flight land, TMEM is freed and the CTA exits.
#include <mutex>

#include "device_common.cuh"
#include "tcgen05.cuh"
#include "tile_common.cuh"

namespace parason {
namespace {

constexpr long long kDrainLimitNs = 1000000000LL;
constexpr int kRows = 128;                         // rows of a tile
constexpr int kDim = 128;                          // head_dim
constexpr int kHalfTokens = 64;                    // keys of half a block
constexpr int kBlockPages = kPrefillBoxPages;                  // 8
constexpr int kBlockTokens = kBlockPages * kPageSize;          // 128
constexpr int kColBlockBytes = kBlockTokens * 128;             // 16 KB: 128 keys x 128 bytes
constexpr int kSlotBytes = 2 * kColBlockBytes;                 // 32 KB: K or V of a block, 16-bit
constexpr int kPagedBytes = kSlotBytes / kBlockPages;          // 4 KB: a page of it
constexpr int kRawSlotBytes = kBlockTokens * 128;              // 16 KB: the same in e4m3
constexpr int kQColBlockBytes = kRows * 128;                   // 16 KB
constexpr int kQBytes = 2 * kQColBlockBytes;                   // 32 KB a tile
constexpr int kMeta = kPrefillMeta;
constexpr int kAheadBlocks = kPrefillAheadBlocks;  // (see the scheduler)
constexpr int kValidRing = 8;
constexpr uint32_t kTmemO = 0, kTmemS = 256;
constexpr int kTmemCols = 512;
constexpr float kRescaleLog2 = 8.f;                // lazy rescale threshold
constexpr float kLn2 = 0.69314718055994530942f;
constexpr int32_t kNoKey0 = -1;                    // the item's rows see all of its keys
constexpr int kProducerWarp = 8, kMmaWarp = 9, kSchedulerWarp = 10, kConvertWarp = 12;

// Launch shapes, with the registers a thread at launch and after the split:
// bf16 384 x 168 = 64512 = 256 x 208 + 128 x 88; e4m3 512 x 128 = 65536 = 256 x
// 152 + 128 x 88 + 128 x 120.
template <bool F8>
struct Cfg;
template <>
struct Cfg<false> {
    static constexpr int kThreads = 384;
    static constexpr int kSlots = 5, kRawSlots = 0;
    static constexpr int kTileRegs = 208, kAuxRegs = 88, kConvertRegs = 0;
    static_assert(256 * kTileRegs + 128 * kAuxRegs <= kThreads * 168, "register split");
};
template <>
struct Cfg<true> {
    static constexpr int kThreads = 512;
    static constexpr int kSlots = 3, kRawSlots = 4;
    static constexpr int kTileRegs = 152, kAuxRegs = 88, kConvertRegs = 120;
    static_assert(256 * kTileRegs + 128 * kAuxRegs + 128 * kConvertRegs <= kThreads * 128,
                  "register split");
};

// shared memory: Q of both tiles, the 16-bit ring, the raw ring
template <bool F8>
constexpr int smem_bytes() {
    return 2 * kQBytes + Cfg<F8>::kSlots * kSlotBytes + Cfg<F8>::kRawSlots * kRawSlotBytes + 1024;
}
static_assert(smem_bytes<false>() <= 225 * 1024 + 1024 && smem_bytes<true>() <= 225 * 1024 + 1024,
              "dynamic shared memory, with room for the static part");

struct Meta {
    WorkItem it, itB;                // the pair's tiles (itB without rows: none)
    int32_t id;                      // -1: the queue is empty
    int32_t key0, key0B;             // causal origins (kNoKey0: none)
    int32_t rows_off;                // the pair's page rows in the stream
};

enum Bar : int {
    kFull = 0,                       // [slots] bf16: TMA bytes; e4m3: 4 converter warps -> issuer
    kEmpty = kFull + 5,              // [slots] MMA commit -> producer (converters)
    kRawFull = kEmpty + 5,           // [raw slots] TMA bytes -> converters
    kRawEmpty = kRawFull + 4,        // [raw slots] 4 converter warps -> producer
    kSFull = kRawEmpty + 4,          // [2] MMA commit and issuer -> tile warps
    kPFull = kSFull + 2,             // [2 tiles x 2 halves] 4 tile warps -> issuer
    kQReady = kPFull + 4,            // [2] 4 tile warps -> issuer
    kOFull = kQReady + 2,            // [2] MMA commit -> tile warps
    kOEmpty = kOFull + 2,            // [2] 4 tile warps -> issuer
    kMetaFull = kOEmpty + 2,         // [kMeta] scheduler -> every role
    kMetaEmpty = kMetaFull + kMeta,  // [kMeta] the 8 tile warps -> scheduler
    kDrain = kMetaEmpty + kMeta,     // MMA commit -> issuer, before TMEM is freed
    kBars
};

__host__ __device__ constexpr int bar_count(int i, bool f8) {
    if (i >= kFull && i < kEmpty) return f8 ? 4 : 1;
    if (i >= kRawEmpty && i < kSFull) return 4;
    if (i >= kSFull && i < kPFull) return 2;
    if (i >= kPFull && i < kOFull) return 4;
    if (i >= kOEmpty && i < kMetaFull) return 4;
    if (i >= kMetaEmpty && i < kDrain) return 8;
    return 1;
}

template <int N>
__device__ __forceinline__ void reg_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void reg_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

__device__ __forceinline__ int blocks_of(int num_pages) {
    return (num_pages + kBlockPages - 1) / kBlockPages;
}

// e4m3 -> f16 of K (or V) of one block by 128 threads, 8 of its 1024 16-byte
// chunks each: 128 rows of 128 bytes (128-byte swizzled) into two 16 KB
// column blocks (128-byte swizzled).  Rows from v0 (first half) and v1
// (second half) on become zeros.  The 8 chunks are loaded before any is
// stored (a load may not pass an earlier shared store); lanes with c >= 4
// store their second half first, so that a quarter warp's eight stores fall
// into eight bank groups.
__device__ __forceinline__ void widen_block(uint32_t src, uint32_t dst, int v0, int v1, int t) {
    uint4 w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int idx = t + kRows * q, r = idx >> 3, c = idx & 7;
        w[q] = lds128(src + r * 128 + ((c ^ (r & 7)) << 4));
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int idx = t + kRows * q, r = idx >> 3, c = idx & 7;
        if ((r & 63) >= (r < kHalfTokens ? v0 : v1)) w[q] = make_uint4(0u, 0u, 0u, 0u);
        const bool second_first = (c & 4) != 0;
        const uint4 v = second_first ? make_uint4(w[q].z, w[q].w, w[q].x, w[q].y) : w[q];
        uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
        e4m3x4_to_f16x2x2(v.x, a0, a1);
        e4m3x4_to_f16x2x2(v.y, a2, a3);
        e4m3x4_to_f16x2x2(v.z, b0, b1);
        e4m3x4_to_f16x2x2(v.w, b2, b3);
        const int c2 = 2 * (c & 3);
        const int first = second_first ? c2 + 1 : c2;
        const uint32_t row = dst + (c >> 2) * kColBlockBytes + r * 128;
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + ((first ^ (r & 7)) << 4)),
                     "r"(a0), "r"(a1), "r"(a2), "r"(a3)
                     : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + (((first ^ 1) ^ (r & 7)) << 4)),
                     "r"(b0), "r"(b1), "r"(b2), "r"(b3)
                     : "memory");
    }
}

// DIRECT: every pair holds its rows' whole paths, and the kernel writes the
// result itself (an instantiation of its own: a run-time test cost the join
// 3%).
template <bool F8, bool DIRECT>
__global__ void __launch_bounds__(Cfg<F8>::kThreads, 1)
    prefill_kernel(const __grid_constant__ KvMaps maps, const AttnArgs a) {
    using C = Cfg<F8>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ int abort_flag;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int progress;                // pairs the producer is at the end of
    __shared__ int valid_ring[kValidRing];           // valid keys of a block's halves (low bytes)
    __shared__ __align__(8) uint64_t bar_mem[kBars];
    __shared__ Meta meta[kMeta];
    const uint32_t q_smem = (dev::smem_addr(smem_raw) + 1023) & ~1023u;
    const uint32_t ring = q_smem + 2 * kQBytes;
    const uint32_t raw = ring + C::kSlots * kSlotBytes;
    const uint32_t bars = dev::smem_addr(bar_mem);
    auto bar = [&](int i) { return bars + 8u * static_cast<uint32_t>(i); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long limit = a.wait_limit_ns;
    volatile int *abort = &abort_flag;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        progress = 0;
        for (int i = 0; i < kBars; ++i) dev::mbar_init(bar(i), bar_count(i, F8));
        dev::fence_mbar_init();
        dev::prefetch_tensormap(F8 ? &maps.k_box : &maps.k);
        dev::prefetch_tensormap(F8 ? &maps.v_box : &maps.v);
    }
    if (warp == kMmaWarp) tc::alloc<kTmemCols>(dev::smem_addr(&tmem_base));
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // (as in attn_kernel)
    dev::grid_wait();
    if (threadIdx.x == 0) dev::grid_launch_dependents();
    const uint32_t tmem = tmem_base;

    if (warp < 8) {
        // ------------------------------------------------------------ tile warps
        reg_inc<C::kTileRegs>();
        const int t = warp >> 2;                         // tile A or B
        const int r = (warp & 3) * 32 + lane;            // tile row == TMEM lane
        const uint32_t lane_base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t tO = lane_base + kTmemO + 128u * t;
        const uint32_t tS = lane_base + kTmemS + 128u * t;
        const uint32_t q_tile = q_smem + t * kQBytes;
        bool ok = true;
        int u = 0, jp = 0;                               // this tile's blocks and pairs so far
        int pos = 0, blk = 0;                            // ring position and number of the CTA's block
        auto warp_arrive = [&](int i) {
            __syncwarp();
            if (lane == 0) dev::mbar_arrive(bar(i));
        };
        auto has_pair = [&](int k) {
            if (!tc_warp_wait(bar(kMetaFull + k % kMeta), (k / kMeta) & 1, limit, abort, lane)) {
                ok = false;
                return false;
            }
            return meta[k % kMeta].id >= 0;
        };
        auto on_in = [&](int k) { return t == 0 || meta[k % kMeta].itB.nrows > 0; };
        // Q row r of the tile in pair k into shared memory (16 chunks of 16
        // bytes, 128-byte swizzle; zeros past the tile's rows): bf16 by
        // asynchronous copies, with e4m3 KV narrowed to f16 on the way
        auto issue_q = [&](int k) {
            const Meta &m = meta[k % kMeta];
            const WorkItem &it = t == 0 ? m.it : m.itB;
            const bool live = r < it.nrows;
            const int nr = live ? it.row0 + r : 0;
            const int leaf = live ? it.leaf_lo + nr / a.group : 0;   // queries are in DFS order
            const int head = live ? it.kv_head * a.group + nr % a.group : 0;
            const char *src = reinterpret_cast<const char *>(
                static_cast<const __nv_bfloat16 *>(a.q) +
                (static_cast<int64_t>(leaf) * a.num_q_heads + head) * kDim);
            auto dst = [&](int c) {
                return q_tile + (c >> 3) * kQColBlockBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4);
            };
            if constexpr (!F8) {
                const uint32_t bytes = live ? 16u : 0u;
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst(c)),
                                 "l"(src + 16 * c), "r"(bytes)
                                 : "memory");
            } else {
                bool big = false;
#pragma unroll
                for (int c0 = 0; c0 < 16; c0 += 8) {
                    uint4 v[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        v[c] = live ? *reinterpret_cast<const uint4 *>(src + 16 * (c0 + c))
                                    : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst(c0 + c)),
                                     "r"(q_pair_to_f16(v[c].x, big)), "r"(q_pair_to_f16(v[c].y, big)),
                                     "r"(q_pair_to_f16(v[c].z, big)), "r"(q_pair_to_f16(v[c].w, big))
                                     : "memory");
                }
                report_q_range(a, big, lane);
            }
        };
        // ... complete, visible to the tensor core and announced
        auto publish_q = [&]() {
            if constexpr (!F8) asm volatile("cp.async.wait_all;" ::: "memory");
            tc::fence_proxy_async_smem();
            warp_arrive(kQReady + t);
        };
        bool have = has_pair(0);
        if (have && on_in(0)) {
            issue_q(0);
            publish_q();
        }
        for (int k = 0; ok && have; ++k) {
            const Meta &m = meta[k % kMeta];
            const int nb = blocks_of(m.it.num_pages);
            bool more = false, loaded_next = false;
            if (on_in(k)) {
                const WorkItem it = t == 0 ? m.it : m.itB;
                const int key0 = t == 0 ? m.key0 : m.key0B;
                // the row's last visible key, relative to the item's first
                const int t_rel = key0 == kNoKey0 ? (1 << 30) : (it.row0 + r) / a.group - key0;
                const float sl = F8 ? a.scale_log2 * a.k_scale[it.kv_head] : a.scale_log2;
                const unsigned long long slp = dev::f32x2(sl, sl);
                float m_use = -INFINITY, l = 0.f;
                for (int i = 0; i < nb; ++i, ++u) {
                    if (!tc_warp_wait(bar(kSFull + t), u & 1, limit, abort, lane)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    const int vv = valid_ring[(blk + i) % kValidRing];
                    // The scores: bf16 holds all 128 of the row from here to
                    // the exponentials; with e4m3 KV, where the converters take
                    // a third of the registers (and are what the pass waits
                    // for), each half is read twice.
                    uint32_t x[F8 ? 2 : 4][32];
                    auto read_half = [&](int h, uint32_t(&x0)[32], uint32_t(&x1)[32]) {
                        tc::ld32(tS + 64 * h, x0);
                        tc::ld32(tS + 64 * h + 32, x1);
                    };
                    // keys the row does not see (past the last token of a
                    // half, or past the row's own token): -inf
                    const int valid[2] = {vv & 0xff, vv >> 8};
                    auto hide_half = [&](int h, uint32_t(&x0)[32], uint32_t(&x1)[32]) {
                        const int seen = min(valid[h], t_rel - (i * kBlockTokens + h * kHalfTokens) + 1);
                        if (seen < kHalfTokens) {
#pragma unroll
                            for (int q = 0; q < 32; ++q) hide_from(x0[q], q, seen);
#pragma unroll
                            for (int q = 0; q < 32; ++q) hide_from(x1[q], q + 32, seen);
                        }
                    };
                    // the max of 64 scores, as two running ones
                    auto max_half = [](const uint32_t(&x0)[32], const uint32_t(&x1)[32]) {
                        float m0 = __uint_as_float(x0[0]), m1 = __uint_as_float(x1[0]);
#pragma unroll
                        for (int q = 1; q + 1 < 32; q += 2) {
                            m0 = dev::max3(m0, __uint_as_float(x0[q]), __uint_as_float(x0[q + 1]));
                            m1 = dev::max3(m1, __uint_as_float(x1[q]), __uint_as_float(x1[q + 1]));
                        }
                        return dev::max3(m0, m1, fmaxf(__uint_as_float(x0[31]), __uint_as_float(x1[31])));
                    };
                    float mx;
                    if constexpr (F8) {
                        read_half(0, x[0], x[1]);
                        tc::wait_ld();
                        hide_half(0, x[0], x[1]);
                        mx = max_half(x[0], x[1]);
                        read_half(1, x[0], x[1]);
                        tc::wait_ld();
                        hide_half(1, x[0], x[1]);
                        mx = fmaxf(mx, max_half(x[0], x[1]));
                    } else {
                        read_half(0, x[0], x[1]);
                        read_half(1, x[2], x[3]);
                        tc::wait_ld();
                    }
                    // the pair's last S is done: the Q buffer takes the next
                    // pair's rows while this block's softmax runs
                    if (i == nb - 1) {
                        more = has_pair(k + 1);
                        if (!ok) break;
                        if (!F8 && more && on_in(k + 1)) {
                            issue_q(k + 1);
                            loaded_next = true;
                        }
                    }
                    if constexpr (!F8) {
                        hide_half(0, x[0], x[1]);
                        hide_half(1, x[2], x[3]);
                        mx = fmaxf(max_half(x[0], x[1]), max_half(x[2], x[3]));
                    }
                    // P of half h as packed 16-bit pairs, against the reference
                    // max m_use (a row that has seen no key: every x is -inf
                    // and P is 0); returns the running row sums
                    auto exponentiate = [&](int h, uint32_t(&pw)[32], unsigned long long sum) {
                        const float m_ref = m_use == -INFINITY ? 0.f : m_use;
                        const unsigned long long nmp = dev::f32x2(-m_ref, -m_ref);
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            const uint32_t(&xc)[32] = x[(F8 ? 0 : 2 * h) + (c >> 4)];
                            float e0, e1;
                            dev::f32x2_split(
                                dev::fma_f32x2(dev::f32x2(__uint_as_float(xc[2 * (c & 15)]),
                                                          __uint_as_float(xc[2 * (c & 15) + 1])),
                                               slp, nmp),
                                e0, e1);
                            const float p0 = dev::fast_exp2(e0), p1 = dev::fast_exp2(e1);
                            sum = dev::add_f32x2(sum, dev::f32x2(p0, p1));
                            pw[c] = F8 ? dev::pack_f16(p0, p1) : dev::pack_bf16(p0, p1);
                        }
                        return sum;
                    };
                    uint32_t pw[32];
                    unsigned long long lsum = 0ull;
                    const float mb = mx * sl;
                    if (i == 0) {
                        m_use = mb;
                    } else if (__any_sync(0xffffffffu, mb > m_use + kRescaleLog2)) {
                        // (this block's S follows the last PV of the tile: O is complete)
                        const float m_new = fmaxf(m_use, mb);
                        const float alpha = m_new == m_use ? 1.f : dev::fast_exp2(m_use - m_new);
#pragma unroll
                        for (int c = 0; c < kDim / 16; ++c) {
                            uint32_t ov[16];
                            tc::ld16(tO + 16 * c, ov);
                            tc::wait_ld();
#pragma unroll
                            for (int q = 0; q < 16; ++q)
                                ov[q] = __float_as_uint(__uint_as_float(ov[q]) * alpha);
                            tc::st16(tO + 16 * c, ov);
                        }
                        tc::wait_st();
                        l *= alpha;
                        m_use = m_new;
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if constexpr (F8) {
                            read_half(h, x[0], x[1]);
                            tc::wait_ld();
                            hide_half(h, x[0], x[1]);
                        }
                        lsum = exponentiate(h, pw, lsum);
                        tc::st32(tS + 32 * h, pw);
                        // V rows past the half's valid tokens may hold anything
                        // (NaN included): P is 0 there, but 0 * NaN is NaN, so
                        // each tile zeroes them before its PV (the same zeros
                        // twice; the e4m3 converters write them as zeros)
                        if (!F8 && valid[h] < kHalfTokens) {
                            const int vs = (pos + 2 * i + 1) % C::kSlots;
                            if (!tc_warp_wait(bar(kFull + vs), ((pos + 2 * i + 1) / C::kSlots) & 1, limit,
                                              abort, lane)) {
                                ok = false;
                                break;
                            }
                            const uint32_t vst = ring + vs * kSlotBytes;
                            const int n16 = (kHalfTokens - valid[h]) * 2 * 8;
                            for (int q = r; q < n16; q += kRows) {
                                const int row = h * kHalfTokens + valid[h] + q / 16, cb = (q / 8) & 1;
                                const uint32_t at = row / kPageSize * kPagedBytes + cb * (kPagedBytes / 2) +
                                                    row % kPageSize * 128;
                                asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                                                 vst + at + ((q & 7) << 4)),
                                             "r"(0u)
                                             : "memory");
                            }
                            tc::fence_proxy_async_smem();
                        }
                        tc::wait_st();
                        tc::fence_before_sync();
                        warp_arrive(kPFull + 2 * t + h);
                    }
                    if (!ok) break;
                    float l0, l1;
                    dev::f32x2_split(lsum, l0, l1);
                    l += l0 + l1;
                }
                if (!ok) break;
                if (F8 && more && on_in(k + 1)) {
                    issue_q(k + 1);
                    loaded_next = true;
                }
                if (loaded_next) publish_q();
                const bool live = r < it.nrows;
                int64_t out_row = 0;
                float inv = 1.f;
                if constexpr (DIRECT) {
                    // what the merge of one partial gives: o / l, natural-log lse
                    const int nr = live ? it.row0 + r : 0;
                    out_row = static_cast<int64_t>(it.leaf_lo + nr / a.group) * a.num_q_heads +
                              it.kv_head * a.group + nr % a.group;
                    const bool empty = !(l > 0.f);
                    inv = empty ? 0.f : 1.f / l;
                    if (live && a.lse) a.lse[out_row] = empty ? -INFINITY : (m_use + log2f(l)) * kLn2;
                } else if (live) {
                    a.part_ml[static_cast<int64_t>(it.slot_base) + r] = make_float2(m_use, l);
                }
                // the tile's O, once its last PV is done
                if (!tc_warp_wait(bar(kOFull + t), jp & 1, limit, abort, lane)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                const float o_scale = F8 ? a.v_scale[it.kv_head] : 1.f;
                float *dst = DIRECT ? nullptr : a.part_o + (static_cast<int64_t>(it.slot_base) + r) * kDim;
#pragma unroll
                for (int c = 0; c < kDim / 32; ++c) {
                    uint32_t ov[32];
                    tc::ld32(tO + 32 * c, ov);
                    tc::wait_ld();
                    if constexpr (!DIRECT) {
                        if (live) store_row32(dst + 32 * c, ov, o_scale);
                    } else if (live) {
                        uint4 *o16 = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(a.out) +
                                                               out_row * kDim + 32 * c);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            uint32_t w[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                w[e] = dev::pack_bf16(__uint_as_float(ov[8 * q + 2 * e]) * o_scale * inv,
                                                      __uint_as_float(ov[8 * q + 2 * e + 1]) * o_scale * inv);
                            o16[q] = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                tc::fence_before_sync();
                warp_arrive(kOEmpty + t);
                ++jp;
            } else {
                // the tile has no rows in this pair; its Q buffer is free
                more = has_pair(k + 1);
                if (!ok) break;
                if (more && on_in(k + 1)) {
                    issue_q(k + 1);
                    publish_q();
                }
            }
            pos += 2 * nb;
            blk += nb;
            warp_arrive(kMetaEmpty + k % kMeta);
            have = more;
        }
        if (!ok && lane == 0) tc_fail(a, abort, kSiteConsumerFull);
    } else if (F8 && warp >= kConvertWarp) {
        // ------------------------------------------------------------ converters
        reg_dec<F8 ? C::kConvertRegs : 96>();
        const int r = (warp - kConvertWarp) * 32 + lane;
        constexpr int NR = F8 ? C::kRawSlots : 1;
        int pos = 0, blk = 0;
        bool ok = true;
        for (int k = 0; ok; ++k) {
            if (!tc_warp_wait(bar(kMetaFull + k % kMeta), (k / kMeta) & 1, limit, abort, lane)) {
                ok = false;
                break;
            }
            if (meta[k % kMeta].id < 0) break;
            const int nb = blocks_of(meta[k % kMeta].it.num_pages);
            for (int i = 0; i < nb && ok; ++i, ++blk)
                for (int op = 0; op < 2; ++op, ++pos) {
                    const int rs = pos % NR, cs = pos % C::kSlots;
                    if (!tc_warp_wait(bar(kRawFull + rs), (pos / NR) & 1, limit, abort, lane) ||
                        (pos >= C::kSlots && !tc_warp_wait(bar(kEmpty + cs), ((pos / C::kSlots) - 1) & 1,
                                                           limit, abort, lane))) {
                        ok = false;
                        break;
                    }
                    const int vv = valid_ring[blk % kValidRing];
                    widen_block(raw + rs * kRawSlotBytes, ring + cs * kSlotBytes, vv & 0xff, vv >> 8, r);
                    tc::fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        dev::mbar_arrive(bar(kFull + cs));
                        dev::mbar_arrive(bar(kRawEmpty + rs));
                    }
                }
        }
        if (!ok && lane == 0) tc_fail(a, abort, kSiteConsumerFull);
    } else {
        reg_dec<C::kAuxRegs>();
        if (warp == kSchedulerWarp) {
            // -------------------------------------------------------- scheduler
            int nbs[kMeta] = {0, 0, 0, 0};                  // blocks of the last pairs
            auto reached = [&](int pairs) {
                int there = 1;
                if (lane == 0 && progress < pairs) {
                    const uint64_t t0 = dev::global_timer_ns();
                    while (progress < pairs) {
                        if (*abort || static_cast<long long>(dev::global_timer_ns() - t0) > limit) {
                            there = 0;
                            break;
                        }
                        __nanosleep(100);
                    }
                }
                return __shfl_sync(0xffffffffu, there, 0) != 0;
            };
            for (int k = 0;; ++k) {
                const int s = k % kMeta;
                // A pair is pulled once the producer is near the end of the one
                // before (a CTA that pulled as soon as a slot was free took
                // pairs that others had time for: join prefill kernel 553 ->
                // 492 us); pairs of a few blocks are pulled up to kMeta ahead,
                // while together they are no more than kAheadBlocks, so that
                // their records' latency does not add up.
                int need = k;                              // pairs the producer has to be through
                for (int ahead = 0; need > 0 && k - need < kMeta - 1; --need) {
                    ahead += nbs[(need - 1) % kMeta];
                    if (ahead > kAheadBlocks) break;
                }
                if (!reached(need) ||
                    (k >= kMeta &&
                     !tc_warp_wait(bar(kMetaEmpty + s), ((k / kMeta) - 1) & 1, limit, abort, lane))) {
                    if (lane == 0) tc_fail(a, abort, kSiteProducerEmpty);
                    break;
                }
                // a CTA owns pair blockIdx.x of the queue
                // (with no more pairs than CTAs the counter is left alone: no
                // merge follows to set it back when the pairs write the result)
                int p = static_cast<int>(blockIdx.x);
                if (k > 0) {
                    if (lane == 0)
                        p = a.num_wide_items <= 2 * a.num_ctas ? a.num_wide_items : atomicAdd(a.queue_next, 1);
                    p = __shfl_sync(0xffffffffu, p, 0);
                }
                int id = !*abort && 2 * p + 1 < a.num_wide_items ? 2 * p : -1;
                if (lane == 0) {
                    Meta &m = meta[s];
                    if (id >= 0) {
                        const WorkItem it = a.items[id], itB = a.items[id + 1];
                        bool bad = it.num_pages <= 0 || it.nrows <= 0 || it.nrows > kRows ||
                                   it.row0 % a.group != 0;
                        if (itB.nrows != 0)
                            bad = bad || itB.nrows < 0 || itB.nrows > kRows || itB.row0 % a.group != 0 ||
                                  itB.num_pages != it.num_pages || itB.page_pos != it.page_pos ||
                                  itB.last_valid != it.last_valid || itB.kv_head != it.kv_head;
                        if (bad) {
                            if (!*abort) {
                                *abort = 1;
                                dev::record_error(a.err, PARASON_EINVAL, kSiteBadItem);
                            }
                            id = -1;
                        } else {
                            m.it = it;
                            m.itB = itB;
                            m.key0 = a.item_key0[id];
                            m.key0B = a.item_key0[id + 1];
                            m.rows_off = a.item_rows[id];
                        }
                    }
                    m.id = id;
                    dev::mbar_arrive(bar(kMetaFull + s));
                }
                if (__shfl_sync(0xffffffffu, id, 0) < 0) break;
                __syncwarp();
                nbs[s] = blocks_of(meta[s].it.num_pages);
            }
        } else if (warp == kProducerWarp) {
            // -------------------------------------------------------- producer
            constexpr int NS = F8 ? C::kRawSlots : C::kSlots;
            constexpr int kLoadBytes = F8 ? kRawSlotBytes : kSlotBytes;
            constexpr int kFullBar = F8 ? kRawFull : kFull, kEmptyBar = F8 ? kRawEmpty : kEmpty;
            const bool skip_first = a.debug_flags & PARASON_DEBUG_SKIP_FIRST_LOAD;
            const int page_rows = a.num_kv_heads * kPageSize;   // TMA rows between consecutive pages
            const uint64_t pol = dev::l2_evict_normal_policy();
            int last_issue[NS];
            for (int s = 0; s < NS; ++s) last_issue[s] = -1;
            int pos = 0, blk = 0, st = 0;                // slot st = pos % NS
            bool ok = true;
            for (int k = 0; ok; ++k) {
                if (!tc_warp_wait(bar(kMetaFull + k % kMeta), (k / kMeta) & 1, limit, abort, lane)) {
                    ok = false;
                    break;
                }
                const Meta &m = meta[k % kMeta];
                if (m.id < 0) break;
                const int np = m.it.num_pages, nb = blocks_of(np);
                const int tokens = (np - 1) * kPageSize + m.it.last_valid;
                const int32_t *rows = a.stream_rows + m.rows_off;
                const int kvh = m.it.kv_head;
                // page rows 32 at a time (4 blocks), the next 32 requested
                // ahead (the stream is padded by 32 entries); what the blocks
                // need of them is worked out for all 32 at once, as bit masks
                // with a bit per page: `ends` (a page that ends a node: it
                // carries 16 - its valid tokens in the row's low bits; or
                // padding) and `follows` (next in the pool to the page before)
                int32_t next = rows[lane], win = 0;
                uint32_t ends = 0, follows = 0, pool = 0;
                for (int i = 0; i < nb && ok; ++i, ++blk) {
                    if (i == max(0, nb - 2) && lane == 0) progress = k + 1;
                    const int pg0 = i * kBlockPages, w0 = pg0 & 31;
                    if (w0 == 0) {
                        // past the item: the first row past the pool, which TMA
                        // fills with zeros
                        win = pg0 + lane < np ? next : a.kv_rows;
                        if (pg0 + 32 < np) next = rows[pg0 + 32 + lane];
                        const int32_t base = win & ~(kPageSize - 1);
                        const int32_t before = __shfl_up_sync(0xffffffffu, base, 1);
                        pool = __ballot_sync(0xffffffffu, win < a.kv_rows);
                        ends = __ballot_sync(0xffffffffu, win >= a.kv_rows || (win & (kPageSize - 1)));
                        follows = __ballot_sync(0xffffffffu, win < a.kv_rows && base == before + page_rows);
                    }
                    int valid[2];
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const uint32_t e4 = (ends >> (w0 + 4 * hh)) & 15u;
                        valid[hh] = kHalfTokens;
                        if (e4) {                        // tokens before and in the first such page
                            const int p = __ffs(e4) - 1;
                            const int32_t w = __shfl_sync(0xffffffffu, win, w0 + 4 * hh + p);
                            valid[hh] = p * kPageSize + (w < a.kv_rows ? kPageSize - (w & (kPageSize - 1)) : 0);
                        }
                        valid[hh] = max(0, min(valid[hh], tokens - (i * kBlockTokens + hh * kHalfTokens)));
                    }
                    if (lane == 0) valid_ring[blk % kValidRing] = valid[0] | (valid[1] << 8);
                    const bool whole = F8 && ((pool >> w0) & 1u) && ((follows >> w0) & 0xfeu) == 0xfeu;
                    const int32_t row0 = __shfl_sync(0xffffffffu, win, w0) & ~(kPageSize - 1);
                    for (int op = 0; op < 2; ++op, ++pos, st = st + 1 == NS ? 0 : st + 1) {
                        if (pos >= NS && !tc_warp_wait(bar(kEmptyBar + st), ((pos / NS) - 1) & 1, limit, abort,
                                                       lane)) {
                            ok = false;
                            break;
                        }
                        if (skip_first && pos == 0) continue;
                        const uint32_t fb = bar(kFullBar + st);
                        const uint32_t dst0 = (F8 ? raw : ring) + st * kLoadBytes;
                        last_issue[st] = pos;
                        if (lane == 0) dev::mbar_arrive_expect_tx(fb, kLoadBytes);
                        if (whole) {                     // 8 pages in a row: one box
                            if (lane == 0)
                                dev::tma_load_5d_hint(dst0, op ? &maps.v_box : &maps.k_box, 0, 0,
                                                      row0 / page_rows, 0, kvh, fb, pol);
                            continue;
                        }
                        __syncwarp();
                        if constexpr (!F8) {
                            // a box of 4 KB per page (lane: page): K as [half][column
                            // block][8 rows], V as [column block][16 rows]
                            const int32_t pr = __shfl_sync(0xffffffffu, win, w0 + (lane & 7));
                            const uint32_t dst = dst0 + (lane & 7) * kPagedBytes;
                            if (lane < kBlockPages) {
                                if (op == 0)
                                    dev::tma_load_5d_hint(dst, &maps.k, 0, 0, 0, 0, pr / kPageSize, fb, pol);
                                else
                                    dev::tma_load_4d_hint(dst, &maps.v, 0, 0, 0, pr / kPageSize, fb, pol);
                            }
                            continue;
                        }
                        // e4m3: a box per run of 4 pages, or per page (lane: page j of half h)
                        const int h = lane >> 2, j = lane & 3;
                        const uint32_t dst = dst0 + h * kHalfTokens * 128;
                        const int lane_pg = w0 + ((4 * h + j) & 7);
                        const int32_t my_row = __shfl_sync(0xffffffffu, win, lane_pg) & ~(kPageSize - 1);
                        const int first = w0 + 4 * (h & 1);
                        const bool my_run = ((pool >> first) & 1u) && ((follows >> first) & 0xeu) == 0xeu;
                        if (lane < kBlockPages && my_run) {
                            if (j == 0)
                                dev::tma_load_5d_hint(dst, op ? &maps.v_run : &maps.k_run, 0, 0, 0, kvh,
                                                      my_row / page_rows, fb, pol);
                        } else if (lane < kBlockPages) {
                            dev::tma_load_3d(dst + j * kPageSize * 128, op ? &maps.v : &maps.k, 0, 0,
                                             my_row, fb);
                        }
                    }
                }
            }
            if (!ok && lane == 0) tc_fail(a, abort, kSiteProducerEmpty);
            // every copy this CTA issued must land before its shared memory goes
            if (lane == 0)
                for (int s = 0; s < NS; ++s)
                    if (last_issue[s] >= 0)
                        dev::mbar_wait_bounded(bar(kFullBar + s), (last_issue[s] / NS) & 1, kDrainLimitNs,
                                               nullptr);
            __syncwarp();
        } else if (warp == kMmaWarp) {
            // -------------------------------------------------------- MMA issuer
            // (the whole warp runs the loop, one elected lane issues: see elect_one)
            constexpr uint32_t kIdS = F8 ? tc::idesc_f16_f32(kRows, kBlockTokens, false)
                                         : tc::idesc_bf16_f32(kRows, kBlockTokens, false);
            constexpr uint32_t kIdPV = F8 ? tc::idesc_f16_f32(kRows, kDim, true)
                                          : tc::idesc_bf16_f32(kRows, kDim, true);
            // A wait that runs out leaves its mark, and the warp goes on together
            // to the next point where it looks (lanes that part would leave the
            // others waiting in elect.sync; what is issued in between works on
            // this CTA's own memory and is thrown away).
            bool bad = false;
            auto wait = [&](int i, int parity) {
                if (!tc_wait(bar(i), static_cast<uint32_t>(parity & 1), limit, abort)) {
                    tc_fail(a, abort, kSiteConsumerFull);
                    bad = true;
                }
            };
            auto failed = [&]() { return __any_sync(0xffffffffu, bad) != 0; };
            // K and V of a block: with bf16 KV page by page (8-row groups of K 2
            // KB apart, column blocks 1 KB; of V a 16-token step 4 KB, column
            // blocks 2 KB), widened e4m3 as column blocks of 128 tokens
            constexpr uint32_t kKGroup = F8 ? 1024 : 2048, kKCol = F8 ? kColBlockBytes : 1024;
            constexpr uint32_t kVStep = F8 ? kPageSize * 128 : kPagedBytes;
            constexpr uint32_t kVCol = F8 ? kColBlockBytes : kPagedBytes / 2;
            const uint64_t desc_k = tc::smem_desc_sw128(ring, 16, kKGroup);
            const uint64_t desc_v = tc::smem_desc_sw128(ring, kVCol, 1024);
            const uint64_t desc_q = tc::smem_desc_sw128(q_smem, 16, 1024);
            int st = 0, ph = 0;              // ring slot of the next operand, and its phase
            auto advance = [&]() {
                if (++st == C::kSlots) {
                    st = 0;
                    ph ^= 1;
                }
            };
            // S_t of the block whose K is in slot st (given back with the last tile's)
            auto issue_s = [&](int t, bool last) {
                const uint64_t kd = desc_k + static_cast<uint64_t>(st * (kSlotBytes >> 4));
                const uint64_t qd = desc_q + static_cast<uint64_t>(t * (kQBytes >> 4));
                const uint32_t tS = tmem + kTmemS + 128u * t;
                if (tc::elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < kDim / 16; ++ks) {
                        const uint32_t off = ((ks >> 2) * kQColBlockBytes + (ks & 3) * 32) >> 4;
                        const uint32_t koff = ((ks >> 2) * kKCol + (ks & 3) * 32) >> 4;
                        tc::mma_bf16(tS, qd + off, kd + koff, kIdS, ks > 0);
                    }
                    // the commit completes with the product; the plain arrive
                    // carries the producer's writes (valid_ring) along
                    tc::commit(bar(kSFull + t));
                    dev::mbar_arrive(bar(kSFull + t));
                    if (last) tc::commit(bar(kEmpty + st));
                }
            };
            int u[2] = {0, 0}, j[2] = {0, 0};                 // blocks and pairs of each tile so far
            for (int k = 0;; ++k) {
                wait(kMetaFull + k % kMeta, k / kMeta);
                if (failed()) break;
                const Meta &m = meta[k % kMeta];
                if (m.id < 0) break;
                const int last = m.itB.nrows > 0 ? 1 : 0;
                const int nb = blocks_of(m.it.num_pages);
                wait(kQReady, j[0]);
                if (last) wait(kQReady + 1, j[1]);
                wait(kFull + st, ph);
                tc::fence_after_sync();
                issue_s(0, last == 0);
                if (last) issue_s(1, true);
                advance();
                for (int i = 0; i < nb; ++i) {
                    if (failed()) break;
                    // V of the block and K of the next one, waited for before P is
                    const int sv = st;
                    const uint64_t vd = desc_v + static_cast<uint64_t>(sv * (kSlotBytes >> 4));
                    wait(kFull + st, ph);
                    advance();
                    if (i + 1 < nb) wait(kFull + st, ph);
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        if (t > last) break;
                        const uint32_t tO = tmem + kTmemO + 128u * t;
                        const uint32_t tP = tmem + kTmemS + 128u * t;
                        if (i == 0 && j[t] > 0) wait(kOEmpty + t, j[t] - 1);
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            wait(kPFull + 2 * t + hf, u[t]);
                            tc::fence_after_sync();
                            if (tc::elect_one()) {
#pragma unroll
                                for (int kk = 4 * hf; kk < 4 * hf + 4; ++kk)
                                    tc::mma_bf16_tmem_a(tO, tP + 8u * kk, vd + ((kk * kVStep) >> 4), kIdPV,
                                                        i > 0 || kk > 0);
                                if (hf == 1 && t == last) tc::commit(bar(kEmpty + sv));
                                if (hf == 1 && i == nb - 1) tc::commit(bar(kOFull + t));
                            }
                        }
                        ++u[t];
                        if (i + 1 < nb) {
                            issue_s(t, t == last);
                            if (t == last) advance();
                        }
                    }
                }
                ++j[0];
                j[1] += last;
            }
            // every MMA must finish before TMEM is freed
            if (tc::elect_one()) tc::commit(bar(kDrain));
            dev::mbar_wait_bounded(bar(kDrain), 0, kDrainLimitNs, nullptr);
            __syncwarp();
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == kMmaWarp) tc::dealloc<kTmemCols>(tmem);
}

// Shared memory is configured once per device; the launch needs one CTA per SM.
constexpr int kMaxConfigDevices = 64;

template <bool F8, bool DIRECT>
cudaError_t configure() {
    static std::mutex mu;
    static bool done[kMaxConfigDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxConfigDevices) return cudaErrorNotSupported;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(prefill_kernel<F8, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_bytes<F8>());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(prefill_kernel<F8, DIRECT>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    done[dev] = true;
    return cudaSuccess;
}

template <bool F8, bool DIRECT>
cudaError_t launch(const AttnArgs &a, const KvMaps &maps, cudaStream_t stream) {
    const cudaError_t e = configure<F8, DIRECT>();
    if (e != cudaSuccess) return e;
    return launch_dependent(a.early != 0, prefill_kernel<F8, DIRECT>, dim3(a.num_ctas),
                            dim3(Cfg<F8>::kThreads), smem_bytes<F8>(), stream, maps, a);
}

}  // namespace

cudaError_t launch_prefill(const AttnArgs &a, const KvMaps &maps, int mode, cudaStream_t stream) {
    if (a.num_items <= 0 || a.num_ctas <= 0) return cudaSuccess;
    if (mode == PARASON_FP8_E4M3_KV)
        return a.out ? launch<true, true>(a, maps, stream) : launch<true, false>(a, maps, stream);
    return a.out ? launch<false, true>(a, maps, stream) : launch<false, false>(a, maps, stream);
}

}  // namespace parason
