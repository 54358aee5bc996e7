// attn_fp32.cu -- node-chunk attention for fp32 q/K/V (the fp32 parity mode).
//
// Same work items as the bf16 kernel (tiles of at most 16 rows in this mode),
// computed with fp32 FMAs so that results stay within 1e-5 of fp64.
//
// One CTA of 4 warps per item, kCtasPerSm of them on an SM.  The item's pages
// (16 tokens of one kv head: contiguous in the pool) come by bulk copies into
// a ring of kRing bytes; the CTAs of an SM keep 192 KB in flight, which is
// what HBM needs.  A warp owns up to 4 rows of the tile (a branch of 4 q
// heads, a quarter of a 16-row tile): a tile of at most 4 rows spreads its
// pages over the 4 warps, one of up to 8 rows over two pairs, wider tiles
// run every page on every warp, so that a page is staged once for its rows.
//
// Inside a warp, the 4 groups of 8 lanes take every 4th token of a page and
// the lanes of a group take 16-byte chunks s, s + 8, ... of the token's row
// (conflict-free 128-byte reads).  A lane then holds partial dots of 4 tokens
// x 4 rows: 14 shuffles reduce and transpose them over the 8 lanes, where 4
// rows took 5 shuffles a token before, and leave 2 scores a lane, so that a
// page costs two exponentials a lane.  P goes back by shuffles, O is kept per
// token group and reduced once per item.  Both products are packed
// fma.rn.f32x2 (each half rounds as an fp32 FMA does).
//
// What bounds it: HBM.  A page of a 4-row tile is 16 KB (d 128) for about 430
// warp instructions.  16 branches of 512 to 4096 tokens under a 2048-token
// prefix, 32 q / 8 kv heads, d 128 (327 MB of KV, 48 us at 6.8 TB/s): 442 us
// with a warp reduction per (token, row) and direct global loads, 70 us with
// K and V of a page copied and awaited together, 65.5 us now.  A tile of at most
// 4 rows has one stage per warp at d 128, which was empty while its copies
// came: its K is now refilled as soon as the scores are made, its V after the
// page (16 kv heads of one q head each: 48.4 -> 45.4 us).  Wider tiles keep one
// copy: there the pages are shared and the FMAs bound it (two-level tree of
// 64 q heads 75 us; 80 us with split copies).
#include "device_common.cuh"
#include "internal.h"

namespace parason {
namespace {

constexpr int kWarps = 4;
constexpr int kThreads = kWarps * 32;
constexpr int kWarpRows = 4;
constexpr int kCtasPerSm = 3;
constexpr int kRing = 64 * 1024;
constexpr long long kDrainNs = 1000000000LL;
constexpr float kGrowLog2 = 8.f;      // the reference max moves once a score passes it by 2^8

template <int D>
struct F32 {
    static constexpr int kTensorBytes = kPageSize * D * 4;    // K (or V) of one (page, kv head)
    static constexpr int kStageBytes = 2 * kTensorBytes;
    static constexpr int kStages = kRing / kStageBytes;       // 4 (d 128) or 8 (d 64)
    static constexpr int kChunks = D / 32;                    // 16-byte chunks of a row per lane
    // (at d 64 a warp has two stages and the split copies were 8% slower)
    static constexpr bool kSplit = D == 128;
    static_assert(kStages % kWarps == 0, "a stage's next page belongs to the same warps");
};

struct alignas(16) Pairs {
    unsigned long long a, b;          // 4 consecutive fp32 values
};

__device__ __forceinline__ Pairs lds_pairs(uint32_t addr) {
    Pairs p;
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(p.a), "=l"(p.b) : "r"(addr));
    return p;
}

// contiguous global bytes into shared memory, completing on `bar`
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

template <int D>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
    attn_fp32_kernel(const AttnArgs a, const float *__restrict__ kp, const float *__restrict__ vp) {
    using S = F32<D>;
    constexpr int NC = S::kChunks, NS = S::kStages;
    extern __shared__ __align__(128) uint8_t ring_mem[];
    __shared__ float sc_o[kWarps][kWarpRows][D];
    __shared__ float2 sc_ml[kWarps][kWarpRows];
    __shared__ __align__(8) uint64_t bars[3 * NS];
    __shared__ int failed;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = lane & 7, tg = lane >> 3;            // chunk and token group of the lane
    const int b0 = lane & 1, b1 = (lane >> 1) & 1, b2 = (lane >> 2) & 1;
    const uint32_t ring = dev::smem_addr(ring_mem);
    const uint32_t full = dev::smem_addr(bars), empty = full + 8 * NS, vfull = empty + 8 * NS;

    dev::grid_wait();
    const WorkItem it = a.items[blockIdx.x];
    const int row_groups = (it.nrows + kWarpRows - 1) / kWarpRows;   // 1 .. 4, each a warp's rows
    const int RG = row_groups == 3 ? 4 : row_groups;
    const int PG = kWarps / RG;                        // warps that share a row group's pages
    const int rgi = warp / PG, pgi = warp % PG;
    // K and V copied, awaited and refilled one by one: a stage's K comes while
    // the page's softmax and V run
    const bool split = S::kSplit && row_groups == 1;
    if (threadIdx.x == 0) {
        failed = 0;
        for (int i = 0; i < NS; ++i) {
            dev::mbar_init(full + 8 * i, 1);
            dev::mbar_init(empty + 8 * i, row_groups);
            dev::mbar_init(vfull + 8 * i, 1);
        }
        dev::fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) dev::grid_launch_dependents();

    // page pg of the item into its stage; pages pg, pg + PG, ... are this
    // warp's, and the warps of row group 0 load them
    const int first_ids = lane < it.num_pages ? a.page_ids[it.page_pos + lane] : 0;
    auto load = [&](int pg, bool k, bool v) {
        const int page = pg < 32 ? __shfl_sync(0xffffffffu, first_ids, pg) : a.page_ids[it.page_pos + pg];
        if (lane == 0) {
            const int64_t off = (static_cast<int64_t>(page) * a.num_kv_heads + it.kv_head) * kPageSize * D;
            const uint32_t dst = ring + (pg % NS) * S::kStageBytes;
            const uint32_t bar = full + 8 * (pg % NS), vbar = split ? vfull + 8 * (pg % NS) : bar;
            if (k) {
                dev::mbar_arrive_expect_tx(bar, split ? S::kTensorBytes : S::kStageBytes);
                bulk_load(dst, kp + off, S::kTensorBytes, bar);
            }
            if (v) {
                if (split) dev::mbar_arrive_expect_tx(vbar, S::kTensorBytes);
                bulk_load(dst + S::kTensorBytes, vp + off, S::kTensorBytes, vbar);
            }
        }
    };
    const bool active = rgi < row_groups;
    int loaded = pgi, used = pgi;                      // next own page to load, to use
    if (rgi == 0)
        for (; loaded < it.num_pages && loaded < NS; loaded += PG) load(loaded, true, true);

    Pairs q[kWarpRows][NC], o[kWarpRows][NC];
#pragma unroll
    for (int r = 0; r < kWarpRows; ++r) {
        const int tr = rgi * kWarpRows + r;
        const float *qrow = nullptr;
        if (tr < it.nrows) {
            const int nr = it.row0 + tr;
            const int leaf = a.dfs_leaf[it.leaf_lo + nr / a.group];
            const int head = it.kv_head * a.group + nr % a.group;
            qrow = static_cast<const float *>(a.q) + (static_cast<int64_t>(leaf) * a.num_q_heads + head) * D;
        }
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            q[r][j] = qrow ? *reinterpret_cast<const Pairs *>(qrow + 4 * (s + 8 * j)) : Pairs{0ull, 0ull};
            o[r][j] = Pairs{0ull, 0ull};
        }
    }
    // this lane's scores: rows 2 b0 and 2 b0 + 1 of token 4 (2 b2 + b1) + tg
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};

    bool ok = true, k_ahead = false;                   // K of page `loaded` is on its way
    for (; active && used < it.num_pages; used += PG) {
        const int st = used % NS;
        if (!dev::mbar_wait_bounded(full + 8 * st, (used / NS) & 1, a.wait_limit_ns, nullptr)) {
            ok = false;
            break;
        }
        const int valid = used == it.num_pages - 1 ? it.last_valid : kPageSize;
        const uint32_t kb = ring + st * S::kStageBytes + 16 * s;
        const uint32_t vb = kb + S::kTensorBytes;
        // partial dots of token 4 i + tg and row r over this lane's chunks
        float d[4][kWarpRows];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            unsigned long long acc[kWarpRows] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const Pairs k = lds_pairs(kb + (4 * i + tg) * (D * 4) + 128 * j);
#pragma unroll
                for (int r = 0; r < kWarpRows; ++r) {
                    acc[r] = dev::fma_f32x2(q[r][j].a, k.a, acc[r]);
                    acc[r] = dev::fma_f32x2(q[r][j].b, k.b, acc[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < kWarpRows; ++r) {
                float lo, hi;
                dev::f32x2_split(acc[r], lo, hi);
                d[i][r] = lo + hi;
            }
        }
        if (split && loaded < it.num_pages) {
            __syncwarp();
            load(loaded, true, false);
            k_ahead = true;
        }
        // sums over the 8 lanes, halving the (token, row) set each time
        float x[2];
        {
            float e[2][kWarpRows], f[kWarpRows];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int r = 0; r < kWarpRows; ++r)
                    e[i][r] = (b2 ? d[2 + i][r] : d[i][r]) +
                              __shfl_xor_sync(0xffffffffu, b2 ? d[i][r] : d[2 + i][r], 4);
#pragma unroll
            for (int r = 0; r < kWarpRows; ++r)
                f[r] = (b1 ? e[1][r] : e[0][r]) + __shfl_xor_sync(0xffffffffu, b1 ? e[0][r] : e[1][r], 2);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                x[h] = (b0 ? f[2 + h] : f[h]) + __shfl_xor_sync(0xffffffffu, b0 ? f[h] : f[2 + h], 1);
        }
        const bool seen = 4 * (2 * b2 + b1) + tg < valid;
#pragma unroll
        for (int h = 0; h < 2; ++h) x[h] = seen ? x[h] * a.scale_log2 : -INFINITY;
        // the reference max moves (and o, l with it) only when a score passes
        // it by 2^8: always at the warp's first page, seldom later
        if (__any_sync(0xffffffffu, x[0] > m[0] + kGrowLog2 || x[1] > m[1] + kGrowLog2)) {
            float al[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float mx = x[h];
#pragma unroll
                for (int w = 2; w < 32; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
                const float mn = fmaxf(m[h], mx);
                al[h] = m[h] == mn ? 1.f : exp2f(m[h] - mn);
                m[h] = mn;
                l[h] *= al[h];
            }
#pragma unroll
            for (int r = 0; r < kWarpRows; ++r) {
                const float ar = __shfl_sync(0xffffffffu, al[r & 1], r >> 1);
                const unsigned long long ar2 = dev::f32x2(ar, ar);
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    o[r][j].a = dev::mul_f32x2(o[r][j].a, ar2);
                    o[r][j].b = dev::mul_f32x2(o[r][j].b, ar2);
                }
            }
        }
        float p[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            p[h] = exp2f(x[h] - m[h]);
            l[h] += p[h];
        }
        if (split && !dev::mbar_wait_bounded(vfull + 8 * st, (used / NS) & 1, a.wait_limit_ns, nullptr)) {
            ok = false;
            break;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            unsigned long long pr[kWarpRows];
#pragma unroll
            for (int r = 0; r < kWarpRows; ++r) {
                const float v = __shfl_sync(0xffffffffu, p[r & 1], (lane & 24) | (i << 1) | (r >> 1));
                pr[r] = dev::f32x2(v, v);
            }
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                Pairs v = lds_pairs(vb + (4 * i + tg) * (D * 4) + 128 * j);
                // slots past the node's length may hold anything (NaN included)
                if (4 * i + tg >= valid) v = Pairs{0ull, 0ull};
#pragma unroll
                for (int r = 0; r < kWarpRows; ++r) {
                    o[r][j].a = dev::fma_f32x2(pr[r], v.a, o[r][j].a);
                    o[r][j].b = dev::fma_f32x2(pr[r], v.b, o[r][j].b);
                }
            }
        }
        __syncwarp();
        // the stage is read: refill it (once every row group has read it)
        if (row_groups > 1 && lane == 0) dev::mbar_arrive(empty + 8 * st);
        if (rgi == 0 && loaded < it.num_pages) {
            if (row_groups > 1 &&
                !dev::mbar_wait_bounded(empty + 8 * st, (used / NS) & 1, a.wait_limit_ns, nullptr)) {
                ok = false;
                used += PG;
                break;
            }
            load(loaded, !split, true);
            k_ahead = false;
            loaded += PG;
        }
    }
    if (!ok) {
        if (lane == 0) {
            dev::record_error(a.err, PARASON_ETIMEOUT, kSiteConsumerFull);
            failed = 1;
        }
        // copies this warp issued must land before the CTA's shared memory goes
        if (rgi == 0)
            for (int pg = used; pg <= loaded && pg < it.num_pages; pg += PG) {
                // k_ahead: the wait for V of page `used` failed, its K was read
                // and K of page `loaded` may be on its way into the same stage
                if (pg < loaded ? !(k_ahead && pg == used) : k_ahead)
                    dev::mbar_wait_bounded(full + 8 * (pg % NS), (pg / NS) & 1, kDrainNs, nullptr);
                if (pg < loaded && split)
                    dev::mbar_wait_bounded(vfull + 8 * (pg % NS), (pg / NS) & 1, kDrainNs, nullptr);
            }
    }

    // l over the tokens; o over the token groups, leaving lane group tg row tg
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int w = 2; w < 32; w <<= 1) l[h] += __shfl_xor_sync(0xffffffffu, l[h], w);
    const int c0 = (lane >> 3) & 1, c1 = lane >> 4;
    float4 t[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        float y[4][4], u[2][4], w[4];
#pragma unroll
        for (int r = 0; r < kWarpRows; ++r) {
            dev::f32x2_split(o[r][j].a, y[r][0], y[r][1]);
            dev::f32x2_split(o[r][j].b, y[r][2], y[r][3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                u[h][e] = (c1 ? y[2 + h][e] : y[h][e]) +
                          __shfl_xor_sync(0xffffffffu, c1 ? y[h][e] : y[2 + h][e], 16);
            w[e] = (c0 ? u[1][e] : u[0][e]) + __shfl_xor_sync(0xffffffffu, c0 ? u[0][e] : u[1][e], 8);
        }
        t[j] = make_float4(w[0], w[1], w[2], w[3]);
    }
    if (PG == 1) {                                     // the warp's rows are whole
        const int tr = rgi * kWarpRows + tg;
        const int64_t slot = static_cast<int64_t>(it.slot_base) + tr;
        if (tr < it.nrows)
#pragma unroll
            for (int j = 0; j < NC; ++j)
                *reinterpret_cast<float4 *>(a.part_o + slot * D + 4 * (s + 8 * j)) = t[j];
        if (lane < 2)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int mr = rgi * kWarpRows + 2 * b0 + h;
                if (mr < it.nrows) a.part_ml[static_cast<int64_t>(it.slot_base) + mr] = make_float2(m[h], l[h]);
            }
        return;
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) *reinterpret_cast<float4 *>(&sc_o[warp][tg][4 * (s + 8 * j)]) = t[j];
    if (lane < 2)
#pragma unroll
        for (int h = 0; h < 2; ++h) sc_ml[warp][2 * b0 + h] = make_float2(m[h], l[h]);
    __syncthreads();
    if (failed) return;
    for (int idx = threadIdx.x; idx < it.nrows * D; idx += kThreads) {
        const int r = idx / D, c = idx % D;
        const int w0 = (r / kWarpRows) * PG, rr = r % kWarpRows;
        float M = -INFINITY;
        for (int w = 0; w < PG; ++w) M = fmaxf(M, sc_ml[w0 + w][rr].x);
        float L = 0.f, acc = 0.f;
        for (int w = 0; w < PG; ++w) {
            const float e = exp2f(sc_ml[w0 + w][rr].x - M);
            L += e * sc_ml[w0 + w][rr].y;
            acc += e * sc_o[w0 + w][rr][c];
        }
        const int64_t slot = static_cast<int64_t>(it.slot_base) + r;
        a.part_o[slot * D + c] = acc;
        if (c == 0) a.part_ml[slot] = make_float2(M, L);
    }
}

template <int D>
cudaError_t launch(const AttnArgs &a, const float *k_pages, const float *v_pages, cudaStream_t stream) {
    // per device and idempotent: set before each launch, as the device may change
    const cudaError_t e = cudaFuncSetAttribute(attn_fp32_kernel<D>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, kRing);
    if (e != cudaSuccess) return e;
    return launch_dependent(a.early != 0, attn_fp32_kernel<D>, dim3(a.num_items), dim3(kThreads), kRing, stream, a,
                            k_pages, v_pages);
}

}  // namespace

cudaError_t launch_attn_fp32(const AttnArgs &a, const float *k_pages, const float *v_pages,
                             int head_dim, cudaStream_t stream) {
    if (a.num_items <= 0) return cudaSuccess;
    if (head_dim == 128) return launch<128>(a, k_pages, v_pages, stream);
    if (head_dim == 64) return launch<64>(a, k_pages, v_pages, stream);
    return cudaErrorNotSupported;
}

}  // namespace parason
