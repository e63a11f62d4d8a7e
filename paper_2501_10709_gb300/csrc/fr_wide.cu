// fr_wide.cu -- the stock ensemble's networks (two hidden layers up to 256
// wide, inputs up to 304, up to 32 outputs; BF16 or FP16) as a batch forward
// with resident weights, for every batch size.
//
// One agent's 303 KB of weights do not fit one SM's operand memory twice
// over, so a pair of CTAs (a cluster of two) shares an agent: CTA c computes
// units 128 c .. 128 c + 127 of both hidden layers for the pair's tile of up
// to 64 rows.  Its halves of the first two layers sit in tensor memory (152 +
// 128 columns at 301-256-256-30) for as long as the CTA lives, where the MMA
// reads them at full rate (an A operand in shared memory takes 1.2 to 1.5
// times as long), and the small output layer in shared memory.  The layers run
// transposed, D[unit][row] = W[unit][k] X[k][row]: M = 128 units, N = the
// tile's rows, so that a batch of eight rows pays for sixteen and not for 128,
// a thread's bias is a register, and eight rows of a unit are one 16-byte
// store (MN-major operand: 8 x 8 core matrices 1,024 bytes apart along k, 128
// along the rows).  Each CTA writes its half of the hidden activations to its
// own and, with asynchronous stores that complete bytes on the other's
// barrier, to its partner's operand.  The output layer of tile i runs on CTA
// i % 2, rows as M = 64 (row r in lane 32 (r / 16) + r % 16).
//
// ensemble_act on a small batch runs the agents' pairs as one cluster: the
// others send their outputs to agent 0's CTAs, which write the weighted mean
// (no per-agent outputs in memory, no second launch, no allocation).
//
// Warps: 0-3 first layer's epilogue, 4-7 second's, 8-11 outputs, 12-19 the
// observation rows (fp32 loads in row order, 16-bit operand out: no tiling
// pass over the batch), 20 issues the MMAs.  Persistent over the tiles of its
// agent: while tile i's first layer runs, tile i - 1 is in its second and
// i - 2 in its third.  Products, their order along k and every rounding are
// those of k_tc_forward: the same bits.
//
// Measured on 3 x 301-256-256-30 (whole calls; before: k_tc_forward below
// 19,456 rows, a tiling pass and k_tc_actor2 above): ensemble_act on 8 rows
// 43.1 -> 12.0 us, on 2,048 rows 51.3 -> 17.4 us; ensemble_forward on 77,824
// rows 151 -> 127 us.  A tile of 64 rows takes about 4,700 cycles there, of
// which the tensor pipe works 1,500: a K = 16 step of 64 rows is 32 cycles of
// MMA but 45 to 70 of issue (its operands go to uniform registers one by one,
// and the code of 21 warps in five roles does not stay in the instruction
// caches: unrolling the issue loops made it slower, compile-time strides
// faster), and the loader's conversion and copies take as long as both layers.
// Small batches are bound by the chain of three layers with an exchange
// between CTAs after each of the first two (about 5,500 cycles), behind the
// weights' 143 KB per SM.
#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>

#include "fr_env_dev.cuh"
#include "fr_ptx.cuh"
#include "fr_tc.cuh"

namespace fr {

namespace {

constexpr int WD_ROWS = 64;                       // most rows of a tile
constexpr int WD_OUTS = 32;                       // outputs, padded
constexpr int WD_UNITS = 128;                     // units per CTA
constexpr int WD_LOADERS = 8;                     // warps loading observations
constexpr int WD_MMA_WARP = 12 + WD_LOADERS;
constexpr int WD_THREADS = 32 * (WD_MMA_WARP + 1);
constexpr int WD_GROUP = 4;                       // rows a loader warp stages at a time: 16 ld bytes apart, so
                                                  // every group of an aligned batch starts on a 16-byte boundary
constexpr int WD_ACT_MAX = 4096, WD_ACT_WAVES = 2;   // most rows, and waves of tiles, combined in the same launch
constexpr int WD_ACT_ROWS = 48;                   // most rows of a tile where the agents are combined
constexpr uint32_t WD_ACC2 = 64u, WD_OUT = 128u, WD_W1 = 160u;   // tensor memory columns

struct WdArgs {
    TcPlan plan;
    const uint8_t *img;
    const float *bias;
    unsigned *err;
    const float *obs;
    int ld, rows;
    float *y;
    int pair, n, tiles, nan0;                     // CTAs per agent, rows per tile, tiles of the batch
    int act;                                      // 1: y is the weighted mean of the agents [rows][outputs]
    const float *w;                               // the agents' weights (device), read by every launch and replay
    uint32_t x_bytes, h_bytes, stage_bytes, w3, x, h1, h2, stage, comb, bars;   // shared memory
    uint32_t cw;                                  // after comb: the weights, a copy per output warp
    int bulk;                                     // rows are packed and 16-byte aligned: bulk copies
};

struct WdBars {
    uint64_t x_full[2], x_empty[2];               // observations of a tile in / read
    uint64_t a1_full, a1_free, a2_full, a2_free;  // the layers' accumulators
    uint64_t h1_full[2], h1_free[2];              // hidden operands: both halves in / read by both CTAs
    uint64_t h2_full, h2_free[2];                 // h2_free[o]: read by owner o's output layer
    uint64_t o_full, o_free;
    uint64_t comb_full, comb_free;                // the other agents' outputs in / read
    uint64_t stage[WD_LOADERS];                   // a loader warp's rows in its stage
    uint64_t drain;
    uint32_t tmem;
    int abort;
};

__device__ __forceinline__ void wd_wait(uint64_t *bar, uint32_t parity, bool remote, volatile int *abort,
                                        unsigned *err, unsigned code)
{
    if (remote) {
        if (__all_sync(0xffffffffu, ptx::mbar_try_wait_cluster(bar, parity))) return;
        ptx::warp_wait_all(bar, parity, true, abort, err, code, TC_WAIT_NS);
    } else {
        quick_wait(bar, parity, abort, err, code);
    }
}

template <int n, bool NAN0>
__device__ __forceinline__ void wd_epilogue(const WdArgs &a, WdBars *bars, uint8_t *base, uint32_t tmem, int layer,
                                            int c, int rank, int agent, int count)
{
    // layer 0 or 1: accumulators -> the next layer's operand
    using namespace ptx;
    const int q = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const bool pair = a.pair == 2, f16 = a.plan.f16 != 0;
    volatile int *abort = &bars->abort;
    const int unit = c * WD_UNITS + q * 32 + lane;
    const float bias = a.bias[((size_t)agent * MAX_LAYERS + layer) * 256 + unit];
    const uint32_t acc = tmem + (layer ? WD_ACC2 : 0u) + ((uint32_t)(q * 32) << 16);
    uint64_t *full = layer ? &bars->a2_full : &bars->a1_full, *freeb = layer ? &bars->a2_free : &bars->a1_free;
    const uint32_t row = (uint32_t)(unit / 8) * (uint32_t)(n * 16) + (uint32_t)(unit % 8) * 16u;
    const uint32_t other = (uint32_t)(rank ^ 1);
    const uint32_t half_bytes = (uint32_t)(WD_UNITS * n * 2);      // the other CTA's half
    const uint32_t r_h1 = pair ? map_shared_rank(smem_u32(base + a.h1), other) : 0u;
    const uint32_t r_h2 = pair ? map_shared_rank(smem_u32(base + a.h2), other) : 0u;
    for (int i = 0; i < count; ++i) {
        quick_wait(full, (uint32_t)i & 1u, abort, a.err, 16u);
        tc_fence_after();
        const int o = pair ? i & 1 : 0;                            // the tile's output layer runs on CTA o
        bool mine = true;
        uint32_t at, rat = 0u, rbar = 0u;
        uint64_t *ready;
        if (layer == 0) {
            const int b = i & 1;
            if (i >= 2) wd_wait(&bars->h1_free[b], (uint32_t)((i >> 1) - 1) & 1u, pair, abort, a.err, 64u);
            at = smem_u32(base + a.h1) + (uint32_t)b * a.h_bytes + row;
            ready = &bars->h1_full[b];
            if (pair) {
                rat = r_h1 + (uint32_t)b * a.h_bytes + row;
                rbar = map_shared_rank(smem_u32(ready), other);
            }
        } else {
            // the second layer has read its operand: both CTAs may refill it
            if (i + 2 < count && q == 0 && lane == 0) {
                mbar_arrive(&bars->h1_free[i & 1]);
                if (pair) mbar_arrive_remote(map_shared_rank(smem_u32(&bars->h1_free[i & 1]), other));
            }
            __syncwarp();
            const int k = pair ? i >> 1 : i;
            if (k >= 1) wd_wait(&bars->h2_free[o], (uint32_t)(k - 1) & 1u, pair, abort, a.err, 64u);
            mine = o == c;
            at = smem_u32(base + a.h2) + row;
            ready = &bars->h2_full;
            if (pair && !mine) {
                rat = r_h2 + row;
                rbar = map_shared_rank(smem_u32(ready), other);
            }
        }
        const bool remote = rat != 0u;
        unit_rows<NAN0>(
            acc, bias, n, f16,
            [&](int g, const uint32_t *w) {
                if (mine) st_shared_v4(at + (uint32_t)g * 128u, w[0], w[1], w[2], w[3]);
                if (remote) st_async_v4(rat + (uint32_t)g * 128u, w[0], w[1], w[2], w[3], rbar);
            },
            [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(freeb);
            });
        if (mine) {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                if (q == 0 && pair)
                    mbar_arrive_expect_tx(ready, half_bytes);
                else
                    mbar_arrive(ready);
            }
        }
        __syncwarp();
    }
}

// Owned tile m's accumulators v of row r (bl: lane k's bias of output k):
// agents 1 .. send their rows' outputs to agent 0's CTA of the same half,
// which forms the weighted mean.
__device__ __forceinline__ void wd_combine(const WdArgs &a, WdBars *bars, uint8_t *base, const uint32_t (&v)[32], float bl,
                                        int n, int r, int c, int agent, int m, int owned, float *yr)
{
    using namespace ptx;
    const TcPlan &p = a.plan;
    const int fout = p.layer[2].fout, lane = threadIdx.x & 31;
    volatile int *abort = &bars->abort;
    const uint32_t comb = smem_u32(base + a.comb);
    const uint32_t w = smem_u32(base + a.cw) + ((threadIdx.x >> 5) & 3u) * (uint32_t)(4 * MAX_AGENTS);
    uint32_t far = 0u, far_bar = 0u;
    if (agent > 0) {
        far = map_shared_rank(comb, (uint32_t)c) + (uint32_t)(((agent - 1) * n + r) * 128);
        far_bar = map_shared_rank(smem_u32(&bars->comb_full), (uint32_t)c);
        if (m > 0) wd_wait(&bars->comb_free, (uint32_t)(m - 1) & 1u, true, abort, a.err, 64u);
    } else if (p.M > 1) {
        wd_wait(&bars->comb_full, (uint32_t)m & 1u, true, abort, a.err, 64u);
    }
#pragma unroll
    for (int k0 = 0; k0 < 32; k0 += 4) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u] = __uint_as_float(v[k0 + u]) + __shfl_sync(FULL_MASK, bl, k0 + u);
            if (p.out_act && k0 + u < fout) x[u] = tanhf(x[u]);
        }
        if (agent > 0) {
            if (lane < 16 && r < n)
                st_async_v4(far + (uint32_t)(k0 * 4), __float_as_uint(x[0]), __float_as_uint(x[1]),
                            __float_as_uint(x[2]), __float_as_uint(x[3]), far_bar);
        } else if (yr) {
            // a_0 + sum w_j (a_j - a_0), rounded at every operation
            float acc[4] = {x[0], x[1], x[2], x[3]};
            for (int j = 1; j < p.M; ++j) {
                const uint4 o = ld_shared_v4(comb + (uint32_t)(((j - 1) * n + r) * 128 + k0 * 4));
                const uint32_t ou[4] = {o.x, o.y, o.z, o.w};
                const float wj = ld_shared_f32(w + 4u * (uint32_t)j);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    acc[u] = __fadd_rn(acc[u], __fmul_rn(wj, __fsub_rn(__uint_as_float(ou[u]), x[u])));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < fout) yr[k0 + u] = acc[u];
        }
    }
    __syncwarp();
    if (agent == 0 && m + 1 < owned && lane < p.M - 1)
        mbar_arrive_remote(map_shared_rank(smem_u32(&bars->comb_free), (uint32_t)((lane + 1) * a.pair + c)));
    __syncwarp();
}

// n: rows per tile, at compile time: descriptors that advance by constants cost
// the issuing warp less than its MMAs (77,824 rows: 139 us, 153 us with n a
// parameter).  QUADS: input widths that are a multiple of 4, whose staged rows
// are read 16 bytes at a time: one float at a time, the four rows of a width of
// 200 or 304 fall on the same banks (forward on 77,824 rows: 3 x 304-256-256-30
// 237 -> 162 us, 3 x 64-256-256-30 105 -> 102 us; inputs up to 32 wide are as
// fast without, 3 x 16-256-256-30 95 us and 100 us with).  At compile time: both
// forms in one kernel cost the odd widths 10 us of 127.
template <int n, bool QUADS>
__global__ void __launch_bounds__(WD_THREADS, 1) k_wide(const __grid_constant__ WdArgs a)
{
    using namespace ptx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const TcPlan &p = a.plan;
    const TcLayer &l1 = p.layer[0], &l2 = p.layer[1], &l3 = p.layer[2];
    const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const bool pair = a.pair == 2, f16 = p.f16 != 0;
    const int size = a.pair * (a.act ? p.M : 1);                // CTAs of the cluster
    const int rank = size > 1 ? (int)cluster_ctarank() : 0, c = pair ? rank & 1 : 0;
    const int cl = (int)blockIdx.x / size, clusters = (int)gridDim.x / size;
    // a cluster is one agent's, or every agent's where their outputs are combined
    const int agent = a.act ? rank / a.pair : cl % p.M, first = a.act ? cl : cl / p.M;
    const int stride = a.act ? clusters : clusters / p.M;
    const int count = first < a.tiles ? (a.tiles - 1 - first) / stride + 1 : 0;
    const int owned = pair ? (count + 1 - c) / 2 : count;        // tiles whose output layer runs here
    WdBars *bars = (WdBars *)(base + a.bars);
    volatile int *abort = &bars->abort;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars->x_full[b], WD_LOADERS);
            mbar_init(&bars->x_empty[b], 1);
            mbar_init(&bars->h1_full[b], 4);
            mbar_init(&bars->h1_free[b], (uint32_t)a.pair);
            mbar_init(&bars->h2_free[b], 1);
        }
        mbar_init(&bars->a1_full, 1);
        mbar_init(&bars->a1_free, 4);
        mbar_init(&bars->a2_full, 1);
        mbar_init(&bars->a2_free, 4);
        mbar_init(&bars->h2_full, 4);
        mbar_init(&bars->o_full, 1);
        mbar_init(&bars->o_free, 4);
        mbar_init(&bars->comb_full, 1);
        mbar_init(&bars->comb_free, 4);
        for (int w = 0; w < WD_LOADERS; ++w) mbar_init(&bars->stage[w], 1);
        mbar_init(&bars->drain, 1);
        bars->abort = 0;
        fence_mbar_init();
    }
    if (warp == WD_MMA_WARP) {
        __syncwarp();
        tmem_alloc(&bars->tmem, 512u);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = uniform(bars->tmem);
    const uint32_t w1t = tmem + WD_W1, w2t = w1t + (uint32_t)l1.K / 2u;
    const int ksteps1 = l1.K / 16, ksteps2 = l2.K / 16, ksteps3 = l3.K / 16;

    // A loader warp stages its groups of rows (g, g + 8, .. of every tile) one
    // after another; the next one's copy is issued as soon as the stage is read.
    float *stage = (float *)(base + a.stage + (uint32_t)(warp - 12) * a.stage_bytes);   // loader warps only
    auto stage_group = [&](int i, int g) {
        const int row = (first + i * stride) * n + g * WD_GROUP;
        const int have = max(0, min(WD_GROUP, a.rows - row));
        if (a.bulk && have == WD_GROUP) {
            if (lane == 0) {
                mbar_arrive_expect_tx(&bars->stage[warp - 12], (uint32_t)(l1.fin * 16));
                bulk_g2s(stage, a.obs + (int64_t)row * a.ld, (uint32_t)(l1.fin * 16), &bars->stage[warp - 12]);
            }
            return true;
        }
        for (int r = 0; r < WD_GROUP; ++r)
#pragma unroll 4
            for (int k = lane; k < l1.fin; k += 32)
                stage[r * l1.fin + k] = r < have ? __ldg(a.obs + (int64_t)(row + r) * a.ld + k) : 0.0f;
        __syncwarp();
        return false;
    };
    grid_launch_next();
    const int groups = n / WD_GROUP;
    bool staged = false;                                   // the stage's rows come by a bulk copy
    if (warp >= 12 && warp < WD_MMA_WARP) {
        grid_wait_previous();                              // whatever wrote the observations
        if (warp - 12 < groups) staged = stage_group(0, warp - 12);
    }

    if (warp < 12) {
        // this CTA's units of the first two layers into tensor memory, lane =
        // unit, the two 16-byte core rows of a K = 16 step into eight columns;
        // four steps' loads in flight.  Units past a layer's get zeros.
        const uint8_t *img = a.img + (size_t)agent * p.agent_bytes;
        const int q = warp & 3, unit = c * WD_UNITS + q * 32 + lane;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        const int all = ksteps1 + ksteps2;
        for (int s0 = warp >> 2; s0 < all; s0 += 12) {
            uint4 v[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int s = s0 + 3 * u;
                const bool second = s >= ksteps1;
                const TcLayer &ly = second ? l2 : l1;
                const int k = second ? s - ksteps1 : s;
                v[u][0] = v[u][1] = make_uint4(0u, 0u, 0u, 0u);
                if (s < all && unit < ly.N) {
                    const uint4 *src = (const uint4 *)(img + ly.off) + (size_t)(2 * k) * ly.N + unit;
                    v[u][0] = __ldg(src);
                    v[u][1] = __ldg(src + ly.N);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int s = s0 + 3 * u;
                if (s < all) {                             // warp-uniform
                    const uint32_t w[8] = {v[u][0].x, v[u][0].y, v[u][0].z, v[u][0].w,
                                           v[u][1].x, v[u][1].y, v[u][1].z, v[u][1].w};
                    __syncwarp();
                    tmem_st8(w1t + 8u * (uint32_t)s + lane_off, w);
                }
            }
        }
        // the output layer's weights, padded to 32 outputs
        const uint4 *src3 = (const uint4 *)(img + l3.off);
        uint4 *dst3 = (uint4 *)(base + a.w3);
        for (int i = threadIdx.x; i < 32 * l3.K / 8; i += 384) {
            const int k = i >> 5, row = i & 31;
            dst3[i] = row < l3.N ? __ldg(src3 + (size_t)k * l3.N + row) : make_uint4(0u, 0u, 0u, 0u);
        }
        tmem_st_wait();
        fence_proxy_async_smem();
        tc_fence_before();
    }
    if (size > 1)
        cluster_sync_all();                                // the barriers of every CTA
    else
        __syncthreads();
    tc_fence_after();

    if (warp < 8) {
        const int layer = warp >> 2;
        if (a.nan0)
            wd_epilogue<n, true>(a, bars, base, tmem, layer, c, rank, agent, count);
        else
            wd_epilogue<n, false>(a, bars, base, tmem, layer, c, rank, agent, count);
    } else if (warp < 12) {
        // ------------------------------------------------------- outputs
        const int q = warp & 3, r = q * 16 + lane;
        const float *b3 = a.bias + ((size_t)agent * MAX_LAYERS + 2) * 256;
        const float bl = lane < l3.N ? b3[lane] : 0.0f;
        grid_wait_previous();                              // whatever still reads the outputs
        if (a.act) {
            if (lane < p.M) ((float *)(base + a.cw))[q * MAX_AGENTS + lane] = a.w[lane];
            __syncwarp();
        }
        for (int m = 0; m < owned; ++m) {
            const int i = pair ? 2 * m + c : m;
            if (n <= WD_ACT_ROWS && a.act && agent == 0 && p.M > 1 && q == 0 && lane == 0)
                mbar_arrive_expect_tx(&bars->comb_full, (uint32_t)((p.M - 1) * n * 128));
            quick_wait(&bars->o_full, (uint32_t)m & 1u, abort, a.err, 16u);
            tc_fence_after();
            if (q == 0 && lane == 0 && i + a.pair < count) {
                // this CTA's hidden operand may be refilled
                mbar_arrive(&bars->h2_free[c]);
                if (pair) mbar_arrive_remote(map_shared_rank(smem_u32(&bars->h2_free[c]), (uint32_t)(rank ^ 1)));
            }
            uint32_t v[32];
            __syncwarp();
            tmem_ld32(tmem + WD_OUT + ((uint32_t)(q * 32) << 16), v);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->o_free);
            const int g = (first + i * stride) * n + r;
            const bool out = lane < 16 && r < n && g < a.rows;
            if (n <= WD_ACT_ROWS && a.act) {               // (its code stays out of the tallest tiles' kernel)
                wd_combine(a, bars, base, v, bl, n, r, c, agent, m, owned, out ? a.y + (size_t)g * l3.fout : nullptr);
            } else {
                float *yr = a.y + ((size_t)agent * a.rows + g) * l3.fout;
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    const float b = __shfl_sync(FULL_MASK, bl, k);
                    if (k < l3.fout && out) {
                        const float x = __uint_as_float(v[k]) + b;
                        yr[k] = p.out_act ? tanhf(x) : x;
                    }
                }
            }
        }
    } else if (warp < WD_MMA_WARP) {
        // -------------------------------------------------- observations
        // lane: row lane % 4 of the group, 8-column chunk lane / 4, + 8, ..
        const int w = warp - 12, r4 = lane & 3;
        const uint32_t xs = smem_u32(base + a.x);
        const int fin = l1.fin, chunks = l1.K / 8;
        const uint32_t xcol = (uint32_t)(n * 16);
        uint32_t sph = 0;
        volatile int no_abort = 0;                         // a copy issued is always waited for
        for (int i = 0; i < count; ++i) {
            const int b = i & 1;
            if (i >= 2) quick_wait(&bars->x_empty[b], (uint32_t)((i >> 1) - 1) & 1u, abort, a.err, 1u);
            for (int g = w; g < groups; g += WD_LOADERS) {
                if (staged) {
                    quick_wait(&bars->stage[w], sph, &no_abort, a.err, 1u);
                    sph ^= 1u;
                }
                const float *src = stage + r4 * fin;
                const int r = g * WD_GROUP + r4;
                const uint32_t at = xs + (uint32_t)b * a.x_bytes + (uint32_t)(r / 8) * 128u + (uint32_t)(r % 8) * 16u;
                for (int ch = lane >> 2; ch < chunks; ch += 8) {
                    float x[8];
                    if constexpr (QUADS) {
#pragma unroll
                        for (int u = 0; u < 8; u += 4)
                            *(float4 *)(x + u) = ch * 8 + u < fin ? *(const float4 *)(src + ch * 8 + u)
                                                                  : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    } else {
#pragma unroll
                        for (int u = 0; u < 8; ++u) x[u] = ch * 8 + u < fin ? src[ch * 8 + u] : 0.0f;
                    }
                    uint32_t v[4];
                    pack8_16(x, v, f16);
                    st_shared_v4(at + (uint32_t)ch * xcol, v[0], v[1], v[2], v[3]);
                }
                __syncwarp();                              // the stage has been read
                if (g + WD_LOADERS < groups)
                    staged = stage_group(i, g + WD_LOADERS);
                else if (i + 1 < count)
                    staged = stage_group(i + 1, w);
                else
                    staged = false;
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->x_full[b]);
        }
    } else {
        // ------------------------------------------------------ MMA issue
        const uint32_t id1 = idesc_16(WD_UNITS, n, f16), id2 = id1 | (1u << 16);
        const uint32_t id3 = idesc_16(WD_ROWS, WD_OUTS, f16) | (1u << 15);
        // a K = 16 step of X or a hidden operand is two columns of n x 16 bytes
        const uint32_t col = (uint32_t)(n * 16);
        const uint64_t xd = smem_desc(smem_u32(base + a.x), col, 128u);
        const uint64_t h1d = smem_desc(smem_u32(base + a.h1), col, 128u);
        const uint64_t h2d = smem_desc(smem_u32(base + a.h2), col, 128u);
        const uint64_t w3d = smem_desc(smem_u32(base + a.w3), (uint32_t)(WD_OUTS * 16), 128u);
        int m = 0;
        // tile t's first layer, tile t - 1's second, tile t - 2's third
        for (int t = 0; t < count + 2; ++t) {
            if (t < count) {
                const int b = t & 1;
                quick_wait(&bars->x_full[b], (uint32_t)(t >> 1) & 1u, abort, a.err, 2u);
                if (t >= 1) quick_wait(&bars->a1_free, (uint32_t)(t - 1) & 1u, abort, a.err, 2u);
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t xb = xd + (uint64_t)(((uint32_t)b * a.x_bytes) >> 4);
                    for (int k = 0; k < ksteps1; ++k)
                        mma_bf16_ta(tmem, w1t + 8u * (uint32_t)k, xb + (uint64_t)(2 * n * k), id1, k ? 1u : 0u);
                    mma_commit(&bars->x_empty[b]);
                    mma_commit(&bars->a1_full);
                }
                __syncwarp();
            }
            if (t >= 1 && t - 1 < count) {
                const int i = t - 1, b = i & 1;
                wd_wait(&bars->h1_full[b], (uint32_t)(i >> 1) & 1u, pair, abort, a.err, 4u);
                if (i >= 1) quick_wait(&bars->a2_free, (uint32_t)(i - 1) & 1u, abort, a.err, 2u);
                fence_proxy_async_smem();                  // the partner's half came by generic stores
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t hb = h1d + (uint64_t)(((uint32_t)b * a.h_bytes) >> 4);
                    for (int k = 0; k < ksteps2; ++k)
                        mma_bf16_ta(tmem + WD_ACC2, w2t + 8u * (uint32_t)k, hb + (uint64_t)(2 * n * k), id2, k ? 1u : 0u);
                    mma_commit(&bars->a2_full);
                }
                __syncwarp();
            }
            if (t >= 2 && (!pair || ((t - 2) & 1) == c)) {
                wd_wait(&bars->h2_full, (uint32_t)m & 1u, pair, abort, a.err, 4u);
                if (m >= 1) quick_wait(&bars->o_free, (uint32_t)(m - 1) & 1u, abort, a.err, 2u);
                fence_proxy_async_smem();
                tc_fence_after();
                if (elect_one()) {
                    for (int k = 0; k < ksteps3; ++k)
                        mma_bf16(tmem + WD_OUT, h2d + (uint64_t)(2 * n * k), w3d + (uint64_t)(2 * WD_OUTS * k), id3,
                                 k ? 1u : 0u);
                    mma_commit(&bars->o_full);
                }
                __syncwarp();
                ++m;
            }
        }
        // every MMA issued completes before tensor memory is released; the
        // partner's bytes of the last tiles have landed too (or timed out)
        if (elect_one()) mma_commit(&bars->drain);
        __syncwarp();
        volatile int no_abort = 0;
        warp_wait_all(&bars->drain, 0u, false, &no_abort, a.err, 128u, TC_WAIT_NS);
        for (int i = count > 2 ? count - 2 : 0; pair && i < count; ++i)
            warp_wait_all(&bars->h1_full[i & 1], (uint32_t)(i >> 1) & 1u, true, &no_abort, a.err, 8u, TC_WAIT_NS);
        if (pair && owned > 0)
            warp_wait_all(&bars->h2_full, (uint32_t)(owned - 1) & 1u, true, &no_abort, a.err, 8u, TC_WAIT_NS);
        if (a.act && agent == 0 && p.M > 1 && owned > 0)
            warp_wait_all(&bars->comb_full, (uint32_t)(owned - 1) & 1u, true, &no_abort, a.err, 8u, TC_WAIT_NS);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == WD_MMA_WARP) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512u);
    }
    __syncwarp();
    if (size > 1) cluster_sync_all();                      // no peer touches this CTA's memory after it exits
}

// by 4-float rows, rows / 16
void (*const wd_kernels[2][4])(const WdArgs) = {
    {k_wide<16, false>, k_wide<32, false>, k_wide<48, false>, k_wide<64, false>},
    {k_wide<16, true>, k_wide<32, true>, k_wide<48, true>, k_wide<64, true>}};
auto wd_kernel(const TcPlan &p, int rows)
{
    return wd_kernels[p.layer[0].fin % 4 == 0 && p.layer[0].fin > 32][rows / 16 - 1];
}

// Shared memory of a launch (bytes, without the alignment slack).  The hidden
// operand of the output layer comes first: its M = 64 rows read past a shorter
// tile's.
uint32_t wd_layout(const TcPlan &p, WdArgs *a)
{
    uint32_t off = 0;
    auto take = [&](uint32_t bytes) {
        const uint32_t at = off;
        off += (bytes + 127u) & ~127u;
        return at;
    };
    a->x_bytes = (uint32_t)(p.layer[0].K / 8 * a->n * 16);
    a->h_bytes = (uint32_t)(256 * a->n * 2);
    a->stage_bytes = (uint32_t)(WD_GROUP * 4 * p.layer[0].fin);
    a->h2 = take(a->h_bytes);
    a->h1 = take(2u * a->h_bytes);
    a->x = take(2u * a->x_bytes);
    a->w3 = take((uint32_t)(WD_OUTS * p.layer[2].K) * 2u);
    a->stage = take(WD_LOADERS * a->stage_bytes);
    a->comb = a->act ? take((uint32_t)((p.M - 1) * a->n * WD_OUTS * 4)) : 0u;
    a->cw = a->act ? take(4u * MAX_AGENTS * sizeof(float)) : 0u;
    a->bars = take(sizeof(WdBars));
    return off;
}

// Rows of the tallest tile: 48 where the agents are combined, else 64, or fewer
// where the operands of 64 do not fit the SM (inputs of 303 or 304 before a
// second hidden layer wider than 240 take 48).
int wd_most(const TcPlan &p, bool act, int optin)
{
    WdArgs a;
    memset(&a, 0, sizeof(a));
    a.act = act ? 1 : 0;
    for (a.n = act ? WD_ACT_ROWS : WD_ROWS; a.n > 16 && wd_layout(p, &a) + 1024u > (uint32_t)optin;) a.n -= 16;
    return a.n;
}

// Shared memory of a launch whose operands take `layout` bytes.  The CTAs of a
// cluster wait for each other with the SM's whole tensor memory in hand, so
// nothing else that does may share their SMs (two clusters, each holding one
// SM's tensor memory and waiting for the other's, would wait for ever; beside
// the 64-row kernel's registers a CTA of the first fused crypto kernel fits):
// they take the shared memory too, but for 8 KB, where the combining kernel's
// blocks fit and no such CTA (14 KB at least for its 32 columns).
uint32_t wd_smem(uint32_t layout, int size, int optin)
{
    return size > 1 ? std::max(layout + 1024u, (uint32_t)optin - 8192u) : layout + 1024u;
}

// Clusters of `size` CTAs the device holds at once (each CTA has an SM to
// itself), queried once per device, size and shared memory; 0 when it holds
// none or the query fails.
int wd_clusters(int size, uint32_t smem, int device, int sms)
{
    static std::mutex mu;
    static std::map<std::tuple<int, int, uint32_t>, int> cache;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_tuple(device, size, smem);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(size * std::max(1, sms / size)), 1, 1);
    cfg.blockDim = dim3(WD_THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_wide<WD_ROWS, false>, &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        return 0;
    }
    n = std::min(n, std::max(1, sms / size));
    cache[key] = n;
    return n;
}

int wd_pair(const TcPlan &p) { return p.layer[0].N > WD_UNITS || p.layer[1].N > WD_UNITS ? 2 : 1; }

// y: every agent's outputs, or (act) their weighted mean.
int wd_launch(const fr_ensemble *e, const float *obs, int ld, int n, float *y, bool act, bool nan0, cudaStream_t s)
{
    const TcPlan &p = e->tc->plan;
    WdArgs a;
    memset(&a, 0, sizeof(a));
    a.plan = p;
    a.img = e->tc->img;
    a.bias = e->tc->bias;
    a.err = e->tc->err;
    a.obs = obs;
    a.ld = ld;
    a.rows = n;
    a.y = y;
    a.act = act ? 1 : 0;
    a.w = e->weights;
    a.nan0 = nan0 ? 1 : 0;
    a.bulk = ld == p.layer[0].fin && ((uintptr_t)obs & 15u) == 0;
    a.pair = wd_pair(p);
    const int size = a.pair * (act ? p.M : 1), most = wd_most(p, act, e->tc->optin);
    a.n = most;
    FR_CUDA(set_max_smem_once((const void *)k_wide<WD_ROWS, false>, e->ctx->device));
    const uint32_t smem = wd_smem(wd_layout(p, &a), size, e->tc->optin);
    const int clusters = wd_clusters(size, smem, e->ctx->device, e->ctx->sm_count);
    FR_CHECK(clusters > 0, FR_ECUDA, "no room for clusters of %d CTAs with %u bytes of shared memory each", size, smem);
    // tiles: as few rows each as spread the batch over every cluster in the
    // waves it needs anyway
    const int64_t lanes = std::max(1, act ? clusters : clusters / p.M);       // tiles in flight
    const int64_t waves = (n + most * lanes - 1) / (most * lanes);
    const int64_t per = (n + waves * lanes - 1) / (waves * lanes);
    a.n = (int)std::min<int64_t>(most, (per + 15) / 16 * 16);
    a.tiles = (int)ceil_div(n, a.n);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(size * (act ? 1 : p.M) * (int)std::min<int64_t>(lanes, a.tiles)), 1, 1);
    cfg.blockDim = dim3(WD_THREADS, 1, 1);
    cfg.dynamicSmemBytes = wd_smem(wd_layout(p, &a), size, e->tc->optin);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // the weights load while the stream's previous kernel finishes
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    FR_CUDA(set_max_smem_once((const void *)wd_kernel(p, a.n), e->ctx->device));
    FR_CUDA(cudaLaunchKernelEx(&cfg, wd_kernel(p, a.n), a));
    return FR_OK;
}

}  // namespace

// Networks k_wide takes: tensor memory must hold the first layer's weights.
bool wd_ok(const fr_ensemble *e)
{
    if (!e->tc) return false;
    const TcPlan &p = e->tc->plan;
    return p.esz == 2 && p.split == 1 && p.L == 3 && p.layer[0].K <= 304 && p.layer[0].N <= 256 &&
           p.layer[1].N <= 256 && p.layer[1].K <= 256 && p.layer[2].K <= 256 && p.layer[2].N <= 32;
}

// Whether a forward of n rows of a network wd_ok takes runs here, where the
// tiled large-batch kernel could (from one 128-row tile per SM): the faster by
// this estimate of both, in us per 77,824 rows (four waves of the tiled kernel's
// tiles).  A row here costs much the same whatever its hidden layers' widths
// (26 us per agent over CTA pairs, 15.5 in single CTAs, 4 for more than 16
// outputs, and the loading), while the tiled kernel, which converts the rows
// once for every agent, pays for the columns that there are and for whole waves.
// Fitted to 459 shapes at 19,455 .. 262,144 rows; what it picks is at most 5%
// behind the better one (3 x 10-144-96-3 on 262,144 rows: 212 us tiled, 258
// here; 8 x 304-16-256-30 on 77,824: 267 and 410; 3 x 301-256-256-30: 164 and
// 127).
bool wd_batch(const fr_ensemble *e, int n)
{
    if (tc_small_batch(e, n)) return true;
    const TcPlan &p = e->tc->plan;
    const int fin = p.layer[0].fin, sms = e->ctx->sm_count;
    const double K = p.layer[0].K, tiles = ceil_div(n, 128), outs = p.layer[2].N > 16 ? 1.0 : 0.0;
    const double rows = (double)WD_ROWS / wd_most(p, false, e->tc->optin);
    const double agent = 4.0 * outs + (wd_pair(p) == 2 ? 26.0 + 0.03 * K : 15.5 + 0.012 * K);
    double tiled = 13.0 + 5.0 * outs;
    for (int l = 0; l < 2; ++l)
        tiled += (p.layer[l].N > 128 ? 4.0 : 0.0) + p.layer[l].K * p.layer[l].N / 10200.0;
    // the tiling pass reads rows that share banks at multiples of 16 and 32
    const double pass = 2.0 + K * (fin % 32 == 0 ? 0.26 : fin % 16 == 0 ? 0.18 : 0.09);
    return 4.0 + (0.02 * K + p.M * agent * rows) * tiles / (4.0 * sms) <=
           13.0 + (pass + p.M * tiled) * ceil_div((long long)tiles, sms) / 4.0;
}

// The host queries and kernel attributes of every launch shape, so that a
// first call may be inside a stream capture.
int wd_prepare(const fr_ensemble *e)
{
    WdArgs a;
    memset(&a, 0, sizeof(a));
    const TcPlan &p = e->tc->plan;
    FR_CUDA(set_max_smem_once((const void *)k_wide<WD_ROWS, false>, e->ctx->device));   // the occupancy query's
    for (int r = 16; r <= WD_ROWS; r += 16) FR_CUDA(set_max_smem_once((const void *)wd_kernel(p, r), e->ctx->device));
    a.n = wd_most(p, false, e->tc->optin);
    wd_clusters(wd_pair(p), wd_smem(wd_layout(p, &a), wd_pair(p), e->tc->optin), e->ctx->device, e->ctx->sm_count);
    // Combining in the same launch: a cluster holds every agent (at most eight
    // CTAs), 48 rows a tile.  It spares small batches, which wait for the host,
    // an allocation and a launch (8 rows of 3 x 301-256-256-30: 12.3 us a call),
    // but the GPU holds few such clusters (23 of six, 15 of eight), so that past
    // two waves of them a forward over every SM and a combining launch are faster
    // on the GPU by more than they cost the host: 8 x 61-64-64-30 on 4,096 rows
    // 54 us combined, 20 us in two launches; 3 x 301-256-256-30 on 3,072 rows 24
    // and 17, on 2,048 rows (two waves) 17.4 and 17.1.
    const int size = wd_pair(p) * p.M;
    if (e->combine == FR_COMBINE_MEAN && size <= 8) {
        a.act = 1;
        a.n = wd_most(p, true, e->tc->optin);
        const int clusters =
            wd_clusters(size, wd_smem(wd_layout(p, &a), size, e->tc->optin), e->ctx->device, e->ctx->sm_count);
        e->tc->act_rows = std::min(WD_ACT_MAX, WD_ACT_WAVES * a.n * clusters);
    }
    return FR_OK;
}

int wd_forward(const fr_ensemble *e, const float *obs, int ld, int n, float *y, bool nan0, cudaStream_t s)
{
    return wd_launch(e, obs, ld, n, y, false, nan0, s);
}

bool wd_act_ok(const fr_ensemble *e, int n) { return e->tc && n <= e->tc->act_rows; }

int wd_act(const fr_ensemble *e, const float *obs, int n, float *act, cudaStream_t s)
{
    return wd_launch(e, obs, e->dims[0], n, act, true, tc_small_batch(e, n), s);
}

}  // namespace fr
