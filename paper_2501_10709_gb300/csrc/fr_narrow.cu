// fr_narrow.cu -- narrow networks (inputs up to 16 wide, two hidden layers up
// to 128, up to 16 outputs, up to five agents: the crypto ensemble) with every
// agent's weights resident in one CTA, as a batch forward and as the whole
// rollout in one launch.
//
// The layers run transposed, D[unit][row] = W[unit][k] X[k][row]: the 128
// units fill the MMA's M and a CTA's tile is its N, any multiple of 16 rows up
// to 64, so 8,192 envs spread over 128 SMs instead of the 64 row tiles of 128
// that put a quarter of the work on each SM.  A thread of the epilogue then
// holds one unit: its bias is a register, and eight rows of a unit are one
// 16-byte store into the next layer's operand (k rows, the tile's rows
// contiguous: both operands' MN-major no-swizzle form, 8 x 8 core matrices
// 1,024 bytes apart along k and 128 along the rows).  The output layer runs
// with the rows as M = 64 (row r in lane 32 (r / 16) + r % 16), so a row's
// outputs land in one thread.  Products, their order along k and every
// rounding are those of k_tc_forward and k_rollout_fused: the same bits.
//
// Each agent is a chain of its own, run by four warps (one per TMEM lane
// quarter) that issue their MMAs themselves after a barrier of the group, so
// a layer costs one commit and wake-up and no hand-over to an issuing warp;
// the agents' chains overlap on the tensor pipe.  Second-layer weights sit in
// tensor memory (64 columns per agent beside the 64 accumulator columns) for
// as many agents as its 512 columns hold, the others' in shared memory.
// Four more warps own the rows: they build the input operand and, in the
// rollout, keep a quarter of the tile's envs each, vote and trade.  What a
// step does under each of the three actions (cash, position and the operand
// word of both) is worked out while the networks run, so that between the
// last MMA and the next operand there is only argmax, vote and a select.
//
// Measured: the 8,192-env, 1,024-step crypto rollout of five 10-128-128-3
// networks 16.4 -> 3.3 ms (a step 13.4 -> 3.1 us with one CTA per agent and
// 128-row tile before); Q targets of 65,536 rows, two such forwards, 170 -> 50
// us.  A step is a chain of three MMA
// round trips, two epilogues and the vote (about 5,900 cycles); its 85 MMAs
// take the tensor pipe 2,700 of them (32 to 47 cycles per K = 16 step of 64
// rows with the weights in tensor or shared memory, 24 in the output layer).
// The agents run in lockstep; ordering their second layers so that one's
// epilogue runs under the others' MMAs lost more in hand-overs than it won (a
// turn barrier: 4.4 ms; one issuing warp: 5.2 ms).
#include <algorithm>
#include <cstring>

#include "fr_env_dev.cuh"
#include "fr_ptx.cuh"
#include "fr_tc.cuh"

namespace fr {

namespace {

constexpr int NW_ROWS = 64;                      // most rows of a tile
constexpr int NW_UNITS = 128;                    // units of a hidden layer, padded
constexpr int NW_MAX_AGENTS = 5;
constexpr uint32_t NW_W1 = 4096u, NW_W2 = 32768u, NW_W3 = 4096u, NW_H = 16384u, NW_X = 2048u;
constexpr int64_t NW_FROZEN = INT64_MIN;         // value log: nothing happened

struct NwShape {
    int M, n, ntm;                               // agents, tile rows, agents with W2 in tensor memory
    uint32_t tmem_cols, w1, w3, x, bias, bars, total;
};

struct NwArgs {
    NwShape sh;
    TcPlan plan;
    const uint8_t *img;
    const float *bias;
    unsigned *err;
    // forward
    const float *obs;
    int ld, rows, tiles, nan0;
    float *y;
    // rollout
    EnvView v;
    int T;
    float *tr_obs;
    int obs_ld;
    uint8_t *tr_act;
    int64_t *tr_rew;
    float *tr_rew_f32;
    uint8_t *tr_done;
    int64_t *vlog;                               // [T][N]
    int32_t *t0_out;                             // [N] step counts at the start, the env's then advanced; or NULL
    Explore ex;
};

// Shared memory: hidden operands first (an M = 64 operand of a shorter tile
// reads past its rows), then the second-layer weights that tensor memory does
// not hold, the first and last layers', the inputs, biases and barriers.
NwShape nw_shape(int M, int n)
{
    NwShape s;
    s.M = M;
    s.n = n;
    s.ntm = std::min(M, 8 - M);
    uint32_t c = 32u;
    while (c < 64u * (uint32_t)(M + s.ntm)) c <<= 1;
    s.tmem_cols = c;
    s.w1 = (uint32_t)M * NW_H + (uint32_t)(M - s.ntm) * NW_W2;
    s.w3 = s.w1 + (uint32_t)M * NW_W1;
    s.x = s.w3 + (uint32_t)M * NW_W3;
    s.bias = s.x + 2u * NW_X;
    s.bars = s.bias + (uint32_t)M * 64u;         // [M][16] output biases
    s.total = s.bars + 256u;
    return s;
}

// A hidden layer's epilogue for this thread's unit: its operand row at h_row.
template <bool NAN0>
__device__ __forceinline__ void nw_hidden(uint32_t acc, float bias, uint32_t h_row, int n, bool f16)
{
    unit_rows<NAN0>(
        acc, bias, n, f16,
        [&](int g, const uint32_t *w) { ptx::st_shared_v4(h_row + (uint32_t)g * 128u, w[0], w[1], w[2], w[3]); },
        [] {});
}

struct NwBars {
    uint64_t x_full[2], x_empty[2];              // inputs of a tile / step in, read
    uint64_t acc_full[NW_MAX_AGENTS];            // a layer's MMAs of agent j done
    uint64_t d_full;                             // rollout: every agent's outputs of the step done
    uint64_t drain;
    uint32_t tmem;
    int abort;
};

// The four rows' warps of a rollout: vote, trade, next operand.  Row r of the
// tile is lane r % 16 of quarter r / 16.
__device__ __forceinline__ void nw_env(const NwArgs &a, NwBars *bars, const uint8_t *base, uint32_t tmem, int q,
                                       int lane)
{
    using namespace ptx;
    const EnvView &v = a.v;
    const int M = a.sh.M, n = a.sh.n;
    const bool f16 = a.plan.f16 != 0;
    volatile int *abort = &bars->abort;
    const int r = q * 16 + lane;
    const bool mine = lane < 16 && r < n;
    const int e = mine && blockIdx.x * n + r < v.N ? blockIdx.x * n + r : -1;
    const uint32_t xat = smem_u32(base + a.sh.x) + (uint32_t)(r / 8) * 128u + (uint32_t)(r % 8) * 16u;
    const float *b3 = (const float *)(base + a.sh.bias);
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;

    int64_t cash = 0;
    int t = 0, start = 0, W = 2, pos = 0;
    bool done = true;
    if (e >= 0) {
        cash = v.cash[e];
        t = v.t[e];
        done = v.done[e] != 0;
        start = v.start[e];
        W = v.W[e];
        pos = v.hold[e];
        if (a.t0_out) a.t0_out[e] = t;
    }
    auto word0 = [&](int64_t c, int p) {
        return pack2_16(obs_scale(c, 1e-8f), __fdiv_rn(__int2float_rn(p), __int2float_rn(v.pmax)), f16);
    };
    float4 fa, fb;                               // factors of the row being built
    auto load_fac = [&](int d) {
        const float4 *f = (const float4 *)(v.fac + (int64_t)d * FR_CRYPTO_FACTORS);
        fa = __ldg(f);
        fb = __ldg(f + 1);
    };
    auto publish = [&](uint32_t w0) {
        if (e >= 0) {
            st_shared_v4(xat, w0, pack2_16(fa.x, fa.y, f16), pack2_16(fa.z, fa.w, f16), pack2_16(fb.x, fb.y, f16));
            st_shared_v4(xat + (uint32_t)(NW_ROWS * 16), pack2_16(fb.z, fb.w, f16), 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->x_full[0]);
    };
    if (e >= 0) load_fac(start + t);
    publish(e >= 0 ? word0(cash, pos) : 0u);

    for (int s = 0; s < a.T; ++s) {
        const int d = start + t;
        const int64_t row = (int64_t)s * v.N + e;
        if (e >= 0 && a.tr_obs) {
            float *o = a.tr_obs + row * a.obs_ld;
            o[0] = obs_scale(cash, 1e-8f);
            o[1] = __fdiv_rn(__int2float_rn(pos), __int2float_rn(v.pmax));
            o[2] = fa.x; o[3] = fa.y; o[4] = fa.z; o[5] = fa.w;
            o[6] = fb.x; o[7] = fb.y; o[8] = fb.z; o[9] = fb.w;
        }
        // ------------------------- the step under each action, in advance
        int64_t c_sell = cash, c_buy = cash, m1 = 0, v0 = 0;
        int p_sell = pos, p_buy = pos;
        bool last = done, reset = false;
        uint32_t w_sell = 0, w_hold = 0, w_buy = 0;
        if (e >= 0) {
            if (!done) {
                const int64_t m0 = __ldg(v.mid + d);
                const int64_t sp = (int64_t)__ldg(v.spread + d);
                m1 = __ldg(v.mid + d + 1);
                last = t + 1 == W - 1;
                reset = last && v.auto_reset;
                load_fac(reset ? start : d + 1);
                v0 = cash + (int64_t)pos * m0;
                const int64_t bid = m0 - sp / 2, ask = bid + sp;
                if (pos < v.pmax && cash >= ask) { p_buy = pos + 1; c_buy = cash - ask; }
                if (pos > 0) { p_sell = pos - 1; c_sell = cash + bid; }
            }
            w_hold = reset ? word0(v.init_cash, 0) : word0(cash, pos);
            w_sell = reset ? w_hold : word0(c_sell, p_sell);
            w_buy = reset ? w_hold : word0(c_buy, p_buy);
        }
        // --------------------------------------------- the agents' outputs
        quick_wait(&bars->d_full, (uint32_t)s & 1u, abort, a.err, 32u);
        tc_fence_after();
        uint32_t z[NW_MAX_AGENTS][4];
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NW_MAX_AGENTS; ++j)
            if (j < M) tmem_ld4(tmem + lane_off + 64u * (uint32_t)j, z[j]);
        tmem_ld_wait();
        int c0 = 0, c1 = 0, c2 = 0;
#pragma unroll
        for (int j = 0; j < NW_MAX_AGENTS; ++j) {
            if (j >= M) break;
            const float q0 = __uint_as_float(z[j][0]) + b3[16 * j], q1 = __uint_as_float(z[j][1]) + b3[16 * j + 1],
                        q2 = __uint_as_float(z[j][2]) + b3[16 * j + 2];
            const bool g1 = q1 > q0;
            const bool g2 = q2 > (g1 ? q1 : q0);
            c2 += g2 ? 1 : 0;
            c1 += !g2 && g1 ? 1 : 0;
            c0 += !g2 && !g1 ? 1 : 0;
        }
        // the strictly largest count, else hold
        int u = 1;
        if (c0 > c1 && c0 > c2) u = 0;
        if (c2 > c0 && c2 > c1) u = 2;
        if (e >= 0 && a.ex.kind == FR_EXPLORE_EPS_GREEDY)
            u = explore_greedy(a.ex, (uint32_t)e, a.ex.g0 + (uint32_t)s, u);
        publish(u == 0 ? w_sell : u == 2 ? w_buy : w_hold);
        // ------------------------------- under the next step's networks
        if (e >= 0) {
            int64_t rew = 0, vlog = NW_FROZEN;
            bool dn = true;
            if (!done) {
                cash = u == 0 ? c_sell : u == 2 ? c_buy : cash;
                pos = u == 0 ? p_sell : u == 2 ? p_buy : pos;
                const int64_t v1 = cash + (int64_t)pos * m1;
                rew = v1 - v0;
                t += 1;
                done = last;
                dn = last;
                vlog = last ? -v1 - 1 : v1;
                if (reset) {
                    cash = v.init_cash;
                    pos = 0;
                    t = 0;
                    done = false;
                }
            }
            if (a.tr_act) a.tr_act[row] = (uint8_t)u;
            if (a.tr_rew) a.tr_rew[row] = rew;
            if (a.tr_rew_f32) a.tr_rew_f32[row] = reward_f32(rew);
            if (a.tr_done) a.tr_done[row] = dn ? 1 : 0;
            a.vlog[row] = vlog;
        }
        __syncwarp();
    }
    // steps (unless recorded) and accumulators follow from the value log
    if (e >= 0) {
        if (a.t0_out) v.t[e] = t;
        v.cash[e] = cash;
        v.done[e] = done ? 1 : 0;
        v.hold[e] = pos;
    }
}

// The four rows' warps of a forward: the tiles' input operands.  Thread i
// holds eight columns of row i / 2; a tile's loads run under the wait for the
// buffer it goes to.
__device__ __forceinline__ void nw_inputs(const NwArgs &a, NwBars *bars, const uint8_t *base, int i)
{
    using namespace ptx;
    const int n = a.sh.n, fin = a.plan.layer[0].fin, lane = i & 31;
    const int r = i >> 1, k0 = (i & 1) * 8;
    const bool f16 = a.plan.f16 != 0;
    const uint32_t at = smem_u32(base + a.sh.x) + (uint32_t)(i & 1) * (uint32_t)(NW_ROWS * 16) +
                        (uint32_t)(r / 8) * 128u + (uint32_t)(r % 8) * 16u;
    int k = 0;
    grid_wait_previous();                        // whatever wrote the observations
    for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, ++k) {
        const int g = tile * n + r;
        const bool in = r < n && g < a.rows;
        float x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = in && k0 + u < fin ? __ldg(a.obs + (int64_t)g * a.ld + k0 + u) : 0.0f;
        uint32_t w[4];
        pack8_16(x, w, f16);
        const int b = k & 1;
        if (k >= 2) quick_wait(&bars->x_empty[b], (uint32_t)((k >> 1) - 1) & 1u, &bars->abort, a.err, 1u);
        if (r < n) st_shared_v4(at + (uint32_t)b * NW_X, w[0], w[1], w[2], w[3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->x_full[b]);
    }
}

template <bool ROLL>
__global__ void __launch_bounds__(32 * (4 * NW_MAX_AGENTS + 4), 1) k_narrow(const __grid_constant__ NwArgs a)
{
    using namespace ptx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const NwShape &sh = a.sh;
    const TcPlan &p = a.plan;
    const int M = sh.M, n = sh.n;
    const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int j = warp >> 2, q = warp & 3;       // agent (M: the rows' warps), TMEM lane quarter
    NwBars *bars = (NwBars *)(base + sh.bars);
    volatile int *abort = &bars->abort;
    const bool f16 = p.f16 != 0;
    const TcLayer &l1 = p.layer[0], &l2 = p.layer[1], &l3 = p.layer[2];

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars->x_full[b], 4);
            mbar_init(&bars->x_empty[b], (uint32_t)M);
        }
        for (int i = 0; i < M; ++i) mbar_init(&bars->acc_full[i], 1);
        mbar_init(&bars->d_full, (uint32_t)M);
        mbar_init(&bars->drain, (uint32_t)M);
        bars->abort = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        __syncwarp();
        tmem_alloc(&bars->tmem, sh.tmem_cols);
        tmem_relinquish();
    }
    // weights: the images hold 16-byte core rows (8 columns of k) of N rows
    // per column group; the units past N get zeros
    const uint8_t *img = a.img + (size_t)min(j, M - 1) * p.agent_bytes;
    auto unit16 = [&](const TcLayer &ly, int c, int row) {
        uint4 z = make_uint4(0u, 0u, 0u, 0u);
        if (row < ly.N && c < ly.K / 8) z = __ldg((const uint4 *)(img + ly.off) + (size_t)c * ly.N + row);
        return z;
    };
    const int gi = threadIdx.x & 127;            // thread within the agent's group
    if (j < M) {
        uint4 *h = (uint4 *)(base + (uint32_t)j * NW_H);
        for (int i = gi; i < (int)(NW_H / 16u); i += 128) h[i] = make_uint4(0u, 0u, 0u, 0u);
        uint4 *w1 = (uint4 *)(base + sh.w1 + (uint32_t)j * NW_W1);
        for (int c = 0; c < 2; ++c) w1[c * 128 + gi] = unit16(l1, c, gi);
        uint4 *w3 = (uint4 *)(base + sh.w3 + (uint32_t)j * NW_W3);
        for (int i = gi; i < 256; i += 128) w3[i] = unit16(l3, i / 16, i % 16);
        if (j >= sh.ntm) {
            uint4 *w2 = (uint4 *)(base + (uint32_t)M * NW_H + (uint32_t)(j - sh.ntm) * NW_W2);
            for (int c = 0; c < 16; ++c) w2[c * 128 + gi] = unit16(l2, c, gi);
        }
        if (gi < 16) ((float *)(base + sh.bias))[16 * j + gi] = a.bias[((size_t)j * MAX_LAYERS + 2) * 256 + gi];
    } else {
        ((uint4 *)(base + sh.x))[gi] = make_uint4(0u, 0u, 0u, 0u);
        ((uint4 *)(base + sh.x))[128 + gi] = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = uniform(bars->tmem);
    if (j < sh.ntm) {
        const uint32_t w2 = tmem + 64u * (uint32_t)(M + j) + ((uint32_t)(q * 32) << 16);
#pragma unroll 2
        for (int c = 0; c < 8; ++c) {
            const uint4 lo = unit16(l2, 2 * c, gi), hi = unit16(l2, 2 * c + 1, gi);
            const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            __syncwarp();
            tmem_st8(w2 + 8u * (uint32_t)c, w);
        }
        tmem_st_wait();
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();

    if (!ROLL) grid_launch_next();
    const int steps = ROLL ? a.T : (blockIdx.x < a.tiles ? (a.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0);
    if (j == M) {
        if (ROLL)
            nw_env(a, bars, base, tmem, q, lane);
        else
            nw_inputs(a, bars, base, gi);
    } else {
        // ------------------------------------------------ agent j's chain
        const uint32_t acc = tmem + 64u * (uint32_t)j, acc_row = acc + ((uint32_t)(q * 32) << 16);
        const uint32_t h = smem_u32(base + (uint32_t)j * NW_H);
        const uint32_t h_row = h + (uint32_t)(gi / 8) * 1024u + (uint32_t)(gi % 8) * 16u;
        const float bias1 = a.bias[((size_t)j * MAX_LAYERS + 0) * 256 + gi];
        const float bias2 = a.bias[((size_t)j * MAX_LAYERS + 1) * 256 + gi];
        const uint32_t id12 = idesc_16(NW_UNITS, n, f16), id3 = idesc_16(NW_ROWS, 16, f16) | (1u << 15);
        const uint64_t w1d = smem_desc(smem_u32(base + sh.w1 + (uint32_t)j * NW_W1), 2048u, 128u);
        const uint64_t w2d = smem_desc(smem_u32(base + (uint32_t)M * NW_H + (uint32_t)max(0, j - sh.ntm) * NW_W2),
                                       2048u, 128u);
        const uint32_t w2t = tmem + 64u * (uint32_t)(M + j);
        const uint64_t w3d = smem_desc(smem_u32(base + sh.w3 + (uint32_t)j * NW_W3), 256u, 128u);
        const uint64_t xd = smem_desc(smem_u32(base + sh.x), (uint32_t)(NW_ROWS * 16), 128u);
        const uint64_t hd = smem_desc(h, 1024u, 128u);     // MN-major: k groups 1,024 apart, row groups 128
        const int k2 = l2.K / 16, k3 = l3.K / 16;
        uint64_t *full = &bars->acc_full[j];
        uint32_t ph = 0;
        if (!ROLL) grid_wait_previous();         // whatever still reads the outputs
        // no early exit: a wait that gives up sets the abort flag, the later
        // ones return after a poll, and the loop runs to its uniform end
        for (int s = 0; s < steps; ++s) {
            const int b = ROLL ? 0 : s & 1;
            if (q == 0) {
                quick_wait(&bars->x_full[b], (uint32_t)(ROLL ? s : s >> 1) & 1u, abort, a.err, 2u);
                tc_fence_after();
                if (elect_one()) {
                    mma_bf16(acc, w1d, xd + (uint64_t)(((uint32_t)b * NW_X) >> 4), id12, 0u);
                    if (!ROLL) mma_commit(&bars->x_empty[b]);
                    mma_commit(full);
                }
                __syncwarp();
            }
            quick_wait(full, ph, abort, a.err, 16u);
            ph ^= 1u;
            tc_fence_after();
            if (!ROLL && a.nan0)
                nw_hidden<true>(acc_row, bias1, h_row, n, f16);
            else
                nw_hidden<false>(acc_row, bias1, h_row, n, f16);
            fence_proxy_async_smem();
            tc_fence_before();
            named_bar_sync((uint32_t)(1 + j), 128u);
            if (q == 0) {
                tc_fence_after();
                if (elect_one()) {
                    uint64_t hk = hd, wk = w2d;
                    uint32_t wt = w2t, on = 0u;
                    if (j < sh.ntm) {
                        for (int k = 0; k < k2; ++k, wt += 8u, hk += 128u, on = 1u)
                            mma_bf16_ta(acc, wt, hk, id12 | (1u << 16), on);
                    } else {
                        for (int k = 0; k < k2; ++k, wk += 256u, hk += 128u, on = 1u)
                            mma_bf16(acc, wk, hk, id12 | (1u << 16), on);
                    }
                    mma_commit(full);
                }
                __syncwarp();
            }
            quick_wait(full, ph, abort, a.err, 16u);
            ph ^= 1u;
            tc_fence_after();
            if (!ROLL && a.nan0)
                nw_hidden<true>(acc_row, bias2, h_row, n, f16);
            else
                nw_hidden<false>(acc_row, bias2, h_row, n, f16);
            fence_proxy_async_smem();
            tc_fence_before();
            named_bar_sync((uint32_t)(1 + j), 128u);
            if (q == 0) {
                tc_fence_after();
                if (elect_one()) {
                    uint64_t hk = hd, wk = w3d;
                    uint32_t on = 0u;
                    for (int k = 0; k < k3; ++k, hk += 128u, wk += 32u, on = 1u) mma_bf16(acc, hk, wk, id3, on);
                    mma_commit(ROLL ? &bars->d_full : full);
                }
                __syncwarp();
            }
            if (!ROLL) {
                quick_wait(full, ph, abort, a.err, 16u);
                ph ^= 1u;
                tc_fence_after();
                uint32_t z[16];
                __syncwarp();
                tmem_ld16(acc_row, z);
                tmem_ld_wait();
                const int r = q * 16 + lane;
                const int g = ((int)blockIdx.x + s * (int)gridDim.x) * n + r;
                if (lane < 16 && r < n && g < a.rows) {
                    float *y = a.y + ((size_t)j * a.rows + g) * l3.fout;
                    const float *b3 = (const float *)(base + sh.bias) + 16 * j;
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (i < l3.fout) {
                            const float x = __uint_as_float(z[i]) + b3[i];
                            y[i] = p.out_act ? tanhf(x) : x;
                        }
                }
                tc_fence_before();
                named_bar_sync((uint32_t)(1 + j), 128u);    // read before the next tile's first layer
            }
        }
        // every MMA issued completes before tensor memory is released
        if (q == 0) {
            if (elect_one()) mma_commit(&bars->drain);
            __syncwarp();
            volatile int no_abort = 0;
            warp_wait_all(&bars->drain, 0u, false, &no_abort, a.err, 128u, TC_WAIT_NS);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, sh.tmem_cols);
    }
}

// Rows per tile: as few as spread n rows over every SM in the waves they need
// anyway (a step's epilogue and output layer cost per row).
int nw_tile_rows(int64_t n, int sms)
{
    sms = std::max(1, sms);
    const int64_t waves = (n + (int64_t)NW_ROWS * sms - 1) / ((int64_t)NW_ROWS * sms);
    const int64_t per = (n + waves * sms - 1) / (waves * sms);
    return (int)std::min<int64_t>(NW_ROWS, (std::max<int64_t>(per, 1) + 15) / 16 * 16);
}

}  // namespace

// Networks k_narrow takes.
bool nw_ok(const fr_ensemble *e)
{
    if (!e->tc) return false;
    const TcPlan &p = e->tc->plan;
    return p.esz == 2 && p.split == 1 && p.L == 3 && p.M <= NW_MAX_AGENTS && p.layer[0].K == 16 &&
           p.layer[0].N <= NW_UNITS && p.layer[1].N <= NW_UNITS && p.layer[2].N == 16 &&
           p.layer[1].K <= NW_UNITS && p.layer[2].K <= NW_UNITS;
}

// The kernel attributes of a forward, so that a first call may be inside a
// stream capture.
int nw_prepare(const fr_ensemble *e)
{
    FR_CUDA(set_max_smem_once((const void *)k_narrow<false>, e->ctx->device));
    return FR_OK;
}

int nw_forward(const fr_ensemble *e, const float *obs, int ld, int n, float *y, bool nan0, cudaStream_t s)
{
    NwArgs a;
    memset(&a, 0, sizeof(a));
    a.plan = e->tc->plan;
    a.sh = nw_shape(a.plan.M, nw_tile_rows(n, e->ctx->sm_count));
    a.img = e->tc->img;
    a.bias = e->tc->bias;
    a.err = e->tc->err;
    a.obs = obs;
    a.ld = ld;
    a.rows = n;
    a.nan0 = nan0 ? 1 : 0;
    a.tiles = (int)ceil_div(n, a.sh.n);
    a.y = y;
    FR_CUDA(set_max_smem_once((const void *)k_narrow<false>, e->ctx->device));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(a.tiles, std::max(1, e->ctx->sm_count)), 1, 1);
    cfg.blockDim = dim3((unsigned)(32 * (4 * a.sh.M + 4)), 1, 1);
    cfg.dynamicSmemBytes = a.sh.total + 1024u;
    cfg.stream = s;
    // the weights load while the stream's previous kernel finishes
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    FR_CUDA(cudaLaunchKernelEx(&cfg, k_narrow<false>, a));
    return FR_OK;
}

uint64_t nw_rollout_scratch(const fr_env *env, int T)
{
    const uint64_t log = ((uint64_t)T * env->v.N * 8 + 255) & ~255ull, t0 = (4ull * env->v.N + 255) & ~255ull;
    return log + SPLIT_PIECES_MAX * t0;
}

// The crypto rollout: one launch and the replay of its value log, or, where
// the tiles leave SMs idle (8,192 envs: 24 of 152), in pieces whose replays
// run there (3.59 -> 3.31 ms for 1,024 steps).
int nw_rollout(fr_env *env, const fr_ensemble *e, int T, const fr_traj *traj, void *scratch, double *metrics,
               cudaStream_t s)
{
    const EnvView &v = env->v;
    NwArgs a;
    memset(&a, 0, sizeof(a));
    a.plan = e->tc->plan;
    a.sh = nw_shape(a.plan.M, nw_tile_rows(v.N, env->ctx->sm_count));
    a.img = e->tc->img;
    a.bias = e->tc->bias;
    a.err = e->tc->err;
    a.v = v;
    a.T = T;
    a.tr_obs = traj->obs;
    a.obs_ld = traj->obs_ld ? traj->obs_ld : v.D;
    a.tr_act = (uint8_t *)traj->act;
    a.tr_rew = traj->rew;
    a.tr_rew_f32 = traj->rew_f32;
    a.tr_done = traj->done;
    a.vlog = (int64_t *)scratch;
    a.ex = explore_of(env, env->explore_step);
    const int grid = (int)ceil_div(v.N, a.sh.n);
    const bool want_traj = traj->obs || traj->act || traj->rew || traj->rew_f32 || traj->done;
    const int K = !want_traj && !v.auto_reset && !env->split_off && grid < env->ctx->sm_count &&
                          env->scratch_bytes >= nw_rollout_scratch(env, T)
                      ? std::min(SPLIT_PIECES_MAX, T / 64)
                      : 1;
    FR_CUDA(set_max_smem_once((const void *)k_narrow<true>, env->ctx->device));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3((unsigned)(32 * (4 * a.sh.M + 4)), 1, 1);
    cfg.dynamicSmemBytes = a.sh.total + 1024u;
    cfg.stream = s;
    FR_CUDA(env_time_mark(env, 0, s));
    if (K <= 1) {
        FR_CUDA(cudaLaunchKernelEx(&cfg, k_narrow<true>, a));
        FR_CUDA(env_time_mark(env, 1, s));
        FR_CUDA(launch_metrics_replay(v, a.vlog, T, metrics, s));
        return FR_OK;
    }
    const uint64_t t0_b = (4ull * v.N + 255) & ~255ull;
    int32_t *t0a = (int32_t *)((char *)scratch + (((uint64_t)T * v.N * 8 + 255) & ~255ull));
    return split_rollout(env, T, K, a.vlog, t0a, t0_b, metrics, s,
                         [&](int s0, int Tk, int64_t *log, int32_t *t0, cudaStream_t ks, int prio) {
                             cudaLaunchAttribute attr[1];
                             attr[0].id = cudaLaunchAttributePriority;
                             attr[0].val.priority = prio;
                             cudaLaunchConfig_t c = cfg;
                             c.attrs = attr;
                             c.numAttrs = 1;
                             c.stream = ks;
                             NwArgs b = a;
                             b.T = Tk;
                             b.vlog = log;
                             b.t0_out = t0;
                             b.ex.g0 = a.ex.g0 + (uint32_t)s0;
                             return cudaLaunchKernelEx(&c, k_narrow<true>, b);
                         });
}

}  // namespace fr
