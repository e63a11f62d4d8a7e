// fr_prep.cu -- on-device data preparation: the technical indicators of the
// state (Sec. 3.1 f_t; the Sec. 6.1 list: MACD, Bollinger bands, RSI-30,
// CCI-30, DX-30, SMA-30 and SMA-60) computed from daily OHLC on the GPU, and
// the per-env +-1% price perturbations of Sec. 5.1 drawn on the GPU.
//
// The indicators are computed in FP64 with every operation explicitly
// rounded (no contraction into FMA), in the order of their definitions:
// windows summed from the oldest day, recurrences in day order.  So the table
// is a pure function of the price series, identical on any launch shape.
//
// The serial chains set the time.  An FP64 operation occupies its SM
// sub-partition for 64 cycles and a division for 580 (fr_fp64.cuh), so a chain
// carries only its recurrence: the Wilder smoothing in four operations (x - w,
// two for the division by 30, the sum), an EMA in two.  A chain block (four per
// 32 assets, one lane per asset) runs two chains, one warp each -- the SM takes
// one FP64 instruction per 19 cycles, so two chains run at full rate and four
// would not -- while a warp beside each prepares its inputs on the integer
// pipe, 64 days ahead; where the chains set the time every block takes an SM to
// itself (shared memory), so nothing else competes for the pipe.  Window blocks
// in the same launch (two assets x 128 days, one thread per day) stage the tile
// plus a 59-day halo of closes and typical prices in shared memory and compute
// the windowed means, the standard deviation and the mean absolute deviation.
// A second launch, one thread per (day, asset), turns the chains' states into
// MACD, RSI and DX.
// Measured, 1,000 days x 30 assets: one block per three chains, with their
// divisions, conversions and input arithmetic on the chain, 826 us (1,650
// cycles per day); this form 160 us (330 cycles per day), and the whole call
// 835 -> 170 us.
#include "fr_common.cuh"
#include "fr_fp64.cuh"
#include "fr_ptx.cuh"

namespace fr {
namespace {

constexpr int PREP_TILE = 128;     // days per window block
constexpr int PREP_HALO = 59;      // longest window (60 days) minus one
constexpr int N_IND = 8;
constexpr int PREP_SEG = 64;       // days a chain's inputs are prepared ahead
constexpr int PREP_THREADS = 256;
constexpr int N_PLANES = 7;        // chain states: gains, losses, TR, DM+, DM-, EMA-12, EMA-26
constexpr int CHAINS = 2;          // chains per block
constexpr size_t PREP_SMEM = sizeof(double) * CHAINS * 2 * PREP_SEG * 32;   // input buffers of a chain block: 64 KB
constexpr size_t PREP_ALONE = 128 * 1024;  // one block per SM
static_assert(PREP_SMEM >= sizeof(double) * 4 * (PREP_TILE + PREP_HALO), "window blocks' tiles");

__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double ddiv(double a, double b) { return __ddiv_rn(a, b); }

// 1 / 30 and 1 / 100 to 2^-106
constexpr Recip kRecip30 = {0x1.1111111111111p-5, 0x1.1111111111111p-61};
constexpr Recip kRecip100 = {0x1.47ae147ae147bp-7, -0x1.eb851eb851eb8p-63};

// Wilder smoothing with n = 30: w + (x - w) / 30.
__device__ __forceinline__ double wilder30(double w, double x) { return dadd(w, div_recip(dsub(x, w), kRecip30, 30u)); }

__device__ __forceinline__ void put(float *ind, int K, int t, int col, int k, double v)
{
    ind[((int64_t)t * N_IND + col) * K + k] = __double2float_rn(v);
}

// The chain inputs as FP64 operations on the prices rounded to double, out of
// line: only prices of 2^52 cents or more, or negative, take them.
__device__ __noinline__ double chain_input_fp64(int plane, int64_t c, int64_t h, int64_t l, int64_t cp, int64_t hp,
                                                int64_t lp)
{
    if (plane <= 1) {
        const double d = plane == 0 ? dsub((double)c, (double)cp) : dsub((double)cp, (double)c);
        return d > 0.0 ? d : 0.0;
    }
    const double ht = (double)h, lt = (double)l, ct = (double)cp;
    if (plane == 2) {
        double tr = dsub(ht, lt);
        const double th = fabs(dsub(ht, ct)), tl = fabs(dsub(lt, ct));
        if (th > tr) tr = th;
        if (tl > tr) tr = tl;
        return tr;
    }
    const double up = dsub(ht, (double)hp), dn = dsub((double)lp, lt);
    if (plane == 3) return (up > dn && up > 0.0) ? up : 0.0;
    return (dn > up && dn > 0.0) ? dn : 0.0;
}

// Day t's input of chain `plane` from the prices of the day and the one
// before (c_{-1} = c_0 etc., so the first moves are 0): gains / losses of
// c_t - c_{t-1}, true range, DM+ / DM-, or a c_t of an EMA (c_0 itself first).
template <int PLANE>
__device__ __forceinline__ double chain_input(int64_t c, int64_t h, int64_t l, int64_t cp, int64_t hp, int64_t lp,
                                              double a, bool first)
{
    if constexpr (PLANE >= 5) {
        const double x = i64_to_double(c);
        return first ? x : dmul(a, x);
    } else {
        // exact in integers: every price below 2^52
        uint64_t any = (uint64_t)c | (uint64_t)cp;
        if constexpr (PLANE >= 2) any |= (uint64_t)h | (uint64_t)l | (uint64_t)hp | (uint64_t)lp;
        if ((any >> 52) != 0) return chain_input_fp64(PLANE, c, h, l, cp, hp, lp);
        int64_t x;
        if constexpr (PLANE == 0) {
            x = c - cp;
        } else if constexpr (PLANE == 1) {
            x = cp - c;
        } else if constexpr (PLANE == 2) {
            const int64_t th = h > cp ? h - cp : cp - h, tl = l > cp ? l - cp : cp - l;
            x = h - l;                                   // negative when low > high: the others win
            if (th > x) x = th;
            if (tl > x) x = tl;
        } else {
            const int64_t up = h - hp, dn = lp - l;
            x = PLANE == 3 ? (up > dn ? up : 0) : (dn > up ? dn : 0);
        }
        return u53_to_double((uint64_t)(x > 0 ? x : 0));
    }
}

// The warp beside a chain: segment after segment of its inputs into the two
// buffers x[2][PREP_SEG][32] (lane = asset), one segment ahead of the chain.
// Both warps meet on named barrier `bar` once per segment.
template <int PLANE>
__device__ void chain_inputs(const int64_t *__restrict__ close, const int64_t *__restrict__ high,
                             const int64_t *__restrict__ low, int T, int K, int k, bool live, double a, double *x,
                             uint32_t bar)
{
    constexpr bool hl = PLANE >= 2 && PLANE <= 4;
    const int lane = threadIdx.x & 31;
    int64_t cp = 1, hp = 1, lp = 1;
    if (live) {
        cp = close[k];
        if (hl) {
            hp = high[k];
            lp = low[k];
        }
    }
    for (int t0 = 0, b = 0; t0 < T; t0 += PREP_SEG, b ^= 1) {
        const int len = min(PREP_SEG, T - t0);
        double *xb = x + b * PREP_SEG * 32 + lane;
#pragma unroll 1
        for (int i0 = 0; i0 < len; i0 += 8) {        // eight days' loads in flight
            int64_t c[8], h[8], l[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const bool in = live && i0 + i < len;
                const int64_t at = (int64_t)(t0 + i0 + i) * K + k;
                c[i] = in ? close[at] : 1;
                h[i] = hl && in ? high[at] : 1;
                l[i] = hl && in ? low[at] : 1;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                xb[(i0 + i) * 32] = chain_input<PLANE>(c[i], h[i], l[i], cp, hp, lp, a, t0 + i0 + i == 0);
                cp = c[i];
                hp = h[i];
                lp = l[i];
            }
        }
        ptx::named_bar_sync(bar, 64);                // segment ready; the chain is done with the other buffer
    }
}

// One chain: day by day w = x on day 0, then Wilder or w = x + b w (EMA),
// the state of each day into plane `out`.  Wilder days run in groups of 8 on
// the two-operation division when w enters the group as 0 or at least 2^-400:
// its inputs are 0 or from 1 to 2^64, so a difference x - w is then 0 or no
// smaller than the last bit of w, which a step lowers by 2^-53 at most and 8
// steps leave above 2^-900.  (A smoothed series without moves decays below
// 2^-400 after some 8,000 days; those take the division proper.)
template <bool EMA>
__device__ void chain_run(int T, int K, int k, bool live, double b, const double *x, double *__restrict__ out,
                          uint32_t bar)
{
    constexpr int G = 8;
    const int lane = threadIdx.x & 31;
    double w = 0.0;
    for (int t0 = 0, buf = 0; t0 < T; t0 += PREP_SEG, buf ^= 1) {
        ptx::named_bar_sync(bar, 64);
        const int len = min(PREP_SEG, T - t0);
        const double *xb = x + buf * PREP_SEG * 32 + lane;
        double *o = out + (int64_t)t0 * K + k;
#pragma unroll 1
        for (int i0 = 0; i0 < len; i0 += G) {
            double xs[G], ws[G];
#pragma unroll
            for (int i = 0; i < G; ++i) xs[i] = xb[(i0 + i) * 32];      // past len: stale and dropped
            const uint32_t wh = (uint32_t)__double2hiint(w);
            const bool tiny = !EMA && wh < ((1023u - 400u) << 20) && (wh | (uint32_t)__double2loint(w)) != 0u;
            if (__any_sync(0xffffffffu, tiny)) {
#pragma unroll 1
                for (int i = 0; i < G; ++i) {
                    const double x1 = xb[(i0 + i) * 32];
                    w = wilder30(w, x1);
                    if (live && i0 + i < len) o[(int64_t)(i0 + i) * K] = w;
                }
                continue;
            }
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const double nw = EMA ? dadd(xs[i], dmul(b, w)) : dadd(w, div_recip_fast(dsub(xs[i], w), kRecip30));
                w = (i == 0 && t0 + i0 == 0) ? xs[0] : nw;
                ws[i] = w;
            }
#pragma unroll
            for (int i = 0; i < G; ++i)
                if (live && i0 + i < len) o[(int64_t)(i0 + i) * K] = ws[i];
        }
    }
}

__device__ __forceinline__ void chain_block(const int64_t *close, const int64_t *high, const int64_t *low, int T, int K,
                                            double *st, double *xs)
{
    // warps 0 and 1 the chains, 2 and 3 their inputs: one per sub-partition
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = warp & 1;
    const int plane = (blockIdx.x & 3) * CHAINS + c;
    const int k = (blockIdx.x >> 2) * 32 + lane;
    if (warp >= 2 * CHAINS || plane >= N_PLANES) return;
    const bool live = k < K;
    // a = 2 / (n + 1), n = 12 or 26
    const double a = plane == 5 ? 2.0 / 13.0 : 2.0 / 27.0;
    double *x = xs + c * 2 * PREP_SEG * 32;
    const uint32_t bar = 1u + (uint32_t)c;
    if (warp < CHAINS) {
        double *out = st + (int64_t)plane * T * K;
        if (plane >= 5)
            chain_run<true>(T, K, k, live, dsub(1.0, a), x, out, bar);
        else
            chain_run<false>(T, K, k, live, 0.0, x, out, bar);
        return;
    }
    switch (plane) {
    case 0: chain_inputs<0>(close, high, low, T, K, k, live, a, x, bar); break;
    case 1: chain_inputs<1>(close, high, low, T, K, k, live, a, x, bar); break;
    case 2: chain_inputs<2>(close, high, low, T, K, k, live, a, x, bar); break;
    case 3: chain_inputs<3>(close, high, low, T, K, k, live, a, x, bar); break;
    case 4: chain_inputs<4>(close, high, low, T, K, k, live, a, x, bar); break;
    default: chain_inputs<5>(close, high, low, T, K, k, live, a, x, bar); break;
    }
}

// MACD / c, RSI-30 / 100 and DX-30 / 100 of (day, asset) from the chains'
// states, the same operations as if they ran on the chain.
__global__ void k_ind_final(const int64_t *__restrict__ close, int T, int K, const double *__restrict__ st,
                            float *__restrict__ ind)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t TK = (int64_t)T * K;
    if (i >= TK) return;
    const int t = (int)(i / K), k = (int)(i % K);
    const double ct = i64_to_double(close[i]);
    put(ind, K, t, 0, k, ddiv(dsub(st[5 * TK + i], st[6 * TK + i]), ct));
    const double gain = st[i], loss = st[TK + i];
    double rsi;
    if (gain == 0.0 && loss == 0.0) rsi = 50.0;
    else if (loss > 0.0) rsi = dsub(100.0, ddiv(100.0, dadd(1.0, ddiv(gain, loss))));
    else rsi = 100.0;
    put(ind, K, t, 3, k, div_recip(rsi, kRecip100, 100u));
    const double str = st[2 * TK + i], spd = st[3 * TK + i], snd = st[4 * TK + i];
    const double den = str > 0.0 ? str : 1.0;
    const double pdi = ddiv(dmul(100.0, spd), den), ndi = ddiv(dmul(100.0, snd), den);
    const double s = dadd(pdi, ndi);
    const double dx = s > 0.0 ? ddiv(dmul(100.0, fabs(dsub(pdi, ndi))), s) : 0.0;
    put(ind, K, t, 5, k, div_recip(dx, kRecip100, 100u));
}

// Mean of x[j - m + 1 .. j] in shared memory, m = min(n, t + 1) days ending at
// day t (local index j), summed from the oldest.
__device__ __forceinline__ double win_mean(const double *x, int j, int t, int n, int &m)
{
    m = t + 1 < n ? t + 1 : n;
    double s = 0.0;
    for (int u = j - m + 1; u <= j; ++u) s = dadd(s, x[u]);
    return ddiv(s, (double)m);
}

__global__ void __launch_bounds__(PREP_THREADS, 1) k_indicators(const int64_t *__restrict__ close,
                                                                const int64_t *__restrict__ high,
                                                                const int64_t *__restrict__ low, int T, int K,
                                                                float *__restrict__ ind, int n_chain, int n_tiles,
                                                                double *__restrict__ st)
{
    extern __shared__ double prep_sm[];
    if ((int)blockIdx.x < n_chain) {
        chain_block(close, high, low, T, K, st, prep_sm);
        return;
    }
    // two assets per block, one thread per day of the tile
    const int sub = threadIdx.x / PREP_TILE, td = threadIdx.x % PREP_TILE;
    double *c_s = prep_sm + sub * 2 * (PREP_TILE + PREP_HALO), *tp_s = c_s + PREP_TILE + PREP_HALO;
    const int b = blockIdx.x - n_chain;
    const int k = 2 * (b / n_tiles) + sub, t0 = (b % n_tiles) * PREP_TILE;
    for (int j = td; j < PREP_TILE + PREP_HALO; j += PREP_TILE) {
        const int u = t0 - PREP_HALO + j;
        if (u >= 0 && u < T && k < K) {
            const int64_t i = (int64_t)u * K + k;
            const double c = (double)close[i];
            c_s[j] = c;
            tp_s[j] = ddiv(dadd(dadd((double)high[i], (double)low[i]), c), 3.0);
        }
    }
    __syncthreads();
    const int t = t0 + td;
    if (t >= T || k >= K) return;
    const int j = PREP_HALO + td;
    const double ct = c_s[j];
    int m;
    // Bollinger(20, 2): SMA20 +- 2 population standard deviations
    const double sma20 = win_mean(c_s, j, t, 20, m);
    double v = 0.0;
    for (int u = j - m + 1; u <= j; ++u) {
        const double z = dsub(c_s[u], sma20);
        v = dadd(v, dmul(z, z));
    }
    const double sd20 = __dsqrt_rn(ddiv(v, (double)m));
    put(ind, K, t, 1, k, dsub(ddiv(dadd(sma20, dmul(2.0, sd20)), ct), 1.0));
    put(ind, K, t, 2, k, dsub(ddiv(dsub(sma20, dmul(2.0, sd20)), ct), 1.0));
    // CCI-30 = (tp - SMA30(tp)) / (0.015 MAD30(tp))
    const double smatp = win_mean(tp_s, j, t, 30, m);
    double mad = 0.0;
    for (int u = j - m + 1; u <= j; ++u) mad = dadd(mad, fabs(dsub(tp_s[u], smatp)));
    mad = ddiv(mad, (double)m);
    const double cci = mad > 0.0 ? ddiv(dsub(tp_s[j], smatp), dmul(0.015, mad)) : 0.0;
    put(ind, K, t, 4, k, ddiv(cci, 100.0));
    // SMA30 / c - 1, SMA60 / c - 1
    put(ind, K, t, 6, k, dsub(ddiv(win_mean(c_s, j, t, 30, m), ct), 1.0));
    put(ind, K, t, 7, k, dsub(ddiv(win_mean(c_s, j, t, 60, m), ct), 1.0));
}

__global__ void k_perturb(EnvView v, uint64_t seed, int R)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)v.N * KP) return;
    const int e = (int)(i / KP), k = (int)(i % KP);
    ((int16_t *)v.bps)[i] = (k < v.K && R > 0) ? perturb_bps(seed, (uint32_t)e, (uint32_t)k, R) : (int16_t)0;
}

}  // namespace

cudaError_t launch_indicators(const int64_t *close, const int64_t *high, const int64_t *low, int T, int K,
                              float *ind, cudaStream_t s)
{
    const int n_chain = 4 * ((K + 31) / 32), n_tiles = (T + PREP_TILE - 1) / PREP_TILE;
    const long long blocks = (long long)n_chain + (long long)((K + 1) / 2) * n_tiles;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    int dev = 0, sms = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // Blocks share SMs (three each) where they are more than the chains' length
    // pays for alone, about 75 days a wave: 60 days x 3,000 assets 214 us shared, 256
    // alone, 1,000 x 600 604 and 642; 1,000 x 300 368 and 335, 2,520 x 100 535 and
    // 419.
    const size_t smem = blocks > sms && blocks * 75 > (long long)sms * T ? PREP_SMEM : PREP_ALONE;
    if (e == cudaSuccess) e = set_max_smem_once((const void *)k_indicators, dev);
    // the chains' states, stream-ordered scratch: 7 doubles per (day, asset)
    double *st = nullptr;
    if (e == cudaSuccess) e = cudaMallocAsync((void **)&st, 8ull * N_PLANES * (uint64_t)T * K, s);
    if (e != cudaSuccess) return e;
    k_indicators<<<(unsigned)blocks, PREP_THREADS, smem, s>>>(close, high, low, T, K, ind, n_chain, n_tiles, st);
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        k_ind_final<<<ceil_div((int64_t)T * K, 256), 256, 0, s>>>(close, T, K, st, ind);
        e = cudaGetLastError();
    }
    const cudaError_t f = cudaFreeAsync(st, s);
    return e != cudaSuccess ? e : f;
}

}  // namespace fr

using namespace fr;

extern "C" {

int market_indicators(const int64_t *close, const int64_t *high, const int64_t *low, int32_t n_days,
                      int32_t n_assets, float *ind, void *stream)
{
    FR_NVTX("market_indicators");
    FR_CHECK(close && high && low && ind, FR_EINVAL, "market_indicators: NULL table");
    FR_CHECK(n_days >= 1 && n_assets >= 1 && (int64_t)n_days * n_assets <= ((int64_t)1 << 40), FR_EINVAL,
             "market_indicators: n_days %d and n_assets %d must be >= 1", n_days, n_assets);
    FR_CUDA(launch_indicators(close, high, low, n_days, n_assets, ind, (cudaStream_t)stream));
    return FR_OK;
}

int env_perturb(fr_env *env, uint64_t seed, int32_t bps_range, void *stream)
{
    FR_NVTX("env_perturb");
    FR_CHECK(env, FR_EINVAL, "env_perturb: NULL env");
    FR_CHECK(env->v.task == FR_TASK_STOCK, FR_EINVAL, "env_perturb: stock envs only");
    FR_CHECK(bps_range >= 0 && bps_range <= 100, FR_EINVAL, "env_perturb: bps_range %d not in 0..100",
             bps_range);
    FR_CUDA(cudaSetDevice(env->ctx->device));
    const int64_t n = (int64_t)env->v.N * KP;
    k_perturb<<<ceil_div(n, 256), 256, 0, (cudaStream_t)stream>>>(env->v, seed, bps_range);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

}  // extern "C"
