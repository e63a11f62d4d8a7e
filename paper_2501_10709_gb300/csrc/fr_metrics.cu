// fr_metrics.cu -- episode statistics in FP64: the Sec. 6.1 metric list and
// the Sec. 4.3 discounted return of stored trajectories (the consumer side of
// the T x N sample tensors), and the replay of a rollout's value log through
// the episode accumulators (Sharpe ratio, maximum drawdown).  Every operation
// is an explicitly rounded intrinsic in the order of the step-by-step
// definitions, so no contraction or reordering changes a result.
//
// What bounds it: FP64 instructions.  Each occupies its SM sub-partition for
// 64 cycles whatever the number of active lanes, and the mean
// mu += (r - mu) / n is a chain through every step (fr_fp64.cuh).  So the work
// is split by warps into a pipeline over segments of EP_SEG steps, one lane
// per env, each serial sum on a sub-partition of its own:
//   scan      values v_t (integers) and the running peak
//   producers returns v_t / v_{t-1} - 1 (six operations and the subtraction in
//             place of a division); 1 / n as hi + lo, once per step when the
//             block's envs have taken equally many steps; the worst v / peak
//             (a pair of integers compared by cross products: division and
//             rounding are monotone, so one division at the end gives the
//             minimum of the rounded drawdowns)
//   mean      the chain: subtract, two for the division by n, add
//   m2        sum of (r - mu_old)(r - mu), one segment behind the mean
//   signs, discount (trajectories): the sums behind Sortino and Omega, and
//             the discounted return
// Segment k is scanned while k - 1 is produced and k - 2 summed.
// Measured: trajectory_metrics of 2,048 envs x 256 steps took 495 us with one
// thread per env and three divisions per step in series, 77 us now; the
// replay of 8,192 envs x 1,024 steps 1.56 ms with the mean's division on the
// chain and the returns' beside it, 0.44 ms now (FP64 pipe 76% busy).
#include <algorithm>

#include "fr_common.cuh"
#include "fr_env_dev.cuh"
#include "fr_fp64.cuh"
#include "fr_ptx.cuh"

namespace fr {
namespace {

constexpr int EP_SEG = 8;                       // steps per pipeline segment
constexpr int EP_WARPS = 16, EP_THREADS = 32 * EP_WARPS;
constexpr int EP_ACTIVE = 32 * 13;              // threads of the working warps
constexpr int EP_PROD = 8;                      // producer warps
constexpr int64_t EP_NONE = INT64_MIN;          // value log: the env took no step

struct EpArgs {
    EnvView v;                  // replay: accumulators in and out
    const int64_t *in;          // [T][N] value log, or rewards
    const uint8_t *done;        // trajectories: [T][N] or NULL
    const int32_t *t0;          // replay: step counts before the log, NULL = the env's own (and advance them)
    double *out;                // replay: metrics [N][3] or NULL; trajectories: [N][11]
    int T, N;
    int64_t v0;                 // trajectories
    double ann, gamma;
};

// Working warps.  Warps w and w + 4 share a sub-partition: the mean has its
// own (warps 4, 8 and 12 end at once), the other sums one each beside
// producers.
constexpr int W_MEAN = 0, W_M2 = 1, W_SIGN = 2, W_DISC = 3, W_SCAN = 7;
__device__ __forceinline__ int producer_of(int warp)      // 0..7, -1 for the others
{
    switch (warp) {
    case 5: return 0;
    case 6: return 1;
    case 9: return 2;
    case 10: return 3;
    case 11: return 4;
    case 13: return 5;
    case 14: return 6;
    case 15: return 7;
    }
    return -1;
}

template <int EN>
struct EpShared {
    int64_t v[2][EP_SEG + 1][EN];       // values before the segment and after each of its steps
    int64_t peak[2][EP_SEG][EN];        // running peak after each step
    int64_t wv[EP_PROD][32], wp[EP_PROD][32];   // each producer lane's worst v / peak (wp 0: none)
    double wd[EP_PROD][32];             // and worst drawdown of values past 2^53
    double rho[3][EP_SEG][EN];
    Recip rn[2][EP_SEG][EN];            // 1 / n of each step ([.][0] when common to the block)
    double delta[2][EP_SEG][EN], mu[2][EP_SEG][EN];
    int len[4][EN];                     // steps each env takes in the segment
    int odd[4];                         // 1: a return of the segment is no ratio of values 0 <= v1 < 2^53, 1 <= v0 < 2^31
    int n0[EN];                         // its steps before the log
    int64_t vlast[EN];
    double mean[EN], m2[EN], mdd[EN], up[EN], dn[EN], down2[EN], disc[EN], cr[EN], annual[EN];
    int cnt[EN];
};

// TRAJ: stored trajectories, else the replay of a value log.  EN envs per
// block (16: two steps per producer instruction; 32).
template <bool TRAJ, int EN>
__global__ void __launch_bounds__(EP_THREADS, 1) k_episodes(const __grid_constant__ EpArgs a)
{
    __shared__ EpShared<EN> sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 4 || warp == 8 || warp == 12) return;
    const EnvView &v = a.v;
    const int T = a.T, N = a.N;
    const int el = lane & (EN - 1);                    // env of the block; lanes >= EN repeat one and store nothing
    const int e = blockIdx.x * EN + el;
    const bool in = e < N, own = in && lane < EN;
    const int nseg = (T + EP_SEG - 1) / EP_SEG;
    const int pi = producer_of(warp);
    auto sync = [] { ptx::named_bar_sync(1u, EP_ACTIVE); };

    int n0 = 0;
    if (!TRAJ && in) n0 = a.t0 ? a.t0[e] : v.t[e];
    // one step count for the whole block: 1 / n is computed once per step
    const int n_first = __shfl_sync(FULL_MASK, n0, 0);
    const bool common = TRAJ || __all_sync(FULL_MASK, n0 == n_first || !in);

    // role state
    int64_t vv = 1, peak = 1;                          // scan: value and peak
    int64_t bv = 0, bp = 0;                            // producers: worst ratio bv / bp (bp 0: none)
    double ddx = 0.0;                                  // and worst drawdown of values past 2^53
    int cnt = 0;
    bool live = in;
    int64_t row[EP_SEG];                               // scan: the next segment's rows
    uint32_t drow = 0u;                                // and done flags
    double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0;         // the sums of this warp
    auto fetch = [&](int k) {
        drow = 0u;
#pragma unroll
        for (int i = 0; i < EP_SEG; ++i) {
            const int t = k * EP_SEG + i;
            row[i] = in && t < T ? __ldg(a.in + (int64_t)t * N + e) : EP_NONE;
            if (TRAJ && a.done && in && t < T && __ldg(a.done + (int64_t)t * N + e)) drow |= 1u << i;
        }
    };
    if (warp == W_SCAN) {
        if (TRAJ) {
            vv = peak = a.v0;
        } else if (in) {
            vv = v.vlast[e];
            peak = v.peak[e];
        }
        fetch(0);
    } else if (warp == W_MEAN) {
        acc0 = !TRAJ && in ? v.mu[e] : 0.0;
    } else if (warp == W_M2) {
        acc0 = !TRAJ && in ? v.m2[e] : 0.0;
    } else if (warp == W_DISC) {
        acc1 = 1.0;
    }

    for (int tick = 0; tick < nseg + 3; ++tick) {
        if (warp == W_SCAN && tick < nseg) {
            const int b = tick & 1;
            int64_t cur[EP_SEG];
            const uint32_t dcur = drow;
#pragma unroll
            for (int i = 0; i < EP_SEG; ++i) cur[i] = row[i];
            if (tick + 1 < nseg) fetch(tick + 1);
            if (lane < EN) sm.v[b][0][el] = vv;
            int len = 0;
#pragma unroll
            for (int i = 0; i < EP_SEG; ++i) {
                const int64_t x = cur[i];
                if (tick * EP_SEG + i >= T || (!TRAJ && x == EP_NONE)) live = false;
                if (live) {
                    vv = TRAJ ? vv + x : (x < 0 ? -x - 1 : x);
                    len = i + 1;
                    if (vv > peak) peak = vv;
                    if (TRAJ && ((dcur >> i) & 1u)) live = false;
                }
                if (lane < EN) {
                    sm.v[b][i + 1][el] = vv;
                    sm.peak[b][i][el] = peak;
                }
            }
            cnt += len;
            if (lane < EN) sm.len[tick & 3][el] = len;
            if (lane == 0) sm.odd[tick & 3] = 0;
        }
        const int kp = tick - 1;                       // segment of the producers and the discounted sum
        if (pi >= 0 && kp >= 0 && kp < nseg) {
            const int b = kp & 1;
            constexpr int PER = 32 / EN;               // steps per instruction
            for (int it = pi; it < EP_SEG / PER; it += EP_PROD) {
                const int i = it * PER + lane / EN;
                // (past an env's last step the value and the peak stay as they are)
                const int64_t v1 = sm.v[b][i + 1][el], pk = sm.peak[b][i][el];
                const int64_t v0 = sm.v[b][i][el];
                sm.rho[kp % 3][i][el] = __dsub_rn(i64_ratio(v1, v0), 1.0);
                if (!i64_ratio_fast(v1, v0)) sm.odd[kp & 3] = 1;
                if (v1 < pk && i < sm.len[kp & 3][el]) {
                    if ((((uint64_t)v1 | (uint64_t)pk) >> 53) != 0) {
                        const double dd = __dsub_rn(fp64_int_ratio(v1, pk), 1.0);
                        if (dd < ddx) ddx = dd;
                    } else if (bp == 0 || ratio_less((uint64_t)v1, (uint64_t)pk, (uint64_t)bv, (uint64_t)bp)) {
                        bv = v1;
                        bp = pk;
                    }
                }
                if (!common) {
                    const uint32_t n = (uint32_t)(n0 + kp * EP_SEG + i + 1);
                    sm.rn[b][i][el] = recip_of(n, u53_to_double(n));
                }
            }
            if (common && pi == (EN == 16 ? 7 : (kp & 7)) && lane < EP_SEG) {
                const uint32_t n = (uint32_t)(n_first + kp * EP_SEG + lane + 1);
                sm.rn[b][lane][0] = recip_of(n, u53_to_double(n));
            }
        }
        if (TRAJ && warp == W_DISC && kp >= 0 && kp < nseg) {
            const int b = kp & 1, len = sm.len[kp & 3][el], most = __reduce_max_sync(FULL_MASK, len);
            for (int i = 0; i < most; ++i) {
                const int64_t r = sm.v[b][i + 1][el] - sm.v[b][i][el];
                const uint64_t m = r < 0 ? 0ull - (uint64_t)r : (uint64_t)r;
                const double ad = u53_to_double(m), rd = (m >> 53) == 0 ? (r < 0 ? -ad : ad) : fp64_of_int(r);
                acc1 = __dmul_rn(acc1, a.gamma);       // gamma^t, the same for every env of the block
                const double s = __dadd_rn(acc0, __dmul_rn(acc1, rd));
                if (i < len) acc0 = s;
            }
        }
        const int kc = tick - 2;                       // segment of the sums over returns
        if (warp == W_MEAN && kc >= 0 && kc < nseg) {
            const int b = kc & 1, len = sm.len[kc & 3][el], most = __reduce_max_sync(FULL_MASK, len);
            const int re = common ? 0 : el;
            if (most > 0) {
                // every step of the segment (what lies past an env's last step
                // is dropped), on the two-operation division when every return
                // is an ordinary ratio less one (0 or 2^-54 to 2^53) and the
                // mean enters as 0 or at least 2^-400: a difference is then 0
                // or no smaller than the last bit of either, and 8 steps leave
                // the mean above 2^-900
                const uint32_t mh = (uint32_t)__double2hiint(acc0) & 0x7fffffffu;
                const bool plain = (mh - ((1023u - 400u) << 20) < (800u << 20) || (mh | (uint32_t)__double2loint(acc0)) == 0u) &&
                                   sm.odd[kc & 3] == 0;
                if (__all_sync(FULL_MASK, plain)) {
                    double r[EP_SEG], d[EP_SEG], m[EP_SEG];
                    Recip rn[EP_SEG];
#pragma unroll
                    for (int i = 0; i < EP_SEG; ++i) {
                        r[i] = sm.rho[kc % 3][i][el];
                        rn[i] = sm.rn[b][i][re];
                    }
                    double mu = acc0;
#pragma unroll
                    for (int i = 0; i < EP_SEG; ++i) {
                        d[i] = __dsub_rn(r[i], mu);
                        mu = __dadd_rn(mu, div_recip_fast(d[i], rn[i]));
                        m[i] = mu;
                    }
#pragma unroll
                    for (int i = 0; i < EP_SEG; ++i) {
                        if (lane < EN) {
                            sm.delta[b][i][el] = d[i];
                            sm.mu[b][i][el] = m[i];
                        }
                        if (i < len) acc0 = m[i];
                    }
                } else {
#pragma unroll 1
                    for (int i = 0; i < EP_SEG; ++i) {
                        const double d = __dsub_rn(sm.rho[kc % 3][i][el], acc0);
                        const double m =
                            __dadd_rn(acc0, div_recip(d, sm.rn[b][i][re], (uint32_t)(n0 + kc * EP_SEG + i + 1)));
                        if (lane < EN) {
                            sm.delta[b][i][el] = d;
                            sm.mu[b][i][el] = m;
                        }
                        if (i < len) acc0 = m;
                    }
                }
            }
        }
        if (TRAJ && warp == W_SIGN && kc >= 0 && kc < nseg) {
            // EN = 16: lanes 0..15 sum the gains, 16..31 the losses
            const int len = sm.len[kc & 3][el], most = __reduce_max_sync(FULL_MASK, len);
            for (int i = 0; i < most; ++i) {
                const double r = sm.rho[kc % 3][i][el];
                // r < 0 on the integer pipe: sign set, not -0 (a return never is), not a NaN
                const uint32_t rh = (uint32_t)__double2hiint(r);
                const bool neg = rh >= 0x80000000u && rh <= 0xfff00000u;
                if (i < len) {
                    if (EN == 16) {
                        const bool dn_lane = lane >= 16;
                        if (neg == dn_lane) acc0 = __dadd_rn(acc0, dn_lane ? -r : r);
                    } else if (neg) {
                        acc1 = __dadd_rn(acc1, -r);
                    } else {
                        acc0 = __dadd_rn(acc0, r);
                    }
                    if (neg) acc2 = __dadd_rn(acc2, __dmul_rn(r, r));
                }
            }
        }
        const int km = tick - 3;                       // segment of m2
        if (warp == W_M2 && km >= 0 && km < nseg) {
            const int b = km & 1, len = sm.len[km & 3][el], most = __reduce_max_sync(FULL_MASK, len);
            for (int i = 0; i < most; ++i) {
                const double s = __dadd_rn(
                    acc0, __dmul_rn(sm.delta[b][i][el], __dsub_rn(sm.rho[km % 3][i][el], sm.mu[b][i][el])));
                if (i < len) acc0 = s;
            }
        }
        sync();
    }

    // the producers' worst ratios, then the sums, into shared memory and the
    // env's accumulators
    if (pi >= 0) {
        sm.wv[pi][lane] = bv;
        sm.wp[pi][lane] = bp;
        sm.wd[pi][lane] = ddx;
    }
    sync();
    if (warp == W_SCAN && own) {
        double m = TRAJ ? 0.0 : v.mdd[e];
        for (int w = 0; w < EP_PROD; ++w) {
            for (int l = el; l < 32; l += EN) {
                const int64_t pv = sm.wv[w][l], pp = sm.wp[w][l];
                if (pp != 0 && (bp == 0 || ratio_less((uint64_t)pv, (uint64_t)pp, (uint64_t)bv, (uint64_t)bp))) {
                    bv = pv;
                    bp = pp;
                }
                if (sm.wd[w][l] < ddx) ddx = sm.wd[w][l];
            }
        }
        if (bp != 0) {
            const double dd = __dsub_rn(i64_ratio(bv, bp), 1.0);
            if (dd < m) m = dd;
        }
        if (ddx < m) m = ddx;
        sm.mdd[el] = m;
        sm.cnt[el] = n0 + cnt;
        sm.cr[el] = __dsub_rn(i64_ratio(vv, TRAJ ? a.v0 : v.init_cash), 1.0);
        if (TRAJ) {
            sm.vlast[el] = vv;
        } else {
            v.mdd[e] = m;
            v.peak[e] = peak;
            v.vlast[e] = vv;
            if (!a.t0) v.t[e] = n0 + cnt;
        }
    } else if (warp == W_MEAN && own) {
        sm.mean[el] = acc0;
        if (!TRAJ) v.mu[e] = acc0;
    } else if (warp == W_M2 && own) {
        sm.m2[el] = acc0;
        if (!TRAJ) v.m2[e] = acc0;
    } else if (TRAJ && warp == W_SIGN && in) {
        if (lane < EN) sm.up[el] = acc0;
        if (EN == 16 ? lane >= 16 : true) sm.dn[el] = EN == 16 ? acc0 : acc1;
        if (lane < EN) sm.down2[el] = acc2;
    } else if (TRAJ && warp == W_DISC && own) {
        sm.disc[el] = acc0;
    }
    sync();
    if (!own || !a.out) return;
    const int n = sm.cnt[el];
    if (!TRAJ) {
        // env_metrics: the last auto-reset episode while the env has taken no step since
        double *o = a.out + (int64_t)e * 3;
        const double *Lt = v.latched + (int64_t)e * 4;
        const bool latched = n == 0 && Lt[3] != 0.0;
        if (warp == W_SCAN) {
            o[0] = latched ? Lt[0] : sm.cr[el];
            o[2] = latched ? Lt[2] : sm.mdd[el];
        } else if (warp == W_M2) {
            o[1] = latched ? Lt[1] : sharpe_of(sm.mean[el], acc0, n, v.ann);
        }
        return;
    }
    double *o = a.out + (int64_t)e * FR_TRAJ_METRICS;
    const double nd = (double)n, dd_max = -sm.mdd[el];
    if (warp == W_SCAN) {
        const double cr = sm.cr[el];
        o[0] = cr;
        o[2] = sm.mdd[el];
        o[5] = dd_max != 0.0 ? __ddiv_rn(cr, dd_max) : 0.0;
        o[10] = nd;
    } else if (warp == W_MEAN) {
        const double annual =
            n > 0 ? __dsub_rn(pow(i64_ratio(sm.vlast[el], a.v0), __ddiv_rn(a.ann, nd)), 1.0) : 0.0;
        o[3] = annual;
        o[7] = dd_max != 0.0 ? __ddiv_rn(annual, dd_max) : 0.0;
    } else if (warp == W_M2) {
        o[1] = sharpe_of(sm.mean[el], acc0, n, a.ann);
        o[4] = n >= 2 ? __dmul_rn(__dsqrt_rn(__ddiv_rn(acc0, __dsub_rn(nd, 1.0))), __dsqrt_rn(a.ann)) : 0.0;
    } else if (warp == W_SIGN) {
        const double ddown = n > 0 ? __dsqrt_rn(__ddiv_rn(sm.down2[el], nd)) : 0.0;
        o[6] = ddown != 0.0 ? __dmul_rn(__ddiv_rn(sm.mean[el], ddown), __dsqrt_rn(a.ann)) : 0.0;
        o[8] = sm.dn[el] != 0.0 ? __ddiv_rn(sm.up[el], sm.dn[el]) : 0.0;
    } else if (warp == W_DISC) {
        o[9] = sm.disc[el];
    }
}

// Trajectories that episodes_short() takes: one thread per env, step by step,
// with plain divisions (a warp alone waits 6% less for one of them than for the
// six operations in its place, and many warps fill the pipe either way).
__global__ void __launch_bounds__(128) k_episodes_short(const __grid_constant__ EpArgs a)
{
    const int e = blockIdx.x * 128 + threadIdx.x;
    if (e >= a.N) return;
    double mu = 0.0, m2 = 0.0, mdd = 0.0, down2 = 0.0, up = 0.0, dn = 0.0, disc = 0.0, g = 1.0;
    int64_t peak = a.v0, v = a.v0;
    int n = 0;
    for (int t = 0; t < a.T; ++t) {
        const int64_t r = __ldg(a.in + (int64_t)t * a.N + e), v1 = v + r;
        const double rho = __dsub_rn(__ddiv_rn((double)v1, (double)v), 1.0);
        n += 1;
        const double delta = __dsub_rn(rho, mu);
        mu = __dadd_rn(mu, __ddiv_rn(delta, (double)n));
        m2 = __dadd_rn(m2, __dmul_rn(delta, __dsub_rn(rho, mu)));
        if (v1 > peak) peak = v1;
        if (v1 < peak) {
            const double dd = __dsub_rn(__ddiv_rn((double)v1, (double)peak), 1.0);
            if (dd < mdd) mdd = dd;
        }
        if (rho < 0.0) {
            down2 = __dadd_rn(down2, __dmul_rn(rho, rho));
            dn = __dadd_rn(dn, -rho);
        } else {
            up = __dadd_rn(up, rho);
        }
        g = __dmul_rn(g, a.gamma);
        disc = __dadd_rn(disc, __dmul_rn(g, (double)r));
        v = v1;
        if (a.done && __ldg(a.done + (int64_t)t * a.N + e)) break;
    }
    double *o = a.out + (int64_t)e * FR_TRAJ_METRICS;
    acc_final(mu, m2, mdd, v, a.v0, n, a.ann, o);
    const double nd = (double)n, cr = o[0], dd_max = -mdd;
    const double annual =
        n > 0 ? __dsub_rn(pow(__ddiv_rn((double)v, (double)a.v0), __ddiv_rn(a.ann, nd)), 1.0) : 0.0;
    const double ddown = n > 0 ? __dsqrt_rn(__ddiv_rn(down2, nd)) : 0.0;
    o[3] = annual;
    o[4] = n >= 2 ? __dmul_rn(__dsqrt_rn(__ddiv_rn(m2, __dsub_rn(nd, 1.0))), __dsqrt_rn(a.ann)) : 0.0;
    o[5] = dd_max != 0.0 ? __ddiv_rn(cr, dd_max) : 0.0;
    o[6] = ddown != 0.0 ? __dmul_rn(__ddiv_rn(mu, ddown), __dsqrt_rn(a.ann)) : 0.0;
    o[7] = dd_max != 0.0 ? __ddiv_rn(annual, dd_max) : 0.0;
    o[8] = dn != 0.0 ? __ddiv_rn(up, dn) : 0.0;
    o[9] = disc;
    o[10] = nd;
}

// 16 envs per block while that leaves at most one block per SM (a block's
// mean chain then has its sub-partition to itself: 260 cycles a step); 32
// beyond, where the FP64 pipes are the limit and full warps halve the sums'
// instructions.  SM count of the GB300.
constexpr int EP_SMS = 152;

template <bool TRAJ>
cudaError_t launch_episodes(const EpArgs &a, cudaStream_t s)
{
    if (TRAJ && episodes_short(true, a.T, a.N))
        k_episodes_short<<<ceil_div(a.N, 128), 128, 0, s>>>(a);
    else if (a.N <= 16 * EP_SMS)
        k_episodes<TRAJ, 16><<<ceil_div(a.N, 16), EP_THREADS, 0, s>>>(a);
    else
        k_episodes<TRAJ, 32><<<ceil_div(a.N, 32), EP_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Few steps of many envs: a block of k_episodes fills and drains its pipeline
// for 32 envs, one block per SM, which costs a wave of them 10 us (4 the replay)
// before its 0.27 us a step; a thread per env waits 1.65 us a step (1.2 the
// replay) and, past a block of 128 per SM, the FP64 pipe has 1.57 us a step of
// work for each (7.6 at 131,072 envs the replay).  The faster by these figures.
// Trajectories of 131,072 envs x 1 step take 70 us, 280 us by k_episodes; x 64
// steps 774 and 740; 8,192 envs x 4 steps 19 and 23, x 8 steps 26 and 26.
bool episodes_short(bool traj, int T, int N)
{
    const double waves = ceil_div(ceil_div(N, N <= 16 * EP_SMS ? 16 : 32), EP_SMS);
    if (traj)
        return T <= 1 || std::max(12.0 + 1.65 * T, ceil_div(N, 128 * EP_SMS) * (9.4 + 1.57 * T)) <
                             waves * (10.4 + 0.27 * T);
    return std::max(0.4 + 1.2 * T, N / 131072.0 * (12.0 + 7.6 * T)) < waves * (4.4 + 0.27 * T);
}

cudaError_t launch_episode_replay(const EnvView &v, const int64_t *vlog, int T, double *metrics, cudaStream_t s,
                                  const int32_t *t0)
{
    EpArgs a = {};
    a.v = v;
    a.in = vlog;
    a.t0 = t0;
    a.out = metrics;
    a.T = T;
    a.N = v.N;
    return launch_episodes<false>(a, s);
}

}  // namespace fr

using namespace fr;

extern "C" int trajectory_metrics(const int64_t *rew, const uint8_t *done, int32_t T, int32_t N, int64_t v0,
                                  double ann, double gamma, double *out, void *stream)
{
    FR_NVTX("trajectory_metrics");
    FR_CHECK(T >= 0 && N >= 0 && v0 > 0 && ann > 0.0 && isfinite(gamma), FR_EINVAL,
             "trajectory_metrics: need T, N >= 0, v0 > 0, ann > 0, finite gamma");
    if (N == 0) return FR_OK;
    FR_CHECK(out && (rew || T == 0), FR_EINVAL, "trajectory_metrics: NULL rew or out");
    EpArgs a = {};
    a.in = rew;
    a.done = done;
    a.out = out;
    a.T = T;
    a.N = N;
    a.v0 = v0;
    a.ann = ann;
    a.gamma = gamma;
    FR_CUDA(launch_episodes<true>(a, (cudaStream_t)stream));
    return FR_OK;
}
