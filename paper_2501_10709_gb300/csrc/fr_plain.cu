// fr_plain.cu -- the plain, unfused FP32 actor path: the whole network in one
// SIMT launch (k_mlp_f32: layer inputs up to 304 wide, outputs up to 256), or a
// dense-layer launch per layer (k_dense_f32: wider inputs), all agents of the
// ensemble in one grid; then a separate combine launch.  It is the comparison
// path for the fused BF16 rollout and the fp32 reference the tensor-core kernels
// are held to.
#include "fr_common.cuh"
#include "fr_ptx.cuh"

namespace fr {

namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;

// Y[a][r][o] = act( sum_k X[a][r][k] * W_a[o][k] + b_a[o] ), ACT: 0 ReLU,
// 1 tanh, 2 identity.  W_a / b_a live at P + a*p_stride + w_off / b_off.
template <int ACT>
__global__ void __launch_bounds__(NT) k_dense_f32(const float *__restrict__ X, int64_t x_stride, int ldx,
                                                  const float *__restrict__ P, int64_t p_stride,
                                                  int64_t w_off, int64_t b_off,
                                                  float *__restrict__ Y, int64_t y_stride, int ldy,
                                                  int n, int fin, int fout)
{
    const int a = blockIdx.z;
    X += a * x_stride;
    const float *W = P + a * p_stride + w_off;
    const float *B = P + a * p_stride + b_off;
    Y += a * y_stride;
    __shared__ float As[BK][BM + 1];
    __shared__ float Bs[BK][BN + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int row0 = blockIdx.y * BM, col0 = blockIdx.x * BN;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    for (int k0 = 0; k0 < fin; k0 += BK) {
        for (int i = threadIdx.x; i < BM * BK; i += NT) {
            const int r = i / BK, kk = i % BK;
            const int gr = row0 + r, gk = k0 + kk;
            As[kk][r] = (gr < n && gk < fin) ? X[(int64_t)gr * ldx + gk] : 0.0f;
        }
        for (int i = threadIdx.x; i < BN * BK; i += NT) {
            const int o = i / BK, kk = i % BK;
            const int go = col0 + o, gk = k0 + kk;
            Bs[kk][o] = (go < fout && gk < fin) ? W[(int64_t)go * fin + gk] : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) av[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = row0 + ty * 4 + i;
        if (r >= n) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int o = col0 + tx * 4 + j;
            if (o >= fout) continue;
            float y = acc[i][j] + B[o];
            if (ACT == 0) y = fmaxf(y, 0.0f);
            else if (ACT == 1) y = tanhf(y);
            Y[(int64_t)r * ldy + o] = y;
        }
    }
}

// The whole fp32 network of one agent for a tile of BM rows in one block.
// k_dense_f32 above runs 4 x 4 outputs per thread from scalar shared-memory
// reads (8 reads per 16 FMAs: 18 TFLOP/s of the 80 the FP32 pipes give) in one
// launch per layer, with every hidden activation through HBM.  Here:
//  * the hidden activations stay in shared memory, k-major as the next layer
//    reads them; a layer's outputs are all in registers when its last k is
//    done, so one buffer serves every layer;
//  * a thread holds TM x TN outputs (8 x 8 at 64 rows x 256 columns) and reads
//    16-byte vectors: a warp is 4 row groups x 8 column groups, so each read is
//    one wavefront, 4 of them per 64 FMAs;
//  * the FMAs run two columns per instruction (fma.rn.f32x2);
//  * weights come from global memory (L2) through registers into a
//    double-buffered k-major tile, the next one's loads under the current
//    one's FMAs.
// Every output is the same chain of FMAs over k as in k_dense_f32: the same
// bits.  3 x 301-256-256-30, whole call: 8,192 rows 415 -> 211 us (35
// TFLOP/s), 256 rows 130 -> 53 us, one row 99 -> 53 us.
constexpr int ML_THREADS = 256;
constexpr int ML_MAX_K = 304;                 // widest layer input
constexpr uint32_t ML_STAGE = 8704;           // bytes of a weight tile (2,048 floats, rows padded by 4)

struct MlpArgs {
    const float *X;
    int ldx, n;
    const float *params;
    int64_t P;
    int64_t w_off[MAX_LAYERS], b_off[MAX_LAYERS];
    int dims[MAX_LAYERS + 1];
    int L, out_act, kmax;
    float *Y;                                 // [M][n][dims[L]]
};

__device__ __forceinline__ uint64_t pack2f(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2f(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// d = a * b + d on both halves, each rounded once
__device__ __forceinline__ void fma2(uint64_t &d, uint64_t a, uint64_t b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// One layer.  NPAD columns (32, 64, 128 or 256 >= fout), weight tiles of BK
// rows.  As [fin][BM + 4] holds the layer's input and receives its output
// unless it is the last layer.
template <int BM, int NPAD>
__device__ __forceinline__ void mlp_layer(const MlpArgs &a, int l, const float *__restrict__ W,
                                          const float *__restrict__ B, float *As, float *Ws, int row0, int agent)
{
    constexpr int BK = NPAD == 32 ? 32 : 2048 / NPAD;
    constexpr int TN = NPAD >= 128 ? 8 : 4;
    constexpr int CW = NPAD / (8 * TN);                   // warps side by side
    constexpr int RW = 8 / CW;
    constexpr int TM = BM / (4 * RW) > 0 ? BM / (4 * RW) : 1;
    constexpr int SA = BM + 4, SW = NPAD + 4;
    constexpr int QUADS = BK * NPAD / 4 / ML_THREADS;     // 4-column groups of a tile per thread
    static_assert((uint32_t)(BK * SW * 4) <= ML_STAGE && QUADS >= 1, "weight tile");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int fin = a.dims[l], fout = a.dims[l + 1];
    const bool last = l == a.L - 1;
    const int r0 = (warp / CW) * 4 * TM + (lane >> 3) * TM;            // rows r0 .. r0 + TM - 1
    const int c0 = (warp % CW) * 8 * TN + (lane & 7) * 4;              // columns c0 .. + 3 (and + 32 ..)
    const bool active = r0 < BM;

    float stage[QUADS][4];
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < QUADS; ++q) {
            const int i = threadIdx.x + q * ML_THREADS, k = k0 + i % BK, c = 4 * (i / BK);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                stage[q][u] = (k < fin && c + u < fout) ? __ldg(W + (int64_t)(c + u) * fin + k) : 0.0f;
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int q = 0; q < QUADS; ++q) {
            const int i = threadIdx.x + q * ML_THREADS;
            *(float4 *)(Ws + b * (ML_STAGE / 4) + (i % BK) * SW + 4 * (i / BK)) =
                make_float4(stage[q][0], stage[q][1], stage[q][2], stage[q][3]);
        }
    };

    uint64_t acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
    auto step = [&](const float *ap, const float *wp) {
        float x[TM];
        if constexpr (TM >= 4) {
#pragma unroll
            for (int i = 0; i < TM; i += 4) *(float4 *)(x + i) = *(const float4 *)(ap + i);
        } else if constexpr (TM == 2) {
            *(float2 *)x = *(const float2 *)ap;
        } else {
            x[0] = ap[0];
        }
        ulonglong2 w[TN / 4];
#pragma unroll
        for (int j = 0; j < TN / 4; ++j) w[j] = *(const ulonglong2 *)(wp + 32 * j);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const uint64_t xx = pack2f(x[i], x[i]);
#pragma unroll
            for (int j = 0; j < TN / 4; ++j) {
                fma2(acc[i][2 * j], xx, w[j].x);
                fma2(acc[i][2 * j + 1], xx, w[j].y);
            }
        }
    };

    load(0);
    store(0);
    __syncthreads();                                      // the tile, and the layer's input
    int b = 0;
    for (int k0 = 0; k0 < fin; k0 += BK, b ^= 1) {
        const bool more = k0 + BK < fin;
        if (more) load(k0 + BK);
        const float *ap = As + k0 * SA + r0, *wp = Ws + b * (ML_STAGE / 4) + c0;
        const int kn = min(BK, fin - k0);
        if (active) {
            if (kn == BK) {
#pragma unroll
                for (int k = 0; k < BK; ++k) step(ap + k * SA, wp + k * SW);
            } else {
#pragma unroll 1
                for (int k = 0; k < kn; ++k) step(ap + k * SA, wp + k * SW);
            }
        }
        if (more) store(b ^ 1);
        __syncthreads();                                  // next tile stored, this one (and at the end As) read
    }

    if (!active) return;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const int c = c0 + (j & 3) + (j >> 2) * 32;
        const float bias = c < fout ? __ldg(B + c) : 0.0f;
        float y[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            float lo, hi;
            unpack2f(acc[i][j / 2], lo, hi);
            y[i] = (j & 1 ? hi : lo) + bias;
        }
        if (last) {
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const int r = row0 + r0 + i;
                if (r < a.n && c < fout)
                    a.Y[((int64_t)agent * a.n + r) * fout + c] = a.out_act ? tanhf(y[i]) : y[i];
            }
        } else if (c < fout) {
            float *h = As + c * SA + r0;
#pragma unroll
            for (int i = 0; i < TM; ++i) y[i] = fmaxf(y[i], 0.0f);
            if constexpr (TM >= 4) {
#pragma unroll
                for (int i = 0; i < TM; i += 4) *(float4 *)(h + i) = *(const float4 *)(y + i);
            } else if constexpr (TM == 2) {
                *(float2 *)h = *(const float2 *)y;
            } else {
                h[0] = y[0];
            }
        }
    }
}

template <int BM>
__global__ void __launch_bounds__(ML_THREADS, 2) k_mlp_f32(const __grid_constant__ MlpArgs a)
{
    extern __shared__ float4 ml_smem[];
    constexpr int SA = BM + 4;
    float *As = (float *)ml_smem;
    float *Ws = As + a.kmax * SA;
    const int agent = blockIdx.y;
    const int row0 = blockIdx.x * BM;
    const float *P = a.params + (int64_t)agent * a.P;
    // the tile's input rows, k-major: four rows per thread, consecutive lanes
    // consecutive k, one 16-byte store each (conflict-free: rows of 4 (BM + 4)
    // bytes shift by 16 bytes per k)
    const int fin = a.dims[0];
    for (int i = threadIdx.x; i < fin * (BM / 4); i += ML_THREADS) {
        const int g = i / fin, k = i - g * fin, r = row0 + 4 * g;
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = r + u < a.n ? __ldg(a.X + (int64_t)(r + u) * a.ldx + k) : 0.0f;
        *(float4 *)(As + k * SA + 4 * g) = make_float4(v[0], v[1], v[2], v[3]);
    }
    for (int l = 0; l < a.L; ++l) {
        const float *W = P + a.w_off[l], *B = P + a.b_off[l];
        const int N = a.dims[l + 1];
        if (N > 128)
            mlp_layer<BM, 256>(a, l, W, B, As, Ws, row0, agent);
        else if (N > 64)
            mlp_layer<BM, 128>(a, l, W, B, As, Ws, row0, agent);
        else if (N > 32)
            mlp_layer<BM, 64>(a, l, W, B, As, Ws, row0, agent);
        else
            mlp_layer<BM, 32>(a, l, W, B, As, Ws, row0, agent);
    }
}

uint32_t mlp_smem(int bm, int kmax) { return (uint32_t)(kmax * (bm + 4) * 4) + 2u * ML_STAGE; }

// a = a_0 + sum_{j>=1} w_j (a_j - a_0), rounded at every operation
__global__ void k_combine_mean(const float *Y, int64_t y_stride, int ldy,
                               const float *__restrict__ w, int M, int n, int K,
                               float *__restrict__ out, int ldo)
{
    ptx::grid_wait_previous();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)n * K) return;
    const int64_t r = i / K, k = i % K;
    const float a0 = Y[r * ldy + k];
    float acc = a0;
    for (int j = 1; j < M; ++j)
        acc = __fadd_rn(acc, __fmul_rn(w[j], __fsub_rn(Y[j * y_stride + r * ldy + k], a0)));
    out[r * ldo + k] = acc;
}

// per-agent argmax (lowest index on ties), then the action with the strictly
// largest count, else hold (1)
__global__ void k_combine_vote(const float *Y, int64_t y_stride, int ldy, int M,
                               int n, int nact, uint32_t dueling, uint8_t *__restrict__ out)
{
    ptx::grid_wait_previous();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    int cnt[3] = {0, 0, 0};
    for (int j = 0; j < M; ++j) {
        const int best = HeadQ(Y + j * y_stride + (int64_t)r * ldy, (dueling >> j) & 1u, nact).argmax();
        if (best < 3) cnt[best]++;
    }
    int best = 0, bc = cnt[0];
    bool tie = false;
    for (int c = 1; c < 3; ++c) {
        if (cnt[c] > bc) { bc = cnt[c]; best = c; tie = false; }
        else if (cnt[c] == bc) tie = true;
    }
    out[r] = (uint8_t)(tie ? 1 : best);
}

// Q-values after each agent's head: q[j][r][a], a < nact.
__global__ void k_heads(const float *Y, int64_t y_stride, int ldy, int M, int n, int nact,
                        uint32_t dueling, float *__restrict__ q)
{
    ptx::grid_wait_previous();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)M * n) return;
    const int j = (int)(i / n), r = (int)(i % n);
    const HeadQ h(Y + j * y_stride + (int64_t)r * ldy, (dueling >> j) & 1u, nact);
    for (int a = 0; a < nact; ++a) q[i * nact + a] = h.q(a);
}

// DQN / Double DQN learning targets y[j][r] = r + (done ? 0 : gamma Q_target(s', a*)).
__global__ void k_q_targets(const float *Yon, const float *Ytg, int64_t y_stride, int ldy,
                            int M, int n, int nact, uint32_t dueling, const float *__restrict__ rew,
                            const uint8_t *__restrict__ done, float gamma, int double_q, float *__restrict__ y)
{
    ptx::grid_wait_previous();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)M * n) return;
    const int j = (int)(i / n), r = (int)(i % n);
    const bool d = (dueling >> j) & 1u;
    const HeadQ tg(Ytg + j * y_stride + (int64_t)r * ldy, d, nact);
    const int a = double_q ? HeadQ(Yon + j * y_stride + (int64_t)r * ldy, d, nact).argmax() : tg.argmax();
    const float rr = rew[r];
    y[i] = (done && done[r]) ? rr : __fadd_rn(rr, __fmul_rn(gamma, tg.q(a)));
}

}  // namespace

// Networks k_mlp_f32 takes: every input up to 304 wide, every output up to 256.
bool mlp_f32_ok(const fr_ensemble *e)
{
    for (int l = 0; l < e->L; ++l)
        if (e->dims[l] > ML_MAX_K || e->dims[l + 1] > 256) return false;
    return true;
}

cudaError_t launch_mlp_f32(const fr_ensemble *e, const float *obs, int ld, int n, float *y, cudaStream_t s)
{
    MlpArgs a = {};
    a.X = obs;
    a.ldx = ld;
    a.n = n;
    a.params = e->params;
    a.P = e->P;
    a.L = e->L;
    a.out_act = e->out_act;
    a.Y = y;
    for (int l = 0; l <= e->L; ++l) a.dims[l] = e->dims[l];
    for (int l = 0; l < e->L; ++l) {
        a.w_off[l] = e->w_off[l];
        a.b_off[l] = e->b_off[l];
        a.kmax = e->dims[l] > a.kmax ? e->dims[l] : a.kmax;
    }
    // Rows per block: an SM's time is its blocks x (rows + a fixed part), so
    // small batches take short tiles that reach every SM, large ones tall
    // tiles that read each weight less often (measured, 3 x 301-256-256-30:
    // 16 rows 53 us up to 810 rows, 64 rows 211 us at 8,192).
    const int sms = e->ctx->sm_count > 0 ? e->ctx->sm_count : 1;
    int bm = 64;
    int64_t best = -1;
    for (int c : {64, 32, 16}) {
        const int64_t cost = (int64_t)ceil_div((int64_t)ceil_div(n, c) * e->M, sms) * (c + 12);
        if (best < 0 || cost < best) {
            best = cost;
            bm = c;
        }
    }
    const dim3 grid(ceil_div(n, bm), e->M);
    const uint32_t smem = mlp_smem(bm, a.kmax);
    const void *f = bm == 64 ? (const void *)k_mlp_f32<64> : bm == 32 ? (const void *)k_mlp_f32<32>
                                                                   : (const void *)k_mlp_f32<16>;
    const cudaError_t err = set_max_smem_once(f, e->ctx->device);
    if (err != cudaSuccess) return err;
    if (bm == 64)
        k_mlp_f32<64><<<grid, ML_THREADS, smem, s>>>(a);
    else if (bm == 32)
        k_mlp_f32<32><<<grid, ML_THREADS, smem, s>>>(a);
    else
        k_mlp_f32<16><<<grid, ML_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_heads(const float *Y, int64_t y_stride, int ldy, int M, int n, int nact, uint32_t dueling,
                         float *q, cudaStream_t s)
{
    return launch_after(k_heads, ceil_div((int64_t)M * n, 256), 256u, s, Y, y_stride, ldy, M, n, nact, dueling, q);
}

cudaError_t launch_q_targets(const float *Yon, const float *Ytg, int64_t y_stride, int ldy, int M, int n, int nact,
                             uint32_t dueling, const float *rew, const uint8_t *done, float gamma, int double_q,
                             float *y, cudaStream_t s)
{
    return launch_after(k_q_targets, ceil_div((int64_t)M * n, 256), 256u, s, Yon, Ytg, y_stride, ldy, M, n, nact, dueling,
                        rew, done, gamma, double_q, y);
}

cudaError_t launch_dense_f32(const float *X, int64_t x_stride, int ldx, const float *P,
                             int64_t p_stride, int64_t w_off, int64_t b_off, float *Y,
                             int64_t y_stride, int ldy, int n, int fin, int fout, int act, int M,
                             cudaStream_t s)
{
    dim3 grid(ceil_div(fout, BN), ceil_div(n, BM), M);
    if (act == 0)
        k_dense_f32<0><<<grid, NT, 0, s>>>(X, x_stride, ldx, P, p_stride, w_off, b_off, Y, y_stride, ldy, n, fin, fout);
    else if (act == 1)
        k_dense_f32<1><<<grid, NT, 0, s>>>(X, x_stride, ldx, P, p_stride, w_off, b_off, Y, y_stride, ldy, n, fin, fout);
    else
        k_dense_f32<2><<<grid, NT, 0, s>>>(X, x_stride, ldx, P, p_stride, w_off, b_off, Y, y_stride, ldy, n, fin, fout);
    return cudaGetLastError();
}

namespace {
// Maximum of |x| over `count` floats of matrix j (at x + j * stride), as float
// bits atomically maxed into out[j * out_stride] (non-negative floats order
// like their bit patterns).
__global__ void k_absmax(const float *__restrict__ x, int64_t stride, int64_t count, unsigned *out,
                         int out_stride)
{
    const float *xj = x + (int64_t)blockIdx.y * stride;
    float m = 0.0f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(xj[i]));
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out + (int64_t)blockIdx.y * out_stride, __float_as_uint(m));
}
}  // namespace

cudaError_t launch_absmax(const float *x, int64_t stride, int64_t count, int M, unsigned *out, int out_stride,
                          cudaStream_t s)
{
    const long long b = ((long long)count + 255) / 256;
    const unsigned blocks = (unsigned)(b < 1024 ? (b > 0 ? b : 1) : 1024);
    k_absmax<<<dim3(blocks, M), 256, 0, s>>>(x, stride, count, out, out_stride);
    return cudaGetLastError();
}

cudaError_t launch_combine_mean(const float *Y, int64_t y_stride, int ldy, const float *w, int M,
                                int n, int K, float *out, int ldo, cudaStream_t s)
{
    const int64_t tot = (int64_t)n * K;
    return launch_after(k_combine_mean, ceil_div(tot, 256), 256u, s, Y, y_stride, ldy, w, M, n, K, out, ldo);
}

cudaError_t launch_combine_vote(const float *Y, int64_t y_stride, int ldy, int M, int n, int nact,
                                uint32_t dueling, uint8_t *out, cudaStream_t s)
{
    return launch_after(k_combine_vote, ceil_div(n, 256), 256u, s, Y, y_stride, ldy, M, n, nact, dueling, out);
}

}  // namespace fr
