// The learned correction's network on the CUDA cores, FP32: forward pass,
// mean-squared-error loss, backward pass (reverse-mode chain rule, layer by
// layer), Adam (Kingma & Ba 2015, Algorithm 1) and the input standardisation.
// Training runs here; so does the FP32 form of learned inference.
//
// Every product is one tiled SGEMM: the operand forms (plain, transposed, and
// rows of x gathered and standardised as they are loaded) and the elementwise
// epilogue (bias, GELU, GELU', the residual) are template parameters, so a
// gradient is three forward products, two backward ones, one launch for all
// weight and bias gradients and one for their sum.  Sums over the batch are
// split over CTAs into partial parameter vectors and added in a fixed order by
// the last kernel (with Adam's update in a training step), so the gradient is
// bit-for-bit repeatable (no atomics anywhere in training).
#include <algorithm>
#include <cmath>

#include "learned.cuh"
#include "ptx.cuh"

namespace cd {
namespace {

constexpr int BK = 16, kGemmStages = 3;

// Operand forms: element (r, k) of a tile's operand, r a row of A or a column of
// B, is p[r ld + k] or p[k ld + r]
enum { OP_N = 0, OP_T = 1 };

enum { EPI_STORE = 0, EPI_BIAS = 1, EPI_BIAS_GELU = 2, EPI_GELU_BWD = 3, EPI_RESIDUAL = 4, EPI_OCT_GELU = 5 };

struct Gemm {
    int M, N, K;
    const float *A;
    int64_t lda;
    const float *B;
    int64_t ldb;
    float *C;
    int64_t ldc;
    const float *bias;     // EPI_BIAS, EPI_BIAS_GELU, EPI_RESIDUAL: [N]; EPI_OCT_GELU: [M / 8][ldc], row m / 8
    float *Z;              // EPI_BIAS_GELU: pre-activation out (ldc), may be NULL
    const float *Zin;      // EPI_GELU_BWD: pre-activation (ldc); may alias C
    const float *Y;        // EPI_RESIDUAL: targets [.][N]; C = scale (C - Y[rows])
    const int64_t *rows;   // EPI_RESIDUAL: target row of each row, or NULL
    float scale;
    float *sq;             // EPI_RESIDUAL: sum of squared residuals of each CTA
    float *rowsum;         // EPI_STORE: sum over k of A's rows (a bias gradient), may be NULL
    int kps;               // K per split, a multiple of BK; the split is the CTA's z
    int fold;              // EPI_STORE: slabs of a chain (fold_slabs)
    int64_t split_stride;  // floats between consecutive splits' C (and rowsum) blocks
};

constexpr float kGeluC = 0.7978845608028654f;   // sqrt(2 / pi)
constexpr float kGeluA = 0.044715f;

__device__ __forceinline__ float gelu_f(float z)
{
    return 0.5f * z * (1.f + tanhf(kGeluC * fmaf(kGeluA * z, z * z, z)));
}

__device__ __forceinline__ float gelu_grad_f(float z)
{
    const float t = tanhf(kGeluC * fmaf(kGeluA * z, z * z, z));
    return 0.5f * (1.f + t) + 0.5f * z * (1.f - t * t) * kGeluC * fmaf(3.f * kGeluA * z, z, 1.f);
}

// A thread's share of one BR x BK operand slab, copied k-major into shared
// memory by 4-byte asynchronous copies (zero outside the matrix).  Consecutive
// threads take consecutive k (row-major form) or consecutive r (transposed
// form), so global reads are coalesced whatever the leading dimension.
template <int BR, int FORM, int THREADS, int PITCH>
__device__ __forceinline__ void slab_async(float (*S)[PITCH], const float *p, int64_t ld, int r0, int R, int k0, int ke)
{
    static_assert(THREADS % BK == 0, "a thread keeps its k");
    constexpr int E = (BR * BK + THREADS - 1) / THREADS;
    const int tid = threadIdx.x;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int idx = tid + e * THREADS;
        if (BR * BK % THREADS && idx >= BR * BK) break;
        const int r = FORM == OP_N ? idx / BK : idx % BR, k = FORM == OP_N ? tid % BK : idx / BR;
        const bool in = r0 + r < R && k0 + k < ke;
        const float *src = FORM == OP_N ? p + (int64_t)(r0 + r) * ld + k0 + k : p + (int64_t)(k0 + k) * ld + r0 + r;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(&S[k][r])), "l"(in ? src : p),
                     "r"(in ? 4 : 0)
                     : "memory");
    }
}

template <int BM, int BN>
struct TileSmem {
    float A[kGemmStages][BK][BM + 4];
    float B[kGemmStages][BK][BN + 4];
};

// row (or column) i of a thread's TM (TN): groups of four, spread over the tile
// so that a warp's fragment reads have no bank conflicts
template <int BR, int TR>
__device__ __forceinline__ int frag(int t, int i)
{
    return (i / 4) * (BR / (TR / 4)) + t * 4 + i % 4;
}

// One BM x BN tile of C = A B (+ epilogue), TM x TN outputs per thread, K in
// slabs of 16 through a three-stage ring of asynchronous copies (packed FP32x2
// FMAs over row pairs).
//
// What bounds it: the FP32 pipes (75 TFLOP/s measured) and beside them the
// latency of a slab's copies, which the ring hides.  Hidden layer 1 of 2^20
// rows at 48 directions and 128 units (128 x 128 tiles): 2.12 ms, 49 TFLOP/s,
// against 3.18 ms for 64 x 64 tiles of 4 x 4 a thread with the slab's loads
// waited for between two barriers; 8 192 rows (64 x 64 tiles): 32 against
// 45 us.  Moving the standardisation into the copies of layer 1 made them wait
// for their loads again (67 us at 8 192 rows); a fourth stage changed nothing.
// KS = 2 gives a tile two sets of threads, each with half of every slab's k; the
// second set's sums are added at the end.  The 32 x 32 tiles of small batches take
// it: one set is two warps, too few to hide a slab's reads (gradient and Adam
// steps of 256 rows, 48 directions, 192 units: 132 -> 115 us; 2 000 rows 194 -> 183).  In
// 64 x 64 tiles it loses (8 192 rows, 128 units: 283 against 296 us).
template <int BM, int BN, int TM, int TN, int FA, int FB, int EPI, int KS = 1>
__device__ __forceinline__ void gemm_tile(const Gemm &g, int bm, int bn, int z, TileSmem<BM, BN> &sm)
{
    constexpr int SET = (BM / TM) * (BN / TN), THREADS = KS * SET;
    static_assert(TM % 4 == 0 && TN % 4 == 0, "fragments of four");
    static_assert(KS == 1 || (KS == 2 && sizeof(TileSmem<BM, BN>) >= BM * BN * sizeof(float)), "room for a set's sums");
    const int tid = threadIdx.x, set = KS == 1 ? 0 : tid / SET, at = KS == 1 ? tid : tid % SET;
    const int tx = at % (BN / TN), ty = at / (BN / TN);
    const int m0 = bm * BM, n0 = bn * BN;
    const int kb = z * g.kps, ke = min(g.K, kb + g.kps);
    float2 acc[TM / 2][TN];                // pairs of rows
#pragma unroll
    for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
    // sums over the batch (EPI_STORE): chains of g.fold slabs, summed in total
    constexpr bool kFold = EPI == EPI_STORE;
    float2 total[kFold ? TM / 2 : 1][kFold ? TN : 1];
    if (kFold)
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) total[i][j] = make_float2(0.f, 0.f);
    float rsum[2] = {0.f, 0.f};            // this chain, those before it
    int chain = kFold ? g.fold : 0;        // slabs left of it
    const bool want_rsum = EPI == EPI_STORE && g.rowsum && bn == 0;

    const auto issue = [&](int k0, int st) {
        if (k0 < ke) {
            slab_async<BM, FA, THREADS>(sm.A[st], g.A, g.lda, m0, g.M, k0, ke);
            slab_async<BN, FB, THREADS>(sm.B[st], g.B, g.ldb, n0, g.N, k0, ke);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int st = 0; st < kGemmStages - 1; ++st) issue(kb + st * BK, st);
    int cur = 0;
    for (int k0 = kb; k0 < ke; k0 += BK) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGemmStages - 2) : "memory");
        __syncthreads();   // slab k0 has landed for every thread, and the slab before it is done with
        issue(k0 + (kGemmStages - 1) * BK, cur == 0 ? kGemmStages - 1 : cur - 1);
#pragma unroll 4
        for (int q = 0; q < BK / KS; ++q) {
            const int kk = set * (BK / KS) + q;
            float4 b[TN / 4];
#pragma unroll
            for (int j = 0; j < TN; j += 4)
                b[j / 4] = *reinterpret_cast<const float4 *>(&sm.B[cur][kk][frag<BN, TN>(tx, j)]);
#pragma unroll
            for (int i = 0; i < TM; i += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(&sm.A[cur][kk][frag<BM, TM>(ty, i)]);
                const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float4 v = b[j / 4];
                    const float w = j % 4 == 0 ? v.x : j % 4 == 1 ? v.y : j % 4 == 2 ? v.z : v.w;
                    acc[i / 2][j] = __ffma2_rn(a0, make_float2(w, w), acc[i / 2][j]);
                    acc[i / 2 + 1][j] = __ffma2_rn(a1, make_float2(w, w), acc[i / 2 + 1][j]);
                }
            }
        }
        if (want_rsum && tid < BM) {
            float slab = 0.f;
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) slab += sm.A[cur][kk][tid];
            rsum[0] += slab;
        }
        if (kFold && --chain == 0) {
            chain = g.fold;
#pragma unroll
            for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    total[i][j] = __fadd2_rn(total[i][j], acc[i][j]);
                    acc[i][j] = make_float2(0.f, 0.f);
                }
            rsum[1] += rsum[0];
            rsum[0] = 0.f;
        }
        cur = cur + 1 == kGemmStages ? 0 : cur + 1;
    }

    if (kFold)
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = __fadd2_rn(total[i][j], acc[i][j]);
    if (KS == 2) {
        float2 *sums = reinterpret_cast<float2 *>(&sm);
        __syncthreads();                   // the slabs are done with
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (set) sums[(i * TN + j) * SET + at] = acc[i][j];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (!set) acc[i][j] = __fadd2_rn(acc[i][j], sums[(i * TN + j) * SET + at]);
    }
    if (want_rsum && tid < BM && m0 + tid < g.M)
        g.rowsum[(int64_t)z * g.split_stride + m0 + tid] = rsum[1] + rsum[0];
    float *C = g.C + (int64_t)z * g.split_stride;
    const bool vec = g.ldc % 4 == 0 && ((uintptr_t)C & 15) == 0 &&
                     (EPI != EPI_BIAS_GELU || !g.Z || ((uintptr_t)g.Z & 15) == 0);
    float sq = 0.f;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + frag<BM, TM>(ty, i);
        if (m >= g.M || set) continue;
        const int64_t src = EPI == EPI_RESIDUAL && g.rows ? g.rows[m] : (int64_t)m;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            constexpr int W = 4;
            const int n = n0 + frag<BN, TN>(tx, j);
            if (n >= g.N) continue;
            const int64_t o = (int64_t)m * g.ldc + n;
            float c[4] = {}, zz[4] = {};
#pragma unroll
            for (int q = 0; q < W; ++q) {
                const float2 p = acc[i / 2][j + q];
                float v = (i & 1) ? p.y : p.x;
                if (n + q < g.N) {
                    if (EPI == EPI_BIAS || EPI == EPI_BIAS_GELU || EPI == EPI_RESIDUAL) v += g.bias[n + q];
                    if (EPI == EPI_BIAS_GELU) {
                        zz[q] = v;
                        v = gelu_f(v);
                    }
                    if (EPI == EPI_OCT_GELU) v = gelu_f(v + g.bias[(int64_t)(m >> 3) * g.ldc + n + q]);
                    if (EPI == EPI_GELU_BWD) v *= gelu_grad_f(g.Zin[o + q]);
                    if (EPI == EPI_RESIDUAL) {
                        const float res = v - g.Y[src * g.N + n + q];
                        sq = fmaf(res, res, sq);
                        v = g.scale * res;
                    }
                }
                c[q] = v;
            }
            if (vec && n + W <= g.N) {
                *reinterpret_cast<float4 *>(C + o) = make_float4(c[0], c[1], c[2], c[3]);
                if (EPI == EPI_BIAS_GELU && g.Z) *reinterpret_cast<float4 *>(g.Z + o) = make_float4(zz[0], zz[1], zz[2], zz[3]);
            } else {
#pragma unroll
                for (int q = 0; q < W; ++q)
                    if (n + q < g.N) {
                        C[o + q] = c[q];
                        if (EPI == EPI_BIAS_GELU && g.Z) g.Z[o + q] = zz[q];
                    }
            }
        }
    }
    if (EPI == EPI_RESIDUAL) {
        // the tile's squared residuals in a fixed order (the slabs are done with)
        float *red = &sm.A[0][0][0];
        __syncthreads();
        red[tid] = sq;
        __syncthreads();
        if (tid < 32) {
            float t = 0.f;
            for (int q = tid; q < THREADS; q += 32) t += red[q];
#pragma unroll
            for (int w = 16; w > 0; w >>= 1) t += __shfl_xor_sync(0xffffffffu, t, w);
            if (tid == 0) g.sq[blockIdx.x] = t;
        }
    }
}

template <int BM, int BN, int TM, int TN, int FA, int FB, int EPI, int KS>
__global__ void __launch_bounds__(KS * (BM / TM) * (BN / TN), BM == 128 ? 2 : 4)
    sgemm(const __grid_constant__ Gemm g)
{
    extern __shared__ __align__(16) unsigned char smem[];
    TileSmem<BM, BN> &sm = *reinterpret_cast<TileSmem<BM, BN> *>(smem);
    const int ntn = (g.N + BN - 1) / BN;
    gemm_tile<BM, BN, TM, TN, FA, FB, EPI, KS>(g, (int)(blockIdx.x / ntn), (int)(blockIdx.x % ntn), 0, sm);
}

template <int BM, int BN, int TM, int TN, int FA, int FB, int EPI, int KS = 1>
cd_status launch_gemm(const Gemm &g, cudaStream_t s)
{
    const int64_t tiles = (int64_t)((g.M + BM - 1) / BM) * ((g.N + BN - 1) / BN);
    constexpr int smem = sizeof(TileSmem<BM, BN>);
    const auto kern = sgemm<BM, BN, TM, TN, FA, FB, EPI, KS>;
    CD_ALLOW_SMEM(kern, smem, smem);
    LaunchScope ls(CD_K_NET, s);
    kern<<<(unsigned)tiles, KS * (BM / TM) * (BN / TN), smem, s>>>(g);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

int64_t tiles_of(int64_t M, int N, int bm, int bn) { return (M + bm - 1) / bm * ((N + bn - 1) / bn); }

// Tile of a product over M rows: the largest that still gives every SM two
// CTAs (large) or most SMs one (medium), since a small batch is bound by how
// many SMs it reaches and a large one by the FMAs per shared-memory read (a
// gradient at 8 192 rows: 145 us this way, 147 with each line at half as many
// tiles; its layer 2 takes 13.7 us in 64 x 64 tiles).
struct TileShape {
    int bm, bn;
};

TileShape tile_shape(int64_t M, int N)
{
    const int wide = N <= 48 ? 48 : N <= 64 ? 64 : 128;
    if (tiles_of(M, N, 128, wide) >= 2 * 152) return {128, wide};
    return tiles_of(M, N, 64, 64) >= 152 ? TileShape{64, 64} : TileShape{32, 32};
}

template <int FA, int FB, int EPI>
cd_status run_gemm(Gemm g, cudaStream_t s)
{
    if (g.M <= 0 || g.N <= 0) return CD_OK;
    g.kps = 1 << 30;
    const TileShape t = tile_shape(g.M, g.N);
    if (t.bm == 32) return launch_gemm<32, 32, 4, 4, FA, FB, EPI, 2>(g, s);
    if (t.bm == 64) return launch_gemm<64, 64, 8, 4, FA, FB, EPI>(g, s);
    if (t.bn == 48) return launch_gemm<128, 48, 8, 4, FA, FB, EPI>(g, s);
    if (t.bn == 64) return launch_gemm<128, 64, 8, 4, FA, FB, EPI>(g, s);
    return launch_gemm<128, 128, 8, 8, FA, FB, EPI>(g, s);
}

// The three weight gradients (and with them the bias gradients, the sums over
// the batch of the same dz) as one launch: split blockIdx.y of every tile adds
// its rows into its own partial parameter vector, laid out as the parameters.
struct Grads {
    Gemm g[3];          // dW1, dW2, dW3
    int first[4];       // first tile of each, then the tile count
};

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), 4) weight_grads(const __grid_constant__ Grads G)
{
    __shared__ __align__(16) TileSmem<BM, BN> sm;
    const int t = (int)blockIdx.x, j = t >= G.first[2] ? 2 : t >= G.first[1] ? 1 : 0;
    const Gemm &g = G.g[j];
    const int q = t - G.first[j], ntn = (g.N + BN - 1) / BN;
    gemm_tile<BM, BN, TM, TN, OP_T, OP_T, EPI_STORE>(g, q / ntn, q % ntn, (int)blockIdx.y, sm);
}

// U[r][i] = (x[row r][i] - mu[i]) sinv[i], clipped to [-kUMax, kUMax]; a warp a
// row, so that the row index is read once
__global__ void __launch_bounds__(256) gather_normalise(int64_t B, int n_in, const float *__restrict__ X,
                                                        const int64_t *__restrict__ rows, const float *__restrict__ mu,
                                                        const float *__restrict__ sinv, float *__restrict__ U)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t r = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5); r < B; r += warps) {
        const float *x = X + (rows ? rows[r] : r) * n_in;
        float *u = U + r * n_in;
#pragma unroll 4
        for (int i = lane; i < n_in; i += 32) u[i] = fminf(fmaxf((x[i] - mu[i]) * sinv[i], -kUMax), kUMax);
    }
}

constexpr int kRedThreads = 256;

struct AdamArgs {
    float *p, *m, *v;
    float lr, b1, b2, eps, c1, c2;   // bias corrections c1 = 1 / (1 - beta1^t), c2 = 1 / (1 - beta2^t)
};

// out[i] = sum over the splits of the partial gradients, in increasing order;
// with kAdam the parameters take their step from it at once.  The last CTA
// sums the loss: loss[0] = loss_scale * sum_b sq[b] in a fixed order.
template <bool kAdam>
__global__ void __launch_bounds__(kRedThreads) reduce_grads(int64_t n, int splits, const float *__restrict__ part,
                                                            float *__restrict__ out, AdamArgs a, int n_sq,
                                                            const float *__restrict__ sq, float loss_scale,
                                                            float *__restrict__ loss)
{
    if (blockIdx.x == gridDim.x - 1) {
        if (!loss) return;
        __shared__ float sh[kRedThreads];
        float acc = 0.f;
        for (int i = threadIdx.x; i < n_sq; i += kRedThreads) acc += sq[i];
        sh[threadIdx.x] = acc;
        __syncthreads();
        for (int w = kRedThreads / 2; w > 0; w >>= 1) {
            if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) loss[0] = loss_scale * sh[0];
        return;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)(gridDim.x - 1) * blockDim.x) {
        float gi = 0.f;
        int z = 0;
        for (; z + 8 <= splits; z += 8) {
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = part[(int64_t)(z + q) * n + i];
#pragma unroll
            for (int q = 0; q < 8; ++q) gi += v[q];
        }
        for (; z < splits; ++z) gi += part[(int64_t)z * n + i];
        if (out) out[i] = gi;
        if (kAdam) {
            const float mi = fmaf(a.b1, a.m[i], (1.f - a.b1) * gi);
            const float vi = fmaf(a.b2, a.v[i], (1.f - a.b2) * gi * gi);
            a.m[i] = mi;
            a.v[i] = vi;
            a.p[i] -= a.lr * (mi * a.c1) / (sqrtf(vi * a.c2) + a.eps);
        }
    }
}

// Column sums of x (pass 0) or of (x - mu)^2 (pass 1) over a row range, in
// FP64: partial[split][col].  32 columns per CTA (one per lane), 8 warps
// striding the rows.
constexpr int kNormSplits = 128;

__global__ void __launch_bounds__(256) column_moments(int64_t n, int n_in, const float *__restrict__ x,
                                                      const float *__restrict__ mu, int pass,
                                                      double *__restrict__ partial)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int col = blockIdx.x * 32 + lane;
    const int64_t per = (n + gridDim.y - 1) / gridDim.y;
    const int64_t r0 = blockIdx.y * per, r1 = min(n, r0 + per);
    double acc = 0.0;
    if (col < n_in) {
        const double m = pass ? (double)mu[col] : 0.0;
        for (int64_t r = r0 + w; r < r1; r += 8) {
            const double v = (double)x[r * n_in + col] - m;
            acc += pass ? v * v : v;
        }
    }
    sh[w][lane] = acc;
    __syncthreads();
    if (w == 0 && col < n_in) {
        double t = 0.0;
        for (int i = 0; i < 8; ++i) t += sh[i][lane];
        partial[(int64_t)blockIdx.y * n_in + col] = t;
    }
}

// pass 0: mu = sum / n; pass 1: sinv = 1 / sqrt(sum / n), or 0 for a column
// whose spread is at most kSdMin (it carried no information: ignored)
constexpr double kSdMin = 1e-3;

__global__ void finish_moments(int n_in, int splits, int64_t n, const double *__restrict__ partial, int pass,
                               float *__restrict__ mu, float *__restrict__ sinv)
{
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= n_in) return;
    double t = 0.0;
    for (int z = 0; z < splits; ++z) t += partial[(int64_t)z * n_in + col];
    t /= (double)n;
    if (pass == 0) {
        mu[col] = (float)t;
    } else {
        const double sd = sqrt(t);
        sinv[col] = sd > kSdMin ? (float)(1.0 / sd) : 0.f;
    }
}

// Slabs of a chain when a split adds n slabs of the batch.  One FP32 chain over
// all of them loses about sqrt(n) roundings; chains of n1 rows, n2 of them, lose
// sqrt(n1 / n2 + n2) where the terms share a sign, least at n2^3 = 2 n1 n2, and
// sqrt((n1 + n2) / 2) where they cancel.  Wide networks have tiles enough for one
// or two splits, whatever the batch.  Relative error of dW2, db2 and dW3 at 48 directions,
// 1 024 units, 8 192 rows: 1.3e-6, 1.2e-6 and 1.3e-6 in one chain, 1.1e-7, 0.9e-7 and
// 1.1e-7 in these; 100 000 rows 4.6e-6 and 1.4e-7.  The sums cost nothing (steps of 1.89
// and 1.88 ms; 128 units: 0.140 and 0.139 ms).
int fold_slabs(int64_t n)
{
    const double n2 = std::ceil(std::cbrt(2.0 * BK * (double)n));
    return (int)std::max<int64_t>(1, (int64_t)std::ceil((double)n / n2));
}

// partial gradients of one batch: at most 64 MiB
constexpr int64_t kPartFloats = (int64_t)16 << 20;

int grid_for(int64_t n, int threads)
{
    const int64_t b = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

template <typename T>
cd_status grow(T **p, size_t *cap, size_t need)
{
    if (*cap >= need) return CD_OK;
    if (*p) cd::lib_free(*p);
    *p = nullptr;
    *cap = 0;
    if (cudaMalloc(p, need * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        set_error("device allocation of %zu bytes failed", need * sizeof(T));
        return CD_ENOMEM;
    }
    *cap = need;
    return CD_OK;
}

// activations of `rows` rows: the two layers' outputs, before them the
// standardised inputs unless the caller has its own, after them the
// pre-activations and the backward scratch of training
enum { kOwnInputs = 1, kTraining = 2 };

cd_status net_reserve(cd_net net, int64_t rows, int what)
{
    Activations &a = net->act;
    const size_t h = (size_t)net->lay.H, d = (size_t)net->lay.nd, width[7] = {(size_t)net->lay.n_in, h, h, h, h, h, d};
    float **p[7] = {&a.U, &a.A1, &a.A2, &a.Z1, &a.Z2, &a.G, &a.D};
    for (int i = what & kOwnInputs ? 0 : 1; i < (what & kTraining ? 7 : 3); ++i) {
        const cd_status st = grow(p[i], &a.cap[i], rows * width[i]);
        if (st != CD_OK) return st;
    }
    return CD_OK;
}

// rows standardised, the two hidden layers; the pre-activations are kept for a
// backward pass
cd_status hidden_layers(cd_net net, int64_t B, const float *x, const int64_t *rows, bool train, cudaStream_t s)
{
    const NetLayout &L = net->lay;
    cd_status st = net_reserve(net, B, train ? kOwnInputs | kTraining : kOwnInputs);
    if (st != CD_OK) return st;
    Activations &a = net->act;
    const float *P = net->p;
    {
        LaunchScope ls(CD_K_NET, s);
        gather_normalise<<<(unsigned)std::min<int64_t>((B + 7) / 8, 152 * 32), 256, 0, s>>>(B, L.n_in, x, rows, net->mu,
                                                                                           net->sinv, a.U);
        CD_CHECK_LAUNCH();
    }
    Gemm g = {};
    g.M = (int)B;
    // z1 = W1 u + b1, a1 = gelu(z1)
    g.N = L.H; g.K = L.n_in; g.A = a.U; g.lda = L.n_in; g.B = P + L.W1; g.ldb = L.n_in;
    g.C = a.A1; g.ldc = L.H; g.bias = P + L.b1; g.Z = train ? a.Z1 : nullptr;
    if ((st = run_gemm<OP_N, OP_N, EPI_BIAS_GELU>(g, s)) != CD_OK) return st;
    // z2 = W2 a1 + b2, a2 = gelu(z2)
    g.N = L.H; g.K = L.H; g.A = a.A1; g.lda = L.H; g.B = P + L.W2; g.ldb = L.H;
    g.C = a.A2; g.ldc = L.H; g.bias = P + L.b2; g.Z = train ? a.Z2 : nullptr;
    return run_gemm<OP_N, OP_N, EPI_BIAS_GELU>(g, s);
}

}  // namespace

cd_status mlp_forward(cd_net net, int64_t B, const float *x, float *delta, cudaStream_t s)
{
    if (B > 0x7fffffff / 2) {
        set_error("batch of %lld rows too large", (long long)B);
        return CD_EINVAL;
    }
    cd_status st = hidden_layers(net, B, x, nullptr, false, s);
    if (st != CD_OK) return st;
    // delta = W3 a2 + b3
    const NetLayout &L = net->lay;
    Gemm g = {};
    g.M = (int)B;
    g.N = L.nd; g.K = L.H; g.A = net->act.A2; g.lda = L.H; g.B = net->p + L.W3; g.ldb = L.H;
    g.C = delta; g.ldc = L.nd; g.bias = net->p + L.b3;
    return run_gemm<OP_N, OP_N, EPI_BIAS>(g, s);
}

// Wl[h][0 .. nd] = columns 0 .. nd-1 and 8 nd of W1 (slot 0 and the density)
static __global__ void local_weights(int H, int nd, const float *__restrict__ W1, float *__restrict__ Wl)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < H * (nd + 1); i += gridDim.x * blockDim.x) {
        const int h = i / (nd + 1), j = i - h * (nd + 1);
        Wl[i] = W1[(int64_t)h * (kSlots * nd + 1) + (j < nd ? j : kSlots * nd)];
    }
}

// Layer 1 by octs: the seven external slots are the same for an oct's 8 leaves,
// so their part of z1 (and b1) is one product over the octs and a leaf adds its
// own nd + 1 inputs: 91 instead of 385 multiply-adds a leaf and unit at 48
// directions.
cd_status mlp_forward_octs(cd_net net, int64_t octs, const float *ue, const float *ul, float *h, float *wl, float *delta,
                           cudaStream_t s)
{
    const NetLayout &L = net->lay;
    cd_status st = net_reserve(net, 8 * octs, 0);
    if (st != CD_OK) return st;
    Activations &a = net->act;
    const float *P = net->p;
    {
        LaunchScope ls(CD_K_NET, s);
        local_weights<<<grid_for((int64_t)L.H * (L.nd + 1), 256), 256, 0, s>>>(L.H, L.nd, P + L.W1, wl);
        CD_CHECK_LAUNCH();
    }
    Gemm g = {};
    g.M = (int)octs;
    g.N = L.H; g.K = (kSlots - 1) * L.nd; g.A = ue; g.lda = g.K; g.B = P + L.W1 + L.nd; g.ldb = L.n_in;
    g.C = h; g.ldc = L.H; g.bias = P + L.b1;
    if ((st = run_gemm<OP_N, OP_N, EPI_BIAS>(g, s)) != CD_OK) return st;
    g.M = (int)(8 * octs);
    g.K = L.nd + 1; g.A = ul; g.lda = g.K; g.B = wl; g.ldb = g.K;
    g.C = a.A1; g.bias = h;
    if ((st = run_gemm<OP_N, OP_N, EPI_OCT_GELU>(g, s)) != CD_OK) return st;
    g.K = L.H; g.A = a.A1; g.lda = L.H; g.B = P + L.W2; g.ldb = L.H;
    g.C = a.A2; g.bias = P + L.b2;
    if ((st = run_gemm<OP_N, OP_N, EPI_BIAS_GELU>(g, s)) != CD_OK) return st;
    g.N = L.nd; g.A = a.A2; g.B = P + L.W3;
    g.C = delta; g.ldc = L.nd; g.bias = P + L.b3;
    return run_gemm<OP_N, OP_N, EPI_BIAS>(g, s);
}

// loss and gradient; grad (device, may be NULL) takes the gradient, adam (may
// be NULL) the step it gives
static cd_status loss_grad(cd_net net, int64_t B, const float *x, const float *y, const int64_t *rows, float *loss_out,
                           float *grad, const AdamArgs *adam, cudaStream_t s)
{
    const NetLayout &L = net->lay;
    cd_status st = hidden_layers(net, B, x, rows, true, s);
    if (st != CD_OK) return st;
    Activations &a = net->act;
    const float *P = net->p;
    Gemm g = {};
    g.M = (int)B;
    g.rows = rows;
    // delta = W3 a2 + b3; d loss / d delta = 2 (delta - y) / (B nd) and the squared residuals
    const TileShape t = tile_shape(B, L.nd);
    const int n_sq = (int)tiles_of(B, L.nd, t.bm, t.bn);
    // dW1 = dz1^T u, dW2 = dz2^T a1, dW3 = G3^T a2, each with its bias gradient,
    // split over the batch so that four CTAs reach every SM
    constexpr int BM = 64, BN = 64;
    const int64_t tiles = tiles_of(L.H, L.n_in, BM, BN) + tiles_of(L.H, L.H, BM, BN) + tiles_of(L.nd, L.H, BM, BN);
    const int64_t slabs = (B + BK - 1) / BK,
                  z_most = std::max<int64_t>(1, std::min<int64_t>(4 * 152 / tiles, kPartFloats / L.total));
    int64_t z = std::min(slabs, z_most);
    const int64_t per = (slabs + z - 1) / z;
    z = (slabs + per - 1) / per;
    // Scratch for any batch up to this one, with or without a gradient: neither the
    // splits nor the tiles of a smaller batch need be fewer, and a call whose buffers
    // exist can be captured
    if ((st = grow(&a.red, &a.red_cap, (size_t)tiles_of(B, L.nd, 32, 32))) != CD_OK) return st;
    if ((st = grow(&a.part, &a.part_cap, (size_t)(z_most * L.total))) != CD_OK) return st;
    g.N = L.nd; g.K = L.H; g.A = a.A2; g.lda = L.H; g.B = P + L.W3; g.ldb = L.H;
    g.C = a.D; g.ldc = L.nd; g.bias = P + L.b3; g.Y = y; g.sq = a.red;
    g.scale = (float)(2.0 / ((double)B * L.nd));
    if ((st = run_gemm<OP_N, OP_N, EPI_RESIDUAL>(g, s)) != CD_OK) return st;
    const float loss_scale = (float)(1.0 / ((double)B * L.nd));
    if (!grad && !adam) {   // the loss alone
        if (!loss_out) return CD_OK;
        LaunchScope ls(CD_K_NET, s);
        reduce_grads<false><<<1, kRedThreads, 0, s>>>(0, 0, nullptr, nullptr, AdamArgs{}, n_sq, a.red, loss_scale,
                                                      loss_out);
        CD_CHECK_LAUNCH();
        return CD_OK;
    }
    // dz2 = (G3 W3) * gelu'(z2)
    g = {};
    g.M = (int)B; g.N = L.H; g.K = L.nd; g.A = a.D; g.lda = L.nd; g.B = P + L.W3; g.ldb = L.H;
    g.C = a.G; g.ldc = L.H; g.Zin = a.Z2;
    if ((st = run_gemm<OP_N, OP_T, EPI_GELU_BWD>(g, s)) != CD_OK) return st;
    // dz1 = (dz2 W2) * gelu'(z1), written over z1
    g = {};
    g.M = (int)B; g.N = L.H; g.K = L.H; g.A = a.G; g.lda = L.H; g.B = P + L.W2; g.ldb = L.H;
    g.C = a.Z1; g.ldc = L.H; g.Zin = a.Z1;
    if ((st = run_gemm<OP_N, OP_T, EPI_GELU_BWD>(g, s)) != CD_OK) return st;
    Grads G = {};
    const auto job = [&](int j, int M, int N, const float *A, const float *Bp, int64_t w, int64_t b) {
        Gemm &q = G.g[j];
        q.M = M; q.N = N; q.K = (int)B; q.A = A; q.lda = M; q.B = Bp; q.ldb = N;
        q.C = a.part + w; q.ldc = N; q.rowsum = a.part + b;
        q.kps = (int)(per * BK);
        q.fold = fold_slabs(per);
        q.split_stride = L.total;
        G.first[j + 1] = G.first[j] + (int)tiles_of(M, N, BM, BN);
    };
    job(0, L.H, L.n_in, a.Z1, a.U, L.W1, L.b1);
    job(1, L.H, L.H, a.G, a.A1, L.W2, L.b2);
    job(2, L.nd, L.H, a.D, a.A2, L.W3, L.b3);
    {
        LaunchScope ls(CD_K_NET, s);
        weight_grads<BM, BN, 8, 4><<<dim3((unsigned)tiles, (unsigned)z), 128, 0, s>>>(G);
        CD_CHECK_LAUNCH();
    }
    LaunchScope ls(CD_K_NET, s);
    const unsigned blocks = (unsigned)grid_for(L.total, kRedThreads) + 1;
    if (adam)
        reduce_grads<true><<<blocks, kRedThreads, 0, s>>>(L.total, (int)z, a.part, grad, *adam, n_sq, a.red, loss_scale,
                                                          loss_out);
    else
        reduce_grads<false><<<blocks, kRedThreads, 0, s>>>(L.total, (int)z, a.part, grad, AdamArgs{}, n_sq, a.red,
                                                           loss_scale, loss_out);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

cd_status mlp_loss_grad(cd_net net, int64_t B, const float *x, const float *y, const int64_t *rows, float *loss_out,
                        float *grad, cudaStream_t s)
{
    return loss_grad(net, B, x, y, rows, loss_out, grad, nullptr, s);
}

cd_status mlp_train_step(cd_net net, int64_t B, const float *x, const float *y, const int64_t *rows, const cd_adam &hp,
                         float *loss_out, cudaStream_t s)
{
    const double t = (double)(net->step + 1);
    AdamArgs a;
    a.p = net->p;
    a.m = net->m;
    a.v = net->v;
    a.lr = (float)hp.lr;
    a.b1 = (float)hp.beta1;
    a.b2 = (float)hp.beta2;
    a.eps = (float)hp.eps;
    a.c1 = (float)(1.0 / (1.0 - pow(hp.beta1, t)));
    a.c2 = (float)(1.0 / (1.0 - pow(hp.beta2, t)));
    const cd_status st = loss_grad(net, B, x, y, rows, loss_out, nullptr, &a, s);
    if (st != CD_OK) return st;
    net->step += 1;
    net->version += 1;
    return CD_OK;
}

cd_status mlp_fit_normaliser(cd_net net, int64_t n, const float *x, cudaStream_t s)
{
    const int n_in = net->lay.n_in;
    const int splits = (int)std::min<int64_t>(kNormSplits, std::max<int64_t>(1, n / 64));
    double *partial = nullptr;
    if (cudaMallocAsync(&partial, sizeof(double) * splits * n_in, s) != cudaSuccess) {
        cudaGetLastError();
        set_error("normaliser scratch allocation failed");
        return CD_ENOMEM;
    }
    const dim3 grid((unsigned)((n_in + 31) / 32), (unsigned)splits);
    for (int pass = 0; pass < 2; ++pass) {
        {
            LaunchScope ls(CD_K_NET, s);
            column_moments<<<grid, 256, 0, s>>>(n, n_in, x, net->mu, pass, partial);
        }
        LaunchScope ls(CD_K_NET, s);
        finish_moments<<<(n_in + 127) / 128, 128, 0, s>>>(n_in, splits, n, partial, pass, net->mu, net->sinv);
    }
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(partial, s);
    if (e != cudaSuccess) {
        set_error("normaliser launch: %s", cudaGetErrorString(e));
        return CD_ECUDA;
    }
    net->version += 1;
    return CD_OK;
}

}  // namespace cd
