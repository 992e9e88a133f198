// The learned form of cd_column_density in BF16 on the tcgen05 tensor cores
// (weights and activations BF16, accumulation FP32 in tensor memory).
//
// Layer 1 is split along its inputs.  The external slots (Delta_l = 1..7, 7
// n_dir inputs) are the same for the 8 leaves of an oct, so
//   z1[leaf] = W1c u_cell[leaf] + h[oct],   h[oct] = W1e u_ext[oct] + b1
// with u_cell = the standardised own-oct slot (n_dir inputs) and ln n.  Two
// kernels:
//   learned_oct_tc   one GEMM row per oct: builds u_ext from the per-level
//                    sums (ln, standardise, BF16) straight into the operand
//                    layout in shared memory, one MMA chain of K = 7 n_dir
//                    against the resident W1e, writes h (BF16) and the oct's
//                    external column sum_s c[s] (FP32).
//   learned_cell_tc  one GEMM row per leaf, 128 leaves per tile: the internal +
//                    local term as a small MMA (the oct's 8 densities against
//                    dx K_loc), u_cell on the CUDA cores, then
//                    MMA1 (W1c, + h) -> GELU -> MMA2 (W2, + b2) -> GELU ->
//                    MMA3 (W3, + b3) = delta log2(e) -> N = N_tree 2^(...),
//                    A_V and the shield; the tile's N rows leave as one bulk
//                    copy.  Three independent groups of eight warps share the
//                    weights, so one group's CUDA-core work overlaps the
//                    others' MMAs.
//
// Additions folded into the MMAs.  Every chain ends with one extra K-step of
// 16 whose A is a constant one-hot block, A1h[m][k] = (k == m / 8): row m
// (leaf m of the tile) selects column m / 8, its oct.  With B[n][k] = h[oct
// k][n] this adds h[oct(m)][n] (the tile's 16 layer-1 parts, which
// learned_oct_tc writes directly in this operand layout); with B[n][k] = b[n]
// for every k it adds the bias b[n].
//
// Every operand is K-major without swizzle: element (row, k) of a [rows x K]
// tile sits at byte (row/8) (K/8) 128 + (k/8) 128 + (row%8) 16 + (k%8) 2,
// i.e. LBO = 128 bytes along K and SBO = 16 K bytes between 8-row groups.
// Waits on the tensor cores are bounded; a timeout sets a device flag
// (cd_device_status) and the kernel leaves its loop with all threads together.
#include <algorithm>
#include <cfloat>
#include <vector>

#include "learned.cuh"
#include "umma.cuh"

namespace cd {
namespace {

constexpr int kH = 128;                     // hidden width of the tensor-core form
constexpr int kKW = kH + 16;                // K of the W2 / W3 images: 128 inputs + the bias block
constexpr int kMaxNd = 48;
constexpr uint32_t kMaxPolls = 1u << 26;
constexpr float kGeluC = 0.7978845608028654f;
constexpr float kGeluA = 0.044715f;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kHBlock = 128 * 16;           // BF16 elements of one tile's layer-1 block (16 octs)

static __device__ int g_ltc_fault;

__host__ __device__ constexpr int round16(int v) { return (v + 15) & ~15; }
__host__ __device__ constexpr size_t align128(size_t v) { return (v + 127) & ~(size_t)127; }

__host__ __device__ inline uint32_t op_off(int row, int k, int K)
{
    return (uint32_t)((row >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// Byte offsets of the packed tensor-core weights in one device buffer.
struct TcLayout {
    int nd, NP, KC, KE, n_in;
    size_t w1c, w1e, w2, w3;           // BF16 operand images [128 x KC], [128 x KE], [128 x kKW], [NP x kKW]
    size_t b1;                         // FP32 [128]
    size_t muc, sic, mue, sie;         // FP32 standardisation u = a lg2(x) + b: a then b for the cell inputs
                                       // [KC] and for the external inputs [KE]
    size_t total;
};

TcLayout make_layout(int nd)
{
    TcLayout T;
    T.nd = nd;
    T.NP = round16(nd);
    T.KC = round16(nd + 1);
    T.KE = round16(7 * nd);
    T.n_in = kSlots * nd + 1;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t r = o; o = align128(o + bytes); return r; };
    T.w1c = take((size_t)kH * T.KC * 2);
    T.w1e = take((size_t)kH * T.KE * 2);
    T.w2 = take((size_t)kH * kKW * 2);
    T.w3 = take((size_t)T.NP * kKW * 2);
    T.b1 = take(kH * 4);
    T.muc = take((size_t)T.KC * 4);
    T.sic = take((size_t)T.KC * 4);
    T.mue = take((size_t)T.KE * 4);
    T.sie = take((size_t)T.KE * 4);
    T.total = o;
    return T;
}

struct TcState {
    TcLayout lay;
    unsigned char *buf = nullptr;
    __nv_bfloat16 *h = nullptr;        // per-leaf-tile blocks [128 n x 16 octs] of the layer-1 parts
    float *ext = nullptr;              // [n_oct][nd] external column
    int64_t cap = 0;                   // octs h / ext hold
};

// ---- packing of the FP32 master parameters ----------------------------------

struct PackArgs {
    TcLayout T;
    const float *p;        // packed FP32 parameters
    const float *mu, *sinv;
    NetLayout N;
    unsigned char *buf;
};

// An input with a negative scale is packed as its negative, together with its
// weights: the same products, and the kernels may count on a >= 0 (std_input2).
// W2 and W3 carry the half of GELU.  W3 and b3 are scaled by log2(e) so that the last chain gives delta log2(e)
// and N = N_tree 2^(that).
__global__ void pack_tc(PackArgs A)
{
    const TcLayout &T = A.T;
    const NetLayout &N = A.N;
    const int nd = T.nd;
    const float *W1 = A.p + N.W1, *W2 = A.p + N.W2, *W3 = A.p + N.W3;
    const int64_t n1c = (int64_t)kH * T.KC, n1e = (int64_t)kH * T.KE, n2 = (int64_t)kH * kKW,
                  n3 = (int64_t)T.NP * kKW;
    const int64_t total = n1c + n1e + n2 + n3 + kH + 2 * T.KC + 2 * T.KE;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = e;
        if (i < n1c) {
            const int n = (int)(i / T.KC), k = (int)(i % T.KC);
            const int src = k < nd ? k : kSlots * nd;
            const float w = k <= nd ? W1[(int64_t)n * N.n_in + src] : 0.f, v = A.sinv[src] < 0.f ? -w : w;
            reinterpret_cast<__nv_bfloat16 *>(A.buf + T.w1c + op_off(n, k, T.KC))[0] = __float2bfloat16_rn(v);
            continue;
        }
        i -= n1c;
        if (i < n1e) {
            const int n = (int)(i / T.KE), k = (int)(i % T.KE);
            const float w = k < 7 * nd ? W1[(int64_t)n * N.n_in + nd + k] : 0.f,
                        v = k < 7 * nd && A.sinv[nd + k] < 0.f ? -w : w;
            reinterpret_cast<__nv_bfloat16 *>(A.buf + T.w1e + op_off(n, k, T.KE))[0] = __float2bfloat16_rn(v);
            continue;
        }
        i -= n1e;
        if (i < n2) {
            const int n = (int)(i / kKW), k = (int)(i % kKW);
            const float v = k < kH ? 0.5f * W2[(int64_t)n * kH + k] : A.p[N.b2 + n];
            reinterpret_cast<__nv_bfloat16 *>(A.buf + T.w2 + op_off(n, k, kKW))[0] = __float2bfloat16_rn(v);
            continue;
        }
        i -= n2;
        if (i < n3) {
            const int n = (int)(i / kKW), k = (int)(i % kKW);
            const float v = n >= nd ? 0.f : kLog2e * (k < kH ? 0.5f * W3[(int64_t)n * kH + k] : A.p[N.b3 + n]);
            reinterpret_cast<__nv_bfloat16 *>(A.buf + T.w3 + op_off(n, k, kKW))[0] = __float2bfloat16_rn(v);
            continue;
        }
        i -= n3;
        if (i < kH) { reinterpret_cast<float *>(A.buf + T.b1)[i] = A.p[N.b1 + i]; continue; }
        i -= kH;
        // standardisation as u = a lg2(x) + b: a = ln(2) |sinv|, b = -mu |sinv|
        if (i < 2 * T.KC) {
            const int k = (int)(i % T.KC);
            const int src = k < nd ? k : (k == nd ? kSlots * nd : -1);
            const bool is_a = i < T.KC;
            const float v = src < 0 ? 0.f : (is_a ? kLn2 * fabsf(A.sinv[src]) : -A.mu[src] * fabsf(A.sinv[src]));
            reinterpret_cast<float *>(A.buf + (is_a ? T.muc : T.sic))[k] = v;
            continue;
        }
        i -= 2 * T.KC;
        {
            const int k = (int)(i % T.KE);
            const bool is_a = i < T.KE;
            const float v = k < 7 * nd ? (is_a ? kLn2 * fabsf(A.sinv[nd + k]) : -A.mu[nd + k] * fabsf(A.sinv[nd + k])) : 0.f;
            reinterpret_cast<float *>(A.buf + (is_a ? T.mue : T.sie))[k] = v;
        }
    }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ uint32_t bf2(float v)   // a BF16 constant in both halves
{
    return pack_bf16x2(v, v);
}

// Twice the GELU (tanh form) of two BF16 values in packed BF16 arithmetic:
// 2 g = z (1 + tanh(z (c + c a z^2))).  The result is an operand of the next
// BF16 product, whose packed weights carry the half (exact in BF16).
__device__ __forceinline__ uint32_t gelu2_bf16x2(uint32_t z)
{
    uint32_t z2, p, inner, t, g;
    const uint32_t ca = bf2(kGeluC * kGeluA), c = bf2(kGeluC);
    asm("mul.rn.bf16x2 %0, %1, %1;" : "=r"(z2) : "r"(z));
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(p) : "r"(z2), "r"(ca), "r"(c));
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(inner) : "r"(p), "r"(z));
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(t) : "r"(inner));
    asm("fma.rn.bf16x2 %0, %1, %2, %1;" : "=r"(g) : "r"(z), "r"(t));
    return g;
}

__device__ __forceinline__ float fast_log2(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// standardised, clipped input from a positive quantity: a lg2(max(x, floor)) + b
__device__ __forceinline__ float std_input(float x, float floor_, float a, float b)
{
    return fminf(fmaxf(fmaf(a, fast_log2(fmaxf(x, floor_)), b), -kUMax), kUMax);
}

// Two standardised, clipped inputs in BF16.  Rounding keeps order, so clipping
// after it gives the same values; lo = max(a lg2(floor) + b, -clip) does for the
// floor and the lower clip (a >= 0: pack_tc sees to it; an ignored input has
// a = b = 0, and its 0 x inf falls back to lo = 0).
__device__ __forceinline__ uint32_t std_input2(float2 x, float2 a, float2 b, uint32_t lo)
{
    const float2 u = __ffma2_rn(a, make_float2(fast_log2(x.x), fast_log2(x.y)), b);
    uint32_t v = pack_bf16x2(u.x, u.y);
    const uint32_t hi = pack_bf16x2(kUMax, kUMax);
    asm("max.bf16x2 %0, %0, %1;" : "+r"(v) : "r"(lo));
    asm("min.bf16x2 %0, %0, %1;" : "+r"(v) : "r"(hi));
    return v;
}

__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void named_barrier(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// D (+)= A[128 x K] * B[N x K]^T over K-steps of 16; A and B are K-major
// images whose K (hence SBO) may differ.
__device__ __forceinline__ void mma_steps(uint32_t tmem_d, uint32_t a0, int Ka, uint32_t b0, int Kb, int steps, int N,
                                          bool accumulate_first)
{
    const uint32_t idesc = umma_idesc_bf16(128, N);
    // a K-step is 256 bytes: 16 in the descriptor's address field
    uint64_t da = umma_smem_desc(a0, 128, (uint32_t)Ka * 16), db = umma_smem_desc(b0, 128, (uint32_t)Kb * 16);
    for (int ks = 0; ks < steps; ++ks, da += 16, db += 16)
        umma_bf16(tmem_d, da, db, idesc, (ks > 0 || accumulate_first) ? 1u : 0u);
}

// ---- per-oct part ---------------------------------------------------------------

struct OctArgs {
    TcLayout T;
    const unsigned char *tc;
    int64_t n_oct, ntiles;
    int L;
    const float *Et[4];
    const float *C[CD_MAXL + 1];
    __nv_bfloat16 *h;      // layer-1 blocks, kHBlock elements per 16 octs
    float *ext;            // [n_oct][nd]
};

constexpr int kOctThreads = 128 * kMaxNd / 8;                // a (row, 8 directions) unit each: 24 warps
constexpr int kFarRows = 20;                                 // rows above a tile of octs: 16 + 2 + 1 + 1

// Far slots of a tile of 128 consecutive octs o0 .. o0+127 (o0 a multiple of
// 128): Delta_l = 4 reads the 16 parents o0/8 + r/8, Delta_l = 5 the 2
// grandparents, every coarser level one ancestor; rows 0-15, 16-17, 18 and 19
// (the tail, Delta_l >= 7 summed) of sT.
__device__ __forceinline__ float far_slot_entry(const OctArgs &A, int64_t o0, int row, int d, int nd)
{
    const int L = A.L;
    if (row < 16) return L >= 5 ? A.C[L - 2][((o0 >> 3) + row) * nd + d] : 0.f;
    if (row < 18) return L >= 6 ? A.C[L - 3][((o0 >> 6) + row - 16) * nd + d] : 0.f;
    if (row == 18) return L >= 7 ? A.C[L - 4][(o0 >> 9) * nd + d] : 0.f;
    float t = 0.f;
    for (int dl = 7; dl <= L - 1; ++dl) t += A.C[L - dl + 2][(o0 >> (3 * (dl - 3))) * nd + d];
    return t;
}

// 32 bytes (one sector) in one access, 32-byte aligned.
__device__ __forceinline__ void ld_sector(const float *src, float4 &a, float4 &b)
{
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(src));
}

__device__ __forceinline__ void st_sector(float *dst, float4 a, float4 b)
{
    asm volatile("st.global.v8.f32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w),
                 "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w), "l"(dst)
                 : "memory");
}

struct OctSmem {
    size_t b, h, mu, si, lo, b1, far, ufar, bar, total;   // the operand [128 x KE] at 0
};

__host__ __device__ inline OctSmem oct_smem(const TcLayout &T)
{
    OctSmem S;
    size_t o = align128((size_t)128 * T.KE * 2);
    auto take = [&](size_t bytes) { const size_t r = o; o = align128(o + bytes); return r; };
    S.b = take((size_t)128 * T.KE * 2);
    S.h = take((size_t)8 * kHBlock * 2);
    S.mu = take((size_t)T.KE * 4);
    S.si = take((size_t)T.KE * 4);
    S.lo = take((size_t)T.KE * 2);
    S.b1 = take(kH * 4);
    S.far = take((size_t)kFarRows * T.nd * 4);
    S.ufar = take((size_t)kFarRows * T.nd * 2);
    S.bar = take(64);
    S.total = o;
    return S;
}

// A tile is 128 octs: u_ext straight into the operand layout, one chain of
// MMAs, the epilogue.  What bounds it: these follow one another (operand and
// weights, 84 KB each, leave room for one tile), so a tile's epilogue runs under the
// next one's chain and its loads under the one before's; each part is spread
// over 24 warps, a thread building one row's piece of 8 directions, and the slots
// that the octs of a parent share (Delta_l >= 4) are standardised once per parent
// and copied.  The tables come in whole sectors, 32 bytes a lane: with 16 the
// loads alone kept the L1 busy for longer than the chain.  256^3 leaves, 48
// directions: 1.13 -> 0.74 ms (12 warps, one after the other, a row a lane before);
// its 2.1 GB take 0.31 ms at the copy rate.
__global__ void __launch_bounds__(kOctThreads, 1) learned_oct_tc(OctArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    const TcLayout &T = A.T;
    const OctSmem S = oct_smem(T);
    const int nd = T.nd, KE = T.KE;
    unsigned char *sA = smem, *sB = smem + S.b, *sHb = smem + S.h;   // [128 x KE] operand, W1e image, 8 h blocks
    float *sMu = reinterpret_cast<float *>(smem + S.mu), *sSi = reinterpret_cast<float *>(smem + S.si);
    __nv_bfloat16 *sLo = reinterpret_cast<__nv_bfloat16 *>(smem + S.lo);
    float *sB1 = reinterpret_cast<float *>(smem + S.b1);             // [128]
    float *sT = reinterpret_cast<float *>(smem + S.far);             // [20][nd] far slots of the tile
    __nv_bfloat16 *sU = reinterpret_cast<__nv_bfloat16 *>(smem + S.ufar);   // the same, standardised
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + S.bar);      // [0] weights, [1] MMA
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 2);
    int *sflag = reinterpret_cast<int *>(tslot + 1);                 // [2] by iteration parity: a wait was given up

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
        sflag[0] = sflag[1] = 0;
    }
    for (int k = tid; k < KE; k += kOctThreads) {
        const float a = reinterpret_cast<const float *>(A.tc + T.mue)[k], b = reinterpret_cast<const float *>(A.tc + T.sie)[k];
        sMu[k] = a;
        sSi[k] = b;
        sLo[k] = __float2bfloat16_rn(fmaxf(fmaf(a, fast_log2(kCFloor), b), -kUMax));
    }
    for (int i = tid; i < kH; i += kOctThreads) sB1[i] = reinterpret_cast<const float *>(A.tc + T.b1)[i];
    for (int e = tid; e < 128 * (KE - 7 * nd) / 8; e += kOctThreads)   // K padding
        *reinterpret_cast<uint4 *>(sA + op_off(e & 127, 7 * nd + 8 * (e >> 7), KE)) = make_uint4(0, 0, 0, 0);
    if (warp == 0) tmem_alloc(tslot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tslot;
    if (tid == 0) {
        const uint32_t bytes = (uint32_t)(128 * KE * 2);
        mbar_expect_tx(&bar[0], bytes);
        bulk_g2s(sB, A.tc + T.w1e, bytes, &bar[0]);
    }
    // this thread's unit: a row of the tile, 8 consecutive directions.  A warp
    // takes 8 rows of 4 such pieces: runs of 128 bytes in the tables, and eight
    // rows side by side in the operand (no bank conflicts)
    const int piece = tid >> 3, r = 8 * (piece / (nd >> 3)) + (tid & 7), d0 = 8 * (piece % (nd >> 3));
    const bool unit = r < 128;
    // its entries of the far slots: row of sT, direction
    constexpr int kFs = (kFarRows * kMaxNd + kOctThreads - 1) / kOctThreads;
    int frow[kFs], fd[kFs];
#pragma unroll
    for (int q = 0; q < kFs; ++q) {
        const int e = tid + q * kOctThreads;
        frow[q] = e / nd;
        fd[q] = e - frow[q] * nd;
    }

    float4 c[3][2];
    float fs[kFs];
    auto issue_loads = [&](int64_t tile) {   // rows past the end repeat the last one
        const int64_t o0 = tile * 128, o = std::min<int64_t>(o0 + r, A.n_oct - 1);
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            c[t][0] = c[t][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (unit && t + 1 <= A.L - 1) {
                ld_sector(A.Et[t + 1] + o * nd + d0, c[t][0], c[t][1]);
            }
        }
#pragma unroll
        for (int q = 0; q < kFs; ++q) fs[q] = frow[q] < kFarRows ? far_slot_entry(A, o0, frow[q], fd[q], nd) : 0.f;
    };
    const int64_t first = blockIdx.x, stride = gridDim.x;
    const int n_tile = (int)((A.ntiles - first + stride - 1) / stride);   // at least 1
    issue_loads(first);
    bool ok = mbar_wait_bounded(&bar[0], 0, kMaxPolls), fault = false;
    auto rows_of = [&](int64_t o0) { return (int)std::min<int64_t>(128, A.n_oct - o0); };

    int it = 0;
    for (; it <= n_tile; ++it) {
        const int64_t tile = first + it * stride, o0 = tile * 128;
        const bool more = it < n_tile;
        if (it > 0) ok = mbar_wait_bounded(&bar[1], (it - 1) & 1, kMaxPolls);   // the operand is free, D is complete
        if (!ok) sflag[it & 1] = 1;
        tc_fence_after();
        float2 tot[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) tot[p] = make_float2(0.f, 0.f);
        auto add = [&](float4 a, float4 b) {
            tot[0] = __fadd2_rn(tot[0], make_float2(a.x, a.y));
            tot[1] = __fadd2_rn(tot[1], make_float2(a.z, a.w));
            tot[2] = __fadd2_rn(tot[2], make_float2(b.x, b.y));
            tot[3] = __fadd2_rn(tot[3], make_float2(b.z, b.w));
        };
        if (more) {
#pragma unroll
            for (int q = 0; q < kFs; ++q) {
                if (frow[q] < kFarRows) {
                    const int e = tid + q * kOctThreads;
                    const int k = (frow[q] < 16 ? 3 : frow[q] < 18 ? 4 : frow[q] - 13) * nd + fd[q];
                    sT[e] = fs[q];
                    sU[e] = __float2bfloat16_rn(std_input(fs[q], kCFloor, sMu[k], sSi[k]));
                }
            }
            // near slots -> operand rows
            if (unit) {
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    const float2 x[4] = {make_float2(c[s][0].x, c[s][0].y), make_float2(c[s][0].z, c[s][0].w),
                                         make_float2(c[s][1].x, c[s][1].y), make_float2(c[s][1].z, c[s][1].w)};
                    const int k = s * nd + d0;
                    const uint4 lo = *reinterpret_cast<const uint4 *>(sLo + k);
                    const uint32_t l[4] = {lo.x, lo.y, lo.z, lo.w};
                    uint32_t v[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        v[p] = std_input2(x[p], *reinterpret_cast<const float2 *>(sMu + k + 2 * p),
                                          *reinterpret_cast<const float2 *>(sSi + k + 2 * p), l[p]);
                    *reinterpret_cast<uint4 *>(sA + op_off(r, k, KE)) = make_uint4(v[0], v[1], v[2], v[3]);
                    add(c[s][0], c[s][1]);
                }
            }
            if (it + 1 < n_tile) issue_loads(tile + stride);   // in flight until the next iteration
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        if (sflag[it & 1]) {
            fault = true;
            break;
        }
        if (tid == 0 && it > 1) {       // the h blocks of the last iteration's epilogue
            const int64_t p0 = o0 - 2 * 128 * stride;
            bulk_s2g(A.h + (p0 >> 4) * kHBlock, sHb, (uint32_t)((rows_of(p0) + 15) / 16 * kHBlock * 2));
            bulk_commit();
        }
        // far slots: copies; the external column -> HBM
        if (more && unit) {
#pragma unroll
            for (int s = 3; s < 7; ++s) {
                const int e = (s == 3 ? (r >> 3) : s == 4 ? 16 + (r >> 6) : s == 5 ? 18 : 19) * nd + d0;
                *reinterpret_cast<uint4 *>(sA + op_off(r, s * nd + d0, KE)) = *reinterpret_cast<const uint4 *>(sU + e);
                add(*reinterpret_cast<const float4 *>(sT + e), *reinterpret_cast<const float4 *>(sT + e + 4));
            }
            if (o0 + r < A.n_oct) {
                st_sector(A.ext + (o0 + r) * nd + d0, make_float4(tot[0].x, tot[0].y, tot[1].x, tot[1].y),
                          make_float4(tot[2].x, tot[2].y, tot[3].x, tot[3].y));
            }
        }
        if (tid == 0) bulk_wait_read<0>();   // sHb is free
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (more && tid == 0) {
            mma_steps(tbase + 128 * (it & 1), smem_u32(sA), KE, smem_u32(sB), KE, KE / 16, kH, false);
            umma_commit(&bar[1]);
        }
        __syncwarp();
        // Epilogue of the tile before: h = D + b1 -> the B-operand blocks of the
        // per-leaf kernel, block r / 16, element (n, r % 16); rows past the end are
        // zero (a 0 x NaN in the product would poison a real row).  Warps w,
        // w + 4, .. share TMEM lanes 32 (w % 4) .. and take 8 columns in turn.  Two
        // rows of one column make a word: even lanes store the even columns of a
        // pair of rows, odd lanes the odd ones.
        if (it > 0) {
            const int quarter = warp & 3, row = quarter * 32 + lane;
            const bool odd = lane & 1, live = row < rows_of(o0 - 128 * stride);
            unsigned char *blk = sHb + (row >> 4) * kHBlock * 2;
            const uint32_t src = tbase + 128 * ((it - 1) & 1) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
            for (int c0 = 8 * (warp >> 2); c0 < kH; c0 += 8 * (kOctThreads / 128)) {
                uint32_t v[8];
                tmem_ld8(src + (uint32_t)c0, v);
                tmem_ld_wait(v);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float2 b = *reinterpret_cast<const float2 *>(sB1 + c0 + 2 * p);
                    const float x = live ? __uint_as_float(v[2 * p]) + b.x : 0.f,
                                y = live ? __uint_as_float(v[2 * p + 1]) + b.y : 0.f;
                    const float got = __shfl_xor_sync(0xffffffffu, odd ? x : y, 1);
                    *reinterpret_cast<uint32_t *>(blk + op_off(c0 + 2 * p + (odd ? 1 : 0), row & 14, 16)) =
                        odd ? pack_bf16x2(got, y) : pack_bf16x2(x, got);
                }
            }
        }
    }
    if (!fault) {
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        if (tid == 0) {
            const int64_t p0 = (first + (n_tile - 1) * stride) * 128;
            bulk_s2g(A.h + (p0 >> 4) * kHBlock, sHb, (uint32_t)((rows_of(p0) + 15) / 16 * kHBlock * 2));
            bulk_commit();
        }
    }
    if (tid == 0) {
        if (fault) {
            atomicExch(&g_ltc_fault, 1);
            mbar_wait_bounded(&bar[0], 0, kMaxPolls);
            if (it > 0) mbar_wait_bounded(&bar[1], (it - 1) & 1, kMaxPolls);   // let an issued chain finish
        }
        bulk_wait_all<0>();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tbase, 256);
    }
}

// ---- per-leaf part --------------------------------------------------------------

struct CellArgs {
    TcLayout T;
    const unsigned char *tc;
    int64_t n_leaf, ntiles;
    float dx_leaf, av_per_nh, c2;    // c2 = -shield_k av_per_nh log2(e)
    float dlo2, dhi2;                // trusted delta range x log2(e)
    const float *rho_leaf;           // Morton
    const float *kloc;               // [8][8][nd]
    const __nv_bfloat16 *h;          // layer-1 blocks
    const float *ext;                // [n_oct][nd]
    float *n_h, *a_v, *shield;
    int vec;                         // n_h is 16-byte aligned: a tile's rows leave as one bulk copy
};

constexpr int kGroups = 3;                       // tiles in flight per CTA
constexpr int kGroupThreads = 256;               // two threads per leaf row, each half the columns
constexpr int kCellThreads = kGroups * kGroupThreads;
constexpr int kMaxGq = (kMaxNd / 8 + 1) / 2;      // 8-direction groups a thread takes

// Shared memory of learned_cell_tc.  Shared: the weight images, the one-hot
// block, the local-term operand B_loc [NP x 64] = dx K_loc[t][s][d] at
// k = 8 t + s, the cell standardisation.  Per group: the operand buffer (the
// leaf inputs [128 x KC] for MMA1, then the activations [128 x 128] for MMA2
// and MMA3, then the tile's N rows [128 x nd] FP32 on their way out), and two
// stages of the tile's inputs that bulk copies bring in one tile ahead (the 16
// octs' layer-1 block, which MMA1 reads in place, densities of the 128 leaves
// and external columns of their 16 octs).
struct CellSmem {
    size_t w1c, w2, w3, onehot, bloc, muc, sic, lo, bar, grp, grp_stride, a, stage, stage_bytes, st_rho, st_ext, st_h,
        total;
};

__host__ __device__ inline CellSmem cell_smem(const TcLayout &T)
{
    CellSmem S;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t r = o; o = align128(o + bytes); return r; };
    S.w1c = take((size_t)kH * T.KC * 2);
    S.w2 = take((size_t)kH * kKW * 2);
    S.w3 = take((size_t)T.NP * kKW * 2);
    S.onehot = take((size_t)kHBlock * 2);
    S.bloc = take((size_t)T.NP * 64 * 2);
    S.muc = take((size_t)T.KC * 4);
    S.sic = take((size_t)T.KC * 4);
    S.lo = take((size_t)T.KC * 2);
    S.bar = take(128);
    S.grp = o;
    S.a = 0;
    S.st_h = 0;
    S.st_rho = (size_t)kHBlock * 2;
    S.st_ext = S.st_rho + 128 * 4;
    S.stage_bytes = align128(S.st_ext + (size_t)16 * T.nd * 4);
    S.stage = align128((size_t)128 * kH * 2);
    S.grp_stride = S.stage + 2 * S.stage_bytes;
    S.total = S.grp + kGroups * S.grp_stride;
    return S;
}

// a tile's inputs: the layer-1 block, 128 densities, 16 external columns
__device__ __forceinline__ void prefetch_tile(const CellArgs &A, const CellSmem &S, int64_t tile, unsigned char *st,
                                              uint64_t *bar)
{
    const int64_t c0 = tile * 128;
    const int rows = (int)(A.n_leaf - c0 < 128 ? A.n_leaf - c0 : 128);   // a multiple of 8
    const uint32_t b_rho = (uint32_t)rows * 4, b_ext = (uint32_t)(rows / 8) * A.T.nd * 4, b_h = kHBlock * 2;
    mbar_expect_tx(bar, b_rho + b_ext + b_h);
    bulk_g2s(st + S.st_h, A.h + tile * kHBlock, b_h, bar);
    bulk_g2s(st + S.st_rho, A.rho_leaf + c0, b_rho, bar);
    bulk_g2s(st + S.st_ext, A.ext + (c0 >> 3) * A.T.nd, b_ext, bar);
}

// What bounds it: the CUDA cores' work of a tile (GELU of 256 values a leaf,
// logarithms, exponentials) and the latencies of its four MMA chains, which
// follow one another; shared memory is at two thirds of its rate (operands of the
// chains, activations, rows).  Hence three tiles in flight, as many as shared
// memory holds: every thread polls its chain's mbarrier itself, so that a chain
// costs one barrier (its operands are ready), and the local term of a tile is
// issued with the rows of the one before.  A_loc lies in tensor memory, where its
// zeros cost nothing; activations there too, with two tiles in flight (TMEM has
// room for no more), take 2.91 ms.  256^3 leaves, 48 directions: 3.25 -> 2.37 ms
// (0.54 TFLOP of products; two tiles in flight and two barriers a chain before).
__global__ void __launch_bounds__(kCellThreads, 1) learned_cell_tc(CellArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    const TcLayout &T = A.T;
    const CellSmem S = cell_smem(T);
    const int nd = T.nd, KC = T.KC, NP = T.NP;
    const int tid = threadIdx.x, warp = tid >> 5;
    // group g (warps 8g .. 8g+7); row i (TMEM lane quarter warp % 4); half of the columns
    const int g = warp >> 3, quarter = warp & 3, half = (warp >> 2) & 1, i = quarter * 32 + (tid & 31);
    const bool lead = half == 0 && i == 0;     // issues the group's copies and MMAs
    const float *sMu = reinterpret_cast<const float *>(smem + S.muc);
    const float *sSi = reinterpret_cast<const float *>(smem + S.sic);
    const __nv_bfloat16 *sLo = reinterpret_cast<const __nv_bfloat16 *>(smem + S.lo);
    // [0] weights, [1 + g] group MMAs, [1 + kGroups + 2 g + stage] group input stages
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + S.bar);
    uint64_t *mma_bar = bar + 1 + g, *stage_bar = bar + 1 + kGroups + 2 * g;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 1 + 3 * kGroups);
    // fault flags [group][barrier parity]: set between barriers n - 1 and n, read after n
    int *sflag = reinterpret_cast<int *>(tslot + 1);
    unsigned char *G = smem + S.grp + g * S.grp_stride;
    unsigned char *sOp = G + S.a;
    __shared__ float sAcc[kGroups][2][128];     // [group][half][row] screening partial sums
    static_assert((1 + 3 * kGroups) * 8 + 4 + 2 * kGroups * 4 <= 128, "barrier block");

    if (tid == 0) {
        for (int b = 0; b < 1 + 3 * kGroups; ++b) mbar_init(&bar[b], 1);
        fence_mbar_init();
        for (int b = 0; b < 2 * kGroups; ++b) sflag[b] = 0;
    }
    // B_loc[d][8 t + s] = dx K_loc[t][s][d] (directions past nd are zero)
    for (int e = tid; e < NP * 64; e += kCellThreads) {
        const int n = e >> 6, k = e & 63;
        const float v = n < nd ? A.dx_leaf * A.kloc[(k >> 3) * 8 * nd + (k & 7) * nd + n] : 0.f;
        *reinterpret_cast<__nv_bfloat16 *>(smem + S.bloc + op_off(n, k, 64)) = __float2bfloat16_rn(v);
    }
    for (int k = tid; k < KC; k += kCellThreads) {
        const float a = reinterpret_cast<const float *>(A.tc + T.muc)[k], b = reinterpret_cast<const float *>(A.tc + T.sic)[k];
        reinterpret_cast<float *>(smem + S.muc)[k] = a;
        reinterpret_cast<float *>(smem + S.sic)[k] = b;
        reinterpret_cast<__nv_bfloat16 *>(smem + S.lo)[k] =
            __float2bfloat16_rn(fmaxf(fmaf(a, fast_log2(k == nd ? kNFloor : kCFloor), b), -kUMax));
    }
    for (int e = tid; e < kHBlock; e += kCellThreads) {   // one-hot: row m selects column m / 8
        const int m = e >> 4, k = e & 15;
        *reinterpret_cast<__nv_bfloat16 *>(smem + S.onehot + op_off(m, k, 16)) =
            __float2bfloat16_rn(k == (m >> 3) ? 1.f : 0.f);
    }
    fence_proxy_async_smem();
    if (warp == 0) tmem_alloc(tslot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tslot;
    if (tid == 0) {
        const uint32_t b1 = (uint32_t)(kH * KC * 2), b2 = (uint32_t)(kH * kKW * 2), b3 = (uint32_t)(NP * kKW * 2);
        mbar_expect_tx(&bar[0], b1 + b2 + b3);
        bulk_g2s(smem + S.w1c, A.tc + T.w1c, b1, &bar[0]);
        bulk_g2s(smem + S.w2, A.tc + T.w2, b2, &bar[0]);
        bulk_g2s(smem + S.w3, A.tc + T.w3, b3, &bar[0]);
    }
    // per group 160 TMEM columns: D (128: D1, D2 in turn, each read out before
    // the next chain; then D3 in columns 0 .. NP-1), the local term in columns
    // 64 .. 64 + NP-1 of it (before D1 and again beside D3), and A_loc (32: row m
    // holds its oct's 8 densities in block t = m % 8, zero elsewhere)
    const uint32_t tD = tbase + (uint32_t)(g * 160), tL = tD + 64, tA = tD + 128;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const uint32_t a_op = smem_u32(sOp), a_1h = smem_u32(smem + S.onehot);
    const int first = blockIdx.x + gridDim.x * g, stride = gridDim.x * kGroups, ntiles = (int)A.ntiles;
    uint32_t phase = 0, sphase = 0;            // sphase: a bit per stage
    uint32_t nbar = 0;                         // group barriers passed
    uint32_t pending = 0;                      // leader, a bit per stage: its prefetch has not been waited for
    bool fault = false;
    if (lead) {
        for (int b = 0; b < 2; ++b)
            if (first + b * stride < ntiles) {
                prefetch_tile(A, S, first + b * stride, G + S.stage + b * S.stage_bytes, &stage_bar[b]);
                pending |= 1u << b;
            }
    }
    const bool bulk_out = A.n_h && A.vec;

    auto give_up = [&]() { sflag[2 * g + (nbar & 1)] = 1; };
    auto wait_mma = [&]() {
        if (!mbar_wait_bounded(mma_bar, phase, kMaxPolls)) give_up();
        phase ^= 1;
        tc_fence_after();
    };
    auto wait_stage = [&](int b) {
        if (mbar_wait_bounded(&stage_bar[b], (sphase >> b) & 1, kMaxPolls)) pending &= ~(1u << b);
        else give_up();
        sphase ^= 1u << b;
    };
    // Everything this group wrote is ready for the next chain (or copy); false
    // if any of its threads gave up a wait.
    auto ready = [&]() {
        fence_proxy_async_smem();
        tc_fence_before();
        named_barrier(1 + g, kGroupThreads);
        tc_fence_after();
        fault = sflag[2 * g + (nbar & 1)] != 0;
        ++nbar;
        return !fault;
    };
    // A_loc of a tile: this thread writes its half of the row's blocks
    auto put_densities = [&](int b, int tile) {
        const float *sR = reinterpret_cast<const float *>(G + S.stage + b * S.stage_bytes + S.st_rho);
        const bool valid = (int64_t)tile * 128 + i < A.n_leaf;
        const float4 r0 = *reinterpret_cast<const float4 *>(sR + (i & ~7));
        const float4 r1 = *reinterpret_cast<const float4 *>(sR + (i & ~7) + 4);
        const uint32_t w[4] = {pack_bf16x2(r0.x, r0.y), pack_bf16x2(r0.z, r0.w), pack_bf16x2(r1.x, r1.y),
                               pack_bf16x2(r1.z, r1.w)};
        const int t = valid ? (i & 7) - 4 * half : -1;
        uint32_t v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = (c >> 2) == t ? w[c & 3] : 0u;
        tmem_st16(tA + lane_off + (uint32_t)(16 * half), v);
        tmem_st_wait();
    };
    auto issue_local = [&]() {
        for (int ks = 0; ks < 4; ++ks)
            umma_bf16_ta(tL, tA + 8 * ks, umma_smem_desc(smem_u32(smem + S.bloc) + ks * 256, 128, 64 * 16),
                         umma_idesc_bf16(128, NP), ks > 0 ? 1u : 0u);
    };

    // GELU of a 128-column accumulator row -> the operand buffer; the next 16
    // columns are on their way while 16 are worked on
    auto gelu_row = [&]() {
        const uint32_t src = tD + lane_off + (uint32_t)(64 * half);
        unsigned char *dst = sOp + op_off(i, 64 * half, kH);
        uint32_t v[2][16];
        tmem_ld16(src, v[0]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t(&w)[16] = v[k & 1];
            tmem_ld_wait(w);
            if (k < 3) tmem_ld16(src + 16 * (k + 1), v[(k + 1) & 1]);
            uint32_t o[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) o[p] = gelu2_bf16x2(pack_bf16x2(__uint_as_float(w[2 * p]), __uint_as_float(w[2 * p + 1])));
            *reinterpret_cast<uint4 *>(dst + (2 * k) * 128) = make_uint4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<uint4 *>(dst + (2 * k + 1) * 128) = make_uint4(o[4], o[5], o[6], o[7]);
        }
    };
    // the row's 8-direction groups this thread takes: [gq0, gq1) of nd / 8
    const int ngq = nd >> 3, gq0 = half * ((ngq + 1) >> 1), gq1 = half ? ngq : (ngq + 1) >> 1;

    // weights, and the first tile's local term
    if (!mbar_wait_bounded(&bar[0], 0, kMaxPolls)) give_up();
    if (first < ntiles) {
        wait_stage(0);
        put_densities(0, first);
    }
    if (ready() && lead && first < ntiles) {
        issue_local();
        umma_commit(mma_bar);
    }

    int stg = 0;
    for (int tile = first; tile < ntiles && !fault; tile += stride, stg ^= 1) {
        const int64_t c0 = (int64_t)tile * 128;
        const int rows = (int)std::min<int64_t>(128, A.n_leaf - c0);
        const int64_t m = c0 + i;
        const bool valid = i < rows, more = tile + stride < ntiles;
        unsigned char *st = G + S.stage + stg * S.stage_bytes;
        const float *sE = reinterpret_cast<const float *>(st + S.st_ext) + (i >> 3) * nd;

        // ---- u_cell = standardised ln(local term) (8 directions per 16-byte
        //      store), then ln n and the K padding ----
        wait_mma();
        {
            uint32_t v[2][8];
            if (gq0 < gq1) tmem_ld8(tL + lane_off + (uint32_t)(8 * gq0), v[0]);
#pragma unroll
            for (int k = 0; k < kMaxGq; ++k) {
                if (gq0 + k >= gq1) break;
                uint32_t(&w)[8] = v[k & 1];
                const int d0 = 8 * (gq0 + k);
                tmem_ld_wait(w);
                if (gq0 + k + 1 < gq1) tmem_ld8(tL + lane_off + (uint32_t)(d0 + 8), v[(k + 1) & 1]);
                const uint4 lo = *reinterpret_cast<const uint4 *>(sLo + d0);
                const uint32_t lw[4] = {lo.x, lo.y, lo.z, lo.w};
                uint32_t o[4];
#pragma unroll
                for (int p = 0; p < 4; ++p)
                    o[p] = std_input2(make_float2(__uint_as_float(w[2 * p]), __uint_as_float(w[2 * p + 1])),
                                      *reinterpret_cast<const float2 *>(sMu + d0 + 2 * p),
                                      *reinterpret_cast<const float2 *>(sSi + d0 + 2 * p), lw[p]);
                *reinterpret_cast<uint4 *>(sOp + op_off(i, d0, KC)) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        for (int d0 = nd + 8 * half; d0 < KC; d0 += 16) {      // ln n at column nd, zeros after it
            const float n = reinterpret_cast<const float *>(st + S.st_rho)[i];
            const float un = d0 == nd ? std_input(n, kNFloor, sMu[nd], sSi[nd]) : 0.f;
            *reinterpret_cast<uint4 *>(sOp + op_off(i, d0, KC)) = make_uint4(pack_bf16x2(un, 0.f), 0, 0, 0);
        }
        if (!ready()) break;
        if (lead) {
            mma_steps(tD, a_op, KC, smem_u32(smem + S.w1c), KC, KC / 16, kH, false);
            mma_steps(tD, a_1h, 16, smem_u32(st + S.st_h), 16, 1, kH, true);
            umma_commit(mma_bar);
        }

        // ---- a1 = gelu(D1) (D1 includes h[oct] + b1) ----
        wait_mma();
        gelu_row();
        if (!ready()) break;
        if (lead) {
            const uint32_t w = smem_u32(smem + S.w2);
            mma_steps(tD, a_op, kH, w, kKW, kH / 16, kH, false);
            mma_steps(tD, a_1h, 16, w + (kH / 16) * 256, kKW, 1, kH, true);
            umma_commit(mma_bar);
        }

        // ---- a2 = gelu(D2) (D2 includes b2; MMA2 has finished reading a1); the
        //      local term once more, beside D3 ----
        wait_mma();
        gelu_row();
        if (!ready()) break;
        if (lead) {
            const uint32_t w = smem_u32(smem + S.w3);
            mma_steps(tD, a_op, kH, w, kKW, kH / 16, NP, false);
            mma_steps(tD, a_1h, 16, w + (kH / 16) * 256, kKW, 1, NP, true);
            issue_local();
            umma_commit(mma_bar);
        }

        // ---- N = (local + external) 2^D3 -> the operand buffer as FP32 rows; shield ----
        wait_mma();
        {
            float *nrow = reinterpret_cast<float *>(sOp) + (size_t)i * nd;
            float *av = A.a_v && valid ? A.a_v + m * nd : nullptr;
            float *nh = A.n_h && valid && !bulk_out ? A.n_h + m * nd : nullptr;
            const bool swap = (i >> (nd & 8 ? 2 : nd & 16 ? 1 : 0)) & 1;
            float2 acc = make_float2(0.f, 0.f);
            const float2 c2 = make_float2(A.c2, A.c2);
#pragma unroll 1
            for (int k = 0; k < kMaxGq; ++k) {
                if (gq0 + k >= gq1) break;
                const int c = 8 * (gq0 + k);
                uint32_t v[8], w[8];
                tmem_ld8(tD + lane_off + (uint32_t)c, v);
                tmem_ld8(tL + lane_off + (uint32_t)c, w);
                tmem_ld_wait(v);
                tmem_ld_wait(w);
                float2 N[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float2 e = *reinterpret_cast<const float2 *>(sE + c + 2 * p);
                    const float2 nt = __fadd2_rn(
                        make_float2(__uint_as_float(w[2 * p]), __uint_as_float(w[2 * p + 1])), e);
                    const float d0 = __uint_as_float(v[2 * p]), d1 = __uint_as_float(v[2 * p + 1]);
                    N[p] = __fmul2_rn(nt, make_float2(fast_exp2(d0 >= A.dlo2 && d0 <= A.dhi2 ? d0 : 0.f),
                                                      fast_exp2(d1 >= A.dlo2 && d1 <= A.dhi2 ? d1 : 0.f)));
                    const float2 x = __fmul2_rn(c2, N[p]);
                    acc = __fadd2_rn(acc, make_float2(fast_exp2(x.x), fast_exp2(x.y)));
                }
                // rows 32 k bytes apart start on 128 / (32 k, 128) banks of 16 bytes: every
                // other run of them takes its two pieces in the other order
                const float4 p0 = make_float4(N[0].x, N[0].y, N[1].x, N[1].y),
                             p1 = make_float4(N[2].x, N[2].y, N[3].x, N[3].y);
                *reinterpret_cast<float4 *>(nrow + c + (swap ? 4 : 0)) = swap ? p1 : p0;
                *reinterpret_cast<float4 *>(nrow + c + (swap ? 0 : 4)) = swap ? p0 : p1;
                if (nh || av) {
                    const float f[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if (nh) nh[c + q] = f[q];
                        if (av) av[c + q] = f[q] * A.av_per_nh;
                    }
                }
            }
            sAcc[g][half][i] = acc.x + acc.y;
        }
        // the next tile's densities (A_loc's last reader was the chain just waited for)
        if (more) {
            wait_stage(stg ^ 1);
            put_densities(stg ^ 1, tile + stride);
        }
        if (!ready()) break;
        if (lead) {
            if (bulk_out) {
                bulk_s2g(A.n_h + c0 * nd, sOp, (uint32_t)(rows * nd * 4));
                bulk_commit();
            }
            if (more) {
                issue_local();
                if (tile + 2 * stride < ntiles) {
                    prefetch_tile(A, S, tile + 2 * stride, st, &stage_bar[stg]);
                    pending |= 1u << stg;
                }
                // the next chain's commit also says that the rows have left the operand buffer
                if (bulk_out) bulk_wait_read<0>();
                umma_commit(mma_bar);
            }
        }
        // the row's screening factor: the two halves' sums, in a fixed order
        if (half == 0 && A.shield && valid) A.shield[m] = (sAcc[g][0][i] + sAcc[g][1][i]) / (float)nd;
    }
    if (fault && lead) {
        atomicExch(&g_ltc_fault, 1);
        mbar_wait_bounded(mma_bar, phase ^ 1, kMaxPolls);   // let an issued chain finish
    }
    // a prefetch still in flight must land, and the output copies must have
    // read the operand buffer, before the CTA exits
    if (lead) {
        for (int b = 0; b < 2; ++b)
            if ((pending >> b) & 1) mbar_wait_bounded(&stage_bar[b], (sphase >> b) & 1, kMaxPolls);
        bulk_wait_all<0>();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tbase, 512);
    }
}

int num_sms()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 152;
}

int max_smem_optin()
{
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}

// Packs the BF16 operands when the master weights changed since the last pack.
cd_status ensure_packed(cd_net net, cudaStream_t s)
{
    TcState *st = static_cast<TcState *>(net->tc);
    if (!st) {
        st = new TcState();
        st->lay = make_layout(net->lay.nd);
        if (cudaMalloc(&st->buf, st->lay.total) != cudaSuccess) {
            cudaGetLastError();
            delete st;
            set_error("cannot allocate the packed tensor-core weights");
            return CD_ENOMEM;
        }
        net->tc = st;
        net->tc_version = 0;
    }
    if (net->tc_version == net->version) return CD_OK;
    PackArgs P;
    P.T = st->lay;
    P.p = net->p;
    P.mu = net->mu;
    P.sinv = net->sinv;
    P.N = net->lay;
    P.buf = st->buf;
    LaunchScope ls(CD_K_NET, s);
    pack_tc<<<num_sms() * 4, 256, 0, s>>>(P);
    CD_CHECK_LAUNCH();
    net->tc_version = net->version;
    return CD_OK;
}

}  // namespace

bool learned_tc_supported(int nd, int hidden) { return hidden == kH && nd >= 8 && nd <= kMaxNd && nd % 8 == 0; }

cd_status column_density_learned_tc(cd_tree t, cd_geom g, const cd_opts &o, float *n_h, float *a_v, float *shield,
                                    cudaStream_t s)
{
    cd_net net = (cd_net)o.net;
    const int nd = g->n_dir;
    if (!learned_tc_supported(nd, net->lay.H)) {
        set_error("the BF16 learned form needs hidden = %d and n_dir a multiple of 8 up to %d (got %d, %d); "
                  "use CD_FP32", kH, kMaxNd, net->lay.H, nd);
        return CD_EUNSUPPORTED;
    }
    if (t->L < 2) {
        set_error("the BF16 learned form needs at least two tree levels");
        return CD_EUNSUPPORTED;
    }
    // the kernels index the tables, the scratch and the outputs, all sized by the
    // geometry, with the network's direction count
    if (net->lay.nd != nd) {
        set_error("the network has %d directions, the geometry %d", net->lay.nd, nd);
        return CD_EINVAL;
    }
    const int sms = num_sms(), smax = max_smem_optin();
    const TcLayout lay = make_layout(nd);
    const size_t smem_oct = oct_smem(lay).total, smem_cell = cell_smem(lay).total;
    if ((int)smem_oct > smax || (int)smem_cell > smax) {
        set_error("the learned kernels need %zu / %zu bytes of shared memory, the device offers %d", smem_oct,
                  smem_cell, smax);
        return CD_EUNSUPPORTED;
    }
    cd_status st = ensure_level_sums(t, g, CD_BF16, s);
    if (st != CD_OK) return st;
    if ((st = ensure_packed(net, s)) != CD_OK) return st;
    TcState *ts = static_cast<TcState *>(net->tc);
    const TcLayout &T = ts->lay;
    const int64_t n_blocks = (t->n_oct + 15) / 16;
    if (ts->cap < t->n_oct) {
        if (ts->h) cd::lib_free(ts->h);
        if (ts->ext) cd::lib_free(ts->ext);
        ts->h = nullptr;
        ts->ext = nullptr;
        ts->cap = 0;
        if (cudaMalloc(&ts->h, (size_t)n_blocks * kHBlock * 2) != cudaSuccess ||
            cudaMalloc(&ts->ext, (size_t)t->n_oct * nd * 4) != cudaSuccess) {
            cudaGetLastError();
            set_error("cannot allocate the per-oct buffers of the learned form");
            return CD_ENOMEM;
        }
        ts->cap = t->n_oct;
    }
    {
        OctArgs A = {};
        A.T = T;
        A.tc = ts->buf;
        A.n_oct = t->n_oct;
        A.ntiles = (t->n_oct + 127) / 128;
        A.L = t->L;
        for (int i = 0; i < 4; ++i) A.Et[i] = t->lv.Et[i];
        for (int k = 0; k <= CD_MAXL; ++k) A.C[k] = t->lv.C[k];
        A.h = ts->h;
        A.ext = ts->ext;
        CD_ALLOW_SMEM(learned_oct_tc, smem_oct, oct_smem(make_layout(kMaxNd)).total);
        const int grid = (int)std::min<int64_t>(A.ntiles, sms);
        LaunchScope ls(CD_K_NET, s);
        learned_oct_tc<<<grid, kOctThreads, smem_oct, s>>>(A);
        CD_CHECK_LAUNCH();
    }
    {
        CellArgs A = {};
        A.T = T;
        A.tc = ts->buf;
        A.n_leaf = t->n_leaf;
        A.ntiles = (t->n_leaf + 127) / 128;
        A.dx_leaf = (float)(t->box_cm / (double)((int64_t)1 << t->L));
        A.av_per_nh = (float)o.av_per_nh;
        A.c2 = (float)(-o.shield_k * o.av_per_nh * 1.4426950408889634);
        // finite bounds: the kernel's comparisons then refuse an infinite correction as well
        A.dlo2 = std::max((float)((double)net->dlo * 1.4426950408889634), -FLT_MAX);
        A.dhi2 = std::min((float)((double)net->dhi * 1.4426950408889634), FLT_MAX);
        A.rho_leaf = t->rho_leaf;
        A.kloc = g->kloc;
        A.h = ts->h;
        A.ext = ts->ext;
        A.n_h = n_h;
        A.a_v = a_v;
        A.shield = shield;
        A.vec = (uintptr_t)n_h % 16 == 0;
        CD_ALLOW_SMEM(learned_cell_tc, smem_cell, cell_smem(make_layout(kMaxNd)).total);
        const int grid = (int)std::min<int64_t>(A.ntiles, sms);
        LaunchScope ls(CD_K_LEARNED, s);
        learned_cell_tc<<<grid, kCellThreads, smem_cell, s>>>(A);
        CD_CHECK_LAUNCH();
    }
    return CD_OK;
}

cd_status learned_tc_fault_check()
{
    int v = 0;
    CD_CUDA(cudaMemcpyFromSymbol(&v, g_ltc_fault, sizeof(int)));
    if (v) {
        const int zero = 0;
        CD_CUDA(cudaMemcpyToSymbol(g_ltc_fault, &zero, sizeof(int)));
        set_error("a learned tensor-core kernel gave up a bounded wait");
        return CD_ETIMEOUT;
    }
    return CD_OK;
}

void net_free_tc(cd_net net)
{
    TcState *st = static_cast<TcState *>(net->tc);
    if (!st) return;
    if (st->buf) cd::lib_free(st->buf);
    if (st->h) cd::lib_free(st->h);
    if (st->ext) cd::lib_free(st->ext);
    delete st;
    net->tc = nullptr;
}

}  // namespace cd
