// Per-leaf combine and epilogue of the BF16 form, with the internal + local
// term (§3.2) on the tensor cores:
//   loc[t][d] = dx_L sum_s rho[oct][s] Kloc[t][s][d]
// is one small product per tile of 128 leaves (16 octs).  Row m of the A
// operand holds the oct's eight densities (BF16) in the block of its own
// octant t = m % 8 (K = 8 blocks x 8; zeros elsewhere, written once);
// B[d][8 t + s] = dx_L Kloc[t][s][d] in BF16.  The product lands in TMEM
// (FP32): the local term carries at most 2^-8 relative error from the two
// roundings, which enters N_H weighted by its share of the column (measured:
// the BF16 path's largest N_H error is unchanged).  The epilogue adds the oct's
// external column E and the parent's far-shell prefix Sp (§3.3), forms the
// screening factor (Eqs. eq_chi, chi_discret) and stages the tile's N_H rows
// for one bulk store.
//
// Tiles are 128 consecutive leaves in Morton order, so E, Sp, the densities and
// the N_H rows of a tile are contiguous spans; bulk copies bring the next
// tile's inputs in while the current one is computed.  Groups of four warps
// (four per CTA when shared memory allows) work on independent tiles so that
// one group's epilogue overlaps another's MMA.  Every wait is bounded; a
// timeout sets a device flag (cd_device_status).
#include <algorithm>
#include <atomic>
#include <string.h>
#include <type_traits>

#include "common.cuh"
#include "umma.cuh"

namespace cd {
namespace {

constexpr uint32_t kMaxPolls = 1u << 26;
constexpr int kK = 64;                  // 8 octant blocks x 8 siblings

static __device__ int g_leaftc_fault;
// cd_debug_wait_polls: < 0 = the default limit
static std::atomic<int64_t> g_pipe_polls{-1};
// cd_debug_leaf_span: list tiles stage their parents' prefix rows as one span
// of up to this many rows (else one row per oct)
constexpr int kSpanRows = 16;
static std::atomic<int> g_span_max{kSpanRows};

__host__ __device__ constexpr size_t align128(size_t v) { return (v + 127) & ~(size_t)127; }
__host__ __device__ constexpr int round16(int v) { return (v + 15) & ~15; }

__host__ __device__ inline uint32_t op_off(int row, int k, int K)
{
    return (uint32_t)((row >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

struct LeafTcArgs {
    LeafLaunch a;
    int NP, G;                 // padded directions (MMA N), groups of 128 threads
    int64_t n_leaf, ntiles;
    float c2;                  // -shield_k av_per_nh log2(e)
    int out_bulk;              // n_h is 16-byte aligned: tile rows leave by bulk copies
    int list;                  // AMR list mode (a.oleaf): tiles of 16 octs, rows scattered
    uint32_t pipe_polls;       // poll limit of the pipeline waits (cd_debug_wait_polls); the exit
                               // waits for the CTA's own copies and products keep kMaxPolls
    int form;                  // kForm* bits; batched: the same for every job of the launch
    int span_max;              // list tiles with Sp: the widest parent span staged as one copy (<= 16)
};

// what a leaf row reads and writes: the parent prefix, staged rows (bulk
// stores) or direct n_h rows, A_V, the screening factor, list tiles
constexpr int kFormSp = 1, kFormBulk = 2, kFormNh = 4, kFormAv = 8, kFormShield = 16, kFormList = 32,
              kFormAvRows = 64;   // A_V alone: its rows are the staged ones, n_h points at a_v

__host__ __device__ inline int leaf_form(const LeafLaunch &a, bool out_bulk, bool list)
{
    return (a.Sp ? kFormSp : 0) | (out_bulk ? kFormBulk : (a.n_h ? kFormNh : 0)) | (a.a_v ? kFormAv : 0) |
           (a.shield ? kFormShield : 0) | (list ? kFormList : 0);
}

struct LeafTcSmem {
    size_t bloc, bar, grp, grp_stride, aloc, out, stage, stage_bytes, st_e, st_p, st_r, st_l, total;
};

__host__ __device__ constexpr LeafTcSmem leaf_tc_smem(int nd, int NP, int G, bool list)
{
    LeafTcSmem S = {};
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t r = o; o = align128(o + bytes); return r; };
    S.bloc = take((size_t)NP * kK * 2);
    S.bar = take(128);
    S.grp = o;
    S.aloc = 0;
    S.out = align128((size_t)128 * kK * 2);
    S.st_e = 0;
    S.st_p = align128((size_t)16 * nd * 4);
    S.st_r = S.st_p + align128((size_t)(list ? 16 : 2) * nd * 4);   // list tiles: up to 16 parent rows
    S.st_l = S.st_r + 128 * 4;                     // list mode: the 16 octs' leaf rows
    S.stage_bytes = align128(S.st_l + (list ? 128 * 4 : 0));
    S.stage = S.out + align128((size_t)128 * nd * 4);
    S.grp_stride = S.stage + 2 * S.stage_bytes;
    S.total = S.grp + (size_t)G * S.grp_stride;
    return S;
}

// groups that fit smax bytes, at most four
constexpr int leaf_tc_groups(int nd, bool list, size_t smax)
{
    int G = 4;
    while (G > 1 && leaf_tc_smem(nd, round16(nd), G, list).total > smax) --G;
    return G;
}

constexpr size_t leaf_tc_smem_most(bool list)
{
    size_t most = 0;
    for (int nd = 4; nd <= 64; nd += 4) {
        const size_t v = leaf_tc_smem(nd, round16(nd), leaf_tc_groups(nd, list, kSmemOptin), list).total;
        most = v > most ? v : most;
    }
    return most;
}

__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ void named_barrier(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// octs in a tile (16, fewer in a list's last tile)
__device__ __forceinline__ int tile_octs(const LeafTcArgs &P, int64_t tile, bool list)
{
    if (!list) return 16;
    const int64_t left = P.a.n_oct - tile * 16;
    return left < 16 ? (int)left : 16;
}

// a tile's inputs: E rows of its 16 octs, Sp rows of their 2 parents, 128
// densities (list mode: plus the octs' 128 leaf rows, and with Sp the parent
// rows of the tile's octs: the span pf .. pl in one copy when it is at most
// 16 rows, else one row per oct; returns the first staged row, or -1 for the
// per-oct layout)
__device__ __forceinline__ int prefetch(const LeafTcArgs &P, const LeafTcSmem &S, int64_t tile, unsigned char *st,
                                        uint64_t *bar, bool list, int pf = 0, int pl = 0)
{
    const int nd = P.a.nd;
    const uint32_t nb = (uint32_t)tile_octs(P, tile, list);
    const bool lsp = list && P.a.Sp;
    const bool per_oct = lsp && pl - pf >= P.span_max;
    // checked builds: a tile outside its job's octs (or parents) copies nothing
    const int64_t o0 = tile * 16, n_oct = P.a.n_oct;
    bool sp_ok = true;
    if (lsp && !per_oct)
        sp_ok = pf <= pl && in_bounds(pf, P.a.n_sp, kCheckLeafTcIn) && in_bounds(pl, P.a.n_sp, kCheckLeafTcIn);
    else if (P.a.Sp && !list)
        sp_ok = in_bounds(tile * 2 + 1, n_oct / 8, kCheckLeafTcIn);
    if (!(in_bounds(o0, n_oct, kCheckLeafTcIn) && in_bounds(o0 + nb - 1, n_oct, kCheckLeafTcIn) && sp_ok)) {
        mbar_expect_tx(bar, 0);
        return pf;
    }
    const uint32_t bp = !P.a.Sp ? 0u : !list ? 2u * nd * 4 : per_oct ? nb * nd * 4 : (uint32_t)(pl - pf + 1) * nd * 4;
    const uint32_t be = nb * nd * 4, br = nb * 32, bl = list ? nb * 32 : 0u;
    mbar_expect_tx(bar, be + bp + br + bl);
    bulk_g2s(st + S.st_e, P.a.E + tile * 16 * nd, be, bar);
    if (per_oct) {
        // a span with parents that have no octs of this level in it: row by row
        for (uint32_t o = 0; o < nb; ++o) {
            int r = __ldg(P.a.oparent + o0 + o);
            if (!in_bounds(r, P.a.n_sp, kCheckLeafTcIn)) r = 0;
            bulk_g2s(st + S.st_p + (size_t)o * nd * 4, P.a.Sp + (int64_t)r * nd, nd * 4, bar);
        }
    } else if (P.a.Sp) {
        bulk_g2s(st + S.st_p, P.a.Sp + (list ? (int64_t)pf : tile * 2) * nd, bp, bar);
    }
    bulk_g2s(st + S.st_r, P.a.rho_leaf + tile * 128, br, bar);
    if (list) bulk_g2s(st + S.st_l, P.a.oleaf + tile * 128, bl, bar);
    return per_oct ? -1 : pf;
}

// Leaf jobs of many boxes (cd_batch) walked by one persistent launch: global
// tile g is tile tile_ref[g].y of job tile_ref[g].x.  All jobs
// of a launch share the direction set; their leaf cell sizes differ, so the
// local-term operand holds Kloc in units of dx and the epilogue scales it.
struct LeafBatch {
    const LeafTcArgs *jobs;
    const int2 *tile_ref;        // global tile -> {job, tile within the job}
    int64_t total;
};

template <class T>
__device__ __forceinline__ T ldg_copy(const T *p)
{
    static_assert(sizeof(T) % 8 == 0, "8-byte words");
    T v;
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(p);
    unsigned long long *dst = reinterpret_cast<unsigned long long *>(&v);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(T) / 8); ++i) dst[i] = __ldg(src + i);
    return v;
}

__device__ __forceinline__ void swap_if(bool s, float4 &a, float4 &b)
{
    const float4 t = a;
    a = s ? b : a;
    b = s ? t : b;
}

// The order in which a lane stores the 16-byte pieces of its row of nd words: 4 q
// directions with q odd spread over the bank groups by themselves; else the
// rows fall on 128 / gcd(4 nd, 128) offsets, and every further run of as many
// rows turns.
__device__ __forceinline__ int row_turn(int nd, int row)
{
    return nd & 4 ? 0 : (row >> (nd & 8 ? 2 : nd & 16 ? 1 : 0)) & 3;
}

// One leaf row of a tile: N_H[d] = loc[d] (x dx when kScale) + E[d] (+ Sp[d]),
// written to the staging row (kOut & 1; as A_V with kOut & 4) and / or straight
// to n_h (kOut & 2, rows with ok only); returns sum_d 2^(c2 N_H[d]).  All 32 lanes of a warp take the
// same instance (the form is a launch constant).
// A staging row is nd words, so rows of 16 k directions start on the same one or
// two of the eight 16-byte bank groups: lanes store the four pieces of 16
// directions in an order of their own (piece q ^ turn, row_turn) instead of four or eight
// lanes at a time on one group.  Lists alone (kTurn): uniform tiles wait for HBM,
// and shorter loads of the product cost them 2 % (256^3, 48 directions).
template <bool kSp, int kOut, bool kScale, bool kTurn>
__device__ __forceinline__ float leaf_rows(uint32_t taddr, int nd, int turn, const float *Ei, const float *Pi,
                                           float *orow, float *nh, bool ok, float c2, float dxs, float avk)
{
    float acc = 0.f;
    if (!kTurn) {
#pragma unroll 1
        for (int c = 0; c < nd; c += 32) {
            uint32_t v[32];
            tmem_ld32(taddr + (uint32_t)c, v);
            tmem_ld_wait();
#pragma unroll
            for (int j4 = 0; j4 < 32; j4 += 4) {
                if (c + j4 >= nd) break;       // nd is a multiple of 4
                float4 e = *reinterpret_cast<const float4 *>(Ei + c + j4);
                if (kSp) {
                    const float4 p = *reinterpret_cast<const float4 *>(Pi + c + j4);
                    e.x += p.x;
                    e.y += p.y;
                    e.z += p.z;
                    e.w += p.w;
                }
                float4 N;
                if (kScale) {
                    N = make_float4(fmaf(__uint_as_float(v[j4]), dxs, e.x), fmaf(__uint_as_float(v[j4 + 1]), dxs, e.y),
                                    fmaf(__uint_as_float(v[j4 + 2]), dxs, e.z), fmaf(__uint_as_float(v[j4 + 3]), dxs, e.w));
                } else {
                    N = make_float4(__uint_as_float(v[j4]) + e.x, __uint_as_float(v[j4 + 1]) + e.y,
                                    __uint_as_float(v[j4 + 2]) + e.z, __uint_as_float(v[j4 + 3]) + e.w);
                }
                acc += (fast_exp2(c2 * N.x) + fast_exp2(c2 * N.y)) + (fast_exp2(c2 * N.z) + fast_exp2(c2 * N.w));
                if (kOut & 4)
                    *reinterpret_cast<float4 *>(orow + c + j4) = make_float4(N.x * avk, N.y * avk, N.z * avk, N.w * avk);
                else if (kOut & 1)
                    *reinterpret_cast<float4 *>(orow + c + j4) = N;
                if ((kOut & 2) && ok) {
                    nh[c + j4] = N.x;
                    nh[c + j4 + 1] = N.y;
                    nh[c + j4 + 2] = N.z;
                    nh[c + j4 + 3] = N.w;
                }
            }
        }
        return acc;
    }
    // kQ pieces from direction c (16 columns of the product are loaded)
    const auto pieces = [&](auto count, int c) {
        constexpr int kQ = decltype(count)::value;
        uint32_t v[16];
        tmem_ld16(taddr + (uint32_t)c, v);
        tmem_ld_wait(v);
        float4 N[kQ];
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            float4 e = *reinterpret_cast<const float4 *>(Ei + c + 4 * q);
            if (kSp) {
                const float4 p = *reinterpret_cast<const float4 *>(Pi + c + 4 * q);
                e.x += p.x;
                e.y += p.y;
                e.z += p.z;
                e.w += p.w;
            }
            const float l[4] = {__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]), __uint_as_float(v[4 * q + 2]),
                                __uint_as_float(v[4 * q + 3])};
            N[q] = kScale ? make_float4(fmaf(l[0], dxs, e.x), fmaf(l[1], dxs, e.y), fmaf(l[2], dxs, e.z),
                                        fmaf(l[3], dxs, e.w))
                          : make_float4(l[0] + e.x, l[1] + e.y, l[2] + e.z, l[3] + e.w);
            acc += (fast_exp2(c2 * N[q].x) + fast_exp2(c2 * N[q].y)) + (fast_exp2(c2 * N[q].z) + fast_exp2(c2 * N[q].w));
            if ((kOut & 2) && ok) {
                nh[c + 4 * q] = N[q].x;
                nh[c + 4 * q + 1] = N[q].y;
                nh[c + 4 * q + 2] = N[q].z;
                nh[c + 4 * q + 3] = N[q].w;
            }
            if (kOut & 4) N[q] = make_float4(N[q].x * avk, N[q].y * avk, N[q].z * avk, N[q].w * avk);
        }
        if (!(kOut & 5)) return;
        float4 *row = reinterpret_cast<float4 *>(orow + c);
        const int x = kQ == 4 ? turn : kQ == 2 ? turn & 1 : 0;
        if constexpr (kQ == 2 || kQ == 4) swap_if(x & 1, N[0], N[1]);
        if constexpr (kQ == 4) {
            swap_if(x & 1, N[2], N[3]);
            swap_if(x & 2, N[0], N[2]);
            swap_if(x & 2, N[1], N[3]);
        }
#pragma unroll
        for (int q = 0; q < kQ; ++q) row[q ^ x] = N[q];
    };
    int c = 0;
#pragma unroll 1
    for (; c + 16 <= nd; c += 16) pieces(std::integral_constant<int, 4>{}, c);
    const int left = (nd - c) >> 2;            // nd is a multiple of 4
    if (left == 1) pieces(std::integral_constant<int, 1>{}, c);
    else if (left == 2) pieces(std::integral_constant<int, 2>{}, c);
    else if (left == 3) pieces(std::integral_constant<int, 3>{}, c);
    return acc;
}

// kMode 0: uniform tiles (P0); 1: list tiles (P0); 2: the jobs of Bt (P0 holds
// the launch-wide nd, NP, G, kloc and screening constant)
template <int kMode>
__global__ void __launch_bounds__(512, 1) leaf_tc(LeafTcArgs P0, LeafBatch Bt)
{
    constexpr bool kList = kMode == 1;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int nd = P0.a.nd, NP = P0.NP, G = P0.G;
    const LeafTcSmem S = leaf_tc_smem(nd, NP, G, kMode != 0);
    const int64_t total = kMode == 2 ? Bt.total : P0.ntiles;
    // global tile -> its job's arguments, the tile within the job and its kind
    auto job_of = [&](int64_t gt, int64_t &lt, bool &list) -> LeafTcArgs {
        if (kMode == 2) {
            const int2 ref = __ldg(Bt.tile_ref + gt);
            lt = ref.y;
            const LeafTcArgs J = ldg_copy(Bt.jobs + ref.x);
            list = J.list != 0;
            return J;
        }
        lt = gt;
        list = kList;
        return P0;
    };
    const int tid = threadIdx.x, warp = tid >> 5;
    const int g = warp >> 2, quarter = warp & 3, i = tid & 127;   // group, TMEM lane quarter, row
    // batched: job arguments and tile index per group in three rotating slots
    // (iteration n uses slot n % 3; during n the group's thread 0 fills slot
    // (n + 1) % 3 for the next tile's prefetch while threads finishing n - 1
    // may still read slot (n - 1) % 3); a job's arguments are copied only when
    // the slot held another job
    __shared__ LeafTcArgs s_job[kMode == 2 ? 4 : 1][3];
    __shared__ int s_job_id[kMode == 2 ? 4 : 1][3];
    __shared__ int s_tile[kMode == 2 ? 4 : 1][3];
    __shared__ int s_run[4][4];                  // list tiles: per group and warp, rows form one run
    // [0 .. G) group MMAs, [G + 2 g + stage] input stages
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + S.bar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 3 * G);
    int *sflag = reinterpret_cast<int *>(tslot + 1);
    unsigned char *Gb = smem + S.grp + (size_t)g * S.grp_stride;
    unsigned char *sA = Gb + S.aloc;
    float *sO = reinterpret_cast<float *>(Gb + S.out);

    if (tid == 0) {
        for (int b = 0; b < 3 * G; ++b) mbar_init(&bar[b], 1);
        fence_mbar_init();
        for (int q = 0; q < G; ++q) sflag[q] = 0;
    }
    // B[d][8 t + s] = dx Kloc[t][s][d] (BF16; batched: dx = 1, the epilogue scales), directions past nd zero
    for (int e = tid; e < NP * kK; e += blockDim.x) {
        const int n = e / kK, k = e % kK;
        const int t = k >> 3, s = k & 7;
        const float v = n < nd ? (kMode == 2 ? 1.f : P0.a.dx_leaf) * P0.a.kloc[(t * 8 + s) * nd + n] : 0.f;
        *reinterpret_cast<__nv_bfloat16 *>(smem + S.bloc + op_off(n, k, kK)) = __float2bfloat16_rn(v);
    }
    // every group's A starts all zero; a tile rewrites only each row's own block
    for (int e = tid; e < G * 128 * kK / 8; e += blockDim.x) {
        const int gg = e / (128 * kK / 8), r = e % (128 * kK / 8);
        reinterpret_cast<uint4 *>(smem + S.grp + (size_t)gg * S.grp_stride + S.aloc)[r] = make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async_smem();
    if (warp == 0) tmem_alloc(tslot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tD = *tslot + (uint32_t)(g * 64);
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const int bid = 1 + g;
    const int64_t first = (int64_t)blockIdx.x * G + g, stride = (int64_t)gridDim.x * G;
    const uint32_t idesc = umma_idesc_bf16(128, NP);
    uint32_t phase = 0, sphase[2] = {0, 0};
    bool pending[2] = {false, false};
    bool fault = false;
    // thread 0 (batched): the reference of the tile after the next one
    int2 ref_next = make_int2(0, 0);
    auto fill_slot = [&](int sl, int2 ref) {   // thread 0, batched
        if (s_job_id[g][sl] != ref.x) {
            s_job[g][sl] = ldg_copy(Bt.jobs + ref.x);
            s_job_id[g][sl] = ref.x;
        }
        s_tile[g][sl] = ref.y;
    };
    // list tiles with a parent prefix: thread 0 reads the span of parent rows of
    // a tile one tile before its prefetch, so that the loads' latency hides
    // behind the current tile; s_pf holds each stage's first staged row
    const bool lsp = kMode == 1 && P0.a.Sp != nullptr;
    __shared__ int s_pf[4][2];
    int pf_next = 0, pl_next = 0;
    auto span = [&](int64_t t, int &pf, int &pl) {
        const int nb = tile_octs(P0, t, true);
        pf = __ldg(P0.a.oparent + t * 16);
        pl = __ldg(P0.a.oparent + t * 16 + nb - 1);
    };
    if (i == 0 && first < total) {
        if (kMode == 2) {
            for (int sl = 0; sl < 3; ++sl) s_job_id[g][sl] = -1;
            fill_slot(0, __ldg(Bt.tile_ref + first));
            prefetch(s_job[g][0], S, s_tile[g][0], Gb + S.stage, &bar[G + 2 * g], P0.list != 0);
            if (first + stride < total) ref_next = __ldg(Bt.tile_ref + first + stride);
        } else {
            int64_t lt;
            bool lst;
            const LeafTcArgs J = job_of(first, lt, lst);
            int pf = 0, pl = 0;
            if (lsp) {
                span(lt, pf, pl);
                if (first + stride < total) span(first + stride, pf_next, pl_next);
            }
            s_pf[g][0] = prefetch(J, S, lt, Gb + S.stage, &bar[G + 2 * g], lst, pf, pl);
        }
        pending[0] = true;
    }

    int stg = 0, it = 0;
    for (int64_t gt = first; gt < total && !fault; gt += stride, stg ^= 1, ++it) {
        int64_t tile;
        bool lst;
        const int slot = it % 3;
        const LeafTcArgs &P = kMode == 2 ? s_job[g][slot] : P0;
        unsigned char *st = Gb + S.stage + stg * S.stage_bytes;
        if (i == 0) {
            if (gt + stride < total) {
                if (kMode == 2) {
                    const int nsl = (it + 1) % 3;
                    fill_slot(nsl, ref_next);
                    prefetch(s_job[g][nsl], S, s_tile[g][nsl], Gb + S.stage + (stg ^ 1) * S.stage_bytes,
                             &bar[G + 2 * g + (stg ^ 1)], P0.list != 0);
                    if (gt + 2 * stride < total) ref_next = __ldg(Bt.tile_ref + gt + 2 * stride);
                } else {
                    int64_t lt;
                    bool ln;
                    const LeafTcArgs J = job_of(gt + stride, lt, ln);
                    const int pf = pf_next, pl = pl_next;
                    if (lsp && gt + 2 * stride < total) span(gt + 2 * stride, pf_next, pl_next);
                    s_pf[g][stg ^ 1] = prefetch(J, S, lt, Gb + S.stage + (stg ^ 1) * S.stage_bytes,
                                                &bar[G + 2 * g + (stg ^ 1)], ln, pf, pl);
                }
                pending[stg ^ 1] = true;
            }
            // the phase bit advances only once the copy has landed: after a
            // timeout the exit below still waits for this stage's copy
            if (mbar_wait_bounded(&bar[G + 2 * g + stg], sphase[stg], P0.pipe_polls)) {
                pending[stg] = false;
                sphase[stg] ^= 1;
            } else {
                sflag[g] = 1;
            }
        }
        named_barrier(bid, 128);
        if (sflag[g]) {
            fault = true;
            break;
        }
        // read after the barrier: thread 0 filled this tile's slot
        lst = kMode == 2 ? P0.list != 0 : kList;
        tile = kMode == 2 ? (int64_t)s_tile[g][slot] : gt;
        const float *sR = reinterpret_cast<const float *>(st + S.st_r);
        // list tiles with a parent prefix: this row's parent row (its load overlaps the product)
        const int par = lsp && (i >> 3) < tile_octs(P, tile, true) ? __ldg(P0.a.oparent + tile * 16 + (i >> 3)) : 0;
        // ---- A row: the oct's densities in block t ----
        {
            const float4 r0 = *reinterpret_cast<const float4 *>(sR + (i & ~7));
            const float4 r1 = *reinterpret_cast<const float4 *>(sR + (i & ~7) + 4);
            *reinterpret_cast<uint4 *>(sA + op_off(i, 8 * (i & 7), kK)) =
                make_uint4(pack_bf16x2(r0.x, r0.y), pack_bf16x2(r0.z, r0.w), pack_bf16x2(r1.x, r1.y),
                           pack_bf16x2(r1.z, r1.w));
        }
        fence_proxy_async_smem();
        tc_fence_before();
        named_barrier(bid, 128);
        if (i == 0) {
            tc_fence_after();
            const uint32_t a0 = smem_u32(sA), b0 = smem_u32(smem + S.bloc);
            for (int ks = 0; ks < kK / 16; ++ks)
                umma_bf16(tD, umma_smem_desc(a0 + ks * 256, 128, kK * 16), umma_smem_desc(b0 + ks * 256, 128, kK * 16),
                          idesc, ks > 0 ? 1u : 0u);
            umma_commit(&bar[g]);
            if (!mbar_wait_bounded(&bar[g], phase, P0.pipe_polls)) sflag[g] = 1;
            // the previous tile's rows must have left the output buffer
            if (P0.out_bulk && !(kMode == 2 ? P0.list != 0 : kList)) bulk_wait_read<0>();
        }
        // each oct's copies were issued by thread i (list tiles)
        if (P0.out_bulk && (kMode == 2 ? P0.list != 0 : kList) && i < 16) bulk_wait_read<0>();
        phase ^= 1;
        named_barrier(bid, 128);
        if (sflag[g]) {
            fault = true;
            break;
        }
        tc_fence_after();
        // ---- N_H = loc + E[oct] + Sp[parent]; screening factor ----
        const int32_t *sL = reinterpret_cast<const int32_t *>(st + S.st_l);
        const int nb = tile_octs(P, tile, lst);
        const float dxs = kMode == 2 ? P.a.dx_leaf : 1.f;   // batched: Kloc in units of dx
        int av_row = -1;                                     // this thread's output row
        {
            // output row of this leaf: Morton position, or the list's row (-1: none)
            const int64_t m = lst ? ((i >> 3) < nb ? (int64_t)sL[i] : -1) : tile * 128 + i;
            const bool ok = m >= 0 && in_bounds(m, lst ? P.a.n_rows : 8 * P.a.n_oct, kCheckLeafTcOut);
            const int64_t mr = ok ? m : 0;
            const float *Ei = reinterpret_cast<const float *>(st + S.st_e) + (i >> 3) * nd;
            // the row's parent row among the staged ones: uniform tiles hold 2 parents;
            // list tiles the span from s_pf (at most 16 rows), or one row per oct (-1)
            int prow = i >> 6;
            if (lsp) {
                const int f = s_pf[g][stg];
                prow = f < 0 ? (i >> 3) : min(max(par - f, 0), 15);
            }
            const float *Pi = reinterpret_cast<const float *>(st + S.st_p) + prow * nd;
            float *orow = sO + (size_t)i * nd;
            const float c2 = P.c2, avk = P.a.av_per_nh;
            // the output form is a launch constant (kernel parameter): pick the
            // loop once, outside the per-direction work.  A_V rows are staged too
            // and leave after the tile's last barrier
            const int fm = P0.form;
            float *nh = (fm & kFormNh) ? P.a.n_h + mr * nd : nullptr;
            float *shp = (fm & kFormShield) ? P.a.shield + mr : nullptr;
            const int form = (fm & kFormSp ? 1 : 0) |
                             (fm & kFormAvRows ? 8 : (fm & (kFormBulk | kFormAv) ? 2 : 0) | (fm & kFormNh ? 4 : 0));
            const uint32_t taddr = tD + lane_off;
            const int turn = row_turn(nd, i);
            float acc;
            __syncwarp();
            switch (form) {
            case 0: acc = leaf_rows<false, 0, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 1: acc = leaf_rows<true, 0, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 2: acc = leaf_rows<false, 1, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 3: acc = leaf_rows<true, 1, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 4: acc = leaf_rows<false, 2, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 5: acc = leaf_rows<true, 2, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 6: acc = leaf_rows<false, 3, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 7: acc = leaf_rows<true, 3, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            case 8: acc = leaf_rows<false, 5, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            default: acc = leaf_rows<true, 5, kMode == 2, kMode == 1>(taddr, nd, turn, Ei, Pi, orow, nh, ok, c2, dxs, avk); break;
            }
            av_row = ok ? (int)m : -1;
            if ((fm & kFormShield) && ok) *shp = acc / (float)nd;
        }
        // list tiles: do the tile's leaf rows form one run (row of leaf i = row of leaf 0 + i)?
        // then one bulk copy sends the tile, as for Morton tiles (octs whose children are all
        // leaves lie next to each other in the depth-first order); else, do every oct's?
        if (lst && P0.out_bulk) {
            const bool past = (i >> 3) >= nb;
            const bool all = __all_sync(0xffffffffu, past || sL[i] == sL[0] + i);
            const bool octs = __all_sync(0xffffffffu, past || (sL[i & ~7] >= 0 && sL[i] == sL[i & ~7] + (i & 7)));
            if ((i & 31) == 0) s_run[g][quarter] = (all ? 1 : 0) | (octs ? 2 : 0);
        }
        // list tiles: the rows the copies below need, read from the stage before the
        // barrier (after it, thread 0 may already prefetch the tile after next into
        // this stage)
        const int lrow0 = lst ? sL[0] : 0, orow0 = lst && i < nb ? sL[8 * i] : -1;
        fence_proxy_async_smem();
        tc_fence_before();
        named_barrier(bid, 128);
        // staged rows times k to their output rows, each warp its own 32, 16 bytes a
        // lane: whole lines of consecutive rows (scalar where dst is off the boundary)
        const auto rows_out = [&](float *dst, float k) {
            const int nq = nd >> 2, dr = 32 / nq, dq = 32 - dr * nq;
            const bool vec = ((uintptr_t)dst & 15) == 0;
            const float4 *N4 = reinterpret_cast<const float4 *>(sO + (size_t)quarter * 32 * nd) + (i & 31);
            int r = (i & 31) / nq, q = (i & 31) - r * nq;
            for (int n = 0; n < nq; ++n, N4 += 32) {
                const int row = __shfl_sync(0xffffffffu, av_row, r);
                const float4 N = *N4;
                float *at = dst + (int64_t)row * nd + 4 * q;
                if (row < 0) {
                } else if (vec) {
                    *reinterpret_cast<float4 *>(at) = make_float4(N.x * k, N.y * k, N.z * k, N.w * k);
                } else {
                    at[0] = N.x * k;
                    at[1] = N.y * k;
                    at[2] = N.z * k;
                    at[3] = N.w * k;
                }
                r += dr;
                q += dq;
                if (q >= nq) {
                    q -= nq;
                    ++r;
                }
            }
        };
        if (P0.form & kFormAv) rows_out(P.a.a_v, P.a.av_per_nh);
        if (P0.out_bulk && !lst && i == 0 && in_bounds(tile * 128 + 127, 8 * P.a.n_oct, kCheckLeafTcOut)) {
            bulk_s2g(P.a.n_h + tile * 128 * nd, sO, (uint32_t)(128 * nd * 4));
            bulk_commit();
        }
        if (lst && P0.out_bulk) {
            const int runs = s_run[g][0] & s_run[g][1] & s_run[g][2] & s_run[g][3];
            if ((runs & 1) && lrow0 >= 0 && in_bounds(lrow0 + 8 * nb - 1, P.a.n_rows, kCheckLeafTcOut)) {
                if (i == 0) {
                    bulk_s2g(P.a.n_h + (int64_t)lrow0 * nd, sO, (uint32_t)(8 * nb * nd * 4));
                    bulk_commit();
                }
            } else if (runs & 2) {
                // a copy per oct
                if (i < nb && in_bounds(orow0 + 7, P.a.n_rows, kCheckLeafTcOut)) {
                    bulk_s2g(P.a.n_h + (int64_t)orow0 * nd, sO + (size_t)8 * i * nd, (uint32_t)(8 * nd * 4));
                    bulk_commit();
                }
            } else {
                // leaves in an order of the caller's: a copy per row would be 128 of
                // them from one warp.  With the rows' turned order (leaf_rows), 48
                // directions of a 1024^3-effective mesh: 0.509 -> 0.492 ms
                rows_out(P.a.n_h, 1.f);
            }
        }
    }
    if (fault && i == 0) {
        atomicExch(&g_leaftc_fault, 1);
        mbar_wait_bounded(&bar[g], phase ^ 1, kMaxPolls);   // let an issued product finish
    }
    if (i == 0)
        for (int b = 0; b < 2; ++b)
            if (pending[b]) mbar_wait_bounded(&bar[G + 2 * g + b], sphase[b], kMaxPolls);
    if (i == 0 || (kMode != 0 && i < 16)) bulk_wait_all<0>();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(*tslot, 256);
    }
}

// ---- few directions, or the screening factor alone: octs as rows -----------------
//
// Up to 32 directions the tile above is mostly latency: 128 leaves of 12
// directions are 1 536 sums behind three barriers and a product.  Here a row of
// the product is an oct: D[oct][t nd + d] = sum_s rho[oct][s] (dx_L Kloc[t][s][d])
// has M = 128 octs, N = 8 nd columns (at most 256; beyond 32 directions two
// products of four children) and K = 16 (its 8 siblings and 8 zeros; the same
// BF16 operands as above), so that one product and one round of barriers serve
// 1 024 leaves.  A thread has one oct: its external column
// E + Sp stays in registers for the 8 children, and their screening factors are
// 32 contiguous bytes.
// N_H and A_V rows leave through a per-warp transpose, 128 bytes of a row at a
// time.
// What bounds it: the exponentials (16 a clock and SM), with rows the HBM
// stores.  256^3 leaves, 12 directions: 0.068 ms for the screening factor alone,
// 0.189 with N_H, 0.327 with A_V too (4.9 TB/s), against 0.314, 0.339 and 0.691 in
// tiles of 128 leaves; 32 directions: 0.210, 0.456, 0.845 against 0.389, 0.759,
// 3.08.  (Rows stored straight from the threads, 16 bytes each: 0.49 for N_H
// at 12 directions.)
struct LeafOctArgs {
    LeafLaunch a;
    int64_t ntiles;              // of 128 octs
    float c2;                    // -shield_k av_per_nh log2(e)
    uint32_t pipe_polls;
};

template <int ND>
struct LeafOctShape {
    static constexpr int N = 8 * ND;
    static constexpr int kParts = N > 256 ? 2 : 1;                       // products a tile: all children, or four
    static constexpr int kN = N / kParts;
    static_assert(kN % 32 == 0, "a product is drained 32 columns at a time");
    static constexpr int kCols = kN <= 64 ? 64 : kN <= 128 ? 128 : 256;  // TMEM columns of a group
    static constexpr int kGroups = 512 / kCols > 4 ? 4 : 512 / kCols;
    static constexpr uint32_t kB = N * 32, kA = 4096;                    // operand bytes (K = 16)
    static constexpr uint32_t kE = 128 * ND * 4, kP = 16 * ND * 4, kStage = kE + kP + 4096;
    static constexpr uint32_t kGroup = kA + 2 * kStage;
    static constexpr uint32_t kT = 128 * 36 * 4;                         // a group's row transposes
    static constexpr size_t smem(int G, bool rows) { return kB + (size_t)G * (kGroup + (rows ? kT : 0)); }
};

// kRows: N_H or A_V rows are wanted (16-byte aligned)
template <int ND, bool kRows>
__global__ void __launch_bounds__(128 * LeafOctShape<ND>::kGroups, 1) leaf_oct_tc(const __grid_constant__ LeafOctArgs P)
{
    using S = LeafOctShape<ND>;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t bar[3 * S::kGroups];      // [g] products, [G + 2 g + stage] input stages
    __shared__ uint32_t tslot;
    // [0] an input wait, [1] a product wait was given up.  Two flags: a slow warp may still
    // read a tile's last product flag when thread 0 gives up the next tile's input wait,
    // and either flag is read before a barrier that comes before its next write
    __shared__ int sflag[S::kGroups][2];
    const int tid = threadIdx.x, warp = tid >> 5, g = warp >> 2, quarter = warp & 3, i = tid & 127;
    const int G = blockDim.x >> 7;
    unsigned char *sA = smem + S::kB + (size_t)g * S::kGroup;
    unsigned char *stage0 = sA + S::kA;
    const int64_t n_oct = P.a.n_oct;
    const auto octs = [&](int64_t tile) { return (uint32_t)(n_oct - tile * 128 < 128 ? n_oct - tile * 128 : 128); };
    const auto prefetch = [&](int64_t tile, int s) {
        const int64_t o0 = tile * 128;
        const uint32_t nb = octs(tile);
        uint64_t *b = &bar[S::kGroups + 2 * g + s];
        unsigned char *st = stage0 + s * S::kStage;
        if (!(in_bounds(o0, n_oct, kCheckLeafTcIn) && in_bounds(o0 + nb - 1, n_oct, kCheckLeafTcIn) &&
              (!P.a.Sp || in_bounds((o0 + nb - 1) >> 3, n_oct / 8, kCheckLeafTcIn)))) {
            mbar_expect_tx(b, 0);
            return;
        }
        const uint32_t bp = P.a.Sp ? (nb + 7) / 8 * ND * 4 : 0u;
        mbar_expect_tx(b, nb * (ND * 4 + 32) + bp);
        bulk_g2s(st, P.a.E + o0 * ND, nb * ND * 4, b);
        if (P.a.Sp) bulk_g2s(st + S::kE, P.a.Sp + (o0 >> 3) * ND, bp, b);
        bulk_g2s(st + S::kE + S::kP, P.a.rho_leaf + o0 * 8, nb * 32, b);
    };

    if (tid == 0) {
        for (int b = 0; b < 3 * S::kGroups; ++b) mbar_init(&bar[b], 1);
        fence_mbar_init();
        for (int q = 0; q < S::kGroups; ++q) sflag[q][0] = sflag[q][1] = 0;
    }
    for (int n = tid; n < S::N; n += blockDim.x) {
        const float *k = P.a.kloc + (n / ND) * 8 * ND + n % ND;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = P.a.dx_leaf * k[q * ND];
        *reinterpret_cast<uint4 *>(smem + op_off(n, 0, 16)) = make_uint4(
            pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
        *reinterpret_cast<uint4 *>(smem + op_off(n, 8, 16)) = make_uint4(0, 0, 0, 0);
    }
    *reinterpret_cast<uint4 *>(sA + op_off(i, 8, 16)) = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
    // the columns of the groups that there are (a power of two): on a small tree one or two,
    // and CTAs of other calls can have the rest of the SM's (eight evaluations of 32^3
    // at 32 directions on streams of their own, screening factor: 107 us with all
    // groups' columns, 81 so; 64^3: 149 and 122)
    const uint32_t cols = S::kCols * (G > 2 ? 4 : G);
    if (warp == 0) tmem_alloc(&tslot, cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tD = tslot + (uint32_t)(g * S::kCols), taddr = tD + ((uint32_t)(quarter * 32) << 16);
    const int64_t first = (int64_t)blockIdx.x * G + g, stride = (int64_t)gridDim.x * G;
    uint32_t phase = 0, sphase[2] = {0, 0};
    bool pending[2] = {false, false}, fault = false;
    if (i == 0 && first < P.ntiles) {
        prefetch(first, 0);
        pending[0] = true;
    }
    int s = 0;
    for (int64_t tile = first; tile < P.ntiles; tile += stride, s ^= 1) {
        if (i == 0) {
            if (tile + stride < P.ntiles) {
                prefetch(tile + stride, s ^ 1);
                pending[s ^ 1] = true;
            }
            if (mbar_wait_bounded(&bar[S::kGroups + 2 * g + s], sphase[s], P.pipe_polls)) {
                pending[s] = false;
                sphase[s] ^= 1;
            } else {
                sflag[g][0] = 1;
            }
        }
        named_barrier(1 + g, 128);
        if (sflag[g][0]) {
            fault = true;
            break;
        }
        const unsigned char *st = stage0 + s * S::kStage;
        const float *rho = reinterpret_cast<const float *>(st + S::kE + S::kP) + 8 * i;
        const float4 r0 = *reinterpret_cast<const float4 *>(rho), r1 = *reinterpret_cast<const float4 *>(rho + 4);
        *reinterpret_cast<uint4 *>(sA + op_off(i, 0, 16)) = make_uint4(
            pack_bf16x2(r0.x, r0.y), pack_bf16x2(r0.z, r0.w), pack_bf16x2(r1.x, r1.y), pack_bf16x2(r1.z, r1.w));
        float e[ND];
#pragma unroll
        for (int d = 0; d < ND; d += 4) {
            float4 v = *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(st) + i * ND + d);
            if (P.a.Sp) {
                const float4 p = *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(st + S::kE) + (i >> 3) * ND + d);
                v.x += p.x;
                v.y += p.y;
                v.z += p.z;
                v.w += p.w;
            }
            e[d] = v.x;
            e[d + 1] = v.y;
            e[d + 2] = v.z;
            e[d + 3] = v.w;
        }
        fence_proxy_async_smem();
        tc_fence_before();
        named_barrier(1 + g, 128);
        const int64_t oct = tile * 128 + i;
        const bool ok = oct < n_oct && in_bounds(oct, n_oct, kCheckLeafTcOut);
        // rows: 32 columns of the warp's 32 octs at a time turn into 128-byte
        // pieces of the octs' rows through a padded square of shared memory
        float *T = reinterpret_cast<float *>(smem + S::kB + (size_t)G * S::kGroup) + (warp * 32) * 36;
        const int lane = tid & 31;
        const int64_t row0 = tile * 128 + quarter * 32 + (lane >> 3);
        float acc[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[t] = 0.f;
#pragma unroll
        for (int c = 0; c < S::N; c += 32) {
            if (c % S::kN == 0) {
                // the product of the next children (the accumulator is drained: the tile's
                // operands, or the part before, are behind this barrier)
                if (c) {
                    tc_fence_before();
                    named_barrier(1 + g, 128);
                }
                if (i == 0) {
                    tc_fence_after();
                    umma_bf16(tD, umma_smem_desc(smem_u32(sA), 128, 256), umma_smem_desc(smem_u32(smem) + c * 32, 128, 256),
                              umma_idesc_bf16(128, S::kN), 0u);
                    umma_commit(&bar[g]);
                    if (!mbar_wait_bounded(&bar[g], phase, P.pipe_polls)) sflag[g][1] = 1;
                }
                phase ^= 1;
                named_barrier(1 + g, 128);
                if (sflag[g][1]) {
                    fault = true;
                    break;
                }
                tc_fence_after();
            }
            uint32_t v[32];
            __syncwarp();
            tmem_ld32(taddr + (uint32_t)(c % S::kN), v);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const int t = (c + j) / ND, d = (c + j) % ND;
                const float4 N = make_float4(__uint_as_float(v[j]) + e[d], __uint_as_float(v[j + 1]) + e[d + 1],
                                             __uint_as_float(v[j + 2]) + e[d + 2], __uint_as_float(v[j + 3]) + e[d + 3]);
                acc[t] += (fast_exp2(P.c2 * N.x) + fast_exp2(P.c2 * N.y)) + (fast_exp2(P.c2 * N.z) + fast_exp2(P.c2 * N.w));
                if (kRows) *reinterpret_cast<float4 *>(T + lane * 36 + j) = N;
            }
            if (kRows) {
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int64_t o = row0 + 4 * j;
                    if (o >= n_oct || !in_bounds(o, n_oct, kCheckLeafTcOut)) break;
                    const float4 N = *reinterpret_cast<const float4 *>(T + ((lane >> 3) + 4 * j) * 36 + 4 * (lane & 7));
                    const int64_t at = o * S::N + c + 4 * (lane & 7);
                    const float k = P.a.av_per_nh;
                    if (P.a.n_h) *reinterpret_cast<float4 *>(P.a.n_h + at) = N;
                    if (P.a.a_v) *reinterpret_cast<float4 *>(P.a.a_v + at) = make_float4(N.x * k, N.y * k, N.z * k, N.w * k);
                }
            }
        }
        if (fault) break;
        if (P.a.shield && ok) {
            float4 *sh = reinterpret_cast<float4 *>(P.a.shield + oct * 8);
            const float n = (float)ND;
            sh[0] = make_float4(acc[0] / n, acc[1] / n, acc[2] / n, acc[3] / n);
            sh[1] = make_float4(acc[4] / n, acc[5] / n, acc[6] / n, acc[7] / n);
        }
        tc_fence_before();
    }
    if (i == 0) {
        if (fault) {
            atomicExch(&g_leaftc_fault, 1);
            mbar_wait_bounded(&bar[g], phase ^ 1, kMaxPolls);   // let an issued product finish
        }
        for (int b = 0; b < 2; ++b)
            if (pending[b]) mbar_wait_bounded(&bar[S::kGroups + 2 * g + b], sphase[b], kMaxPolls);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tslot, cols);
    }
}

int sms()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 152;
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }

template <int ND>
cd_status launch_leaf_oct(const LeafOctArgs &P, cudaStream_t s)
{
    using S = LeafOctShape<ND>;
    // as many groups a CTA as leave every SM one (a small tree's tiles go to more SMs)
    int G = S::kGroups;
    while (G > 1 && (P.ntiles + G - 1) / G < sms()) --G;
    const bool rows = P.a.n_h || P.a.a_v;
    auto kern = leaf_oct_tc<ND, false>;
    if constexpr (S::kParts == 1)
        if (rows) kern = leaf_oct_tc<ND, true>;
    const size_t smem = S::smem(G, rows);
    CD_ALLOW_SMEM(kern, smem, S::smem(S::kGroups, rows));
    const int64_t grid = std::min<int64_t>((P.ntiles + G - 1) / G, sms());
    LaunchScope ls(CD_K_LEAF, s, 2.0 * (double)P.ntiles * 128.0 * 16 * S::N);
    kern<<<(unsigned)grid, 128 * G, smem, s>>>(P);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

// poll limit of the pipeline waits (cd_debug_wait_polls)
uint32_t pipe_polls()
{
    const int64_t cap = g_pipe_polls.load();
    return cap < 0 ? kMaxPolls : (uint32_t)std::min<int64_t>(cap, kMaxPolls);
}

}  // namespace

// The tensor-core leaf kernel serves uniform trees with at least one full tile
// (128 leaves), n_dir a multiple of 4 up to 64, 16-byte aligned inputs.
cd_status launch_leaf_tc(const LeafLaunch &a, cudaStream_t s)
{
    const int nd = a.nd;
    const int64_t n_leaf = a.n_oct * 8;
    const bool list = a.oleaf != nullptr;
    if (nd % 4 != 0 || nd > 64 || !aligned16(a.E) || !aligned16(a.Sp) || !aligned16(a.rho_leaf) || !a.E)
        return CD_EUNSUPPORTED;
    if (!list && (n_leaf < 128 || n_leaf % 128 != 0)) return CD_EUNSUPPORTED;
    if (list && ((a.Sp && !a.oparent) || !aligned16(a.oleaf) || (a.n_h && !aligned16(a.n_h)))) return CD_EUNSUPPORTED;
    if (n_leaf == 0) return CD_OK;
    // 8 n_dir columns fit one product up to 32 directions; from 128 leaves to 256^3
    // the oct form is the faster one there (8.0 against 8.2 us at 16^3, 12.0 against
    // 14.5 at 64^3, 12 directions).  Beyond them it takes two products (of a
    // multiple of 32 columns each) and only calls that want the screening factor
    // alone (256^3, 48 directions: 0.249 against 0.456 ms); N_H rows are bound by
    // their stores, which tiles of 128 leaves send as bulk copies
    if (!list && (nd <= 32 || (nd % 8 == 0 && !a.n_h && !a.a_v)) && aligned16(a.n_h) && aligned16(a.a_v) && aligned16(a.shield)) {
        LeafOctArgs Q;
        Q.a = a;
        Q.ntiles = (a.n_oct + 127) / 128;
        Q.c2 = (float)(-(double)a.shield_k * (double)a.av_per_nh * 1.4426950408889634);
        Q.pipe_polls = pipe_polls();
        using Launch = cd_status (*)(const LeafOctArgs &, cudaStream_t);
        static constexpr Launch kLaunch[16] = {
            launch_leaf_oct<4>, launch_leaf_oct<8>, launch_leaf_oct<12>, launch_leaf_oct<16>, launch_leaf_oct<20>,
            launch_leaf_oct<24>, launch_leaf_oct<28>, launch_leaf_oct<32>, nullptr, launch_leaf_oct<40>,
            nullptr, launch_leaf_oct<48>, nullptr, launch_leaf_oct<56>, nullptr, launch_leaf_oct<64>};
        return kLaunch[nd / 4 - 1](Q, s);
    }
    LeafTcArgs P;
    P.a = a;
    P.list = list;
    P.NP = round16(nd);
    P.n_leaf = n_leaf;
    P.ntiles = (a.n_oct + 15) / 16;
    P.c2 = (float)(-(double)a.shield_k * (double)a.av_per_nh * 1.4426950408889634);
    // A_V alone leaves like N_H, in bulk copies of the staged rows (256^3, 48
    // directions: 0.61 ms; beside N_H it is written from them, 1.13 ms together;
    // both were 4-byte stores of a thread a row, 5.06 and 5.55 ms)
    const bool av_rows = a.a_v && !a.n_h && aligned16(a.a_v);
    if (av_rows) {
        P.a.n_h = a.a_v;
        P.a.a_v = nullptr;
    }
    P.out_bulk = P.a.n_h && aligned16(P.a.n_h);
    P.form = leaf_form(P.a, P.out_bulk, list) | (av_rows ? kFormAvRows : 0);
    P.pipe_polls = pipe_polls();
    P.span_max = g_span_max.load();
    int dev = 0, smax = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    P.G = leaf_tc_groups(nd, list, smax);
    const size_t smem = leaf_tc_smem(nd, P.NP, P.G, list).total;
    if ((int)smem > smax) return CD_EUNSUPPORTED;
    const auto kern = list ? leaf_tc<1> : leaf_tc<0>;
    constexpr size_t most[2] = {leaf_tc_smem_most(false), leaf_tc_smem_most(true)};
    CD_ALLOW_SMEM(kern, smem, most[list]);
    const int64_t grid = std::min<int64_t>((P.ntiles + P.G - 1) / P.G, sms());
    LaunchScope ls(CD_K_LEAF, s, 2.0 * (double)P.ntiles * 128.0 * kK * P.NP);
    kern<<<(unsigned)grid, 128 * P.G, smem, s>>>(P, LeafBatch{});
    CD_CHECK_LAUNCH();
    return CD_OK;
}

size_t leaf_tc_job_bytes() { return sizeof(LeafTcArgs); }

int64_t leaf_tc_job_fill(const LeafLaunch &a, void *dst)
{
    const int nd = a.nd;
    const int64_t n_leaf = a.n_oct * 8;
    const bool list = a.oleaf != nullptr;
    if (nd % 4 != 0 || nd > 64 || !aligned16(a.E) || !aligned16(a.Sp) || !aligned16(a.rho_leaf) || !a.E) return -1;
    if (!list && (n_leaf < 128 || n_leaf % 128 != 0)) return -1;
    if (list && (a.Sp || !aligned16(a.oleaf) || (a.n_h && !aligned16(a.n_h)))) return -1;
    LeafTcArgs P = {};
    P.a = a;
    P.list = list;
    P.NP = round16(nd);
    P.n_leaf = n_leaf;
    P.ntiles = (a.n_oct + 15) / 16;
    P.c2 = (float)(-(double)a.shield_k * (double)a.av_per_nh * 1.4426950408889634);
    P.out_bulk = a.n_h && aligned16(a.n_h);
    P.form = leaf_form(a, P.out_bulk, list);
    P.pipe_polls = kMaxPolls;
    memcpy(dst, &P, sizeof(P));
    return P.ntiles;
}

int leaf_tc_job_form(const void *job)
{
    LeafTcArgs P;
    memcpy(&P, job, sizeof(P));
    return P.form;
}

cd_status launch_leaf_tc_batch(const void *jobs, const int2 *tile_ref, int64_t total, int nd, const float *kloc,
                               int form, double flops, cudaStream_t s)
{
    if (total <= 0) return CD_OK;
    LeafTcArgs P = {};
    P.a.nd = nd;
    P.a.kloc = kloc;
    P.NP = round16(nd);
    P.form = form;
    P.list = (form & kFormList) != 0;
    P.out_bulk = (form & kFormBulk) != 0;
    P.pipe_polls = pipe_polls();
    int dev = 0, smax = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    P.G = leaf_tc_groups(nd, true, smax);
    const size_t smem = leaf_tc_smem(nd, P.NP, P.G, true).total;   // the kernel's layout (mode 2) has the list rows
    if ((int)smem > smax) {
        set_error("the batched leaf kernel needs %zu bytes of shared memory", smem);
        return CD_EUNSUPPORTED;
    }
    LeafBatch Bt;
    Bt.jobs = static_cast<const LeafTcArgs *>(jobs);
    Bt.tile_ref = tile_ref;
    Bt.total = total;
    constexpr size_t most = leaf_tc_smem_most(true);
    CD_ALLOW_SMEM(leaf_tc<2>, smem, most);
    const int64_t grid = std::min<int64_t>((total + P.G - 1) / P.G, sms());
    LaunchScope ls(CD_K_LEAF, s, flops);
    leaf_tc<2><<<(unsigned)grid, 128 * P.G, smem, s>>>(P, Bt);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

double leaf_tc_job_flops(const void *job)
{
    LeafTcArgs P;
    memcpy(&P, job, sizeof(P));
    return 2.0 * (double)P.ntiles * 128.0 * kK * P.NP;
}

void set_leaf_tc_wait_polls(int64_t polls) { g_pipe_polls.store(polls < 0 ? -1 : polls); }

void set_leaf_tc_span_max(int rows) { g_span_max.store(rows < 0 || rows > kSpanRows ? kSpanRows : rows); }

cd_status leaf_tc_fault_check()
{
    int v = 0;
    CD_CUDA(cudaMemcpyFromSymbol(&v, g_leaftc_fault, sizeof(int)));
    if (v) {
        const int zero = 0;
        CD_CUDA(cudaMemcpyToSymbol(g_leaftc_fault, &zero, sizeof(int)));
        set_error("a tensor-core leaf kernel gave up a bounded wait");
        return CD_ETIMEOUT;
    }
    return CD_OK;
}

}  // namespace cd
