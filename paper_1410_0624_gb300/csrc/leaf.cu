// Per-leaf combine and epilogue (§3.2 internal + local contributions; Eqs.
// eq_chi / chi_discret for the direction average):
//   N_H[t][d] = E[oct][d] + Sp[oct / 8][d] + sum_s rho_leaf[oct][s] dx_L Kloc[t][s][d]
//   A_V = N_H av_per_nh,   shield[t] = (1/nd) sum_d exp(-k A_V)
// This kernel writes the N_H array, the dominant HBM traffic of the path
// (4 bytes per cell-direction), so it is built as a streaming pipeline:
//
//   - persistent CTAs, each walking batches of B consecutive octs (Morton
//     order, so every batch is one contiguous span of E, rho and N_H);
//   - E, Sp and rho of the next batch arrive by bulk asynchronous copies (TMA,
//     cp.async.bulk) into a double-buffered shared-memory stage, completed on
//     an mbarrier, while the current batch is computed;
//   - every thread owns one fixed (child t, four directions) slot of the oct,
//     so its 8 x 4 local weights sit in registers for the whole kernel;
//   - results are staged in shared memory in output layout and leave by bulk
//     stores, so HBM sees full-line writes;
//   - the direction sum of the screening factor goes through a shared-memory
//     partial array (no atomics).
// Direction counts that are not a multiple of four and unaligned output pointers
// go to a kernel of one warp per child of 32 octs, or with very few or very many
// of them to a generic one-thread-per-leaf kernel.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace cd {
namespace {

constexpr uint32_t kMaxPolls = 1u << 26;   // bounded mbarrier waits (seconds at worst)

static __device__ int g_leaf_fault;         // set when a bounded wait gives up

constexpr int kLoadStages = 4;             // E / rho batches in flight per CTA

struct LeafTmaArgs {
    LeafLaunch a;
    int G;           // thread groups; one group = 2 nd threads = one oct at a time
    int B;           // octs per batch
    int prows;       // parent rows a batch can touch: B / 8 + 2
    int64_t nbatch;
    float c_exp2;    // base-2 exponent per unit N_H: -shield_k * av_per_nh * log2(e)
    float inv_nd;
};

// A leaf's screening partials, one per slot, in shared memory: from three on padded
// (with zeros) to an odd number of 16-byte words, so that a lane per leaf reads
// them 16 bytes at a time without bank conflicts.
__host__ __device__ constexpr int part_pitch(int nd) { return nd <= 8 ? nd / 4 : 4 * (((nd / 4 + 3) / 4) | 1); }

// shared memory of G groups: the input stages, the screening sums and partials, the
// rows of two batches if they are wanted
constexpr size_t leaf_tma_smem(int nd, int G, bool rows)
{
    const size_t B = 4 * (size_t)G, prows = B / 8 + 2;
    return 128 + sizeof(float) * (kLoadStages * (B * (nd + 8) + prows * nd) + 3 * B * 8 + 2 * B * 8 * part_pitch(nd) +
                                  (rows ? 2 * B * 8 * nd : 0));
}

constexpr int leaf_tma_groups(int nd) { return 384 / (2 * nd) > 1 ? 384 / (2 * nd) : 1; }

constexpr size_t leaf_tma_smem_most()
{
    size_t most = 0;
    for (int nd = 4; 2 * nd <= 384; nd += 4) {
        const size_t v = leaf_tma_smem(nd, leaf_tma_groups(nd), true);
        most = v > most ? v : most;
    }
    return most;
}

// Thread group g takes octs 4 g .. 4 g + 3 of a batch: siblings, so their
// parent's prefix is read once.  The screening partials of batch i are summed in a
// fixed order while batch i+1 is computed and their store trails the N_H store
// by one batch, so results are bitwise reproducible with one barrier per batch (it also
// says whether any thread gave up its wait for the batch's inputs).
// ND > 0 fixes the direction count at compile time (every offset folds to an
// immediate); ND = 0 reads it from the arguments.
// What bounds it: issue slots (the product's 32 FMA2 cycles of some 60 a unit), the
// barrier of a batch and the N_H stores.  256^3 FP32 with N_H: 48 directions 0.804 ->
// 0.653 ms (5.2 TB/s; the stores alone take 0.55), 40 directions 1.068 -> 0.668, 84
// 2.342 -> 1.373, 12 0.222 -> 0.180, with a load of the prefix for every oct, a check
// of every output in the loop, conflicts in the screening sums and a second barrier
// (one thread polled for the inputs: 0.696, 0.704, 1.553 and 0.192) before.
template <int ND>
__global__ void __launch_bounds__(384, 2) leaf_tma(LeafTmaArgs P)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kG = ND ? leaf_tma_groups(ND ? ND : 1) : 0;
    const int nd = ND ? ND : P.a.nd;
    const int G = ND ? kG : P.G;
    const int B = ND ? 4 * kG : P.B;
    const int prows = ND ? (4 * kG) / 8 + 2 : P.prows;
    const int q4 = nd >> 2, slots = 2 * nd, lp = part_pitch(nd);
    const bool want_nh = P.a.n_h != nullptr, want_sh = P.a.shield != nullptr;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    float *Eb = reinterpret_cast<float *>(smem + 128);      // [kLoadStages][B nd]
    float *Rb = Eb + kLoadStages * B * nd;                  // [kLoadStages][B 8]
    float *Pb = Rb + kLoadStages * B * 8;                   // [kLoadStages][(B/8 + 2) nd] parent rows
    float *Sb = Pb + kLoadStages * prows * nd;              // [3][B 8]
    float *part = Sb + 3 * B * 8;                           // [2][B 8][lp]
    float *Ob = part + 2 * B * 8 * lp;                      // [2][B 8 nd]

    const int tid = threadIdx.x;
    const int g = tid / slots, r = tid - g * slots;
    const int t = r / q4, d0 = 4 * (r - t * q4);
    // dx_L * Kloc[t][s][d0 + i] for sibling pairs j = (2j, 2j+1) and directions i
    float2 KP[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            KP[j][i] = make_float2(P.a.dx_leaf * P.a.kloc[(t * 8 + 2 * j) * nd + d0 + i],
                                   P.a.dx_leaf * P.a.kloc[(t * 8 + 2 * j + 1) * nd + d0 + i]);

    // this thread's offsets in the stages (oct 4 g of the batch, the next three follow)
    const bool has_E = P.a.E != nullptr, has_Sp = P.a.Sp != nullptr;
    const int b0 = 4 * g, eoff = b0 * nd + d0, roff = b0 * 8, ooff = (b0 * 8 + t) * nd + d0,
              poff = (b0 * 8 + t) * lp + (d0 >> 2);

    const int64_t n_oct = P.a.n_oct;
    const int64_t first = blockIdx.x, stride = gridDim.x;
    const int n_iter = first < P.nbatch ? (int)((P.nbatch - first + stride - 1) / stride) : 0;
    auto batch_o0 = [&](int it) { return (first + (int64_t)it * stride) * B; };
    auto batch_nb = [&](int it) {
        const int64_t o0 = batch_o0(it);
        return (int)(n_oct - o0 < (int64_t)B ? n_oct - o0 : (int64_t)B);
    };

    auto issue = [&](int it) {
        const int st = it % kLoadStages;
        const int64_t o0 = batch_o0(it);
        const int nb = batch_nb(it);
        const uint32_t eb = P.a.E ? (uint32_t)nb * nd * 4 : 0u;
        const int64_t p0 = o0 >> 3;
        const uint32_t pb = P.a.Sp ? (uint32_t)(((o0 + nb - 1) >> 3) - p0 + 1) * nd * 4 : 0u;
        // checked builds: a batch outside the octs (or their parents) copies nothing
        if (!(in_bounds(o0, n_oct, kCheckLeafIn) && in_bounds(o0 + nb - 1, n_oct, kCheckLeafIn) &&
              (!P.a.Sp || in_bounds((o0 + nb - 1) >> 3, (n_oct + 7) / 8, kCheckLeafIn)))) {
            mbar_expect_tx(&bar[st], 0);
            return;
        }
        mbar_expect_tx(&bar[st], eb + pb + (uint32_t)nb * 32);
        if (P.a.E) bulk_g2s(Eb + st * B * nd, P.a.E + o0 * nd, eb, &bar[st]);
        if (P.a.Sp) bulk_g2s(Pb + st * prows * nd, P.a.Sp + p0 * nd, pb, &bar[st]);
        bulk_g2s(Rb + st * B * 8, P.a.rho_leaf + o0 * 8, (uint32_t)nb * 32, &bar[st]);
    };
    // screening factor of batch `it` from its partials, in a fixed order
    auto shield_sum = [&](int it) {
        const float *pp = part + (it & 1) * B * 8 * lp;
        float *S = Sb + (it % 3) * B * 8;
        for (int j = tid; j < B * 8; j += blockDim.x) {
            if (nd <= 8) {
                S[j] = (nd == 4 ? pp[j] : pp[2 * j] + pp[2 * j + 1]) * P.inv_nd;
                continue;
            }
            float2 acc = make_float2(0.f, 0.f);
            for (int q = 0; q < lp; q += 4) {
                const float4 p = *reinterpret_cast<const float4 *>(pp + j * lp + q);
                acc = __fadd2_rn(acc, __fadd2_rn(make_float2(p.x, p.y), make_float2(p.z, p.w)));
            }
            S[j] = (acc.x + acc.y) * P.inv_nd;
        }
    };
    for (int j = tid; j < 2 * B * 8; j += blockDim.x)
        for (int q = q4; q < lp; ++q) part[j * lp + q] = 0.f;

    if (tid == 0) {
        for (int s = 0; s < kLoadStages; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
        for (int it = 0; it < kLoadStages - 1 && it < n_iter; ++it) issue(it);
    }
    __syncthreads();

    int it = 0;
    bool fault = false;
    for (; it < n_iter; ++it) {
        const int ls = it % kLoadStages, os = it & 1;
        // the stage of batch it - 1 is free: every thread has passed its barrier
        if (tid == 0 && it + kLoadStages - 1 < n_iter) issue(it + kLoadStages - 1);
        const bool ok = mbar_wait_bounded(&bar[ls], (it / kLoadStages) & 1, kMaxPolls);
        if (want_sh && it > 0) shield_sum(it - 1);

        const int64_t o0 = batch_o0(it);
        const int nb = batch_nb(it);
        const float *E = Eb + ls * B * nd + eoff;
        const float *R = Rb + ls * B * 8 + roff;
        float *O = Ob + os * B * 8 * nd + ooff;
        float *pp = part + (it & 1) * B * 8 * lp + poff;
        float *AV = P.a.a_v ? P.a.a_v + o0 * 8 * nd + ooff : nullptr;
        float2 s01 = make_float2(0.f, 0.f), s23 = s01;
        if (has_Sp) {   // octs o0 + 4 g .. have one parent (o0 is a multiple of 4)
            const float4 p4 = *reinterpret_cast<const float4 *>(
                Pb + ls * prows * nd + (((int)(o0 & 7) + b0) >> 3) * nd + d0);
            s01 = make_float2(p4.x, p4.y);
            s23 = make_float2(p4.z, p4.w);
        }
        // all: a whole batch with E, Sp and the screening factor, without A_V (the
        // checks of the other forms cost a seventh); rows: N_H is wanted
        const auto octs = [&](auto all, auto rows) {
            constexpr bool kAll = decltype(all)::value;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (!kAll && b0 + k >= nb) break;
                float2 n01 = make_float2(0.f, 0.f), n23 = n01;
                if (kAll || has_E) {
                    const float4 e4 = *reinterpret_cast<const float4 *>(E + k * nd);
                    n01 = make_float2(e4.x, e4.y);
                    n23 = make_float2(e4.z, e4.w);
                }
                if (kAll || has_Sp) {
                    n01 = __fadd2_rn(n01, s01);
                    n23 = __fadd2_rn(n23, s23);
                }
                const float4 r0 = *reinterpret_cast<const float4 *>(R + k * 8);
                const float4 r1 = *reinterpret_cast<const float4 *>(R + k * 8 + 4);
                // packed FP32x2 FMAs over sibling pairs (s, s+1): acc[i] holds the
                // even- and odd-sibling partial sums of direction d0 + i
                const float2 rp[4] = {make_float2(r0.x, r0.y), make_float2(r0.z, r0.w), make_float2(r1.x, r1.y),
                                      make_float2(r1.z, r1.w)};
                float2 acc[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[i] = __fmul2_rn(rp[0], KP[0][i]);
#pragma unroll
                    for (int j = 1; j < 4; ++j) acc[i] = __ffma2_rn(rp[j], KP[j][i], acc[i]);
                }
                n01.x += acc[0].x + acc[0].y;
                n01.y += acc[1].x + acc[1].y;
                n23.x += acc[2].x + acc[2].y;
                n23.y += acc[3].x + acc[3].y;
                if (rows)
                    *reinterpret_cast<float4 *>(O + k * 8 * nd) = make_float4(n01.x, n01.y, n23.x, n23.y);
                if (!kAll && AV) {
                    const float2 a2 = make_float2(P.a.av_per_nh, P.a.av_per_nh);
                    const float2 x = __fmul2_rn(n01, a2), y = __fmul2_rn(n23, a2);
                    *reinterpret_cast<float4 *>(AV + k * 8 * nd) = make_float4(x.x, x.y, y.x, y.y);
                }
                if (kAll || want_sh) {
                    // exp(-k A_V) = 2^(c2 N_H), c2 = -k av log2(e) precomputed on the host
                    const float2 c2 = make_float2(P.c_exp2, P.c_exp2);
                    const float2 a = __fmul2_rn(c2, n01), b = __fmul2_rn(c2, n23);
                    pp[k * 8 * lp] = (exp2f(a.x) + exp2f(a.y)) + (exp2f(b.x) + exp2f(b.y));
                }
            }
        };
        // (a third copy of the loop pays with runtime offsets alone: 40 directions
        // of 256^3 0.706 against 0.759 ms, 48 at compile time 0.709 against 0.686, both
        // with a second barrier)
        if (nb != B || !has_E || !has_Sp || !want_sh || AV) octs(std::false_type{}, want_nh);
        else if (ND) octs(std::true_type{}, want_nh);
        else if (want_nh) octs(std::true_type{}, std::true_type{});
        else octs(std::true_type{}, std::false_type{});
        if (tid == 0) bulk_wait_read<0>();   // the last batch's stores have read O[os ^ 1] and their S
        fence_proxy_async_smem();
        if (__syncthreads_or(!ok)) {
            fault = true;
            break;
        }
        if (tid == 0) {
            if (want_nh) bulk_s2g(P.a.n_h + o0 * 8 * nd, Ob + os * B * 8 * nd, (uint32_t)nb * 32 * nd);
            if (want_sh && it > 0)
                bulk_s2g(P.a.shield + batch_o0(it - 1) * 8, Sb + ((it - 1) % 3) * B * 8, (uint32_t)batch_nb(it - 1) * 32);
            bulk_commit();
        }
    }
    if (!fault && want_sh && n_iter > 0) {
        // the last batch's screening factor
        if (tid == 0) bulk_wait_read<1>();
        __syncthreads();
        shield_sum(n_iter - 1);
        fence_proxy_async_smem();
        __syncthreads();
        if (tid == 0) {
            bulk_s2g(P.a.shield + batch_o0(n_iter - 1) * 8, Sb + ((n_iter - 1) % 3) * B * 8,
                     (uint32_t)batch_nb(n_iter - 1) * 32);
            bulk_commit();
        }
    }
    if (tid == 0) {
        if (fault) {
            atomicExch(&g_leaf_fault, 1);
            // let the loads already issued land before shared memory is released
            for (int j = it; j < it + kLoadStages && j < n_iter; ++j)
                mbar_wait_bounded(&bar[j % kLoadStages], (j / kLoadStages) & 1, kMaxPolls);
        }
        bulk_wait_all<0>();
    }
}

// One thread per leaf; any direction count and alignment.
__global__ void __launch_bounds__(256) leaf_generic(LeafLaunch P, float c_exp, float inv_nd)
{
    extern __shared__ float s_k[];   // [8 s][nd][8 t], times dx
    const int nd = P.nd;
    for (int i = threadIdx.x; i < 64 * nd; i += blockDim.x) {
        const int t = i & 7, sd = i >> 3, s = sd / nd, d = sd - s * nd;
        s_k[i] = P.dx_leaf * P.kloc[(t * 8 + s) * nd + d];
    }
    __syncthreads();
    const int64_t n_leaf = P.n_oct * 8;
    for (int64_t leaf = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; leaf < n_leaf;
         leaf += (int64_t)gridDim.x * blockDim.x) {
        const int64_t oct = leaf >> 3;
        const int t = (int)(leaf & 7);
        float rs[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) rs[s] = P.rho_leaf[oct * 8 + s];
        float acc = 0.f;
        for (int d = 0; d < nd; ++d) {
            float n = P.E ? P.E[oct * nd + d] : 0.f;
            if (P.Sp) n += P.Sp[(oct >> 3) * nd + d];
#pragma unroll
            for (int s = 0; s < 8; ++s) n = fmaf(rs[s], s_k[(s * nd + d) * 8 + t], n);
            if (P.n_h) P.n_h[leaf * nd + d] = n;
            if (P.a_v) P.a_v[leaf * nd + d] = n * P.av_per_nh;
            acc += __expf(c_exp * n);
        }
        if (P.shield) P.shield[leaf] = acc * inv_nd;
    }
}

// Direction counts that are not a multiple of four, and unaligned outputs: a
// CTA takes 32 octs, a warp one of their children and a lane one oct, which
// walks the directions.  The local weights are then the same for a warp (two
// 16-byte broadcasts for eight FMAs), the oct's densities stay in registers, the
// external columns E + Sp come from shared memory (odd pitch: no bank
// conflicts), and 32 directions of the 32 octs at a time turn into coalesced row
// pieces through a padded square.
// What bounds it: shared memory, about eight wavefronts per 32 outputs.  An FP32
// evaluation of 256^3 at 35 directions took 6.20 ms with a thread a leaf (32 rows
// a store) and takes 1.83, at 81 directions 14.6 and 4.7, of 64^3 at 9
// directions 32 and 25 us.
constexpr int kOctWarps = 8;   // one per child
constexpr size_t kOctSmemMost = 200 * 1024;

__host__ __device__ constexpr int oct_pitch(int nd) { return nd | 1; }

size_t leaf_oct_smem(int nd, bool rows)
{
    return sizeof(float) * (64 * (size_t)nd + (size_t)32 * oct_pitch(nd) + (rows ? kOctWarps * 32 * 33 : 0));
}

template <bool kRows>
__global__ void __launch_bounds__(32 * kOctWarps) leaf_oct_fp32(LeafLaunch P, float c_exp, float inv_nd)
{
    extern __shared__ __align__(16) float sm[];
    const int nd = P.nd, pitch = oct_pitch(nd);
    const int t = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *sK = sm;                                                        // [8 t][nd][8 s], times dx
    float *sE = sK + 64 * nd;                                              // [32 octs][pitch]
    float *T = sE + 32 * pitch + t * 32 * 33;                              // [32 octs][33]
    for (int i = threadIdx.x; i < 64 * nd; i += blockDim.x) {
        const int d = i % nd, ts = i / nd;                                 // kloc[t][s][d]
        sK[((ts >> 3) * nd + d) * 8 + (ts & 7)] = P.dx_leaf * P.kloc[i];
    }
    const int64_t tiles = (P.n_oct + 31) / 32;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t o0 = tile * 32, oct = o0 + lane;
        const int nb = (int)(P.n_oct - o0 < 32 ? P.n_oct - o0 : 32);
        if (!in_bounds(o0 + nb - 1, P.n_oct, kCheckLeafIn)) break;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 r0 = lane < nb ? *reinterpret_cast<const float4 *>(P.rho_leaf + oct * 8) : z;
        const float4 r1 = lane < nb ? *reinterpret_cast<const float4 *>(P.rho_leaf + oct * 8 + 4) : z;
        for (int i = threadIdx.x; i < nb * nd; i += blockDim.x) {
            const int o = i / nd, d = i - o * nd;
            float e = P.E ? P.E[o0 * nd + i] : 0.f;
            if (P.Sp) e += P.Sp[((o0 + o) >> 3) * nd + d];
            sE[o * pitch + d] = e;
        }
        __syncthreads();
        const float *E = sE + lane * pitch, *K = sK + t * nd * 8;
        float acc = 0.f;
        for (int d0 = 0; d0 < nd; d0 += 32) {
            const int w = min(32, nd - d0);
#pragma unroll 4
            for (int j = 0; j < w; ++j) {
                const float4 k0 = *reinterpret_cast<const float4 *>(K + (d0 + j) * 8),
                             k1 = *reinterpret_cast<const float4 *>(K + (d0 + j) * 8 + 4);
                float v = E[d0 + j];
                v = fmaf(r0.x, k0.x, v);
                v = fmaf(r0.y, k0.y, v);
                v = fmaf(r0.z, k0.z, v);
                v = fmaf(r0.w, k0.w, v);
                v = fmaf(r1.x, k1.x, v);
                v = fmaf(r1.y, k1.y, v);
                v = fmaf(r1.z, k1.z, v);
                v = fmaf(r1.w, k1.w, v);
                if (kRows) T[lane * 33 + j] = v;
                acc += __expf(c_exp * v);
            }
            if (!kRows) continue;
            __syncwarp();
            if (lane < w) {
                const int64_t at = (o0 * 8 + t) * nd + d0 + lane;
                if (P.n_h) {
                    float *out = P.n_h + at;
#pragma unroll 8
                    for (int o = 0; o < nb; ++o) out[(int64_t)o * 8 * nd] = T[o * 33 + lane];
                }
                if (P.a_v) {
                    float *out = P.a_v + at;
#pragma unroll 8
                    for (int o = 0; o < nb; ++o) out[(int64_t)o * 8 * nd] = T[o * 33 + lane] * P.av_per_nh;
                }
            }
            __syncwarp();
        }
        if (P.shield && lane < nb) P.shield[oct * 8 + t] = acc * inv_nd;
        __syncthreads();   // every warp is done with the external columns
    }
}

struct DevInfo {
    int sms = 0;
};
std::mutex g_mu;
DevInfo g_dev[64];

int sm_count()
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 152;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_dev[dev].sms) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        g_dev[dev].sms = n > 0 ? n : 152;
    }
    return g_dev[dev].sms;
}

bool aligned16(const void *p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

cd_status launch_leaf(const LeafLaunch &a, cudaStream_t s)
{
    const int nd = a.nd;
    const float c_exp = -a.shield_k * a.av_per_nh;
    const float inv_nd = 1.0f / (float)nd;
    const bool tma = (nd % 4 == 0) && 2 * nd <= 384 && aligned16(a.n_h) && aligned16(a.a_v) &&
                     aligned16(a.shield) && aligned16(a.E) && aligned16(a.Sp) && aligned16(a.rho_leaf);
    if (tma) {
        auto kern = nd == 48 ? leaf_tma<48> : nd == 12 ? leaf_tma<12> : leaf_tma<0>;
        LeafTmaArgs P;
        P.a = a;
        P.G = leaf_tma_groups(nd);
        // small trees: smaller batches, so that every SM gets one (16^3, 48 directions,
        // the whole evaluation as a graph 16.4 -> 14.4 us, 12 directions the same)
        while (P.G > 1 && P.G * nd >= 96 && a.n_oct < (int64_t)4 * P.G * sm_count()) {
            P.G /= 2;
            kern = leaf_tma<0>;
        }
        P.B = 4 * P.G;
        P.prows = P.B / 8 + 2;
        P.nbatch = (a.n_oct + P.B - 1) / P.B;
        P.c_exp2 = (float)(-(double)a.shield_k * (double)a.av_per_nh * 1.4426950408889634);
        P.inv_nd = inv_nd;
        const int threads = P.G * 2 * nd;
        const size_t smem = leaf_tma_smem(nd, P.G, a.n_h != nullptr);
        constexpr size_t most = leaf_tma_smem_most();
        CD_ALLOW_SMEM(kern, smem, most);
        int per_sm = 1;
        if (P.nbatch > sm_count()) CD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
        if (per_sm < 1) per_sm = 1;
        const int64_t grid = std::min<int64_t>(P.nbatch, (int64_t)per_sm * sm_count());
        LaunchScope ls(CD_K_LEAF, s);
        kern<<<(unsigned)grid, threads, smem, s>>>(P);
        CD_CHECK_LAUNCH();
        return CD_OK;
    }
    const bool rows = a.n_h || a.a_v;
    // hardly any directions leave a warp too little to do per tile: up to 4 at any
    // size (256^3 at 3 directions 0.39 against 0.26 ms), 5 where N_H or A_V is written (128^3
    // 41 against 35 us; both 60 against 61, the screening factor alone 23 against 25; 6
    // directions with N_H 43 against 47).  Below 32^3 a tile is a CTA's only one: rows
    // of up to 8 directions (16^3 at 6: 12.3 against 10.4 us) and the screening factor
    // alone of up to 31 (8^3 at 10: 6.6 against 6.2 us, 15: 7.6 against 6.9, 16^3 at 27:
    // 8.8 against 8.2)
    const bool tiny = a.n_oct < 4096;
    const bool one = (a.n_h != nullptr) != (a.a_v != nullptr);
    const int least = tiny ? (rows ? 9 : 32) : one ? 6 : 5;
    if (nd >= least && leaf_oct_smem(nd, rows) <= kOctSmemMost && aligned16(a.rho_leaf)) {
        const auto kern = rows ? leaf_oct_fp32<true> : leaf_oct_fp32<false>;
        const size_t smem = leaf_oct_smem(nd, rows);
        CD_ALLOW_SMEM(kern, smem, kOctSmemMost);
        int per_sm = 0;
        CD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kOctWarps, smem));
        const int64_t grid = std::min<int64_t>((a.n_oct + 31) / 32, (int64_t)sm_count() * std::max(1, per_sm));
        LaunchScope ls(CD_K_LEAF, s);
        kern<<<(unsigned)std::max<int64_t>(grid, 1), 32 * kOctWarps, smem, s>>>(a, c_exp, inv_nd);
        CD_CHECK_LAUNCH();
        return CD_OK;
    }
    const size_t smem = sizeof(float) * 64 * nd;
    CD_ALLOW_SMEM(leaf_generic, smem, sizeof(float) * 64 * CD_MAXDIR);
    int64_t blocks = (a.n_oct * 8 + 255) / 256;
    blocks = std::min<int64_t>(blocks, (int64_t)sm_count() * 8);
    LaunchScope ls(CD_K_LEAF, s);
    leaf_generic<<<(unsigned)std::max<int64_t>(blocks, 1), 256, smem, s>>>(a, c_exp, inv_nd);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

// Returns CD_ETIMEOUT (and clears the flag) if a leaf kernel gave up a wait.
cd_status leaf_fault_check()
{
    int v = 0;
    CD_CUDA(cudaMemcpyFromSymbol(&v, g_leaf_fault, sizeof(int)));
    if (v) {
        const int zero = 0;
        CD_CUDA(cudaMemcpyToSymbol(g_leaf_fault, &zero, sizeof(int)));
        set_error("a leaf kernel gave up waiting for its input copies");
        return CD_ETIMEOUT;
    }
    return CD_OK;
}

}  // namespace cd
