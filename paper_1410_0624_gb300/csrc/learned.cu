// The learned correction (include/colden_learned.h): the tree method's terms
// level by level, the exact ray-marcher that gives the training targets, the
// combine N = N_tree exp(delta), the network handle and the FP32 learned form
// of cd_column_density.
//
// Per-level terms.  The plain evaluation folds the far shells into prefix
// sums; here every shell stays apart.  For a uniform tree with leaves at level
// L (octs at L-1) the shell Delta_l = L - l of leaf m comes from
//   Delta_l = 1, 2, 3:  Et[Delta_l][m >> 3]    (oct level, table Delta_l alone)
//   Delta_l >= 4:       C[k][m >> 3 (L - k)]   with k = L - Delta_l + 2
// (C[k] = shell of level k - 2 seen from the centre of the level-k ancestor,
// table 3, §3.3), and Delta_l = 0 is the internal + local term of §3.2.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "learned.cuh"

namespace cd {
namespace {

constexpr int kThreads = 256;
constexpr int64_t kChunkRows = 1 << 20;   // leaves per chunk of the FP32 learned path

float dx_of(const cd_tree t, int l) { return (float)(t->box_cm / (double)((int64_t)1 << l)); }

int grid_for(int64_t n, int threads)
{
    const int64_t b = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 32));
}

struct FeatArgs {
    int64_t n, first, n_leaf;
    const int64_t *leaves;
    int L, nd;
    float dx_leaf;
    const float *rho_leaf;          // Morton
    const float *kloc;              // [8][8][nd], units of dx
    const float *Et[4];             // [n_oct][nd] or NULL
    const float *C[CD_MAXL + 1];    // [8^k][nd] or NULL
    float *x;                       // [n][8 nd + 1]
    float *n_tree;                  // [n][nd] or NULL
};

// One thread per (row, direction).
__global__ void __launch_bounds__(kThreads) learned_features(FeatArgs A)
{
    const int nd = A.nd, n_in = kSlots * nd + 1;
    const int64_t total = A.n * nd;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / nd;
        const int d = (int)(e - r * nd);
        const int64_t m = A.leaves ? A.leaves[r] : A.first + r;
        float *xr = A.x + r * n_in;
        if (m < 0 || m >= A.n_leaf) {
            for (int sl = 0; sl < kSlots; ++sl) xr[sl * nd + d] = 0.f;
            if (d == 0) xr[kSlots * nd] = 0.f;
            if (A.n_tree) A.n_tree[r * nd + d] = 0.f;
            continue;
        }
        const int t = (int)(m & 7);
        const int64_t oct = m >> 3;
        float c[kSlots];
        // Delta_l = 0: internal + local (§3.2)
        float loc = 0.f;
        for (int sib = 0; sib < 8; ++sib)
            loc = fmaf(A.rho_leaf[oct * 8 + sib], A.kloc[(t * 8 + sib) * nd + d], loc);
        c[0] = A.dx_leaf * loc;
        for (int sl = 1; sl < kSlots; ++sl) c[sl] = 0.f;
#pragma unroll
        for (int dl = 1; dl < CD_MAXL; ++dl) {      // dl constant after unrolling
            if (dl > A.L - 1) break;
            const float v = dl <= 3 ? A.Et[dl][oct * nd + d] : A.C[A.L - dl + 2][(m >> (3 * (dl - 2))) * nd + d];
            c[dl < kSlots ? dl : kSlots - 1] += v;
        }
        float tot = 0.f;
        for (int sl = 0; sl < kSlots; ++sl) {
            tot += c[sl];
            xr[sl * nd + d] = logf(fmaxf(c[sl], kCFloor));
        }
        if (d == 0) xr[kSlots * nd] = logf(fmaxf(A.rho_leaf[m], kNFloor));
        if (A.n_tree) A.n_tree[r * nd + d] = tot;
    }
}

// Inputs of the FP32 learned columns for a run of octs: the external slots once
// per oct, slot 0 and the density per leaf, standardised (mlp.cu,
// mlp_forward_octs), and the plain columns.  One thread per (oct, direction).
struct OctFeatArgs {
    int64_t first, n;               // octs
    int L, nd;
    float dx_leaf;
    const float *rho_leaf;
    const float *kloc;
    const float *Et[4];
    const float *C[CD_MAXL + 1];
    const float *mu, *sinv;         // [8 nd + 1]
    float *ue, *ul, *n_tree;        // [n][7 nd], [8 n][nd + 1], [8 n][nd]
};

__device__ __forceinline__ float standardised_log(float v, float floor, float mu, float sinv)
{
    return fminf(fmaxf((logf(fmaxf(v, floor)) - mu) * sinv, -kUMax), kUMax);
}

__global__ void __launch_bounds__(kThreads) oct_features(const __grid_constant__ OctFeatArgs A)
{
    const int nd = A.nd;
    const int64_t total = A.n * nd;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / nd, oct = A.first + i;
        const int d = (int)(e - i * nd);
        float c[kSlots];
#pragma unroll
        for (int sl = 0; sl < kSlots; ++sl) c[sl] = 0.f;
#pragma unroll
        for (int dl = 1; dl < CD_MAXL; ++dl) {      // dl constant after unrolling
            if (dl > A.L - 1) break;
            const float v = dl <= 3 ? A.Et[dl][oct * nd + d] : A.C[A.L - dl + 2][(oct >> (3 * (dl - 3))) * nd + d];
            c[dl < kSlots ? dl : kSlots - 1] += v;
        }
        float ext = 0.f;
        float *ue = A.ue + i * (kSlots - 1) * nd + d;
#pragma unroll
        for (int sl = 1; sl < kSlots; ++sl) {
            ext += c[sl];
            ue[(sl - 1) * nd] = standardised_log(c[sl], kCFloor, A.mu[sl * nd + d], A.sinv[sl * nd + d]);
        }
        float rho[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) rho[q] = A.rho_leaf[oct * 8 + q];
        const float mu = A.mu[d], sinv = A.sinv[d];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            float loc = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) loc = fmaf(rho[q], A.kloc[(t * 8 + q) * nd + d], loc);
            const float c0 = A.dx_leaf * loc;
            const int64_t row = 8 * i + t;
            A.n_tree[row * nd + d] = c0 + ext;
            A.ul[row * (nd + 1) + d] = standardised_log(c0, kCFloor, mu, sinv);
            if (d == 0)
                A.ul[row * (nd + 1) + nd] = standardised_log(rho[t], kNFloor, A.mu[kSlots * nd], A.sinv[kSlots * nd]);
        }
    }
}

struct MarchArgs {
    int64_t n, n_leaf;
    const int64_t *leaves;    // [n] leaf of each row, or NULL: row r is leaf r
    const uint2 *order;       // [n] {row, leaf (kNoLeaf: out of range)} in spatial order, or NULL
    int L, nd;
    int rows_per_thread;      // a CTA marches 256 x this many rows in one direction
    int64_t items;            // (row chunk, direction) pairs
    float dx_leaf;
    const float *rho_leaf;    // Morton
    const double *dirs;       // [nd][3]
    float *out;               // [n][nd]
};

constexpr uint32_t kDil = 0x09249249u;     // bits of the x coordinate in a Morton code (10 per axis)
constexpr uint32_t kNoLeaf = 0xffffffffu;

// One cell of a direction's path: the ray's length in it (cell units) and the
// step to the next cell, a dilated-integer add on the axis `mask`.
struct __align__(16) MarchStep {
    float len;
    uint32_t mask, add;
    float t;                  // exit distance (len is the difference of two)
};

constexpr int kMarchMaxLevel = 10;         // of a uniform tree
constexpr size_t march_smem(int L) { return ((size_t)3 << L) * (sizeof(MarchStep) + sizeof(uint16_t)); }

// Exact column from the leaf centre to the box edge: Amanatides-Woo DDA over
// the leaf grid in cell units.
//
// All rays of one direction start at cell centres of one grid, so they cross
// the same sequence of faces at the same distances (j + 1/2) / |u_a| and differ
// only in where they leave the box.  A CTA takes one direction and a chunk of
// rows: it builds the sequence once in shared memory (each crossing finds its
// place by counting the earlier crossings of the other two axes; ties go to
// the lower axis, and each distance is computed afresh, so no error
// accumulates), and each ray then walks it with a uniform loop of one table
// read, one density load, one FMA and three integer instructions.  The length
// of a ray's walk is known beforehand: the place of the crossing that leaves
// the box, the first of the three axes'.
//
// What bounds it: the density loads, one 4-byte gather per cell crossed.  With
// the rows in spatial order (march_scatter) a warp's 32 cells move through the
// box as one small block that falls into few lines, and its rays end together.
// 262 144 random leaves of 128^3, 48 directions (1.2e9 cells): 1.09 ms, 2.41
// with the rows as listed, 9.39 with a DDA of its own per (row, direction).
__global__ void __launch_bounds__(kThreads) raymarch(MarchArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = 1 << A.L;
    MarchStep *path = reinterpret_cast<MarchStep *>(smem);                 // [3 n]
    uint16_t *place = reinterpret_cast<uint16_t *>(path + 3 * n);          // [3][n] place of crossing j of axis a
    const int tid = threadIdx.x;
    const int64_t chunk_rows = (int64_t)kThreads * A.rows_per_thread;
    for (int64_t item = blockIdx.x; item < A.items; item += gridDim.x) {
        const int64_t chunk = item / A.nd;
        const int d = (int)(item - chunk * A.nd);
        float ad[3], inv[3];
        bool fwd[3];
        float t_end = INFINITY;             // no ray goes on beyond its first axis' last crossing
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float u = (float)A.dirs[3 * d + a];
            fwd[a] = u > 0.f;
            ad[a] = fabsf(u);
            inv[a] = u != 0.f ? fabsf(1.f / u) : 0.f;
            if (u != 0.f) t_end = fminf(t_end, ((float)n - 0.5f) * inv[a]);
        }
        __syncthreads();                    // the previous item's rays are done with the path
        for (int e = tid; e < 3 * n; e += kThreads) {
            const int a = e >> A.L, j = e & (n - 1);
            const float iv = a == 0 ? inv[0] : a == 1 ? inv[1] : inv[2];
            const float t = ((float)j + 0.5f) * iv;
            int pos = 0xffff;
            if (iv != 0.f && t <= t_end) {
                pos = j;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    if (b == a || inv[b] == 0.f) continue;
                    // crossings of axis b before this one
                    int k = (int)fminf(t * ad[b] + 0.5f, (float)n);
                    const auto before = [&](int i) {
                        const float tb = ((float)i + 0.5f) * inv[b];
                        return tb < t || (tb == t && b < a);
                    };
                    while (k > 0 && !before(k - 1)) --k;
                    while (k < n && before(k)) ++k;
                    pos += k;
                }
                const uint32_t mask = kDil << a;
                const bool f = a == 0 ? fwd[0] : a == 1 ? fwd[1] : fwd[2];
                path[pos].t = t;
                path[pos].mask = mask;
                path[pos].add = f ? 1u << a : mask;   // + 1, or - 1 (all bits) in dilated arithmetic
            }
            place[e] = (uint16_t)pos;
        }
        __syncthreads();
        for (int e = tid; e < 3 * n; e += kThreads) {
            const int pos = place[e];
            if (pos != 0xffff) path[pos].len = path[pos].t - (pos ? path[pos - 1].t : 0.f);
        }
        __syncthreads();
        for (int rr = 0; rr < A.rows_per_thread; ++rr) {
            const int64_t i = chunk * chunk_rows + rr * kThreads + tid;
            int64_t r = i;
            uint32_t m = kNoLeaf;
            if (i < A.n) {
                if (A.order) {
                    const uint2 o = A.order[i];
                    r = o.x;
                    m = o.y;
                } else {
                    const int64_t l = A.leaves ? A.leaves[i] : i;
                    if (l >= 0 && l < A.n_leaf) m = (uint32_t)l;
                }
            }
            int steps = 0;
            if (m != kNoLeaf) {
                steps = 0xffff;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int c = (int)compact3((uint64_t)(m >> a));
                    if (inv[a] != 0.f) steps = min(steps, (int)place[a * n + (fwd[a] ? n - 1 - c : c)]);
                }
                ++steps;
            }
            const int warp_steps = __reduce_max_sync(0xffffffffu, steps);
            float sum = 0.f;
            int s = 0;
            for (; s + 4 <= warp_steps; s += 4) {
                float v[4];
                float len[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const MarchStep p = path[s + q];
                    len[q] = p.len;
                    v[q] = s + q < steps ? __ldg(A.rho_leaf + m) : 0.f;
                    m = (((m | ~p.mask) + p.add) & p.mask) | (m & ~p.mask);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) sum = fmaf(v[q], len[q], sum);
            }
            for (; s < warp_steps; ++s) {
                const MarchStep p = path[s];
                sum = fmaf(s < steps ? __ldg(A.rho_leaf + m) : 0.f, p.len, sum);
                m = (((m | ~p.mask) + p.add) & p.mask) | (m & ~p.mask);
            }
            if (i < A.n) A.out[r * A.nd + d] = sum * A.dx_leaf;
        }
    }
}

// Spatial order of a list of leaves: a counting sort by the leading Morton bits
// (about 16 rows a bucket, at most 2^15 buckets; the order within a bucket does
// not matter, each row's column is its own).  The rows of a warp that share a
// bucket add to it as one: lists sorted already, or of few distinct leaves,
// would queue 32 atomics on one word (1 000 000 rows of 32^3, 12 directions, march
// included: one leaf 1.49 -> 0.25 ms, eight 0.45 -> 0.20, random ones 0.22 either way).
constexpr int kMarchBits = 15;

__device__ __forceinline__ uint32_t march_bucket(int64_t leaf, int64_t n_leaf, int shift)
{
    return leaf >= 0 && leaf < n_leaf ? (uint32_t)(leaf >> shift) : 0u;
}

// Whole warps walk the rows; lanes past the end share a bucket of their own.
// same: the lanes of this lane's bucket; lead: it adds for them
__device__ __forceinline__ bool march_peers(bool live, uint32_t bucket, uint32_t &same)
{
    same = __match_any_sync(0xffffffffu, live ? bucket : 0xffffffffu);
    return live && (int)(threadIdx.x & 31) == __ffs(same) - 1;
}

__global__ void __launch_bounds__(kThreads) march_count(int64_t n, const int64_t *__restrict__ leaves, int64_t n_leaf,
                                                        int shift, uint32_t *__restrict__ count)
{
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = blockIdx.x * (int64_t)kThreads + threadIdx.x - lane; i0 < n; i0 += (int64_t)gridDim.x * kThreads) {
        const bool live = i0 + lane < n;
        const uint32_t b = live ? march_bucket(leaves[i0 + lane], n_leaf, shift) : 0u;
        uint32_t same;
        if (march_peers(live, b, same)) atomicAdd(&count[b], (uint32_t)__popc(same));
    }
}

// counts -> first place of each bucket: one CTA of 1024 threads walks the
// counts in coalesced runs of 4096 (buckets is a multiple of 4)
__global__ void __launch_bounds__(1024) march_scan(int buckets, uint4 *__restrict__ count)
{
    __shared__ uint32_t warp_sum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int b0 = 0; b0 < buckets / 4; b0 += 1024) {
        const int b = b0 + threadIdx.x;
        const uint4 c = b < buckets / 4 ? count[b] : make_uint4(0, 0, 0, 0);
        const uint32_t mine = c.x + c.y + c.z + c.w;
        uint32_t inc = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) warp_sum[w] = inc;
        __syncthreads();
        const uint32_t ws = warp_sum[lane];
        uint32_t wi = ws;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += v;
        }
        const uint32_t base = carry + __shfl_sync(0xffffffffu, wi - ws, w) + inc - mine;
        carry += __shfl_sync(0xffffffffu, wi, 31);
        if (b < buckets / 4) count[b] = make_uint4(base, base + c.x, base + c.x + c.y, base + c.x + c.y + c.z);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kThreads) march_scatter(int64_t n, const int64_t *__restrict__ leaves, int64_t n_leaf,
                                                          int shift, uint32_t *__restrict__ next,
                                                          uint2 *__restrict__ order)
{
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = blockIdx.x * (int64_t)kThreads + threadIdx.x - lane; i0 < n; i0 += (int64_t)gridDim.x * kThreads) {
        const int64_t i = i0 + lane, l = i < n ? leaves[i] : -1;
        const uint32_t b = march_bucket(l, n_leaf, shift);
        uint32_t same, at = 0;
        if (march_peers(i < n, b, same)) at = atomicAdd(&next[b], (uint32_t)__popc(same));
        at = __shfl_sync(0xffffffffu, at, __ffs(same) - 1) + __popc(same & ((1u << lane) - 1));
        if (i < n) order[at] = make_uint2((uint32_t)i, l >= 0 && l < n_leaf ? (uint32_t)l : kNoLeaf);
    }
}

__global__ void targets(int64_t n, const float *__restrict__ n_ray, const float *__restrict__ n_tree,
                        float *__restrict__ y)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = logf(n_ray[i] / n_tree[i]);
}

// per-block minimum and maximum of the finite entries of y (+inf / -inf
// where a block saw none)
__global__ void __launch_bounds__(256) finite_range(int64_t n, const float *__restrict__ y, float *__restrict__ part)
{
    __shared__ float smin[256], smax[256];
    float lo = INFINITY, hi = -INFINITY;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float v = y[i];
        if (isfinite(v)) {
            lo = fminf(lo, v);
            hi = fmaxf(hi, v);
        }
    }
    smin[threadIdx.x] = lo;
    smax[threadIdx.x] = hi;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            smin[threadIdx.x] = fminf(smin[threadIdx.x], smin[threadIdx.x + w]);
            smax[threadIdx.x] = fmaxf(smax[threadIdx.x], smax[threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = smin[0];
        part[2 * blockIdx.x + 1] = smax[0];
    }
}

// N = N_tree exp(delta) (N_tree where delta is not finite or outside
// [dlo, dhi]), A_V and the shield; one warp per leaf, the shield summed by a
// fixed butterfly.
__global__ void __launch_bounds__(kThreads) learned_combine(int64_t n, int nd, const float *__restrict__ n_tree,
                                                            const float *__restrict__ delta, float dlo, float dhi,
                                                            float av_per_nh,
                                                            float shield_k, float *__restrict__ n_h,
                                                            float *__restrict__ a_v, float *__restrict__ shield)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
    for (int64_t r = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5); r < n; r += warps) {
        float acc = 0.f;
        for (int d = lane; d < nd; d += 32) {
            const int64_t o = r * nd + d;
            const float dl = delta[o], nt = n_tree[o];
            const float N = isfinite(dl) && dl >= dlo && dl <= dhi ? nt * expf(dl) : nt;
            const float av = N * av_per_nh;
            if (n_h) n_h[o] = N;
            if (a_v) a_v[o] = av;
            acc += expf(-shield_k * av);
        }
        for (int w = 16; w > 0; w >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, w);
        if (shield && lane == 0) shield[r] = acc / (float)nd;
    }
}

cd_status check_tree_geom(cd_tree t, cd_geom g)
{
    if (!t || !g) {
        set_error("tree or geometry is NULL");
        return CD_EINVAL;
    }
    if (t->amr) {
        set_error("the learned form and the ray-marcher serve uniform trees only");
        return CD_EUNSUPPORTED;
    }
    return CD_OK;
}

template <typename T>
cd_status alloc(T **p, size_t count)
{
    if (cudaMalloc(p, count * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        set_error("device allocation of %zu bytes failed", count * sizeof(T));
        return CD_ENOMEM;
    }
    return CD_OK;
}

cd_status launch_features(cd_tree t, cd_geom g, int64_t n, int64_t first, const int64_t *leaves, float *x,
                          float *n_tree, cudaStream_t s)
{
    FeatArgs A = {};
    A.n = n;
    A.first = first;
    A.n_leaf = t->n_leaf;
    A.leaves = leaves;
    A.L = t->L;
    A.nd = g->n_dir;
    A.dx_leaf = dx_of(t, t->L);
    A.rho_leaf = t->rho_leaf;
    A.kloc = g->kloc;
    for (int i = 0; i < 4; ++i) A.Et[i] = t->lv.Et[i];
    for (int k = 0; k <= CD_MAXL; ++k) A.C[k] = t->lv.C[k];
    A.x = x;
    A.n_tree = n_tree;
    if (n == 0) return CD_OK;
    LaunchScope ls(CD_K_FEATURES, s);
    learned_features<<<grid_for(n * g->n_dir, kThreads), kThreads, 0, s>>>(A);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

// Where the spatial order pays for its four small launches (13 us): enough
// cells to march (rows x directions x cells per side; 52 against 56 us at
// 16 384 rows of 32^3, 48 directions, but 49 against 41 at 16 384 of 64^3, 12
// directions), and at least a row per 64 leaves, so that a warp's 32 rows are
// near one another (4.28 against 4.95 ms at 262 144 rows of 256^3, 48
// directions; sparser lists keep the SMs on one region at a time and lose:
// 1.48 against 1.35 ms at 65 536).  Up to 8^3 the densities are 2 KB, near
// whatever the order (4 000 000 rows of 8^3, 6 directions: 0.18 ms as listed, 1.23
// sorted, of 4^3 0.15 and 1.45; 200 000 of 16^3, 48 directions: 0.19 and 0.13).
bool march_sorted(int64_t n, int nd, int L)
{
    return L >= 4 && n * nd >= (int64_t)25000000 >> L && n >= (int64_t)1 << std::max(14, 3 * L - 6);
}

cd_status launch_march(cd_tree t, cd_geom g, int64_t n, const int64_t *leaves, float *n_ray, cudaStream_t s)
{
    MarchArgs A = {};
    A.n = n;
    A.n_leaf = t->n_leaf;
    A.leaves = leaves;
    A.L = t->L;
    A.nd = g->n_dir;
    A.dx_leaf = dx_of(t, t->L);
    A.rho_leaf = t->rho_leaf;
    A.dirs = g->dirs_dev;
    A.out = n_ray;
    const size_t smem = march_smem(A.L);
    CD_ALLOW_SMEM(raymarch, smem, march_smem(kMarchMaxLevel));
    // rows listed in any order are marched in spatial order.  The order lives in
    // stream-ordered scratch; without it (a capture, no memory, more rows than
    // 32-bit places) the rows are taken as they come
    void *scratch = nullptr;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (leaves && march_sorted(n, A.nd, t->L) && n < (int64_t)1 << 31 && cudaStreamIsCapturing(s, &cs) == cudaSuccess &&
        cs == cudaStreamCaptureStatusNone) {
        int bits = 2;
        while (bits < std::min(3 * t->L, kMarchBits) && (int64_t)32 << bits <= n) ++bits;
        const int shift = 3 * t->L - bits, buckets = 1 << bits;
        const size_t head = sizeof(uint32_t) * buckets;
        if (scratch_alloc(&scratch, head + sizeof(uint2) * n, s) == cudaSuccess) {
            uint32_t *count = static_cast<uint32_t *>(scratch);
            uint2 *order = reinterpret_cast<uint2 *>(static_cast<unsigned char *>(scratch) + head);
            cudaMemsetAsync(count, 0, head, s);
            {
                LaunchScope ls(CD_K_RAYMARCH, s);
                march_count<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, leaves, t->n_leaf, shift, count);
            }
            {
                LaunchScope ls(CD_K_RAYMARCH, s);
                march_scan<<<1, 1024, 0, s>>>(buckets, reinterpret_cast<uint4 *>(count));
            }
            {
                LaunchScope ls(CD_K_RAYMARCH, s);
                march_scatter<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, leaves, t->n_leaf, shift, count, order);
            }
            A.order = order;
        }
    }
    // chunks of up to 1024 rows (the path is built once per chunk and
    // direction), fewer where that would leave SMs without a CTA
    A.rows_per_thread = (int)std::max<int64_t>(1, std::min<int64_t>(4, n * A.nd / (kThreads * 152 * 8)));
    const int64_t chunk = (int64_t)kThreads * A.rows_per_thread;
    A.items = (n + chunk - 1) / chunk * A.nd;
    {
        LaunchScope ls(CD_K_RAYMARCH, s);
        raymarch<<<(unsigned)std::min<int64_t>(A.items, 1 << 20), kThreads, smem, s>>>(A);
    }
    const cudaError_t e = cudaGetLastError();
    if (scratch) scratch_free(scratch, s);
    if (e != cudaSuccess) {
        set_error("ray-march launch: %s", cudaGetErrorString(e));
        return CD_ECUDA;
    }
    return CD_OK;
}

cd_status check_net(cd_net net)
{
    if (!net) {
        set_error("network is NULL");
        return CD_EINVAL;
    }
    return CD_OK;
}

cd_status check_batch(cd_net net, int64_t B, const float *x, const float *y)
{
    const cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (B < 1 || B > kChunkRows * 4 || !x || !y) {
        set_error("batch size %lld outside 1 .. %lld or NULL data", (long long)B, (long long)kChunkRows * 4);
        return CD_EINVAL;
    }
    return CD_OK;
}

}  // namespace

// Computes (or reuses) every shell's sum kept apart: C[k] for k = 3 .. L-2 and
// Et[t] at the oct level.
cd_status ensure_level_sums(cd_tree t, cd_geom g, int precision, cudaStream_t s)
{
    LevelSums &lv = t->lv;
    const int nd = g->n_dir, L = t->L;
    if (lv.ndir == nd && lv.geom_uid == g->uid && lv.rho_version == t->rho_version && lv.precision == precision)
        return CD_OK;
    // BF16: the tensor-core contraction (one table per launch) where it serves
    const bool tc = precision == CD_BF16 && tc_supported(nd) && g->wb != nullptr;
    if (lv.ndir != nd) {
        free_level_sums(t);
        for (int k = 3; k <= L - 2; ++k)
            if (alloc(&lv.C[k], ((size_t)1 << (3 * k)) * nd) != CD_OK) return CD_ENOMEM;
        for (int tt = 1; tt <= 3 && tt <= L - 1; ++tt)
            if (alloc(&lv.Et[tt], (size_t)t->n_oct * nd) != CD_OK) return CD_ENOMEM;
        lv.ndir = nd;
    }
    lv.rho_version = -1;
    for (int k = 3; k <= L - 2; ++k) {
        ExtLaunch a = {};
        a.k = k;
        a.nd = nd;
        a.tmask = 4;
        a.rho[3] = t->rho_lvl[k - 2];
        a.dx[3] = dx_of(t, k - 2);
        a.out = lv.C[k];
        cd_status st = tc && k >= 4 ? launch_ext_tc(a, t->rho_brick, g, s) : launch_ext_fp32(a, g, s);
        if (st != CD_OK) return st;
    }
    const int k = L - 1;
    for (int tt = 1; tt <= 3 && tt <= k; ++tt) {
        ExtLaunch a = {};
        a.k = k;
        a.nd = nd;
        a.tmask = 1 << (tt - 1);
        a.rho[tt] = t->rho_lvl[k - tt + 1];
        a.dx[tt] = dx_of(t, k - tt + 1);
        a.out = lv.Et[tt];
        cd_status st = tc && k >= 4 ? launch_ext_tc(a, t->rho_brick, g, s) : launch_ext_fp32(a, g, s);
        if (st != CD_OK) return st;
    }
    lv.geom_uid = g->uid;
    lv.rho_version = t->rho_version;
    lv.precision = precision;
    return CD_OK;
}

void free_level_sums(cd_tree t)
{
    LevelSums &lv = t->lv;
    for (int k = 0; k <= CD_MAXL; ++k) {
        if (lv.C[k]) cd::lib_free(lv.C[k]);
        lv.C[k] = nullptr;
    }
    for (int i = 0; i < 4; ++i) {
        if (lv.Et[i]) cd::lib_free(lv.Et[i]);
        lv.Et[i] = nullptr;
    }
    if (lv.chunk) cd::lib_free(lv.chunk);
    lv.chunk = nullptr;
    lv.chunk_floats = 0;
    lv.ndir = 0;
    lv.geom_uid = 0;
    lv.rho_version = -1;
    lv.precision = -1;
}

cd_status column_density_learned(cd_tree t, cd_geom g, const cd_opts &o, float *n_h, float *a_v, float *shield,
                                 cudaStream_t s)
{
    cd_status st = check_tree_geom(t, g);
    if (st != CD_OK) return st;
    if (o.precision != CD_FP32 && o.precision != CD_BF16) {
        set_error("unknown precision %d", o.precision);
        return CD_EINVAL;
    }
    cd_net net = (cd_net)o.net;
    const int nd = g->n_dir;
    if (o.precision == CD_BF16) return column_density_learned_tc(t, g, o, n_h, a_v, shield, s);
    if (net->lay.nd != nd) {
        set_error("the network has %d directions, the geometry %d", net->lay.nd, nd);
        return CD_EINVAL;
    }
    if ((st = ensure_level_sums(t, g, CD_FP32, s)) != CD_OK) return st;
    LevelSums &lv = t->lv;
    // chunks of whole octs
    const int64_t chunk = std::min<int64_t>(kChunkRows / 8, t->n_oct), H = net->lay.H;
    const auto pad = [](int64_t n) { return (n + 63) & ~(int64_t)63; };   // 256-byte sub-buffers
    const int64_t n_ue = pad(chunk * (kSlots - 1) * nd), n_ul = pad(8 * chunk * (nd + 1)), n_t = pad(8 * chunk * nd),
                  n_h_ = pad(chunk * H), n_wl = pad(H * (nd + 1)), need = n_ue + n_ul + 2 * n_t + n_h_ + n_wl;
    if (lv.chunk_floats < need) {
        if (lv.chunk) cd::lib_free(lv.chunk);
        lv.chunk = nullptr;
        lv.chunk_floats = 0;
        if (alloc(&lv.chunk, (size_t)need) != CD_OK) return CD_ENOMEM;
        lv.chunk_floats = need;
    }
    OctFeatArgs A = {};
    A.L = t->L;
    A.nd = nd;
    A.dx_leaf = dx_of(t, t->L);
    A.rho_leaf = t->rho_leaf;
    A.kloc = g->kloc;
    for (int i = 0; i < 4; ++i) A.Et[i] = lv.Et[i];
    for (int k = 0; k <= CD_MAXL; ++k) A.C[k] = lv.C[k];
    A.mu = net->mu;
    A.sinv = net->sinv;
    A.ue = lv.chunk;
    A.ul = A.ue + n_ue;
    A.n_tree = A.ul + n_ul;
    float *delta = A.n_tree + n_t, *h = delta + n_t, *wl = h + n_h_;
    for (int64_t c0 = 0; c0 < t->n_oct; c0 += chunk) {
        A.first = c0;
        A.n = std::min(chunk, t->n_oct - c0);
        {
            LaunchScope ls(CD_K_FEATURES, s);
            oct_features<<<grid_for(A.n * nd, kThreads), kThreads, 0, s>>>(A);
            CD_CHECK_LAUNCH();
        }
        if ((st = mlp_forward_octs(net, A.n, A.ue, A.ul, h, wl, delta, s)) != CD_OK) return st;
        LaunchScope ls(CD_K_FEATURES, s);
        const int64_t r0 = 8 * c0, rn = 8 * A.n;
        learned_combine<<<grid_for(rn * 32, kThreads), kThreads, 0, s>>>(
            rn, nd, A.n_tree, delta, net->dlo, net->dhi, (float)o.av_per_nh, (float)o.shield_k,
            n_h ? n_h + r0 * nd : nullptr, a_v ? a_v + r0 * nd : nullptr, shield ? shield + r0 : nullptr);
        CD_CHECK_LAUNCH();
    }
    return CD_OK;
}

}  // namespace cd

using namespace cd;

extern "C" {

void cd_adam_default(cd_adam *a)
{
    if (!a) return;
    a->lr = 1e-3;
    a->beta1 = 0.9;
    a->beta2 = 0.999;
    a->eps = 1e-8;
}

int64_t cd_net_num_params(int n_dir, int hidden)
{
    if (n_dir < 1 || n_dir > CD_MAXDIR || hidden < 1 || hidden > 1024) return -1;
    return NetLayout(n_dir, hidden).total;
}

cd_status cd_raymarch(cd_tree tree, cd_geom geom, int64_t n, const int64_t *leaves, float *n_ray, void *stream)
{
    NvtxRange nvtx_range("colden:raymarch");
    cd_status st = check_tree_geom(tree, geom);
    if (st != CD_OK) return st;
    if (n < 0 || !n_ray || (!leaves && n > tree->n_leaf)) {
        set_error("bad ray-march arguments (n = %lld)", (long long)n);
        return CD_EINVAL;
    }
    if (n == 0) return CD_OK;
    return launch_march(tree, geom, n, leaves, n_ray, (cudaStream_t)stream);
}

cd_status cd_learned_features(cd_tree tree, cd_geom geom, int64_t n, const int64_t *leaves, float *x, float *n_tree,
                              void *stream)
{
    NvtxRange nvtx_range("colden:learned_features");
    cd_status st = check_tree_geom(tree, geom);
    if (st != CD_OK) return st;
    if (geom->mode != CD_MODE_PREC) {
        set_error("the learned inputs are defined on the single-ray precalculated form");
        return CD_EUNSUPPORTED;
    }
    if (n < 0 || !x || (!leaves && n > tree->n_leaf)) {
        set_error("bad feature arguments (n = %lld)", (long long)n);
        return CD_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if ((st = ensure_level_sums(tree, geom, CD_FP32, s)) != CD_OK) return st;
    return launch_features(tree, geom, n, 0, leaves, x, n_tree, s);
}

cd_status cd_learned_targets(int64_t n, const float *n_ray, const float *n_tree, float *y, void *stream)
{
    NvtxRange nvtx_range("colden:learned_targets");
    if (n < 0 || (n > 0 && (!n_ray || !n_tree || !y))) {
        set_error("bad target arguments");
        return CD_EINVAL;
    }
    if (n == 0) return CD_OK;
    cudaStream_t s = (cudaStream_t)stream;
    LaunchScope ls(CD_K_FEATURES, s);
    targets<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, n_ray, n_tree, y);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

cd_status cd_net_create(int n_dir, int hidden, const float *params, cd_net *out)
{
    if (!out) {
        set_error("out is NULL");
        return CD_EINVAL;
    }
    *out = nullptr;
    if (cd_net_num_params(n_dir, hidden) < 0 || !params) {
        set_error("bad network sizes (n_dir %d, hidden %d) or NULL params", n_dir, hidden);
        return CD_EINVAL;
    }
    cd_net net = new cd_net_s();
    net->lay = NetLayout(n_dir, hidden);
    cudaGetDevice(&net->dev);
    const size_t P = (size_t)net->lay.total, I = (size_t)net->lay.n_in;
    bool ok = alloc(&net->p, P) == CD_OK && alloc(&net->m, P) == CD_OK && alloc(&net->v, P) == CD_OK &&
              alloc(&net->mu, I) == CD_OK && alloc(&net->sinv, I) == CD_OK;
    if (!ok) {
        cd_net_free(net);
        return CD_ENOMEM;
    }
    std::vector<float> ones(I, 1.f);
    ok = cudaMemcpy(net->p, params, P * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemset(net->m, 0, P * sizeof(float)) == cudaSuccess &&
         cudaMemset(net->v, 0, P * sizeof(float)) == cudaSuccess &&
         cudaMemset(net->mu, 0, I * sizeof(float)) == cudaSuccess &&
         cudaMemcpy(net->sinv, ones.data(), I * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
         // pageable uploads and memsets may return before they land, ordered only
         // on the legacy default stream: finish them before any stream reads the net
         cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) {
        set_error("network upload failed: %s", cudaGetErrorString(cudaGetLastError()));
        cd_net_free(net);
        return CD_ECUDA;
    }
    *out = net;
    return CD_OK;
}

cd_status cd_net_fit_normaliser(cd_net net, int64_t n, const float *x, void *stream)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (n < 1 || !x) {
        set_error("the normaliser needs at least one row");
        return CD_EINVAL;
    }
    return mlp_fit_normaliser(net, n, x, (cudaStream_t)stream);
}

cd_status cd_net_forward(cd_net net, int64_t n, const float *x, float *delta, void *stream)
{
    NvtxRange nvtx_range("colden:net_forward");
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (n < 0 || (n > 0 && (!x || !delta))) {
        set_error("bad forward arguments");
        return CD_EINVAL;
    }
    const NetLayout &L = net->lay;
    cudaStream_t s = (cudaStream_t)stream;
    for (int64_t c0 = 0; c0 < n; c0 += kChunkRows) {
        const int64_t cn = std::min<int64_t>(kChunkRows, n - c0);
        if ((st = mlp_forward(net, cn, x + c0 * L.n_in, delta + c0 * L.nd, s)) != CD_OK) return st;
    }
    return CD_OK;
}

cd_status cd_net_loss_grad(cd_net net, int64_t B, const float *x, const float *y, const int64_t *rows, float *loss,
                           float *grad, void *stream)
{
    NvtxRange nvtx_range("colden:net_loss_grad");
    const cd_status st = check_batch(net, B, x, y);
    if (st != CD_OK) return st;
    return mlp_loss_grad(net, B, x, y, rows, loss, grad, (cudaStream_t)stream);
}

cd_status cd_net_train_step(cd_net net, int64_t B, const float *x, const float *y, const int64_t *rows,
                            const cd_adam *hp, float *loss, void *stream)
{
    NvtxRange nvtx_range("colden:net_train_step");
    const cd_status st = check_batch(net, B, x, y);
    if (st != CD_OK) return st;
    cd_adam h;
    if (hp) h = *hp; else cd_adam_default(&h);
    return mlp_train_step(net, B, x, y, rows, h, loss, (cudaStream_t)stream);
}

cd_status cd_net_get_state(cd_net net, float *params, float *mu, float *sinv, float *adam_m, float *adam_v,
                           int64_t *step)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    CD_CUDA(cudaDeviceSynchronize());
    const size_t P = sizeof(float) * net->lay.total, I = sizeof(float) * net->lay.n_in;
    if (params) CD_CUDA(cudaMemcpy(params, net->p, P, cudaMemcpyDeviceToHost));
    if (adam_m) CD_CUDA(cudaMemcpy(adam_m, net->m, P, cudaMemcpyDeviceToHost));
    if (adam_v) CD_CUDA(cudaMemcpy(adam_v, net->v, P, cudaMemcpyDeviceToHost));
    if (mu) CD_CUDA(cudaMemcpy(mu, net->mu, I, cudaMemcpyDeviceToHost));
    if (sinv) CD_CUDA(cudaMemcpy(sinv, net->sinv, I, cudaMemcpyDeviceToHost));
    if (step) *step = net->step;
    return CD_OK;
}

cd_status cd_net_set_state(cd_net net, const float *params, const float *mu, const float *sinv, const float *adam_m,
                           const float *adam_v, int64_t step)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (step < 0) {
        set_error("negative step count");
        return CD_EINVAL;
    }
    CD_CUDA(cudaDeviceSynchronize());
    const size_t P = sizeof(float) * net->lay.total, I = sizeof(float) * net->lay.n_in;
    if (params) CD_CUDA(cudaMemcpy(net->p, params, P, cudaMemcpyHostToDevice));
    if (adam_m) CD_CUDA(cudaMemcpy(net->m, adam_m, P, cudaMemcpyHostToDevice));
    if (adam_v) CD_CUDA(cudaMemcpy(net->v, adam_v, P, cudaMemcpyHostToDevice));
    if (mu) CD_CUDA(cudaMemcpy(net->mu, mu, I, cudaMemcpyHostToDevice));
    if (sinv) CD_CUDA(cudaMemcpy(net->sinv, sinv, I, cudaMemcpyHostToDevice));
    CD_CUDA(cudaDeviceSynchronize());   // the pageable uploads have landed
    net->step = step;
    net->version += 1;
    return CD_OK;
}

cd_status cd_net_set_delta_range(cd_net net, double lo, double hi)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (std::isnan(lo) || std::isnan(hi)) {
        set_error("the delta range has a NaN end");
        return CD_EINVAL;
    }
    net->dlo = (float)lo;
    net->dhi = (float)hi;
    return CD_OK;
}

cd_status cd_net_get_delta_range(cd_net net, double *lo, double *hi)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (lo) *lo = net->dlo;
    if (hi) *hi = net->dhi;
    return CD_OK;
}

cd_status cd_net_fit_delta_range(cd_net net, int64_t n, const float *y, double margin, void *stream)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (n < 1 || !y || !(margin >= 0.0) || std::isinf(margin)) {
        set_error("the delta range needs n >= 1 targets and a finite margin >= 0");
        return CD_EINVAL;
    }
    constexpr int kBlocks = 256;
    float *part = nullptr;
    if (alloc(&part, 2 * kBlocks) != CD_OK) return CD_ENOMEM;
    cudaStream_t s = (cudaStream_t)stream;
    float h[2 * kBlocks];
    finite_range<<<kBlocks, 256, 0, s>>>(n, y, part);
    const bool ok = cudaGetLastError() == cudaSuccess &&
                    cudaMemcpyAsync(h, part, sizeof(h), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
                    cudaStreamSynchronize(s) == cudaSuccess;
    cd::lib_free(part);
    if (!ok) {
        set_error("delta range reduction failed: %s", cudaGetErrorString(cudaGetLastError()));
        return CD_ECUDA;
    }
    float lo = INFINITY, hi = -INFINITY;
    for (int b = 0; b < kBlocks; ++b) {
        lo = std::min(lo, h[2 * b]);
        hi = std::max(hi, h[2 * b + 1]);
    }
    if (lo > hi) {   // no finite target: an empty range, the plain method everywhere
        net->dlo = INFINITY;
        net->dhi = -INFINITY;
    } else {
        net->dlo = (float)((double)lo - margin);
        net->dhi = (float)((double)hi + margin);
    }
    return CD_OK;
}

cd_status cd_net_info(cd_net net, int *n_dir, int *hidden, int64_t *num_params)
{
    cd_status st = check_net(net);
    if (st != CD_OK) return st;
    if (n_dir) *n_dir = net->lay.nd;
    if (hidden) *hidden = net->lay.H;
    if (num_params) *num_params = net->lay.total;
    return CD_OK;
}

void cd_net_free(cd_net net)
{
    if (!net) return;
    cudaDeviceSynchronize();
    for (float *p : {net->p, net->m, net->v, net->mu, net->sinv, net->act.U, net->act.Z1, net->act.A1,
                     net->act.Z2, net->act.A2, net->act.D, net->act.G, net->act.part, net->act.red})
        if (p) cd::lib_free(p);
    net_free_tc(net);
    delete net;
}

}  // extern "C"
