// FP32 CUDA-core forms of the shell contraction (Eq. N_discret, one level of
// receiving cells per launch): the row form below serves whole levels above 16^3
// and lists of enough receivers, the block form the few cells of coarser levels
// and what the row form has no lists for.  For every cell c at level k and direction d:
//   out[c][d] = prefix_in[parent(c)][d]
//             + sum_{t in tmask} dx_{k-t+1} sum_s rho_{k-t+1}(stencil_t(c), s) K_t[cfg_t(c)][d][s]
// with the 6^3 stencil of table t anchored at the ancestor A_{k-t} of c and
// cfg_t(c) the Morton tail of c (geometry.cu).
//
// One CTA takes the 8^span descendants of one level-q cell (q = k - span,
// span <= 3, smaller on coarse levels so that every launch has at least two
// CTAs per SM): a Morton-contiguous run, so the output rows are written
// coalesced.  The
// density regions its stencils touch (at most 12^3, 8^3 and 6^3 cells for
// tables 1, 2, 3) are staged once in shared memory, zero outside the box
// (§3.2: the shells stop at the box border).  Lanes walk consecutive (cell,
// direction) pairs; the sparse weights are stored [cfg][entry][direction] as
// {shared-memory offset, weight} pairs, so a warp's loads of one entry are
// contiguous, and each (cfg) row is walked to the largest non-zero count of
// its directions (padding entries have weight 0).
#include <algorithm>

#include "common.cuh"
#include "umma.cuh"

namespace cd {
namespace {

constexpr int kExtThreads = 256;

struct ExtArgs {
    ExtLaunch a;
    int span;
    const int2 *tab[4];
    const int *cmax[4];
    int maxe;           // entries per table row
};

// The level-k cells below one CTA root (Morton index at level k - span).
__device__ __forceinline__ void shell_block(const ExtArgs &P, const uint64_t root)
{
    __shared__ float s_rho[kRegionTotal];

    const int k = P.a.k, nd = P.a.nd;
    const int span = P.span;                                  // levels below the CTA root
    const uint32_t Qx = compact3(root), Qy = compact3(root >> 1), Qz = compact3(root >> 2);

    // stage the density regions (level k - t + 1, origin 2 (P_min - 1))
    for (int t = 1; t <= 3; ++t) {
        if (!(P.a.tmask & (1 << (t - 1)))) continue;
        const int l = k - t + 1;
        const int64_t n = (int64_t)1 << l;
        // ancestors A_{k-t} of the CTA's cells: nP per axis from P_min
        const int nP = span >= t ? 1 << (span - t) : 1;
        const int ext = 2 * nP + 4, R = region_side(t);
        const int64_t ox = 2 * ((((int64_t)Qx << span) >> t) - 1), oy = 2 * ((((int64_t)Qy << span) >> t) - 1),
                      oz = 2 * ((((int64_t)Qz << span) >> t) - 1);
        const float *rho = P.a.rho[t];
        for (int r = threadIdx.x; r < R * R * R; r += blockDim.x) {
            const int rx = r % R, ry = (r / R) % R, rz = r / (R * R);
            const int64_t gx = ox + rx, gy = oy + ry, gz = oz + rz;
            float v = 0.f;
            if (rx < ext && ry < ext && rz < ext && gx >= 0 && gy >= 0 && gz >= 0 && gx < n && gy < n && gz < n)
                v = rho[(gz * n + gy) * n + gx];
            s_rho[region_base(t) + r] = v;
        }
    }
    __syncthreads();

    const int ncell = 1 << (3 * span);
    const uint64_t first = root << (3 * span);
    for (int p = threadIdx.x; p < ncell * nd; p += blockDim.x) {
        const int j = p / nd, d = p - j * nd;
        const uint64_t m = first + (uint64_t)j;
        const uint32_t cx = compact3((uint64_t)j), cy = compact3((uint64_t)j >> 1), cz = compact3((uint64_t)j >> 2);
        float acc = P.a.prefix_in && in_bounds((long long)(m >> 3), 1ll << (3 * (k - 1)), kCheckFp32Prefix)
                        ? P.a.prefix_in[(m >> 3) * nd + d]
                        : 0.f;
#pragma unroll
        for (int t = 1; t <= 3; ++t) {
            if (!(P.a.tmask & (1 << (t - 1)))) continue;
            const int R = region_side(t);
            // stencil origin of A_{k-t} relative to the staged region
            const int ax = span >= t ? 2 * (cx >> t) : 0, ay = span >= t ? 2 * (cy >> t) : 0,
                      az = span >= t ? 2 * (cz >> t) : 0;
            const int anchor = region_base(t) + ax + R * (ay + R * az);
            const int cfg = (int)(m & ((1u << (3 * t)) - 1));
            const int2 *row = P.tab[t] + (size_t)cfg * P.maxe * nd + d;
            const int n = P.cmax[t][cfg];
            float part = 0.f;
            for (int e = 0; e < n; ++e) {
                const int2 v = row[(size_t)e * nd];
                if (in_bounds(anchor + v.x - region_base(t), R * R * R, kCheckFp32Region))
                    part = fmaf(s_rho[anchor + v.x], __int_as_float(v.y), part);
            }
            acc = fmaf(P.a.dx[t], part, acc);
        }
        if (in_bounds((long long)m, 1ll << (3 * k), kCheckFp32Out)) P.a.out[m * nd + d] = acc;
    }
}

__global__ void __launch_bounds__(kExtThreads) shell_sum_fp32(ExtArgs P)
{
    shell_block(P, blockIdx.x);
}

// Two levels that do not depend on one another.  (One kernel for both, the job
// picked at run time, reads every argument through a register: 16^3 octs of 12
// directions 11.1 -> 12.1 us.)
struct ExtPair {
    ExtArgs job[2];
    unsigned first;     // CTAs of job 0
};

__global__ void __launch_bounds__(kExtThreads) shell_pair_fp32(const __grid_constant__ ExtPair P)
{
    if (blockIdx.x < P.first) shell_block(P.job[0], blockIdx.x);
    else shell_block(P.job[1], blockIdx.x - P.first);
}


// ---- row form (receiving levels >= 4) -------------------------------------------
//
// The kernel above reads a table entry (8 bytes, mostly from L2) and a density
// from shared memory per lane, whose 32 directions hit random banks; its rows
// are padded to the longest direction (18 entries where 10 are not zero).  Here
// a warp computes four directions of 32 receiving cells of one configuration: a
// lane has one direction and four cells, so that one entry (a broadcast read
// for the eight lanes of a direction) serves four densities that lie next to
// one another (16-byte reads without bank conflicts), and four directions walk
// only as many entries as the longest of them has.
//
// One CTA takes 32 parents P of one class (the six Morton bits that, with the
// child, select the weight rows): every cell of a level has the 64 classes of a
// uniform tree, a list (AMR) groups its receivers' parents by class.  The
// stencils of the three tables around every P are staged once as X[s][parent]
// (648 densities per P, for 8 children x n_dir sums of about ten entries); 16
// warps take the 8 children and halves of the directions.  A warp's entries are
// one stream that comes through a small ring of asynchronous copies.  A 4 x 4
// exchange between the lanes of a cell group turns the sums into rows of four
// directions.
//
// What bounds it: shared memory, one wavefront per 32 (cell, direction) and
// entry (L1 data pipe 93 % busy).  Octs of 256^3, 48 directions: 0.424 ms
// against 1.400 with the kernel above; 40 cone-averaged directions at 128^3
// (39 entries): 0.117 against 0.917; far shells of 64^3 cells 0.049 against
// 0.130.  Steps on the way: one direction and lane-wise rows 0.49 ms (140
// instructions an output row, entries read by every warp), the entries from L1
// instead of the ring 0.68 (their latency).
constexpr int kRowThreads = 512, kRowPitch = 36, kRowCells = CD_STENCIL, kRingQuads = 4;
constexpr int kRowMinEntries = 48;       // directions x longest row
constexpr int kRowMinReceivers = 1024;   // of a list
constexpr int kRowShort = 24;            // longest row of a table: single rays have about ten entries, cones over thirty

struct RowArgs {
    int k, nd;
    int t0, nt;                  // tables t0 .. t0 + nt - 1 are staged
    const float *rho[4];         // dense level arrays by table
    float scale;                 // dx of the weights' unit
    const RowQuad *quad;
    const int *start;
    int width, cfg_mask;         // quad chunks per four directions at most; the configuration bits of the largest table
    const float *prefix;         // S_{k-1} or NULL
    float *out;
    int64_t nG, nblk;            // uniform: 8^(k-3) rows per class in blocks of 32
    const int4 *tiles;           // list: {class, first row, rows, half} in pairs, 128 rows at most
    const uint64_t *row_key;     // list: parent Morton keys
    const int32_t *row_out;      // list: [row][8] output row of child o, -1 if not a receiver
    const int32_t *prefix_row;   // list: prefix row of each output row
    int64_t n_out, n_prefix;     // rows (bounds checks)
};

template <bool kList>
__global__ void __launch_bounds__(kRowThreads, 2) shell_rows_fp32(const __grid_constant__ RowArgs A)
{
    extern __shared__ __align__(128) float smem[];
    float *X = smem;                                                  // [nt 216 + 1][36], the last row zero
    __shared__ int s_p[3][32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nd = A.nd, nq = (nd + 3) >> 2;
    RowQuad *ring = reinterpret_cast<RowQuad *>(smem + ((A.nt * kRowCells + 1) * kRowPitch + 31) / 32 * 32) +
                    warp * 2 * kRingQuads;
    int cls, nrows;
    int64_t first;
    if (kList) {
        const int4 t = A.tiles[2 * (blockIdx.x >> 2)];
        cls = t.x;
        const int sub = 32 * (int)(blockIdx.x & 3);
        first = t.y + sub;
        nrows = min(32, t.z - sub);
        if (nrows <= 0) return;
    } else {
        cls = (int)(blockIdx.x / A.nblk);                             // a class's blocks run together
        first = (int64_t)(blockIdx.x % A.nblk) * 32;
        nrows = (int)(A.nG - first < 32 ? A.nG - first : 32);
    }
    const int o = warp & 7, c9 = (cls << 3) | o, cfg = c9 & A.cfg_mask;
    // this warp's quads of directions [qa, qb) and their stream of quad chunks
    // (a ring block past the lists is allocated)
    const int half = (nq + 1) / 2, qa = (warp >> 3) * half, qb = min(nq, qa + half);
    const int *start = A.start + (size_t)cfg * (nq + 1);
    const int first_quad = qa < qb ? start[qa] : 0, n = qa < qb ? start[qb] - first_quad : 0;
    const char *stream = reinterpret_cast<const char *>(A.quad + (size_t)cfg * nq * A.width + first_quad);
    static_assert(kRingQuads * sizeof(RowQuad) == 32 * 16, "a ring block is one copy per lane");
    const auto issue = [&](int blk) {
        if (blk * kRingQuads < n)
            cp_async16(reinterpret_cast<char *>(ring + (blk & 1) * kRingQuads) + 16 * lane,
                       stream + (size_t)blk * kRingQuads * sizeof(RowQuad) + 16 * lane, 16u);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    issue(0);
    issue(1);
    if (warp == 0) {
        const bool live = lane < nrows;
        const uint64_t P = !live ? 0 : kList ? A.row_key[first + lane] : (uint64_t)(first + lane) << 6 | (uint64_t)cls;
        s_p[0][lane] = live ? (int)compact3(P) : -1;
        s_p[1][lane] = (int)compact3(P >> 1);
        s_p[2][lane] = (int)compact3(P >> 2);
    }
    for (int i = tid; i < kRowPitch; i += kRowThreads) X[A.nt * kRowCells * kRowPitch + i] = 0.f;
    // this lane's output and prefix rows once its sums are exchanged: parent 4 (lane & 7) + (lane >> 3)
    const int g = lane >> 3, r_out = 4 * (lane & 7) + g;
    int64_t orow = -1, prow = -1;
    if (r_out < nrows) {
        orow = kList ? (int64_t)A.row_out[8 * (first + r_out) + o] : (first + r_out) * 512 + c9;
        if (orow >= 0 && !in_bounds(orow, A.n_out, kCheckFp32Out)) orow = -1;
        if (orow >= 0 && A.prefix) prow = kList ? (int64_t)A.prefix_row[orow] : (first + r_out) * 64 + cls;
        if (prow >= 0 && !in_bounds(prow, A.n_prefix, kCheckFp32Prefix)) prow = -1;
    }
    float *out = A.out + (orow < 0 ? 0 : orow) * nd;
    const float *pre = prow < 0 ? nullptr : A.prefix + prow * nd;
    __syncthreads();

    // stage the stencils: a warp takes (y, z) rows of one table's stencils, three
    // reads of a pair of cells for the 32 parents; its lanes take the three pairs
    // of four parents that are neighbours in x on a uniform tree (one line of
    // densities) before the next four
    const int groups = 16 / A.nt, q = warp % A.nt, sub = warp / A.nt;
    if (sub < groups) {
        const int t = A.t0 + q, side = 1 << (A.k - t + 1);
        const float *rho = A.rho[t];
        int base[3], dst[3];
        uint32_t in_y[3], in_z[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int u = lane + 32 * j, a = 2 * (u % 3), v = u / 3, gr = v >> 2;
            const int r = (v & 1) | ((v & 2) << 2) | ((gr & 3) << 1) | ((gr >> 2) << 4);
            const int px = s_p[0][r];
            const int x = 2 * ((px >> (t - 1)) - 1) + a, y = 2 * ((s_p[1][r] >> (t - 1)) - 1),
                      z = 2 * ((s_p[2][r] >> (t - 1)) - 1);
            base[j] = (z * side + y) * side + x;
            dst[j] = (q * kRowCells + a) * kRowPitch + r;
            in_y[j] = in_z[j] = 0;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                in_y[j] |= (uint32_t)(y + i >= 0 && y + i < side) << i;
                in_z[j] |= (uint32_t)(z + i >= 0 && z + i < side) << i;
            }
            if (px < 0 || x < 0 || x >= side) in_y[j] = 0;
        }
        for (int bc0 = sub; bc0 < 36; bc0 += 4 * groups) {
            float2 f[4][3];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int bc = bc0 + i * groups, b = bc % 6, c = bc / 6, step = (c * side + b) * side;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    f[i][j] = make_float2(0.f, 0.f);
                    if (bc < 36 && ((in_y[j] >> b) & (in_z[j] >> c) & 1u) &&
                        in_bounds((long long)base[j] + step + 1, (long long)side * side * side, kCheckListLevel))
                        f[i][j] = *reinterpret_cast<const float2 *>(rho + (base[j] + step));
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int bc = bc0 + i * groups;
                if (bc >= 36) break;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    float *p = X + 6 * bc * kRowPitch + dst[j];
                    p[0] = f[i][j].x;
                    p[kRowPitch] = f[i][j].y;
                }
            }
        }
    }
    __syncthreads();

    const char *Xl = reinterpret_cast<const char *>(X + 4 * (lane & 7));
    float acc[4] = {0.f, 0.f, 0.f, 0.f};                              // direction 4 quad + g of parents 4 (lane & 7) ..
    int d = 4 * qa;
    const auto cells = [&](int off) { return *reinterpret_cast<const float4 *>(Xl + off); };
    for (int blk = 0; blk * kRingQuads < n; ++blk) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const RowChunk *rb = ring[(blk & 1) * kRingQuads].d + g;
        const int cnt = min(kRingQuads, n - blk * kRingQuads);
#pragma unroll 1
        for (int j = 0; j < cnt; ++j, rb += 4) {
            const RowChunk v = *rb;
            const int ow = v.off.w & ~1;                              // bit 0: the quad's last chunk
            if (in_bounds(max(max(v.off.x, v.off.y), max(v.off.z, ow)), (A.nt * kRowCells + 1) * kRowPitch * 4,
                          kCheckFp32Region)) {
                // four entries at a time: rows of a cone have forty
                const float4 x0 = cells(v.off.x), x1 = cells(v.off.y), x2 = cells(v.off.z), x3 = cells(ow);
                acc[0] += fmaf(x3.x, v.w.w, fmaf(x2.x, v.w.z, fmaf(x1.x, v.w.y, x0.x * v.w.x)));
                acc[1] += fmaf(x3.y, v.w.w, fmaf(x2.y, v.w.z, fmaf(x1.y, v.w.y, x0.y * v.w.x)));
                acc[2] += fmaf(x3.z, v.w.w, fmaf(x2.z, v.w.z, fmaf(x1.z, v.w.y, x0.z * v.w.x)));
                acc[3] += fmaf(x3.w, v.w.w, fmaf(x2.w, v.w.z, fmaf(x1.w, v.w.y, x0.w * v.w.x)));
            }
            if (!(v.off.w & 1)) continue;
            // exchange: lane g of a group of four parents gets its parent's four directions
            const bool g0 = g & 1, g1 = g & 2;
            float s0 = __shfl_xor_sync(0xffffffffu, g0 ? acc[0] : acc[1], 8);
            float s1 = __shfl_xor_sync(0xffffffffu, g0 ? acc[2] : acc[3], 8);
            if (g0) { acc[0] = s0; acc[2] = s1; } else { acc[1] = s0; acc[3] = s1; }
            s0 = __shfl_xor_sync(0xffffffffu, g1 ? acc[0] : acc[2], 16);
            s1 = __shfl_xor_sync(0xffffffffu, g1 ? acc[1] : acc[3], 16);
            if (g1) { acc[0] = s0; acc[1] = s1; } else { acc[2] = s0; acc[3] = s1; }
            if (orow >= 0) {
                if ((nd & 3) == 0) {
                    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (pre) p = *reinterpret_cast<const float4 *>(pre + d);
                    *reinterpret_cast<float4 *>(out + d) =
                        make_float4(fmaf(A.scale, acc[0], p.x), fmaf(A.scale, acc[1], p.y), fmaf(A.scale, acc[2], p.z),
                                    fmaf(A.scale, acc[3], p.w));
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (d + i < nd) out[d + i] = fmaf(A.scale, acc[i], pre ? pre[d + i] : 0.f);
                }
            }
            acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
            d += 4;
        }
        __syncwarp();
        issue(blk + 2);
    }
}

// One warp per configuration of list i, a lane per quad of directions: the
// quads' chunks one after another (at least one each), start[cfg][quad] the
// first of each.  A quad has as many as its longest direction; entries not used
// have weight 0 and point at the zero row, and bit 0 of the last offset marks
// the quad's last chunk.
__global__ void __launch_bounds__(128) row_lists(int i, int nd, int ncfg, const int2 *t1, const int2 *t2,
                                                 const int2 *t3, int maxe, int width, RowQuad *__restrict__ quad,
                                                 int *__restrict__ start)
{
    const int cfg = (int)(blockIdx.x * 4 + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
    if (cfg >= ncfg) return;
    const int nq = (nd + 3) / 4;
    const int ta = i < 3 ? i + 1 : 1, tb = i < 3 ? i + 1 : 3;
    const int zero = (tb - ta + 1) * kRowCells * kRowPitch * 4;
    const auto entry = [&](int t, int q, int d) {   // entries of a row come first, then zeros
        const int2 *tab = t == 1 ? t1 : t == 2 ? t2 : t3;
        return tab[((size_t)(cfg & ((1 << (3 * t)) - 1)) * maxe + q) * nd + d];
    };
    int done = 0;
    for (int q0 = 0; q0 < nq; q0 += 32) {
        const int qd = q0 + lane;
        int chunks = qd < nq ? 1 : 0;
        for (int d = 4 * qd; d < min(nd, 4 * qd + 4); ++d) {
            int count = 0;
            for (int t = ta; t <= tb; ++t)
                for (int q = 0; q < maxe && __int_as_float(entry(t, q, d).y) != 0.f; ++q) ++count;
            chunks = max(chunks, (count + 3) / 4);
        }
        int inc = chunks;
        for (int s = 1; s < 32; s <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, s);
            if (lane >= s) inc += v;
        }
        const int first = done + inc - chunks;
        done += __shfl_sync(0xffffffffu, inc, 31);
        if (qd < nq) {
            start[(size_t)cfg * (nq + 1) + qd] = first;
            for (int j = 0; j < 4; ++j) {
                RowQuad *to = quad + (size_t)cfg * nq * width + first;
                const int d = 4 * qd + j;
                int t = ta, q = 0;
                for (int c = 0; c < chunks; ++c) {
                    float w[4];
                    int off[4];
                    for (int e = 0; e < 4; ++e) {
                        w[e] = 0.f;
                        off[e] = zero;
                        while (d < nd && t <= tb) {
                            const int2 v = q < maxe ? entry(t, q, d) : make_int2(0, 0);
                            if (__int_as_float(v.y) == 0.f) {
                                ++t;
                                q = 0;
                                continue;
                            }
                            const int R = region_side(t);
                            const int s = v.x % R + 6 * ((v.x / R) % R) + 36 * (v.x / (R * R));
                            w[e] = __int_as_float(v.y) * (i < 3 ? 1.f : (float)(1 << (t - 1)));
                            off[e] = ((t - ta) * kRowCells + s) * kRowPitch * 4;
                            ++q;
                            break;
                        }
                    }
                    if (c == chunks - 1) off[3] |= 1;
                    to[c].d[j] = {make_float4(w[0], w[1], w[2], w[3]), make_int4(off[0], off[1], off[2], off[3])};
                }
            }
        }
        __syncwarp();
    }
    if (lane == 0) start[(size_t)cfg * (nq + 1) + nq] = done;
}

size_t row_smem(int nt)
{
    return sizeof(float) * (((size_t)(nt * kRowCells + 1) * kRowPitch + 31) / 32 * 32) +
           16 * 2 * kRingQuads * sizeof(RowQuad);
}

// the list of a table mask, or -1
int row_list(int tmask) { return tmask == 1 ? 0 : tmask == 2 ? 1 : tmask == 4 ? 2 : tmask == 7 ? 3 : -1; }

cd_status launch_rows(const ExtLaunch &a, cd_geom g, cudaStream_t s)
{
    const int li = row_list(a.tmask);
    const cd_geom_s::RowList &L = g->rows[li];
    RowArgs A = {};
    A.k = a.k;
    A.nd = a.nd;
    A.t0 = li < 3 ? li + 1 : 1;
    A.nt = li < 3 ? 1 : 3;
    for (int t = 1; t <= 3; ++t) A.rho[t] = a.rho[t];
    A.scale = a.dx[A.t0];
    A.quad = L.quad;
    A.start = L.start;
    A.width = L.width;
    A.cfg_mask = (li < 3 ? 8 << (3 * li) : 512) - 1;
    A.prefix = a.prefix_in;
    A.out = a.out;
    int64_t grid;
    if (a.list) {
        A.tiles = a.list->tiles;
        A.row_key = a.list->key;
        A.row_out = a.list->out;
        A.prefix_row = a.list->recv_parent;
        A.n_out = a.list->n_recv;
        A.n_prefix = a.n_prefix;
        grid = a.list->ntiles / 2 * 4;
    } else {
        A.nG = (int64_t)1 << (3 * (a.k - 3));
        A.nblk = (A.nG + 31) / 32;
        A.n_out = (int64_t)1 << (3 * a.k);
        A.n_prefix = (int64_t)1 << (3 * (a.k - 1));
        grid = 64 * A.nblk;
    }
    if (grid == 0) return CD_OK;
    const size_t smem = row_smem(A.nt);
    const auto kern = a.list ? shell_rows_fp32<true> : shell_rows_fp32<false>;
    CD_ALLOW_SMEM(kern, smem, row_smem(3));
    LaunchScope ls(CD_K_SHELL, s);
    kern<<<(unsigned)grid, kRowThreads, smem, s>>>(A);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

// arguments of the block form over a whole level; its CTAs
unsigned block_args(const ExtLaunch &a, cd_geom g, ExtArgs &P)
{
    P.a = a;
    // largest span <= min(3, k) that still gives >= 304 CTAs (2 per SM)
    int span = a.k < 3 ? a.k : 3;
    while (span > 0 && (1ull << (3 * (a.k - span))) < 304ull) --span;
    P.span = span;
    for (int t = 0; t < 4; ++t) {
        P.tab[t] = g->tab[t];
        P.cmax[t] = g->cmax[t];
    }
    P.maxe = g->maxe;
    return (unsigned)(1ull << (3 * (a.k - span)));
}

}  // namespace

// the row form has the lists of these tables and something to sum
static bool rows_serve(int k, int tmask, cd_geom g)
{
    // with hardly anything to sum (the six axis rays have three entries at most)
    // staging a parent's stencils costs more than the block form's gathers
    // (64^3: 24.6 against 23.1 us; 12 HEALPix directions 24.4 against 28.7)
    const int li = row_list(tmask);
    return k >= 4 && li >= 0 && g->rows[li].quad != nullptr && g->n_dir * g->maxe >= kRowMinEntries;
}

bool ext_fp32_serves_list(int k, int tmask, cd_geom g, const TcList *list, bool walk)
{
    if (!rows_serve(k, tmask, g)) return false;
    // A CTA reads its class's entries for 32 cells: too few receivers per class
    // leave it little to share them with.  The whole level of 16^3 has eight parents in
    // each of 64 classes (evaluations of 32^3 replayed as graphs, row against block
    // form: 12 directions 22.5 and 18.5 us, 84 directions 37.0 and 28.8, 40
    // cone-averaged ones 48.3 and 35.4; at 64^3 48 directions take 43 and 64).
    if (!list) return k > 4;
    // Lists have slower alternatives.  On 16^3, where a whole class has eight parents,
    // the list kernel's gathers hit few lines: with the short rows of single rays it
    // keeps lists of up to about 131 072 / directions receivers.  Graphs of meshes of 16^3
    // with refined cells, row against list form: 1 050 cells 20 directions 24.6 and
    // 22.7 us, 32 26.8 and 24.6, 84 41.2 and 39.0, but 12 directions 24.6 and 24.7, 192 57
    // and 65, 12 cone-averaged ones 68 and 88; 1 600 cells 32 directions 28.7 and 26.7,
    // 84 41.1 and 41.1; 2 600 cells 48 directions 32.8 and 34.9.  On 32^3 1 050 cells
    // take 48 directions 34.9 and 45.1 us.  In-situ columns would walk instead.
    const bool coarse = k == 4 && !walk && g->maxe <= kRowShort && g->n_dir > 16;
    const int64_t least = coarse ? std::min(2400, 131072 / g->n_dir) : 0;
    return list->n_recv >= std::max<int64_t>(kRowMinReceivers, least);
}

cd_status build_row_lists(cd_geom g, cudaStream_t s)
{
    // rows of a list are as wide as the largest counts allow; direction sets
    // whose lists would take more than 256 MB, or find no room, stay with the
    // tables alone
    constexpr size_t kMaxBytes = (size_t)256 << 20;
    for (int i = 0; i < 4; ++i) {
        cd_geom_s::RowList &L = g->rows[i];
        const int ncfg = i < 3 ? 8 << (3 * i) : 512;
        L.width = ((i < 3 ? 1 : 3) * g->maxe + 3) / 4;
        const int nq = (g->n_dir + 3) / 4;
        const size_t quads = (size_t)ncfg * nq * L.width + kRingQuads;   // the kernel reads whole blocks
        if (quads * sizeof(RowQuad) > kMaxBytes) continue;
        if (cudaMalloc(&L.quad, quads * sizeof(RowQuad)) != cudaSuccess ||
            cudaMalloc(&L.start, sizeof(int) * ncfg * (nq + 1)) != cudaSuccess) {
            cudaGetLastError();           // no room: the other forms serve these tables
            if (L.quad) cudaFree(L.quad);   // no evaluation has seen it: captured graphs stay valid
            L.quad = nullptr;
            L.start = nullptr;
            continue;
        }
        LaunchScope ls(CD_K_OTHER, s);
        row_lists<<<(unsigned)((ncfg + 3) / 4), 128, 0, s>>>(i, g->n_dir, ncfg, g->tab[1], g->tab[2], g->tab[3], g->maxe,
                                                            L.width, L.quad, L.start);
        CD_CHECK_LAUNCH();
    }
    return CD_OK;
}

cd_status launch_ext_fp32(const ExtLaunch &a, cd_geom g, cudaStream_t s)
{
    if (a.list ? rows_serve(a.k, a.tmask, g) : ext_fp32_serves_list(a.k, a.tmask, g, nullptr)) return launch_rows(a, g, s);
    if (a.list) {
        set_error("the FP32 block form serves whole levels only");
        return CD_EUNSUPPORTED;
    }
    ExtArgs P;
    const unsigned grid = block_args(a, g, P);
    LaunchScope ls(CD_K_SHELL, s);
    shell_sum_fp32<<<grid, kExtThreads, 0, s>>>(P);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

// (a's CTAs are placed first: the far shells' rows before the octs', whose 84 directions
// then take 24.7 us a call of 32^3 instead of 26.7, 192 directions 37.0 instead of 41.0)
cd_status launch_ext_fp32_pair(const ExtLaunch &a, const ExtLaunch &b, cd_geom g, cudaStream_t s)
{
    if (!a.list && !b.list && !ext_fp32_serves_list(a.k, a.tmask, g, nullptr) &&
        !ext_fp32_serves_list(b.k, b.tmask, g, nullptr)) {
        ExtPair P;
        P.first = block_args(a, g, P.job[0]);
        const unsigned grid = P.first + block_args(b, g, P.job[1]);
        LaunchScope ls(CD_K_SHELL, s);
        shell_pair_fp32<<<grid, kExtThreads, 0, s>>>(P);
        CD_CHECK_LAUNCH();
        return CD_OK;
    }
    const cd_status st = launch_ext_fp32(a, g, s);
    return st != CD_OK ? st : launch_ext_fp32(b, g, s);
}

}  // namespace cd
