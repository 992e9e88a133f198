// The in-situ variant of the tree method (§4.3): every shell is seen from the
// centre of the target's oct, with no precalculated two-level approximation.
//
// From the oct centre p, the shell of level l (the 6^3 level-l cells covering
// the 3^3 block of level l-1 around the ancestor A_{l-1}, minus the inner
// region: the oct itself at l = l0-1, the 3^3 level-l block around A_l below,
// both clipped to the box; Eq. N_discret) meets the ray p + s u (s >= 0) in the
// single segment between the ray's exits from the two nested boxes, since
// both contain p.  The contribution sum_i n_i dx_i of the shell is therefore
// the line integral of the level-l density over that segment, which a short
// cell-by-cell walk (DDA) over the level-l grid computes exactly: each
// crossing is recomputed from its cell face, so nothing accumulates.
//
// The three nearest shells are the precalculated ones: tables 1 to 3 are seen
// from the oct centre too (§3.3), so there the two-level approximation is exact
// and the row kernel of colden_fp32.cu sums them, in FP64-built weights.  One
// thread per (oct, direction) then walks the coarser levels, whose arrays fit
// L1, and adds them; a shell's inner exit is the outer exit of the shell before.
// What bounds it: the instructions of the walks.  Octs of 128^3, 40 directions:
// 0.052 + 0.184 ms, against 0.941 for walks of every level with lanes over the
// directions (0.377 for the coarse levels alone that way, 0.327 with the
// directions' reciprocals kept and 32-bit indices).
// The leaf kernels add the internal and local terms as in the precalculated
// form.
#include <algorithm>

#include "common.cuh"

namespace cd {
namespace {

struct InsituArgs {
    int64_t n;               // octs
    const uint64_t *keys;    // Morton keys of the octs at level k, or NULL: octs 0 .. n-1
    int k;                   // level of the octs (their children are the leaves, l0 = k + 1)
    int top;                 // first level walked: k, or k - 3 after the precalculated shells
    int nd, chunk;           // directions; how many of them a CTA takes
    const double *dirs;      // [nd][3]
    const float *lvl[CD_MAXL + 1];   // dense row-major volume means of levels 0 .. k
    float box;               // cm
    float *out;              // [n][nd], cm^-2; added to when top < k
};

// exit distance of the ray p + s u from the box [lo, hi] (which contains p)
__device__ __forceinline__ float box_exit(const float p[3], const float u[3], const float inv[3], const float lo[3],
                                          const float hi[3])
{
    float t = INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (u[a] > 0.f) t = fminf(t, (hi[a] - p[a]) * inv[a]);
        else if (u[a] < 0.f) t = fminf(t, (lo[a] - p[a]) * inv[a]);
    }
    return t;
}

constexpr int kOctsPerCta = 32;   // a lane each

// directions and reciprocals, the octs' sums
constexpr size_t insitu_smem(int nc) { return sizeof(float) * (6 * (size_t)nc + kOctsPerCta * (size_t)(nc | 1)); }

__global__ void __launch_bounds__(256) insitu_external(const __grid_constant__ InsituArgs A)
{
    extern __shared__ float s_dir[];     // [nc][6]: direction and reciprocals (0 where a component is 0)
    const int d0 = blockIdx.y * A.chunk, nc = min(A.chunk, A.nd - d0);   // directions d0 .. d0 + nc - 1
    const int nd = A.nd, k = A.k, pitch = nc | 1, lane = threadIdx.x & 31;
    float *s_sum = s_dir + 6 * nc;       // [32 octs][pitch]
    for (int d = threadIdx.x; d < nc; d += blockDim.x)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float u = (float)A.dirs[3 * (d0 + d) + a];
            s_dir[6 * d + a] = u;
            s_dir[6 * d + 3 + a] = u != 0.f ? 1.f / u : 0.f;
        }
    __syncthreads();
    const float hk = 1.f / (float)(1 << k);
    for (int64_t o0 = blockIdx.x * (int64_t)kOctsPerCta; o0 < A.n; o0 += (int64_t)gridDim.x * kOctsPerCta) {
        const int nb = (int)(A.n - o0 < kOctsPerCta ? A.n - o0 : kOctsPerCta);
        // a lane per oct: neighbours' rays of one direction cross the same coarse cells
        // in step (lanes over directions diverge at every crossing)
        const uint64_t key = lane < nb ? (A.keys ? A.keys[o0 + lane] : (uint64_t)(o0 + lane)) : 0;
        for (int d = threadIdx.x >> 5; lane < nb && d < nc; d += blockDim.x >> 5) {
            const int oc[3] = {(int)compact3(key), (int)compact3(key >> 1), (int)compact3(key >> 2)};
            float u[3], inv[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                u[a] = s_dir[6 * d + a];
                inv[a] = s_dir[6 * d + 3 + a];
            }
            // coordinates in units of the box; the oct centre
            const float p[3] = {((float)oc[0] + 0.5f) * hk, ((float)oc[1] + 0.5f) * hk, ((float)oc[2] + 0.5f) * hk};
            float total = 0.f;
            // the exit from the first shell's inner region: the oct, or the 3^3 block
            // around its ancestor
            float t1;
            {
                const int l = A.top, n = 1 << l;
                const float h = 1.f / (float)n;
                float lo[3], hi[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int al = oc[a] >> (k - l);
                    lo[a] = (float)(l == k ? al : max(al - 1, 0)) * h;
                    hi[a] = (float)(l == k ? al + 1 : min(al + 2, n)) * h;
                }
                t1 = box_exit(p, u, inv, lo, hi);
            }
            for (int l = A.top; l >= 1; --l) {
                const int n = 1 << l;
                const float h = 1.f / (float)n;
                float olo[3], ohi[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int am = oc[a] >> (k - l + 1);   // A_{l-1}
                    olo[a] = (float)max(2 * (am - 1), 0) * h;
                    ohi[a] = (float)min(2 * (am + 2), n) * h;
                }
                const float t0 = t1;                       // the shell before ends where this one begins
                t1 = box_exit(p, u, inv, olo, ohi);
                if (!(t1 > t0)) {
                    t1 = t0;
                    continue;
                }
                // first cell: the one the ray enters at t0; face: the coordinate (in cells) of
                // its exit face per axis
                int c[3], step[3];
                float face[3], tnext[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float q = (p[a] + t0 * u[a]) * (float)n;
                    step[a] = u[a] > 0.f ? 1 : u[a] < 0.f ? -1 : 0;
                    c[a] = min(max(u[a] < 0.f ? (int)ceilf(q) - 1 : (int)floorf(q), 0), n - 1);
                    face[a] = (float)(c[a] + (u[a] > 0.f));
                    tnext[a] = u[a] != 0.f ? (face[a] * h - p[a]) * inv[a] : INFINITY;
                }
                const float *rho = A.lvl[l];
                float t = t0, sum = 0.f;
                for (int it = 0; it < 24 && t < t1; ++it) {
                    const bool ay = tnext[1] < tnext[0];                       // ties go to the lower axis
                    const bool az = tnext[2] < (ay ? tnext[1] : tnext[0]);
                    const float tn = fminf(az ? tnext[2] : ay ? tnext[1] : tnext[0], t1);
                    sum = fmaf(rho[(c[2] << (2 * l)) + (c[1] << l) + c[0]], tn - t, sum);
                    t = tn;
                    bool out = false;
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (a == 2 ? az : a == 1 ? ay && !az : !ay && !az) {
                            c[a] += step[a];
                            face[a] += (float)step[a];
                            tnext[a] = (face[a] * h - p[a]) * inv[a];
                            out = (unsigned)c[a] >= (unsigned)n;
                        }
                    if (out) break;
                }
                total += sum;
            }
            s_sum[lane * pitch + d] = total;
        }
        __syncthreads();
        for (int w = threadIdx.x; w < nb * nc; w += blockDim.x) {
            const int i = w / nc, j = w - i * nc;
            float *out = A.out + (o0 + i) * nd + d0 + j;
            const float total = s_sum[i * pitch + j];
            *out = A.top < k ? fmaf(total, A.box, *out) : total * A.box;
        }
        __syncthreads();
    }
}

}  // namespace

cd_status launch_insitu(cd_tree t, cd_geom g, int k, int64_t n, const uint64_t *keys, const TcList *list, float *out,
                        cudaStream_t s)
{
    if (n == 0) return CD_OK;
    InsituArgs A = {};
    A.top = k;
    if (ext_fp32_serves_list(k, 7, g, keys ? list : nullptr, true) && (!keys || (list && list->ntiles))) {
        ExtLaunch e = {};
        e.k = k;
        e.nd = g->n_dir;
        e.tmask = 7;
        for (int q = 1; q <= 3; ++q) {
            e.rho[q] = t->rho_lvl[k - q + 1];
            e.dx[q] = (float)(t->box_cm / (double)((int64_t)1 << (k - q + 1)));
        }
        e.out = out;
        e.list = keys ? list : nullptr;
        const cd_status st = launch_ext_fp32(e, g, s);
        if (st != CD_OK) return st;
        A.top = k - 3;
    }
    A.n = n;
    A.keys = keys;
    A.k = k;
    A.nd = g->n_dir;
    A.dirs = g->dirs_dev;
    for (int l = 0; l <= k && l <= CD_MAXL; ++l) A.lvl[l] = t->rho_lvl[l];
    A.box = (float)t->box_cm;
    A.out = out;
    const int64_t blocks = std::min<int64_t>((n + kOctsPerCta - 1) / kOctsPerCta, 152 * 32);
    // a CTA takes all directions of its octs, or on small trees as many eights as
    // still give two CTAs per SM (16^3, 84 directions:
    // 24.9 -> 9.3 us; 32^3: 31.2 -> 21.4)
    const int64_t eights = (g->n_dir + 7) / 8;
    A.chunk = blocks >= 304 ? g->n_dir : 8 * (int)std::max<int64_t>(1, eights * blocks / 304);
    const dim3 grid((unsigned)std::max<int64_t>(blocks, 1), (unsigned)((g->n_dir + A.chunk - 1) / A.chunk));
    const int nc = std::min(A.chunk, g->n_dir);
    LaunchScope ls(CD_K_SHELL, s);
    const size_t smem = insitu_smem(nc);
    CD_ALLOW_SMEM(insitu_external, smem, insitu_smem(CD_MAXDIR));
    insitu_external<<<grid, 32 * std::min(8, nc), smem, s>>>(A);
    CD_CHECK_LAUNCH();
    return CD_OK;
}

}  // namespace cd
