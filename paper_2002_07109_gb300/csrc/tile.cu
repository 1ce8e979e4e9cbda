// Pair sums over all pairs (droplets and batches of replicas without a
// cutoff; the F_0 share of every pair, Sec. IV.A / V, and BAOAB's full pair
// gradient).
//
// Work: a static list of items (i-tile of 32 atoms, j-block of tj atoms of the
// same replica at or after the i-tile), built on the host when the topology
// or the replica layout is set; every unordered pair of a replica lies in
// exactly one item (two atoms of one tile: in the item whose j-block starts
// at that tile, with j > i).  A second i-tile, tj atoms further on, meets the
// same j-blocks and rides along in the same item where there is work enough
// (setup_tiles).  A resident grid of warps strides over the items: lane l
// holds atom l of each i-tile, the j-block is staged in shared memory 32
// atoms at a time, and in sub-step k lane l evaluates its pairs with atom
// (l + k) mod 32 of the stage, both tiles' in packed arithmetic (pairs.cuh).
// Both sides of every pair are summed once (Newton's third law): the i side
// in the lane's registers, the j side (one sum per i-tile) in registers that
// move to the next lane after every sub-step, so that after 32 sub-steps lane
// l holds the sums of atom l of the stage; all go to int64 fixed-point
// accumulators (2^-32 kcal/mol/A) rounded from FP32 by the int64 conversion,
// so the result does not depend on the order in which warps finish.  The
// j-block length tj is chosen by the autotuner (bounce_autotune).
#include <algorithm>

#include "common.cuh"
#include "pairs.cuh"

namespace {

// The sub-steps of one stage: this lane's i atoms (two, packed) against the 32
// staged j atoms.  GEN: with the index rule j > i (m > dj) and the minimum image.
template <int PART, bool EW, bool CJ, bool GEN>
__device__ __forceinline__ void tile_stage(const PairConsts& k, const float4* sh, const float4* sl, const int* sm,
                                           const float2* lj, const float2 (&h)[3], const float2 (&l)[3], float2 kq,
                                           const int (&mi)[2], const int (&ti)[2], const int (&dj)[2], float2 (&gi)[3],
                                           float2 (&gj)[3], int (&np)[2]) {
    const int lane = threadIdx.x & 31;
#pragma unroll 8
    for (int s = 0; s < 32; ++s) {
        const int m = (lane + s) & 31;
        const float4 hj = sh[m], lw = sl[m];
        const int mj = sm[m], tj = type_of(lw);
        // (one value of j against both: two scalar differences cost what
        // duplicating it for a packed one would)
        float2 dx = make_float2(h[0].x - hj.x, h[0].y - hj.x), ex = make_float2(l[0].x - lw.x, l[0].y - lw.x);
        float2 dy = make_float2(h[1].x - hj.y, h[1].y - hj.y), ey = make_float2(l[1].x - lw.y, l[1].y - lw.y);
        float2 dz = make_float2(h[2].x - hj.z, h[2].y - hj.z), ez = make_float2(l[2].x - lw.z, l[2].y - lw.z);
        if (GEN) {
            image2(k, 0, dx, ex);
            image2(k, 1, dy, ey);
            image2(k, 2, dz, ez);
        }
        dx = __fadd2_rn(dx, ex);
        dy = __fadd2_rn(dy, ey);
        dz = __fadd2_rn(dz, ez);
        const float2 r2 = norm2(dx, dy, dz);
        const bool in0 = mj >= 0 && mi[0] != mj && (!GEN || m > dj[0]);
        const bool in1 = mj >= 0 && mi[1] != mj && (!GEN || m > dj[1]);
        const float2 a = lj[ti[0] + tj], b = lj[ti[1] + tj];
        float2 w = pair_w2<PART, EW, CJ>(k, r2, make_float2(kq.x * hj.w, kq.y * hj.w), make_float2(a.x, b.x),
                                         make_float2(a.y, b.y));
        w.x = in0 ? w.x : 0.f;
        w.y = in1 ? w.y : 0.f;
        np[0] += in0 ? 1 : 0;
        np[1] += in1 ? 1 : 0;
        gi[0] = __ffma2_rn(w, dx, gi[0]);
        gi[1] = __ffma2_rn(w, dy, gi[1]);
        gi[2] = __ffma2_rn(w, dz, gi[2]);
        // the j-side sums move to the lane that meets their atom next
        const int from = (lane + 1) & 31;
        const float2 ax = __ffma2_rn(w, dx, gj[0]), ay = __ffma2_rn(w, dy, gj[1]), az = __ffma2_rn(w, dz, gj[2]);
        gj[0] = make_float2(__shfl_sync(0xffffffffu, ax.x, from), __shfl_sync(0xffffffffu, ax.y, from));
        gj[1] = make_float2(__shfl_sync(0xffffffffu, ay.x, from), __shfl_sync(0xffffffffu, ay.y, from));
        gj[2] = make_float2(__shfl_sync(0xffffffffu, az.x, from), __shfl_sync(0xffffffffu, az.y, from));
    }
}

__device__ __forceinline__ void fix_add2(unsigned long long* a, float v, float w) {
    const unsigned long long f = fix_round<32>(v) + fix_round<32>(w);
    if (f) red_add(a, f);
}

// Bound by instruction issue (the six shuffles and the staged loads of a
// sub-step among it).  64 droplets of 64-1,024 molecules, 115 M pairs, per
// launch: 265 us with two tiles an item, 382 with one; two resident CTAs per
// SM (three spill: the same time there, 18 against 16 us on one droplet).
template <int PART, bool EW, bool CJ>
__global__ void __launch_bounds__(256, 2) k_tile_pairs(const __grid_constant__ DevSys s,
                                                             const __grid_constant__ Params p,
                                                             const __grid_constant__ PairConsts k, int step_off) {
    chain_enter();
    __shared__ float4 sh_h[8][32], sh_l[8][32];
    __shared__ int sh_m[8][32];
    __shared__ float2 s_lj[BOUNCE_MAXT * BOUNCE_MAXT];  // 12 c12, -6 c6 of each pair of types
    if (threadIdx.x < BOUNCE_MAXT * BOUNCE_MAXT)
        s_lj[threadIdx.x] = make_float2(12.f * p.c12[threadIdx.x], -6.f * p.c6[threadIdx.x]);
    __syncthreads();
    const DevTile& t = s.tl;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int cur = (int)((*s.step_base + step_off) & 1);
    const size_t n = (size_t)s.n;
    int npair = 0;
    for (int it = blockIdx.x * 8 + wl; it < t.nitems; it += gridDim.x * 8) {
        // (first atom of the i-tile, atoms of it and of the second tile << 16, first j, number of j)
        const int4 w = t.items[it];
        float2 h[3], l[3], kq;
        int mi[2], ti[2], i[2];
        bool vi[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            i[q] = w.x + q * t.tj + lane;
            // an i atom that does not exist, or takes no part (of a negative molecule), is placed
            // out of reach, without charge, and beyond every j: the minimum image folds its
            // coordinate back into a periodic box
            float4 hi = make_float4(PAIR_FAR, PAIR_FAR, PAIR_FAR, 0.f), lo = make_float4(0.f, 0.f, 0.f, 0.f);
            mi[q] = -1;
            vi[q] = lane < (q ? w.y >> 16 : w.y & 0xffff);
            if (vi[q]) mi[q] = s.mol[i[q]];
            vi[q] = mi[q] >= 0;
            if (vi[q]) {
                hi = s.phi[cur][i[q]];
                lo = s.plo[cur][i[q]];
            } else {
                i[q] = 1 << 30;
            }
            (&h[0].x)[q] = hi.x;
            (&h[1].x)[q] = hi.y;
            (&h[2].x)[q] = hi.z;
            (&l[0].x)[q] = lo.x;
            (&l[1].x)[q] = lo.y;
            (&l[2].x)[q] = lo.z;
            (&kq.x)[q] = -(p.kcoul * hi.w);
            ti[q] = type_of(lo) * BOUNCE_MAXT;
        }
        float2 gi[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        int np[2] = {0, 0};
        for (int jb = 0; jb < w.w; jb += 32) {
            const int nj = min(32, w.w - jb), j0 = w.z + jb;
            __syncwarp();
            // (padding: finite zeros, masked by the molecule)
            sh_h[wl][lane] = lane < nj ? s.phi[cur][j0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            sh_l[wl][lane] = lane < nj ? s.plo[cur][j0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            sh_m[wl][lane] = lane < nj ? s.mol[j0 + lane] : -1;
            __syncwarp();
            float2 gj[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            const int dj[2] = {i[0] - j0, i[1] - j0};  // staged atom of the lane's own i atoms
            const bool gen = p.periodic || j0 < w.x + 32 || ((w.y >> 16) && j0 < w.x + t.tj + 32);
            if (gen)
                tile_stage<PART, EW, CJ, true>(k, sh_h[wl], sh_l[wl], sh_m[wl], s_lj, h, l, kq, mi, ti, dj, gi, gj, np);
            else
                tile_stage<PART, EW, CJ, false>(k, sh_h[wl], sh_l[wl], sh_m[wl], s_lj, h, l, kq, mi, ti, dj, gi, gj, np);
            if (lane < nj) {
                const size_t jj = (size_t)(j0 + lane);
                fix_add2(t.acc + jj, -gj[0].x, -gj[0].y);
                fix_add2(t.acc + n + jj, -gj[1].x, -gj[1].y);
                fix_add2(t.acc + 2 * n + jj, -gj[2].x, -gj[2].y);
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (vi[q]) {
                fix_add(t.acc + i[q], (&gi[0].x)[q]);
                fix_add(t.acc + n + i[q], (&gi[1].x)[q]);
                fix_add(t.acc + 2 * n + i[q], (&gi[2].x)[q]);
                npair += np[q];
            }
    }
    npair = warp_sum_i(npair);
    if (lane == 0 && npair) atomicAdd(&s.cnt[PART == 3 ? CNT_SHORT_PAIRS : CNT_FULL_PAIRS], (unsigned long long)npair);
}

// One i-tile per item and one pair per instruction: batches and droplets with
// few items, where a second tile would only make the items longer.
template <int PART>
__global__ void __launch_bounds__(256) k_tile_pairs1(const __grid_constant__ DevSys s, const __grid_constant__ Params p, int step_off) {
    chain_enter();
    __shared__ float4 sh_h[8][32], sh_l[8][32];
    __shared__ int sh_m[8][32];
    __shared__ float s_c12[BOUNCE_MAXT * BOUNCE_MAXT], s_c6[BOUNCE_MAXT * BOUNCE_MAXT];
    if (threadIdx.x < BOUNCE_MAXT * BOUNCE_MAXT) {  // LJ table: per-lane type pairs read from shared memory
        s_c12[threadIdx.x] = p.c12[threadIdx.x];
        s_c6[threadIdx.x] = p.c6[threadIdx.x];
    }
    __syncthreads();
    const DevTile& t = s.tl;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int cur = (int)((*s.step_base + step_off) & 1);
    const size_t n = (size_t)s.n;
    int npair = 0;
    for (int it = blockIdx.x * 8 + wl; it < t.nitems; it += gridDim.x * 8) {
        const int4 w = t.items[it];  // (first i, number of i, first j, number of j): no second tile
        const bool vi = lane < w.y;
        const int i = w.x + lane;
        float4 hi = make_float4(0.f, 0.f, 0.f, 0.f), lo = hi;
        int mi = -1;
        if (vi) {
            hi = s.phi[cur][i];
            lo = s.plo[cur][i];
            mi = s.mol[i];
        }
        const float qi = p.kcoul * hi.w;
        const int ti = type_of(lo) * BOUNCE_MAXT;
        float gix = 0.f, giy = 0.f, giz = 0.f;
        for (int jb = 0; jb < w.w; jb += 32) {
            const int nj = min(32, w.w - jb), j0 = w.z + jb;
            __syncwarp();
            if (lane < nj) {
                sh_h[wl][lane] = s.phi[cur][j0 + lane];
                sh_l[wl][lane] = s.plo[cur][j0 + lane];
                sh_m[wl][lane] = s.mol[j0 + lane];
            } else {  // padding: finite zeros, masked below
                sh_h[wl][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                sh_l[wl][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                sh_m[wl][lane] = -1;
            }
            __syncwarp();
            float ax = 0.f, ay = 0.f, az = 0.f;  // j-side sum of stage atom (lane + k) mod 32
#pragma unroll 4
            for (int k = 0; k < 32; ++k) {
                const int m = (lane + k) & 31;
                const float4 hj = sh_h[wl][m], lj = sh_l[wl][m];
                const int mj = sh_m[wl][m];
                const float3 d = pair_disp(p, hi, lo, hj, lj);
                const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
                const bool in = mj >= 0 && mi >= 0 && mi != mj && j0 + m > i;
                const int tp = ti + type_of(lj);
                const float w0 = pairsum_w<PART>(p, in ? r2 : 1.f, qi * hj.w, s_c12[tp], s_c6[tp]);
                const float wv = in ? w0 : 0.f;
                npair += in ? 1 : 0;
                gix = fmaf(wv, d.x, gix);
                giy = fmaf(wv, d.y, giy);
                giz = fmaf(wv, d.z, giz);
                ax = fmaf(-wv, d.x, ax);
                ay = fmaf(-wv, d.y, ay);
                az = fmaf(-wv, d.z, az);
                // the j-side sum moves to the lane that meets its atom next
                const int from = (lane + 1) & 31;
                ax = __shfl_sync(0xffffffffu, ax, from);
                ay = __shfl_sync(0xffffffffu, ay, from);
                az = __shfl_sync(0xffffffffu, az, from);
            }
            if (lane < nj) {
                const size_t jj = (size_t)(j0 + lane);
                fix_add(t.acc + jj, ax);
                fix_add(t.acc + n + jj, ay);
                fix_add(t.acc + 2 * n + jj, az);
            }
        }
        if (vi) {
            fix_add(t.acc + i, gix);
            fix_add(t.acc + n + i, giy);
            fix_add(t.acc + 2 * n + i, giz);
        }
    }
    npair = warp_sum_i(npair);
    if (lane == 0 && npair) atomicAdd(&s.cnt[PART == 3 ? CNT_SHORT_PAIRS : CNT_FULL_PAIRS], (unsigned long long)npair);
}

// Accumulated sums added to out (n x 3, FP64); accumulators cleared.
__global__ void k_tile_collect(DevSys s, double* out) {
    const size_t n = (size_t)s.n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.n; i += gridDim.x * blockDim.x)
        for (int d = 0; d < 3; ++d) {
            const long long v = (long long)s.tl.acc[d * n + i];
            s.tl.acc[d * n + i] = 0ull;
            out[3 * (size_t)i + d] += (double)v * CL_UNFIX;
        }
}

}  // namespace

template <int PART, bool CJ>
static void launch_tiles(const DevSys& s, const Params& p, int step_off, int blocks, cudaStream_t st) {
    const PairConsts k = make_pair_consts(p);
    if (!s.tl.pairs) launch_chained(k_tile_pairs1<PART>, blocks, 256, 0, st, s, p, step_off);
    else if (p.ebeta > 0.f) launch_chained(k_tile_pairs<PART, true, CJ>, blocks, 256, 0, st, s, p, k, step_off);
    else launch_chained(k_tile_pairs<PART, false, CJ>, blocks, 256, 0, st, s, p, k, step_off);
}

void launch_tile_pairs(const DevSys& s, const Params& p, int step_off, int part, cudaStream_t st) {
    const int blocks = std::max(1, std::min(s.tl.blocks, (s.tl.nitems + 7) / 8));
    if (part != 3) launch_tiles<5, true>(s, p, step_off, blocks, st);
    else if (p.coul_jump) launch_tiles<3, true>(s, p, step_off, blocks, st);
    else launch_tiles<3, false>(s, p, step_off, blocks, st);
}

void launch_tile_collect(const DevSys& s, double* out, cudaStream_t st) {
    k_tile_collect<<<(s.n + 255) / 256, 256, 0, st>>>(s, out);
}
