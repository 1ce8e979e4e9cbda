// Candidate rows of the jump step and the pair sums (paper Sec. V, first
// paragraph: the partner J of atom i is drawn uniformly among the particles
// interacting with i).  Row of atom i: every atom j of another molecule with
// r_ij^2 < r_list^2 (FP64, minimum image), in ascending j.
//
// GPU design: a cell grid of edge >= r_list / 3 (counting sort: count, scan,
// scatter), then one warp per atom scans the cells that meet its r_list
// sphere, screens each candidate in FP32 from the high position parts and
// settles the few candidates near r_list exactly in FP64.  Accepted
// candidates set a bit in a per-warp bitmap over a window of atom indices
// centred on the atom's own (one per partner type with per-type-pair
// bounds, then a bitmap of the short-row members, r < r_off + skin);
// reading a bitmap back in word order yields the row already in ascending
// order (no sort), and duplicate visits of a cell are harmless.  Members
// outside the window take further passes (rare when atoms are numbered in
// spatial order).
// Every kernel returns at once unless a rebuild is pending (the step kernel
// raises the flag when an atom has moved more than skin/2 since the last
// build), so the sequence can sit in a captured CUDA graph.  Two launches:
// k_bins (counts, scan, scatter into cell order; it bins the clusters' columns
// too), rows (the CTA finishing last clears the flag).
#include <algorithm>

#include "common.cuh"

namespace {

constexpr int ROWS_T = 128, ROWS_CTAS = 7;  // threads of a row CTA, CTAs of an SM (72 registers)
constexpr int BIN_CTAS = 8, BIN_NT = 1024, BIN_PASS = 4;  // k_bins: CTAs, threads of each, atoms in flight per thread
constexpr int RANGE_MAX = 128;  // cell-row runs per atom (<= 2 (2*3+1)^2 = 98)

// Entry of a gated rebuild kernel: after its predecessor in the chain, is a
// rebuild due (or forced)?
__device__ __forceinline__ bool pending(const DevSys& s, int force) {
    chain_enter();
    return force || *s.rebuild;
}

__device__ __forceinline__ void cell_of(const DevSys& s, const Params& p, float4 hi, int& cx, int& cy, int& cz) {
    if (p.periodic) {
        cx = min(max((int)(hi.x * s.ihx), 0), s.ncx - 1);
        cy = min(max((int)(hi.y * s.ihy), 0), s.ncy - 1);
        cz = min(max((int)(hi.z * s.ihz), 0), s.ncz - 1);
    } else {
        cx = min(max((int)floorf((hi.x - s.ox) * s.ihx), 0), s.ncx - 1);
        cy = min(max((int)floorf((hi.y - s.oy) * s.ihy), 0), s.ncy - 1);
        cz = min(max((int)floorf((hi.z - s.oz) * s.ihz), 0), s.ncz - 1);
    }
}

// True in the one CTA of the grid that finishes last (all others have
// completed their global writes); that CTA resets the counter to zero.
__device__ bool last_cta(unsigned int* ctr) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(ctr, 1u) == gridDim.x - 1;
        if (last) atomicExch(ctr, 0u);
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Exclusive scan of nc counts by one CTA into start (nc + 1 values) and fill;
// resets the counts to zero for the next rebuild.  Four counts to a thread, in
// one word of 16 bytes: the 10,000 cells of a box of 27,783 atoms are three
// trips to memory, not ten.
__device__ void bins_scan(int* count, int* start, int* fill, int nc) {
    __shared__ int warp_tot[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int carry = 0;
    for (int base = 0; base < nc; base += BIN_NT * 4) {
        const int c0 = base + threadIdx.x * 4;
        const bool whole = c0 + 4 <= nc;
        int4 v = make_int4(0, 0, 0, 0);  // (read past L1: written by other CTAs' atomics)
        if (whole) {
            v = __ldcg((const int4*)(count + c0));
        } else if (c0 < nc) {
            v.x = __ldcg(count + c0);
            if (c0 + 1 < nc) v.y = __ldcg(count + c0 + 1);
            if (c0 + 2 < nc) v.z = __ldcg(count + c0 + 2);
        }
        const int sum = v.x + v.y + v.z + v.w;
        int x = sum;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_tot[w] = x;
        __syncthreads();
        int t = warp_tot[lane];  // (BIN_NT / 32 = 32 warps)
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        const int before = __shfl_sync(0xffffffffu, t, max(w - 1, 0));
        int4 e;
        e.x = carry + x - sum + (w ? before : 0);
        e.y = e.x + v.x;
        e.z = e.y + v.y;
        e.w = e.z + v.z;
        carry += __shfl_sync(0xffffffffu, t, 31);
        if (whole) {
            *(int4*)(start + c0) = e;
            *(int4*)(fill + c0) = e;
            *(int4*)(count + c0) = make_int4(0, 0, 0, 0);
        } else if (c0 < nc) {
            const int f[3] = {e.x, e.y, e.z};
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (c0 + k < nc) {
                    start[c0 + k] = f[k];
                    fill[c0 + k] = f[k];
                    count[c0 + k] = 0;
                }
        }
        __syncthreads();  // warp_tot is read
    }
    if (threadIdx.x == 0) start[nc] = carry;
}

// Atom i goes into the cells (ROWS_FILTER: only the types some jump row can hold).
__device__ __forceinline__ bool in_cells(const DevSys& s, const Params& p, int mode, int i) {
    return !(mode & ROWS_FILTER) || ((p.jcells >> s.type[i]) & 1);
}

__device__ __forceinline__ int column_of(const DevClu& c, const Params& p, float4 hi) {
    int cx, cy;
    if (p.periodic) {
        cx = min(max((int)(hi.x * c.ihx), 0), c.ncx - 1);
        cy = min(max((int)(hi.y * c.ihy), 0), c.ncy - 1);
    } else {
        cx = min(max((int)floorf((hi.x - c.ox) * c.ihx), 0), c.ncx - 1);
        cy = min(max((int)floorf((hi.y - c.oy) * c.ihy), 0), c.ncy - 1);
    }
    return cy * c.ncx + cx;
}

// All threads of a cluster of CTAs; what they wrote before is visible after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Counting sort of the atoms into the row builder's cells (BIN_CELLS) and the
// clusters' columns (BIN_COLUMNS, arbitrary order inside a column), gated by
// their own flags: counts, their scan and the scatter in one launch, a
// cluster of eight CTAs for each of the two, whose barriers part the phases.
// The two counts, the two scatters and their launches apart cost a step four
// gates of ~1.1 us when nothing is due.
__global__ void __launch_bounds__(BIN_NT) k_bins(const __grid_constant__ DevSys s, const __grid_constant__ Params p,
                                                 int step_off, int force, int which, int mode) {
    chain_enter();
    const bool columns = which == BIN_COLUMNS || blockIdx.x >= BIN_CTAS;
    if (!(force || *(columns ? s.cl.rebuild : s.rebuild))) return;  // the same for the whole cluster
    const int rank = blockIdx.x % BIN_CTAS, cur = (int)((*s.step_base + step_off) & 1);
    const DevClu& c = s.cl;
    int* count = columns ? c.col_count : s.cell_count;
    int* fill = columns ? c.col_fill : s.cell_fill;
    auto bin_of = [&](int i, float4 hi) {
        if (columns) return column_of(c, p, hi);
        int cx, cy, cz;
        cell_of(s, p, hi, cx, cy, cz);
        return (cz * s.ncy + cy) * s.ncx + cx;
    };
    constexpr int STEP = BIN_CTAS * BIN_NT;
    for (int i0 = rank * BIN_NT + threadIdx.x; i0 < s.n; i0 += BIN_PASS * STEP) {
        int b[BIN_PASS];
#pragma unroll
        for (int u = 0; u < BIN_PASS; ++u) {
            const int i = i0 + u * STEP;
            b[u] = i < s.n && (columns || in_cells(s, p, mode, i)) ? bin_of(i, s.phi[cur][i]) : -1;
        }
#pragma unroll
        for (int u = 0; u < BIN_PASS; ++u)
            if (b[u] >= 0) atomicAdd(&count[b[u]], 1);
    }
    cluster_sync();
    if (rank == 0)
        bins_scan(count, columns ? c.col_start : s.cell_start, fill, columns ? c.ncol : s.ncx * s.ncy * s.ncz);
    cluster_sync();
    for (int i0 = rank * BIN_NT + threadIdx.x; i0 < s.n; i0 += BIN_PASS * STEP) {
        int b[BIN_PASS];
        float4 hi[BIN_PASS];
#pragma unroll
        for (int u = 0; u < BIN_PASS; ++u) {
            const int i = i0 + u * STEP;
            b[u] = -1;
            if (i < s.n && (columns || in_cells(s, p, mode, i))) {
                hi[u] = s.phi[cur][i];
                b[u] = bin_of(i, hi[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < BIN_PASS; ++u)
            if (b[u] >= 0) b[u] = atomicAdd(&fill[b[u]], 1);
#pragma unroll
        for (int u = 0; u < BIN_PASS; ++u) {
            const int i = i0 + u * STEP;
            if (b[u] < 0) continue;
            if (columns) {
                c.col_atoms[b[u]] = i;
            } else {
                s.cell_phi[b[u]] = make_float4(hi[u].x, hi[u].y, hi[u].z, __int_as_float(i));
                s.cell_mt[b[u]] = make_int2(s.mol[i], s.type[i]);
            }
        }
    }
}

__device__ __forceinline__ bool in_list_fp64(const DevSys& s, const Params& p, int cur, int i, int j) {
    return exact_r2(s, p, cur, i, j) < p.rlist2_d;
}

// An FP32 minimum-image choice can differ from the FP64 one only when a
// component sits near half a box edge.
__device__ __forceinline__ bool image_ambiguous(const Params& p, float4 hi, float4 hj) {
    float fx = fabsf((hi.x - hj.x) * p.invL[0]), fy = fabsf((hi.y - hj.y) * p.invL[1]),
          fz = fabsf((hi.z - hj.z) * p.invL[2]);
    fx -= floorf(fx);
    fy -= floorf(fy);
    fz -= floorf(fz);
    return fabsf(fx - 0.5f) < 1e-4f || fabsf(fy - 0.5f) < 1e-4f || fabsf(fz - 0.5f) < 1e-4f;
}

// Can that choice decide a membership?  Not when the screening band ends below 0.4999 of the shortest edge: a
// component that near half an edge is then beyond r_list under either image.  (Warp-uniform, once per kernel: the
// test was a fifth of the work per candidate.)
__device__ __forceinline__ bool image_matters(const Params& p) {
    const float h = 0.4999f * fminf(p.Lhi[0], fminf(p.Lhi[1], p.Lhi[2]));
    return p.periodic && !(p.rlist2_hi < h * h);
}

// Candidate runs of atom i (one warp): up to two contiguous runs of cells
// per (z, y) cell row meeting the r_list sphere (periodic wrap), each a
// contiguous run of atoms in the cell-sorted arrays; rb / rl / rp receive
// their starts less their prefixes, their lengths and their exclusive
// prefixes, the return value is the number of candidates and nr the number of
// runs (none of them empty).
__device__ int candidate_runs(const DevSys& s, const Params& p, float4 hi, int* rb, int* rl, int* rp, int& nr) {
    const int lane = threadIdx.x & 31;
    // unclamped cell coordinates of atom i
    const float fx = p.periodic ? hi.x * s.ihx : (hi.x - s.ox) * s.ihx;
    const float fy = p.periodic ? hi.y * s.ihy : (hi.y - s.oy) * s.ihy;
    const float fz = p.periodic ? hi.z * s.ihz : (hi.z - s.oz) * s.ihz;
    int cx, cy, cz;
    cell_of(s, p, hi, cx, cy, cz);
    // geometric culling is valid unless atom i sits outside a droplet grid
    const bool cull = p.periodic || (fx >= 0.f && fy >= 0.f && fz >= 0.f && fx < (float)s.ncx &&
                                     fy < (float)s.ncy && fz < (float)s.ncz);
    const float rc2 = p.rcull * p.rcull;
    // axes narrower than the stencil are scanned once, without culling or wrap
    const bool fullz = s.ncz <= 2 * s.mz + 1, fully = s.ncy <= 2 * s.my + 1, fullx = s.ncx <= 2 * s.mx + 1;
    const int z0 = fullz ? 0 : cz - s.mz, z1 = fullz ? s.ncz - 1 : cz + s.mz;
    const int y0 = fully ? 0 : cy - s.my, y1 = fully ? s.ncy - 1 : cy + s.my;
    // 1) lanes compute the candidate ranges of all (z, y) cell rows in
    //    parallel: up to two contiguous runs of cells per row (periodic
    //    wrap), each a contiguous run of atoms in the cell-sorted array
    const int nzr = z1 - z0 + 1, nyr = y1 - y0 + 1, nrows = nzr * nyr;
    const uint32_t iny = 65536u / nyr + 1u;  // r / nyr = r iny >> 16 for the r < 128 there are
    int nr_tot = 0;
    for (int r0 = 0; r0 < nrows; r0 += 32) {
        const int r = r0 + lane;
        int b0 = 0, l0 = 0, b1 = 0, l1 = 0;
        if (r < nrows) {
            const int rz = r * iny >> 16, zu = z0 + rz, yu = y0 + r - rz * nyr;
            int zz = zu, yy = yu;
            bool ok = true;
            if (!fullz) {
                if (p.periodic) zz = zu < 0 ? zu + s.ncz : zu >= s.ncz ? zu - s.ncz : zu;
                else ok = zu >= 0 && zu < s.ncz;
            }
            if (!fully) {
                if (p.periodic) yy = yu < 0 ? yu + s.ncy : yu >= s.ncy ? yu - s.ncy : yu;
                else ok = ok && yu >= 0 && yu < s.ncy;
            }
            float gz = 0.f, gy = 0.f;
            if (cull && !fullz) gz = fmaxf(fmaxf((float)zu - fz, fz - (float)(zu + 1)), 0.f) * s.hz;
            if (cull && !fully) gy = fmaxf(fmaxf((float)yu - fy, fy - (float)(yu + 1)), 0.f) * s.hy;
            const float g2 = gz * gz + gy * gy;
            if (ok && g2 <= rc2) {
                int xa, xb;
                if (fullx) {
                    xa = 0;
                    xb = s.ncx - 1;
                } else if (cull) {
                    const float hw = sqrtf(rc2 - g2) * s.ihx;
                    xa = max((int)floorf(fx - hw), cx - s.mx);
                    xb = min((int)floorf(fx + hw), cx + s.mx);
                } else {
                    xa = cx - s.mx;
                    xb = cx + s.mx;
                }
                const int rowc = (zz * s.ncy + yy) * s.ncx;
                int ca[3], cb[3], nrr = 0;
                if (fullx) {
                    ca[0] = xa; cb[0] = xb; nrr = 1;
                } else if (p.periodic) {
                    if (xa < 0) { ca[nrr] = xa + s.ncx; cb[nrr] = s.ncx - 1; ++nrr; xa = 0; }
                    if (xb >= s.ncx) { ca[nrr] = 0; cb[nrr] = xb - s.ncx; ++nrr; xb = s.ncx - 1; }
                    if (xa <= xb) { ca[nrr] = xa; cb[nrr] = xb; ++nrr; }
                } else {
                    xa = max(xa, 0);
                    xb = min(xb, s.ncx - 1);
                    if (xa <= xb) { ca[0] = xa; cb[0] = xb; nrr = 1; }
                }
                if (nrr > 0) {
                    b0 = s.cell_start[rowc + ca[0]];
                    l0 = s.cell_start[rowc + cb[0] + 1] - b0;
                }
                if (nrr > 1) {
                    b1 = s.cell_start[rowc + ca[1]];
                    l1 = s.cell_start[rowc + cb[1] + 1] - b1;
                }
                if (nrr > 2) {  // both wraps: the span covers the whole row
                    b0 = s.cell_start[rowc];
                    l0 = s.cell_start[rowc + s.ncx] - b0;
                    l1 = 0;
                }
            }
        }
        // compact non-empty runs into the per-warp list, in row order
        const bool h0 = l0 > 0, h1 = l1 > 0;
        const int cnt = (int)h0 + (int)h1;
        int x = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        int pos = nr_tot + x - cnt;
        if (h0 && pos < RANGE_MAX) { rb[pos] = b0; rl[pos] = l0; ++pos; }
        if (h1 && pos < RANGE_MAX) { rb[pos] = b1; rl[pos] = l1; }
        nr_tot += __shfl_sync(0xffffffffu, x, 31);
    }
    nr_tot = min(nr_tot, RANGE_MAX);
    __syncwarp();
    // 2) exclusive prefix of the run lengths
    int total_c = 0;
    for (int r0 = 0; r0 < nr_tot; r0 += 32) {
        const int r = r0 + lane;
        const int len = r < nr_tot ? rl[r] : 0;
        int x = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (r < nr_tot) {
            rp[r] = total_c + x - len;
            rb[r] -= total_c + x - len;
        }
        total_c += __shfl_sync(0xffffffffu, x, 31);
    }
    __syncwarp();
    nr = nr_tot;
    return total_c;
}

// Position of the set bit of rank r (0-based, r < popc(b)) in b.
__device__ __forceinline__ int select_bit(uint32_t b, int r) {
    int pos = 0;
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
        const int c = __popc(b & ((1u << half) - 1u));
        if (r >= c) {
            r -= c;
            b >>= half;
            pos += half;
        }
    }
    return pos;
}

// Writes the set bits of a warp's bitmap, in ascending order, as indices to
// row[0 .. cap), returns their count (which may exceed cap; cap may be zero or
// negative, then nothing is written) and leaves the bitmap clear; word w of it
// stands for atoms 32 (wbase + w) .. 32 (wbase + w) + 31, and nwords is a
// multiple of 4.  Passes of 128 words, four to a lane: a prefix of their
// popcounts, then the pass's set bits are spread over the lanes, 32 at a time:
// output k finds its lane by a shuffle search over the prefix, its word by the
// lane's own three partial counts and its bit by a popcount halving search, so
// the stores are contiguous and the cost follows the number of set bits.
// (A row of 420 members among 12,288 atoms has some 35 set bits to 64 words:
// one word to a lane left half of the outputs of each pass idle.)
__device__ int expand_bitmap(uint32_t* bm, int nwords, int* row, int cap, int wbase = 0) {
    const int lane = threadIdx.x & 31;
    int total = 0;
    for (int w0 = 0; w0 < nwords; w0 += 128) {
        const int w = w0 + 4 * lane;
        uint4 b = make_uint4(0u, 0u, 0u, 0u);
        if (w < nwords) b = *(const uint4*)(bm + w);
        const uint32_t c1 = __popc(b.x), c2 = c1 + __popc(b.y), c3 = c2 + __popc(b.z);
        const int c = c3 + __popc(b.w);
        if (!__any_sync(0xffffffffu, c != 0)) continue;
        const uint32_t part = c1 << 8 | c2 << 16 | c3 << 24;  // set bits of the lane before each of its words
        int x = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const int excl = x - c;  // set bits of this pass before the lane's words
        const int tc = __shfl_sync(0xffffffffu, x, 31);
        for (int k0 = 0; k0 < tc; k0 += 32) {
            const int k = k0 + lane;
            // last lane l with excl_l <= k (the lanes before it hold fewer than k + 1 bits)
            int l = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int e = __shfl_sync(0xffffffffu, excl, l + step);
                if (e <= k) l += step;
            }
            const uint32_t pl = __shfl_sync(0xffffffffu, part, l);
            uint32_t r = k - __shfl_sync(0xffffffffu, excl, l);
            const int q = (r >= (pl >> 8 & 255u)) + (r >= (pl >> 16 & 255u)) + (r >= pl >> 24);
            r -= __byte_perm(pl, 0u, 0x4440 | q);
            const int pos = total + k;
            if (k < tc && pos < cap) {
                const int v = w0 + 4 * l + q;
                row[pos] = ((wbase + v) << 5) + select_bit(bm[v], r);
            }
        }
        total += tc;
        __syncwarp();
        if (c) *(uint4*)(bm + w) = make_uint4(0u, 0u, 0u, 0u);
    }
    return total;
}

// Member test of candidate j for atom i at r_list: FP32 screen on the high
// parts, settled in FP64 inside the band around r_list or when the minimum
// image is ambiguous in FP32.  r2 receives the FP32 distance squared.
__device__ __forceinline__ bool row_member(const DevSys& s, const Params& p, int cur, int i, float4 hi, float4 hj,
                                           int j, bool images, float& r2) {
    float dx = hi.x - hj.x, dy = hi.y - hj.y, dz = hi.z - hj.z;
    if (p.periodic) {
        dx -= rintf(dx * p.invL[0]) * p.Lhi[0];
        dy -= rintf(dy * p.invL[1]) * p.Lhi[1];
        dz -= rintf(dz * p.invL[2]) * p.Lhi[2];
    }
    r2 = dx * dx + dy * dy + dz * dz;
    const bool in = r2 < p.rlist2_lo;
    if ((in || r2 > p.rlist2_hi) && !(images && image_ambiguous(p, hi, hj))) return in;
    return in_list_fp64(s, p, cur, i, j);
}

// One block of 32 candidates of a warp: lane l holds candidate t0 + l.
struct Cand {
    float4 h;  // position (high parts) and index
    int2 mt;   // molecule, type
    bool on;
};

// Candidate t0 + lane: r0 is the run that holds candidate t0 and moves on to
// the one of t0 + 32.  The runs are not empty, so at most 32 of them start in
// (t0, t0 + 32]: one bit each, and a lane's run is a popcount away (a scan
// along the prefixes per lane cost a dependent shared load and a divergent
// branch per step).  Both loads go out at once, a block ahead of their use.
__device__ __forceinline__ Cand candidate(const DevSys& s, const int* rb, const int* rp, int nr, int total, int t0,
                                          int& r0) {
    const int lane = threadIdx.x & 31;
    Cand c;
    c.h = make_float4(0.f, 0.f, 0.f, 0.f);
    c.mt = make_int2(0, 0);
    c.on = t0 + lane < total;
    const int d = r0 + 1 + lane < nr ? rp[r0 + 1 + lane] - t0 - 1 : 32;
    const uint32_t starts = __reduce_or_sync(0xffffffffu, d < 32 ? 1u << d : 0u);
    if (c.on) {
        const int idx = t0 + lane + rb[r0 + __popc(starts & ((1u << lane) - 1u))];
        c.h = s.cell_phi[idx];
        c.mt = s.cell_mt[idx];
    }
    r0 += __popc(starts);
    return c;
}

// Rows of the cell-list builder, one warp per atom.  Bounded by its
// instructions (75% of the issue slots): the scan of the candidates, of whose
// cells the sphere fills two thirds, and the reading back of the bitmaps, half
// each.  A block of candidates ahead in registers, one record of position,
// index, molecule and type instead of four dependent loads, a popcount instead
// of a search for the run, and the image test only where it can matter took a
// build of 12,288 atoms (419 members a row) from 175 to 84 us, of 27,783 from
// 380 to 175, of 648 from 53 to 27 (there the chain of one atom's warp).  The warp's bitmaps (one
// per partner type with per-type-pair bounds, and one for the short rows)
// cover a window of `ww` words of atom indices centred on the atom's own
// index: reading them back in word order yields the row in ascending order
// without a sort.  The first pass screens the candidates, sets the bits of
// the members inside the window and counts, per type, the members below and
// above it; the window's members go to their final place in the row at
// once.  Members outside the window (index order far from spatial order)
// take further passes over windows below, then above it, each screening the
// candidates again; systems numbered in spatial order need one pass, and a
// window that spans every atom always does.
// mode: ROWS_ALL builds every row; ROWS_ACTIVE leaves the rows of atoms
// whose type has L* = 0 empty (they never propose: valid while the pair sums
// run over clusters or tiles and no short rows exist); ROWS_IDLE builds only
// those rows, at the current positions, keeping the reference positions and
// the rebuild flag of the last build (completing ROWS_ACTIVE rows for the
// energy, histogram and gradient entry points, which read every row);
// ROWS_READER builds every row the same way, into the readers' own row
// buffers.  ROWS_FILTER (with ROWS_ALL or ROWS_ACTIVE): the rows of the
// jump step keep only the partner types of the row's atom (Params::jpart),
// and the cells hold only the types some row can hold.
__global__ void __launch_bounds__(ROWS_T, ROWS_CTAS) k_rows_warp(DevSys s, Params p, int step_off, int force, int ww, int mode_in) {
    if (!pending(s, force)) return;
    extern __shared__ uint32_t smem_bm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int nwords = (s.n + 31) >> 5;
    const int nbm = p.typed ? p.n_types : 1;
    const bool has_short = p.rshort2 < INFINITY;  // only when one window spans every atom
    const int nb = nbm + (has_short ? 1 : 0);
    const int per_warp = nb * ww + 3 * RANGE_MAX;
    uint32_t* bm = smem_bm + (size_t)warp * per_warp;
    uint32_t* bs = bm + (size_t)nbm * ww;  // the short-row bitmap (has_short)
    int* rb = (int*)(bm + (size_t)nb * ww);
    int* rl = rb + RANGE_MAX;
    int* rp = rl + RANGE_MAX;
    const int cur = (int)((*s.step_base + step_off) & 1);
    const int mode = mode_in & 7;
    const bool filt = (mode_in & ROWS_FILTER) != 0;
    // ROWS_IDLE and ROWS_READER builds leave the reference positions, the
    // rebuild flag and the rebuild count to the run's own builds
    const bool own = mode != ROWS_IDLE && mode != ROWS_READER;
    const bool images = image_matters(p);
    if (blockIdx.x == 0 && threadIdx.x == 0 && own) atomicAdd(&s.cnt[CNT_REBUILDS], 1ull);
    // the bitmaps start clear; reading one back clears the words it touched
    for (int w = lane; w < nb * ww; w += 32) bm[w] = 0u;
    __syncwarp();
    // When the pair sums run over clusters or tiles, the rows serve only the
    // jump step, and an atom whose type has the bound L* = 0 never proposes
    // (its Poisson mean is 0).  act_order lists the atoms that can propose,
    // then the others: ROWS_ACTIVE builds the rows of the first n_act (the
    // others get empty rows and their reference positions), ROWS_IDLE the
    // rows of the rest; the warps stride over the listed atoms only, so the
    // work stays balanced whatever the order of the atom types.
    const bool split =
        mode != ROWS_ALL && mode != ROWS_READER && (s.cl.on || s.tl.on) && !has_short && s.act_order != nullptr;
    const int t0 = split && mode == ROWS_IDLE ? s.n_act : 0;
    const int t1 = split && mode == ROWS_ACTIVE ? s.n_act : s.n;
    if (split && mode == ROWS_ACTIVE)
        for (int t = s.n_act + blockIdx.x * blockDim.x + threadIdx.x; t < s.n; t += gridDim.x * blockDim.x) {
            const int i = s.act_order[t];
            if (p.typed)
                for (int u = 0; u < nbm; ++u) s.nseg[(size_t)i * BOUNCE_MAXT + u] = 0;
            s.nlong[i] = 0;
            s.nshort[i] = 0;
            s.refx[i] = s.qx[cur][i];
            s.refy[i] = s.qy[cur][i];
            s.refz[i] = s.qz[cur][i];
        }
    for (int t = t0 + blockIdx.x * wpb + warp; t < t1; t += gridDim.x * wpb) {
        const int i = split ? s.act_order[t] : t;
        const float4 hi = s.phi[cur][i];
        const int mi = s.mol[i];
        const int pm = filt ? p.jpart[s.type[i]] : -1;  // partner types of the row (all without the filter)
        int nr_tot;
        const int total_c = candidate_runs(s, p, hi, rb, rl, rp, nr_tot);
        __syncwarp();
        // window A: ww words centred on the atom's word, inside [0, nwords)
        const int wa = max(0, min((i >> 5) - ww / 2, nwords - ww));
        const int wz = min(wa + ww, nwords);
        int below[BOUNCE_MAXT], above[BOUNCE_MAXT];
#pragma unroll
        for (int t = 0; t < BOUNCE_MAXT; ++t) below[t] = above[t] = 0;
        int wmin = nwords, wmax = -1;  // words of the members outside the window
        int ulo = ww, uhi = -1;        // window words the members touched
        int run = 0;
        Cand nx = candidate(s, rb, rp, nr_tot, total_c, 0, run);
        for (int t0 = 0; t0 < total_c; t0 += 32) {
            const Cand c = nx;
            nx = candidate(s, rb, rp, nr_tot, total_c, t0 + 32, run);
            const int j = __float_as_int(c.h.w);
            float r2;
            if (!c.on || c.mt.x == mi || !((pm >> c.mt.y) & 1) || !row_member(s, p, cur, i, hi, c.h, j, images, r2))
                continue;
            const int ty = p.typed ? c.mt.y : 0, w = j >> 5;
            if (w < wa) {
                wmin = min(wmin, w);
#pragma unroll
                for (int u = 0; u < BOUNCE_MAXT; ++u) below[u] += u == ty;
            } else if (w >= wz) {
                wmax = max(wmax, w);
#pragma unroll
                for (int u = 0; u < BOUNCE_MAXT; ++u) above[u] += u == ty;
            } else {
                atomicOr(&bm[(size_t)ty * ww + (w - wa)], 1u << (j & 31));
                ulo = min(ulo, w - wa);
                uhi = max(uhi, w - wa);
                // short rows: r < r_off + skin (rshort2 carries a 1e-4 margin)
                if (has_short && r2 < p.rshort2) atomicOr(&bs[w - wa], 1u << (j & 31));
            }
        }
        wmin = __reduce_min_sync(0xffffffffu, wmin);
        wmax = __reduce_max_sync(0xffffffffu, wmax);
        ulo = __reduce_min_sync(0xffffffffu, ulo);
        uhi = __reduce_max_sync(0xffffffffu, uhi);
        const bool outside = wmax >= 0 || wmin < nwords;
        if (outside) {
#pragma unroll
            for (int u = 0; u < BOUNCE_MAXT; ++u) {
                below[u] = __reduce_add_sync(0xffffffffu, below[u]);
                above[u] = __reduce_add_sync(0xffffffffu, above[u]);
            }
        }
        __syncwarp();
        // window A in place (touched words only): type group u starts at
        // seg[u], its members below the window first
        ulo &= ~3;
        const int nu = uhi >= ulo ? ((uhi - ulo) | 3) + 1 : 0;  // (ww is a multiple of 4)
        int* row = s.rows + (size_t)i * s.cap;
        int inside[BOUNCE_MAXT], seg[BOUNCE_MAXT], total = 0;
#pragma unroll
        for (int u = 0; u < BOUNCE_MAXT; ++u) {
            seg[u] = total;
            inside[u] = 0;
            if (u >= nbm) continue;
            const int off = total + below[u];
            inside[u] = expand_bitmap(bm + (size_t)u * ww + ulo, nu, row + off, s.cap - off, wa + ulo);
            total = off + inside[u] + above[u];
        }
        const int ns = has_short ? expand_bitmap(bs + ulo, nu, s.srows + (size_t)i * s.caps, s.caps, wa + ulo) : 0;
        __syncwarp();
        // further windows: below window A (ascending from the lowest member), then above it
        if (outside)
            for (int side = 0; side < 2; ++side) {
                int w0 = side == 0 ? wmin : wz;
                const int wend = side == 0 ? wa : wmax + 1;
                int off[BOUNCE_MAXT];
#pragma unroll
                for (int u = 0; u < BOUNCE_MAXT; ++u) off[u] = seg[u] + (side == 0 ? 0 : below[u] + inside[u]);
                for (; w0 < wend; w0 += ww) {
                    const int w1 = min(w0 + ww, wend);
                    run = 0;
                    for (int t0 = 0; t0 < total_c; t0 += 32) {
                        const Cand c = candidate(s, rb, rp, nr_tot, total_c, t0, run);
                        const int j = __float_as_int(c.h.w);
                        const int w = j >> 5;
                        float r2;
                        if (!c.on || w < w0 || w >= w1 || c.mt.x == mi || !((pm >> c.mt.y) & 1) ||
                            !row_member(s, p, cur, i, hi, c.h, j, images, r2))
                            continue;
                        const int ty = p.typed ? c.mt.y : 0;
                        atomicOr(&bm[(size_t)ty * ww + (w - w0)], 1u << (j & 31));
                    }
                    __syncwarp();
                    for (int u = 0; u < nbm; ++u) {
                        int o = 0;
#pragma unroll
                        for (int v = 0; v < BOUNCE_MAXT; ++v) o = v == u ? off[v] : o;
                        const int c = expand_bitmap(bm + (size_t)u * ww, ((w1 - w0) + 3) & ~3, row + o, s.cap - o, w0);
#pragma unroll
                        for (int v = 0; v < BOUNCE_MAXT; ++v) off[v] += v == u ? c : 0;
                    }
                    __syncwarp();
                }
            }
        if (lane == 0) {
            if (p.typed)
                for (int u = 0; u < nbm; ++u) {
                    int c = 0;
#pragma unroll
                    for (int v = 0; v < BOUNCE_MAXT; ++v) c = v == u ? below[v] + inside[v] + above[v] : c;
                    s.nseg[(size_t)i * BOUNCE_MAXT + u] = c;
                }
            s.nlong[i] = min(total, s.cap);
            if (total > s.cap) atomicOr(s.err, BERR_LIST_OVERFLOW);
            s.nshort[i] = min(ns, s.caps);
            if (ns > s.caps) atomicOr(s.err, BERR_SHORT_OVERFLOW);
            if (own) {
                s.refx[i] = s.qx[cur][i];
                s.refy[i] = s.qy[cur][i];
                s.refz[i] = s.qz[cur][i];
            }
        }
        __syncwarp();
    }
    if (last_cta(&s.done_ctr[1]) && own) *s.rebuild = 0;
}

// Rows of a batch of independent all-pairs replicas: every atom of the same
// replica outside the own molecule, ascending (no distance test: replicas
// have no cutoff), then the short rows and reference positions as above.
__global__ void k_rows_batch(DevSys s, Params p, int step_off, int force, int mode_in) {
    if (!pending(s, force)) return;
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const int cur = (int)((*s.step_base + step_off) & 1);
    const bool filt = (mode_in & ROWS_FILTER) != 0;
    const bool own = (mode_in & 7) != ROWS_IDLE && (mode_in & 7) != ROWS_READER;
    if (blockIdx.x == 0 && threadIdx.x == 0 && own) atomicAdd(&s.cnt[CNT_REBUILDS], 1ull);
    for (int i = blockIdx.x * wpb + (threadIdx.x >> 5); i < s.n; i += gridDim.x * wpb) {
        const int r = s.rep_of[i], b = s.rep_off[r], e = s.rep_off[r + 1], mi = s.mol[i];
        const int pm = filt ? p.jpart[s.type[i]] : -1;  // partner types of the row (all without the filter)
        int* row = s.rows + (size_t)i * s.cap;
        int total = 0;
        const int ngroups = p.typed ? p.n_types : 1;
        for (int tb = 0; tb < ngroups; ++tb) {  // typed rows: one pass per partner type
            const int before = total;
            for (int j0 = b; j0 < e; j0 += 32) {
                const int j = j0 + lane;
                const bool keep = j < e && s.mol[j] != mi && (!p.typed || s.type[j] == tb) && ((pm >> s.type[j]) & 1);
                const uint32_t m = __ballot_sync(0xffffffffu, keep);
                const int pos = total + __popc(m & ((1u << lane) - 1u));
                if (keep && pos < s.cap) row[pos] = j;
                total += __popc(m);
            }
            if (p.typed && lane == 0) s.nseg[(size_t)i * BOUNCE_MAXT + tb] = total - before;
        }
        __syncwarp();
        // short rows: ascending over the replica with the same high-part
        // screen as the cell-list builder (independent of the long row's order)
        const float4 hi = s.phi[cur][i];
        const int nl = min(total, s.cap);
        int ns = 0;
        int* srow = s.srows + (size_t)i * s.caps;
        for (int j0 = b; p.rshort2 < INFINITY && j0 < e; j0 += 32) {
            const int j = j0 + lane;
            bool keep = false;
            if (j < e && s.mol[j] != mi) {
                const float4 hj = s.phi[cur][j];
                const float dx = hi.x - hj.x, dy = hi.y - hj.y, dz = hi.z - hj.z;
                keep = dx * dx + dy * dy + dz * dz < p.rshort2;
            }
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int pos = ns + __popc(m & ((1u << lane) - 1u));
                if (pos < s.caps) srow[pos] = j;
            }
            ns += __popc(m);
        }
        if (lane == 0) {
            s.nlong[i] = nl;
            if (total > s.cap) atomicOr(s.err, BERR_LIST_OVERFLOW);
            s.nshort[i] = min(ns, s.caps);
            if (ns > s.caps) atomicOr(s.err, BERR_SHORT_OVERFLOW);
            if (own) {
                s.refx[i] = s.qx[cur][i];
                s.refy[i] = s.qy[cur][i];
                s.refz[i] = s.qz[cur][i];
            }
        }
        __syncwarp();
    }
    if (last_cta(&s.done_ctr[1]) && own) *s.rebuild = 0;
}

__global__ void k_flag_moved(DevSys s, Params p, int cur) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.n; i += gridDim.x * blockDim.x) {
        const double ex = s.qx[cur][i] - s.refx[i], ey = s.qy[cur][i] - s.refy[i], ez = s.qz[cur][i] - s.refz[i];
        if (((s.rows_move >> s.type[i]) & 1) && ex * ex + ey * ey + ez * ez > p.skin_half2) atomicOr(s.rebuild, 1);
    }
}

}  // namespace

void launch_flag_moved(const DevSys& s, const Params& p, int cur, cudaStream_t st) {
    k_flag_moved<<<(s.n + 255) / 256, 256, 0, st>>>(s, p, cur);
}

void launch_bins(const DevSys& s, const Params& p, int step_off, bool force, int which, int mode, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = which == (BIN_CELLS | BIN_COLUMNS) ? 2 * BIN_CTAS : BIN_CTAS;
    cfg.blockDim = BIN_NT;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = BIN_CTAS;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, k_bins, s, p, step_off, force ? 1 : 0, which, mode);
}

void launch_rebuild(const DevSys& s, const Params& p, int step_off, bool force, int window_words, size_t bitmap_bytes,
                    int mode, cudaStream_t st, bool binned) {
    const int f = force ? 1 : 0;
    if (s.rep_of) {
        const int wpb = 8;
        // (one wave of CTAs: the warps stride over the atoms, and the gate is cheap when nothing is due: a CTA
        // per eight atoms took 19 us to find that out on 104,000 atoms)
        launch_chained(k_rows_batch, std::min((s.n + wpb - 1) / wpb, 152 * 8), wpb * 32, 0, st, s, p, step_off, f, mode);
        return;
    }
    if (!binned) launch_bins(s, p, step_off, force, BIN_CELLS, mode, st);
    // Warp per atom, a grid-stride loop over one wave of CTAs where the launch may find nothing to do; a forced
    // build takes up to four waves, so that an SM which is done early gets another CTA (27,783 atoms: 196 -> 175 us).
    // CTAs of four warps, not eight: 418 -> 392 us there, 87.4 -> 84.0 us on 12,288 atoms.
    const int wpb = ROWS_T / 32;
    const size_t smem = bitmap_bytes / 8 * wpb;  // (bitmap_bytes: of eight warps)
    const int per_sm = std::max(1, std::min(ROWS_CTAS, (int)((227u << 10) / std::max<size_t>(smem, 1))));
    const int blocks = std::min((s.n + wpb - 1) / wpb, 152 * per_sm * (force ? 4 : 1));
    launch_chained(k_rows_warp, blocks, ROWS_T, smem, st, s, p, step_off, f, window_words, mode);
}

void nlist_set_smem_limit(size_t bytes) {
    cudaFuncSetAttribute(k_rows_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
