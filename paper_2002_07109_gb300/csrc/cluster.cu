// Pair sums over clusters of atoms (the F_0 share of every pair, Sec. IV.A /
// Sec. V, and BAOAB's full pair gradient), for systems with a finite cutoff.
//
// Build (three gated launches; each returns at once unless the cluster
// rebuild flag is raised -- the step kernel raises it when an atom has moved
// more than half the skin since the build):
//   1. k_bins (nlist.cu): the atoms counted into columns of a grid over (x, y),
//      the counts scanned, the atom indices scattered into column order; one
//      launch, which bins the candidate rows' cells too;
//   2. k_cl_sort: one CTA per column sorts its atoms by (z, index) (bitonic
//      sort in shared memory: the order, hence every cluster, is
//      deterministic), cuts them into clusters of BOUNCE_CL and writes the
//      slot-ordered copies of the split positions, the molecule ids, the slot
//      of every atom and the bounding box of every cluster;
//   3. k_cl_lists: one CTA per cluster I collects the atoms of the clusters
//      J >= I of the columns in reach that lie within the search radius of I's
//      box (minimum image per axis), in a fixed order, with the periodic image
//      of each.
// Prune (in the third launch, which its own flag opens too: the step kernel
// raises it when an atom has moved half the prune skin since the last prune):
// the entries of each list within r + prune skin of some atom of I at the
// current positions, so that the pair kernel reads a list close to the pairs
// it must evaluate while the outer lists, with a larger skin, are rebuilt
// rarely.  A CTA prunes the clusters whose lists it made itself, so that a
// barrier of the CTA parts the two; the CTA finishing last, after every other
// one has read the flags, clears them both.
// Pair kernel: one warp per work item (cluster I, a chunk of its pruned
// entries); lane = one list atom j, the 8 atoms
// of cluster I two at a time from shared memory.  Every unordered pair inside the
// cutoff is evaluated once (Newton's third law): the j-side sum of a lane is
// added once per item, the i-side sums are reduced over the warp at the end
// of the item, both into int64 fixed-point accumulators (2^-32 kcal/mol/A)
// rounded from FP32 by the int64 conversion: integer addition is
// associative, so the result does not depend on the order in which warps
// finish.
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "pairs.cuh"

namespace {

// Threads per CTA of the pair kernel and the resident CTAs per SM it is
// compiled for: 128 registers a thread, 16 warps per SM.  96 registers (20
// warps) spill: 123 against 109 us on the 98,304-atom box; 168 registers (12
// warps): 113 us.
constexpr int PAIRS_NT = 128, PAIRS_CTAS = 4;

constexpr int CL = BOUNCE_CL;
constexpr int EPW = BOUNCE_CL_EPW;
constexpr int SORT_NT = 256;
constexpr int NO_SHIFT = 13;  // image code (kx + 1) * 9 + (ky + 1) * 3 + (kz + 1) of k = 0
constexpr int PER_PAIR = 31;  // the pair's clusters may straddle half a box edge: minimum image per atom pair

__device__ __forceinline__ bool cl_pending(const DevSys& s, int force) {
    chain_enter();
    return force || *s.cl.rebuild;
}

// True in the one CTA of the grid that finishes last; it resets the counter.
__device__ bool cl_last_cta(unsigned int* ctr) {
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

// Order-preserving map of a float onto an unsigned key.
__device__ __forceinline__ uint32_t float_key(float z) {
    const uint32_t b = __float_as_uint(z);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// 2. one CTA per column (binned by k_bins): sort by (z, index), clusters, slots, boxes.
__global__ void __launch_bounds__(SORT_NT) k_cl_sort(DevSys s, Params p, int step_off, int force) {
    if (!cl_pending(s, force)) return;
    __shared__ unsigned long long key[BOUNCE_CL_MAXCOL];
    const DevClu& c = s.cl;
    const int tid = threadIdx.x;
    const int cur = (int)((*s.step_base + step_off) & 1);
    for (int col = blockIdx.x; col < c.ncol; col += gridDim.x) {
        const int b = c.col_start[col];
        int nc = c.col_start[col + 1] - b;
        if (nc > c.maxcol) {  // the column outgrew its capacity: the state is reported invalid
            if (tid == 0) atomicOr(s.err, BERR_LIST_OVERFLOW);
            nc = c.maxcol;
        }
        int P = 1;
        while (P < nc) P <<= 1;
        for (int t = tid; t < P; t += SORT_NT) {
            unsigned long long k = ~0ull;
            if (t < nc) {
                const int a = c.col_atoms[b + t];
                k = ((unsigned long long)float_key(s.phi[cur][a].z) << 32) | (uint32_t)a;
            }
            key[t] = k;
        }
        __syncthreads();
        for (int k = 2; k <= P; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = tid; t < P; t += SORT_NT) {
                    const int l = t ^ j;
                    if (l > t) {
                        const unsigned long long x = key[t], y = key[l];
                        if ((x > y) == ((t & k) == 0)) {
                            key[t] = y;
                            key[l] = x;
                        }
                    }
                }
                __syncthreads();
            }
        const int ncl = (nc + CL - 1) / CL;
        if (tid == 0) c.col_ncl[col] = ncl;
        for (int t = tid; t < ncl * CL; t += SORT_NT) {
            const int slot = (col * c.maxcl + t / CL) * CL + t % CL;
            if (t < nc) {
                const int a = (int)(uint32_t)(key[t] & 0xFFFFFFFFull);
                c.cl_atom[slot] = a;
                c.a2s[a] = slot;
                c.sphi[cur][slot] = s.phi[cur][a];
                c.splo[cur][slot] = s.plo[cur][a];
                c.smol[slot] = s.mol[a];
                const double qa = s.qx[cur][a], qb = s.qy[cur][a], qc = s.qz[cur][a];
                c.crefx[a] = qa;
                c.crefy[a] = qb;
                c.crefz[a] = qc;
                // the image of the wrapped copy in phi (the step kernel's wrap)
                c.cofx[a] = p.periodic ? p.Ld[0] * floor(qa / p.Ld[0]) : 0.0;
                c.cofy[a] = p.periodic ? p.Ld[1] * floor(qb / p.Ld[1]) : 0.0;
                c.cofz[a] = p.periodic ? p.Ld[2] * floor(qc / p.Ld[2]) : 0.0;
            } else {
                c.cl_atom[slot] = -1;
                c.smol[slot] = -1;
                c.sphi[cur][slot] = make_float4(0.f, 0.f, 0.f, 0.f);
                c.splo[cur][slot] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        for (int k = tid; k < ncl; k += SORT_NT) {
            float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f), hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
            for (int u = k * CL; u < min(nc, (k + 1) * CL); ++u) {
                const float4 h = s.phi[cur][(int)(uint32_t)(key[u] & 0xFFFFFFFFull)];
                lo.x = fminf(lo.x, h.x);
                lo.y = fminf(lo.y, h.y);
                lo.z = fminf(lo.z, h.z);
                hi.x = fmaxf(hi.x, h.x);
                hi.y = fmaxf(hi.y, h.y);
                hi.z = fmaxf(hi.z, h.z);
            }
            c.bb_lo[col * c.maxcl + k] = lo;
            c.bb_hi[col * c.maxcl + k] = hi;
        }
        __syncthreads();
    }
}

// Range of columns along one axis that a box [a, b] (extended by the search
// radius) meets: [lo, hi] on the unwrapped grid; `all` when it covers every
// column (periodic wrap would visit one twice).
__device__ __forceinline__ void column_span(int n, float a, float b, float org, float ih, int periodic, int& lo,
                                            int& hi, bool& all) {
    const float fa = (a - org) * ih, fb = (b - org) * ih;
    if (periodic) {
        lo = (int)floorf(fa);
        hi = (int)floorf(fb);
        all = hi - lo + 1 >= n;
        if (all) {
            lo = 0;
            hi = n - 1;
        }
    } else {
        lo = min(max((int)floorf(fa), 0), n - 1);
        hi = min(max((int)floorf(fb), 0), n - 1);
        all = false;
    }
}

// q_j - k L in split form (sh, sl: the high and low parts of k L): the high
// part rounded, its rounding error moved into the low part (two-sum), so the
// pair stays an exact split of the shifted coordinate.
__device__ __forceinline__ void shift_split(float& h, float& l, float sh, float sl) {
    const float t = h - sh;
    const float bb = t - h;
    const float err = (h - (t - bb)) + (-sh - bb);
    h = t;
    l = (l - sl) + err;
}

// 3a. neighbour lists (CTA per cluster I): every atom j of a cluster
// J >= I of the columns in reach whose distance to I's bounding box (minimum
// image per axis) is below the search radius, in a fixed order, as its slot
// with the periodic image of the pair (or the per-pair code when the pair's
// separation could reach half a box edge).  Every unordered pair of atoms
// inside the cutoff then appears once: in the list of the lower cluster, and
// for two atoms of one cluster with the lower slot as i.
//
// Bounded by the chain of one cluster (columns, boxes, atoms, each load
// waiting for the last), so the chain is kept short: the columns in reach are
// one prefix sum over the CTA's threads, the box tests run 128 clusters at a
// time over the columns' concatenation, those that pass queue up in a ring,
// and the atom tests take 64 queued clusters at a time, four loads in flight
// per thread.  Votes and counts of the warps, exchanged once per step, keep
// every entry in the order of (row, column, cluster, atom).  A warp per
// cluster that walked the columns one by one (six clusters of 32 lanes) took
// 97 us for 12,288 atoms, 120 us for 27,783 and 285 us for 98,304; this takes 31,
// 50 and 170.
constexpr int NB_NT = 128, NB_W = NB_NT / 32;  // threads and warps of a search or prune CTA
constexpr int NB_PASS = 4;                     // atoms (entries) in flight per thread
constexpr int NB_QUEUE = NB_PASS * NB_NT / CL;  // clusters of an atom-level step
constexpr int NB_RING = 256;                   // queued clusters: < NB_QUEUE left over + 128 new

__device__ __forceinline__ void cl_search(const DevSys& s, const Params& p, int step_off) {
    __shared__ int run_start[NB_NT], run_off[NB_NT];  // non-empty columns: first candidate, first cluster less it
    __shared__ uint32_t wsum[NB_W];
    __shared__ int ring[NB_RING];
    __shared__ int bcnt[2][NB_W];
    __shared__ uint32_t acnt[2][NB_PASS * NB_W];
    const DevClu& c = s.cl;
    const int tid = threadIdx.x, lane = tid & 31, wl = tid >> 5;
    const int ncl = c.ncol * c.maxcl;
    const int cur = (int)((*s.step_base + step_off) & 1);
    const float Lx = p.Lhi[0], Ly = p.Lhi[1], Lz = p.Lhi[2];
    const uint32_t below = (1u << lane) - 1u;
    bool overflow = false;
    int bpar = 0, apar = 0;  // the count buffers alternate: one barrier per step
    // the first clusters of all columns, then the second ones, ...: the unused slots of the columns come last
    for (int t = blockIdx.x; t < ncl; t += gridDim.x) {
        const int k = t / c.ncol, col = t - k * c.ncol, I = col * c.maxcl + k;
        if (k >= c.col_ncl[col]) {
            if (tid == 0) {
                c.lcnt[0][I] = 0;
                c.lcnt[1][I] = 0;
            }
            continue;
        }
        const float4 lo = c.bb_lo[I], hi = c.bb_hi[I];
        const float cx = 0.5f * (lo.x + hi.x), cy = 0.5f * (lo.y + hi.y), cz = 0.5f * (lo.z + hi.z);
        const float ex = 0.5f * (hi.x - lo.x), ey = 0.5f * (hi.y - lo.y), ez = 0.5f * (hi.z - lo.z);
        const float R = c.rsx[0];
        int xa, xb, ya, yb;
        bool xall, yall;
        column_span(c.ncx, lo.x - R, hi.x + R, p.periodic ? 0.f : c.ox, c.ihx, p.periodic, xa, xb, xall);
        column_span(c.ncy, lo.y - R, hi.y + R, p.periodic ? 0.f : c.oy, c.ihy, p.periodic, ya, yb, yall);
        const int nxs = xb - xa + 1, ncols = nxs * (yb - ya + 1);
        int m0 = 0, m1 = 0;          // entries so far
        int head = 0, tail = 0;      // ring: queued clusters
        // atom level over up to 64 queued clusters: thread = 8 q + t of each pass
        auto atoms = [&](int nq) {
            int sj[NB_PASS], mj[NB_PASS];
            float4 h[NB_PASS];
#pragma unroll
            for (int u = 0; u < NB_PASS; ++u) {
                const int q = u * (NB_NT / CL) + (tid >> 3);
                sj[u] = q < nq ? ring[(head + q) & (NB_RING - 1)] * CL + (tid & 7) : -1;
                mj[u] = -1;
                if (sj[u] >= 0) {
                    mj[u] = c.smol[sj[u]];
                    h[u] = c.sphi[cur][sj[u]];
                }
            }
            uint32_t bl[NB_PASS], bs[NB_PASS];
#pragma unroll
            for (int u = 0; u < NB_PASS; ++u) {
                bool inL = false, inS = false;
                int code = NO_SHIFT;
                if (mj[u] >= 0) {
                    float dx = h[u].x - cx, dy = h[u].y - cy, dz = h[u].z - cz;
                    if (p.periodic) {
                        const int kx = (int)rintf(dx * p.invL[0]);
                        const int ky = (int)rintf(dy * p.invL[1]);
                        const int kz = (int)rintf(dz * p.invL[2]);
                        dx -= kx * Lx;
                        dy -= ky * Ly;
                        dz -= kz * Lz;
                        // image code of q_j - k L (the kernel subtracts k L from q_j)
                        code = (kx + 1) * 9 + (ky + 1) * 3 + (kz + 1);
                        if (fabsf(dx) + 2.f * ex >= 0.49f * Lx || fabsf(dy) + 2.f * ey >= 0.49f * Ly ||
                            fabsf(dz) + 2.f * ez >= 0.49f * Lz)
                            code = PER_PAIR;
                    }
                    const float gx = fmaxf(fabsf(dx) - ex, 0.f), gy = fmaxf(fabsf(dy) - ey, 0.f),
                                gz = fmaxf(fabsf(dz) - ez, 0.f);
                    const float d2 = gx * gx + gy * gy + gz * gz;
                    inL = d2 < c.rs2[0];
                    inS = c.nlists > 1 && d2 < c.rs2[1];
                }
                bl[u] = __ballot_sync(0xffffffffu, inL);
                bs[u] = __ballot_sync(0xffffffffu, inS);
                sj[u] |= code << 27;
                if (lane == 0) acnt[apar][u * NB_W + wl] = __popc(bl[u]) | __popc(bs[u]) << 16;
            }
            __syncthreads();
            // entries of the passes and warps before, both lists packed
            const uint32_t v = lane < NB_PASS * NB_W ? acnt[apar][lane] : 0u;
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < NB_PASS * NB_W; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
#pragma unroll
            for (int u = 0; u < NB_PASS; ++u) {
                const uint32_t before = __shfl_sync(0xffffffffu, x - v, u * NB_W + wl);
                if (bl[u] >> lane & 1) {
                    const int pos = m0 + (int)(before & 0xffffu) + __popc(bl[u] & below);
                    if (pos < c.capj[0]) c.lst[0][(size_t)I * c.capj[0] + pos] = sj[u];
                }
                if (bs[u] >> lane & 1) {
                    const int pos = m1 + (int)(before >> 16) + __popc(bs[u] & below);
                    if (pos < c.capj[1]) c.lst[1][(size_t)I * c.capj[1] + pos] = sj[u];
                }
            }
            const uint32_t all = __shfl_sync(0xffffffffu, x, NB_PASS * NB_W - 1);
            m0 += all & 0xffffu;
            m1 += all >> 16;
            head += nq;
            apar ^= 1;
        };
        for (int cb = 0; cb < ncols; cb += NB_NT) {
            // the clusters J >= I of a column: all of them, or those from I on in I's own column
            int off = 0, len = 0;
            if (cb + tid < ncols) {
                const int ry = (cb + tid) / nxs, yy = ya + ry, xx = xa + (cb + tid) - ry * nxs;
                const int cyn = p.periodic ? (yy % c.ncy + c.ncy) % c.ncy : yy;
                const int cxn = p.periodic ? (xx % c.ncx + c.ncx) % c.ncx : xx;
                const int coln = cyn * c.ncx + cxn;
                const int k0 = coln > col ? 0 : k;
                len = coln >= col ? max(c.col_ncl[coln] - k0, 0) : 0;
                off = coln * c.maxcl + k0;
            }
            // prefix over the columns: candidates (low 24 bits) and non-empty
            // columns (the upper 8: up to NB_NT, which a signed word does not hold)
            static_assert(NB_NT < 256 && NB_NT * (BOUNCE_CL_MAXCOL / CL) < 1 << 24, "both counts fit their bits");
            const uint32_t v = (uint32_t)len | (len > 0 ? 1u << 24 : 0u);
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            __syncthreads();  // (the last batch's runs are read)
            if (lane == 31) wsum[wl] = x;
            __syncthreads();
            uint32_t total = 0u;
#pragma unroll
            for (int w = 0; w < NB_W; ++w) {
                if (w == wl) x += total;
                total += wsum[w];
            }
            x -= v;
            if (len > 0) {
                run_start[x >> 24] = (int)(x & 0xffffffu);
                run_off[x >> 24] = off - (int)(x & 0xffffffu);
            }
            const int nr = (int)(total >> 24), nt = (int)(total & 0xffffffu);
            __syncthreads();
            int t0 = 0;
            do {  // (once where no column has a cluster, for what is left in the ring)
                // cluster level: boxes within the search radius (minimum image per axis)
                const int tt = t0 + tid;
                bool near = false;
                int J = 0;
                if (tt < nt) {
                    int r = 0;  // last run with run_start <= tt
#pragma unroll
                    for (int st = NB_NT / 2; st > 0; st >>= 1)
                        if (r + st < nr && run_start[r + st] <= tt) r += st;
                    J = tt + run_off[r];
                    const float4 lj = c.bb_lo[J], hj = c.bb_hi[J];
                    float dx = cx - 0.5f * (lj.x + hj.x), dy = cy - 0.5f * (lj.y + hj.y),
                          dz = cz - 0.5f * (lj.z + hj.z);
                    if (p.periodic) {
                        dx -= rintf(dx * p.invL[0]) * Lx;
                        dy -= rintf(dy * p.invL[1]) * Ly;
                        dz -= rintf(dz * p.invL[2]) * Lz;
                    }
                    const float gx = fmaxf(fabsf(dx) - (ex + 0.5f * (hj.x - lj.x)), 0.f);
                    const float gy = fmaxf(fabsf(dy) - (ey + 0.5f * (hj.y - lj.y)), 0.f);
                    const float gz = fmaxf(fabsf(dz) - (ez + 0.5f * (hj.z - lj.z)), 0.f);
                    near = gx * gx + gy * gy + gz * gz < c.rs2[0];
                }
                const uint32_t bn = __ballot_sync(0xffffffffu, near);
                if (lane == 0) bcnt[bpar][wl] = __popc(bn);
                __syncthreads();
                int at = tail;
#pragma unroll
                for (int w = 0; w < NB_W; ++w) {
                    if (w == wl && near) ring[(at + __popc(bn & below)) & (NB_RING - 1)] = J;
                    at += bcnt[bpar][w];
                }
                tail = at;
                bpar ^= 1;
                __syncthreads();
                t0 += NB_NT;
                const int least = cb + NB_NT >= ncols && t0 >= nt ? 1 : NB_QUEUE;
                while (tail - head >= least) atoms(min(tail - head, NB_QUEUE));
            } while (t0 < nt);
        }
        if (tid == 0) {
            c.lcnt[0][I] = min(m0, c.capj[0]);
            c.lcnt[1][I] = c.nlists > 1 ? min(m1, c.capj[1]) : 0;
        }
        overflow = overflow || m0 > c.capj[0] || (c.nlists > 1 && m1 > c.capj[1]);
    }
    if (overflow && tid == 0) atomicOr(s.err, BERR_LIST_OVERFLOW);
}

// Whether list entry `ent` (high part hj of the j atom's slot copy) lies
// within sqrt(R2) of some atom of the cluster in shi/slo: high parts with the
// entry's periodic image (their rounding is far below the radius's margin),
// or the per-pair minimum image from the split positions (rare).
__device__ __forceinline__ bool prune_keep(const DevSys& s, const Params& p, int cur, int ent, float4 hj,
                                           const float4* shi, const float4* slo, float R2) {
    const DevClu& c = s.cl;
    const int sj = ent & 0x07FFFFFF, code = (int)((uint32_t)ent >> 27);
    float best = INFINITY;
    if (code == PER_PAIR) {
        const float4 lj = c.splo[cur][sj];
        for (int a = 0; a < CL; ++a) {
            const float3 d = pair_disp(p, shi[a], slo[a], hj, lj);
            best = fminf(best, d.x * d.x + d.y * d.y + d.z * d.z);
        }
    } else {
        if (code != NO_SHIFT) {
            hj.x -= (float)(code / 9 - 1) * p.Lhi[0];
            hj.y -= (float)((code / 3) % 3 - 1) * p.Lhi[1];
            hj.z -= (float)(code % 3 - 1) * p.Lhi[2];
        }
#pragma unroll
        for (int a = 0; a < CL; ++a) {
            const float dx = shi[a].x - hj.x, dy = shi[a].y - hj.y, dz = shi[a].z - hj.z;
            best = fminf(best, dx * dx + dy * dy + dz * dz);
        }
    }
    return best < R2;
}

// 3b. pruned lists (warp per cluster I): the
// entries of each list whose atom j lies within the prune radius of at least
// one atom of I at the current positions (same images as the pair kernel;
// FP32 with a margin, so that no pair the exact test would keep is dropped),
// in list order.  The step kernel raises the flag when an atom's slot copy has moved half the
// prune skin since this launch, which it records here.
//
// Bounded by the chain of one list (entries, their positions, the vote): four
// passes of 32 entries are in flight per warp (two: 30 us for 12,288 atoms, 73 us
// for 98,304; four: 26 and 67).  A CTA per cluster takes 24 and 98 us.
//
// 3. The two in one launch: a CTA prunes the clusters whose lists it has just
// made (new lists), or those it would make (prune flag alone).  Each kernel of
// the gated sequence costs a step ~1.1 us when nothing is due.  (Apart, two
// launches are no faster where both are due: 1447 against 1421 us for the
// forces of two frames of 27,783 atoms.)
__global__ void __launch_bounds__(NB_NT, 8) k_cl_lists(const __grid_constant__ DevSys s, const __grid_constant__ Params p,
                                                       int step_off, int force) {
    chain_enter();
    const DevClu& c = s.cl;
    const bool search = force || *c.rebuild;
    if (!(search || *c.prune)) return;
    if (search) {
        cl_search(s, p, step_off);
        __syncthreads();  // the CTA's lists are written
    }
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    __shared__ float4 s_hi[NB_W][CL], s_lo[NB_W][CL];
    const int ncl = c.ncol * c.maxcl;
    const int cur = (int)((*s.step_base + step_off) & 1);
    const uint32_t below = (1u << lane) - 1u;
    for (int t = blockIdx.x + wl * gridDim.x; t < ncl; t += gridDim.x * NB_W) {
        const int kt = t / c.ncol, I = (t - kt * c.ncol) * c.maxcl + kt;  // the columns' unused slots come last
        int n[2];
        n[0] = c.lcnt[0][I];
        n[1] = c.nlists > 1 ? c.lcnt[1][I] : 0;
        __syncwarp();
        if (lane < CL) {
            // padding slots (no atom) are placed out of reach: their copies in
            // the buffer the step kernel writes are never refreshed
            const bool real = c.smol[I * CL + lane] >= 0;
            const float4 h = c.sphi[cur][I * CL + lane];
            s_hi[wl][lane] = real ? h : make_float4(1e30f, 1e30f, 1e30f, 0.f);
            s_lo[wl][lane] = real ? c.splo[cur][I * CL + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            c.pref[I * CL + lane] = h;
        }
        __syncwarp();
#pragma unroll
        for (int L = 0; L < 2; ++L) {
            if (L >= c.nlists) break;
            const int* src = c.lst[L] + (size_t)I * c.capj[L];
            int* dst = c.plst[L] + (size_t)I * c.capj[L];
            int m = 0;
            const float R2 = c.prs2[L];
            for (int e0 = 0; e0 < n[L]; e0 += 32 * NB_PASS) {
                int ent[NB_PASS];
                float4 h[NB_PASS];
                // (an entry's image code fills its top bits: validity comes from the index)
#pragma unroll
                for (int u = 0; u < NB_PASS; ++u) {
                    const int e = e0 + 32 * u + lane;
                    ent[u] = e < n[L] ? src[e] : 0;
                }
#pragma unroll
                for (int u = 0; u < NB_PASS; ++u)
                    h[u] = e0 + 32 * u + lane < n[L] ? c.sphi[cur][ent[u] & 0x07FFFFFF] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < NB_PASS; ++u) {
                    const bool keep =
                        e0 + 32 * u + lane < n[L] && prune_keep(s, p, cur, ent[u], h[u], s_hi[wl], s_lo[wl], R2);
                    const uint32_t b = __ballot_sync(0xffffffffu, keep);
                    if (keep) dst[m + __popc(b & below)] = ent[u];
                    m += __popc(b);
                }
            }
            if (lane == 0) {
                c.pcnt[L][I] = m;
                // work items of I's pruned list, at slots taken from a counter
                // (their order does not matter: the sums are fixed point)
                const int nch = (m + EPW - 1) / EPW;
                const int b = nch ? atomicAdd(&c.pnitems[2 + L], nch) : 0;
                for (int k = 0; k < nch; ++k)
                    if (b + k < c.capitems) c.pitems[L][b + k] = make_int4(I, k * EPW, min((k + 1) * EPW, m), 0);
            }
        }
    }
    if (!cl_last_cta(&c.done_ctr[1])) return;
    if (threadIdx.x < 2) {
        const int L = threadIdx.x;
        const int n = atomicExch(&c.pnitems[2 + L], 0);
        c.pnitems[L] = min(n, c.capitems);
        if (n > c.capitems) atomicOr(s.err, BERR_LIST_OVERFLOW);
    }
    if (threadIdx.x == 0) {
        *c.prune = 0;
        if (search) *c.rebuild = 0;
    }
}

// The pairs of one list entry (atom slot sj, split position hj/lj in the
// image of the entry) whose FP32 r^2 falls within the rounding band of r_c^2:
// each takes the exact FP64 cutoff test; a pair inside adds its i side
// straight to the accumulator of its slot; the j side gj with the pairs added
// and their number are returned (by value: the caller's sums stay in
// registers).  Rare (the band is 2e-5 of r_c^2 wide), so kept out of the
// unrolled code.
template <int PART>
__device__ __noinline__ float4 near_pairs(const DevSys& s, const Params& p, int cur, int I, int sj, float4 hj, float4 lj,
                                          int mj, int above, float3 gj) {
    const DevClu& c = s.cl;
    int npair = 0;
    const size_t ns = (size_t)c.ncol * c.maxcl * CL;
    for (int a = 0; a < min(CL, above); ++a) {
        const int si = I * CL + a;
        if (c.smol[si] < 0 || c.smol[si] == mj) continue;
        const float4 hi = c.sphi[cur][si], lo = c.splo[cur][si];
        const float3 d = pair_disp(p, hi, lo, hj, lj);
        const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
        if (!(r2 >= p.rc2_lo && r2 <= p.rc2_hi)) continue;
        if (!(exact_r2(s, p, cur, c.cl_atom[si], c.cl_atom[sj]) < p.rc2_d)) continue;
        const int tp = type_of(lo) * BOUNCE_MAXT + type_of(lj);
        const float w = pairsum_w<PART>(p, r2, p.kcoul * hi.w * hj.w, p.c12[tp], p.c6[tp]);
        fix_add(c.acc + si, w * d.x);
        fix_add(c.acc + ns + si, w * d.y);
        fix_add(c.acc + 2 * ns + si, w * d.z);
        gj.x = fmaf(-w, d.x, gj.x);
        gj.y = fmaf(-w, d.y, gj.y);
        gj.z = fmaf(-w, d.z, gj.z);
        ++npair;
    }
    return make_float4(gj.x, gj.y, gj.z, __int_as_float(npair));
}

// Pair sums over the work items of list `L`.  PART 3: the F_0 share
// (1 - chi) W'_sw + W'_fixed; PART 5: the full W'.  A warp takes an item of
// cluster I: lanes hold one list atom j each, the 8 atoms of I are read from
// shared memory two at a time (pairs.cuh); the j side of every pair is summed
// in the lane's registers and added once per entry, the i side is kept per
// lane for the 8 atoms and reduced over the warp at the end of the item.
//
// Bound by instruction issue and the latency that 16 warps per SM leave
// uncovered.  98,304-atom water box, per launch: 109 us for the F_0 share and
// 96 us for the full sums, against 165 and 145 with one pair per instruction;
// 12,288-atom droplet (r_c 12 A) 35 against 55 us.  What it took besides the
// packed arithmetic: the j atoms of the next pass are gathered into registers
// while this one is evaluated, across items too; reductions to global memory
// instead of generic atomics, and near_pairs by value instead of through the
// stack (together 12 us of the box's 117).
template <int PART, bool EW, bool CJ>
__global__ void __launch_bounds__(PAIRS_NT, PAIRS_CTAS) k_cl_pairs(const __grid_constant__ DevSys s,
                                                                   const __grid_constant__ Params p,
                                                                   const __grid_constant__ PairConsts k, int step_off,
                                                                   int L, int early) {
    if (early) chain_next();
    else chain_enter();
    __shared__ IGroup s_g[PAIRS_NT / 32];
    const DevClu& c = s.cl;
    const int lane = threadIdx.x & 31;
    IGroup& g = s_g[threadIdx.x >> 5];
    const int cur = (int)((*s.step_base + step_off) & 1);
    const int capj = c.capj[L];
    const int nit = c.pnitems[L];
    const size_t ns = (size_t)c.ncol * c.maxcl * CL;
    const float4* sphi = c.sphi[cur];
    const float4* splo = c.splo[cur];
    const int* plst = c.plst[L];
    auto entry = [&](int4 it, int e) -> int {  // list entry e of item it (0 beyond its end)
        return e < it.z ? __ldg(plst + (size_t)it.x * capj + e) : 0;
    };
    float4 nh, nl;  // j atom of the next pass
    int nm;
    auto gather = [&](int ent) {
        nh = sphi[ent & 0x07FFFFFF];
        nl = splo[ent & 0x07FFFFFF];
        nm = c.smol[ent & 0x07FFFFFF];
    };
    int npair = 0;
    // items are fetched from a counter, so that no warp idles while its
    // CTA's other warps still work (the items differ in length)
    int nx = 0;
    if (lane == 0) nx = atomicAdd(&c.pnitems[4 + L], 1);
    nx = __shfl_sync(0xffffffffu, nx, 0);
    if (nx < nit) {
        int4 w = c.pitems[L][nx];  // (I, first entry, end, -)
        int ent = entry(w, w.y + lane), ent1 = entry(w, w.y + 32 + lane);
        gather(ent);
        for (;;) {
            const int I = w.x;
            if (lane == 0) nx = atomicAdd(&c.pnitems[4 + L], 1);
            // the next item: its number was asked for just now, its record is
            // read after this item's first pass, its first entries after the second
            int4 wn = make_int4(0, 0, 0, 0);
            int stage = 0, nent = 0;
            auto advance = [&]() {
                if (stage == 0) {
                    nx = __shfl_sync(0xffffffffu, nx, 0);
                    if (nx < nit) wn = c.pitems[L][nx];
                } else if (stage == 1) {
                    nent = entry(wn, wn.y + lane);
                }
                ++stage;
            };
            __syncwarp();
            if (lane < CL) igroup_set(g, p, lane, sphi[I * CL + lane], splo[I * CL + lane], c.smol[I * CL + lane]);
            __syncwarp();
            float2 gi[4][3];
#pragma unroll
            for (int a = 0; a < 4; ++a) gi[a][0] = gi[a][1] = gi[a][2] = make_float2(0.f, 0.f);
            for (int e0 = w.y; e0 < w.z; e0 += 32) {
                const bool valid = e0 + lane < w.z;  // (an entry's image code fills its top bits)
                const int sj = ent & 0x07FFFFFF;
                const int code = valid ? (int)((uint32_t)ent >> 27) : NO_SHIFT;
                JAtom j;
                j.h = nh;
                j.l = nl;
                j.mol = nm;
                // the next pass's atoms, of this item or the next
                if (e0 + 32 < w.z) {
                    ent = ent1;
                    gather(ent);
                    ent1 = entry(w, e0 + 64 + lane);
                } else {
                    while (stage < 2) advance();
                    ent = nent;
                    gather(ent);
                    ent1 = entry(wn, wn.y + 32 + lane);
                }
                j.type = type_of(j.l);
                // pairs within I: the lower slot is i (every other j lies in a later cluster)
                j.above = valid ? sj - I * CL : 0;
                if (code != NO_SHIFT && code != PER_PAIR) {
                    const float kx = (float)(code / 9 - 1), ky = (float)((code / 3) % 3 - 1), kz = (float)(code % 3 - 1);
                    shift_split(j.h.x, j.l.x, kx * p.Lhi[0], kx * p.Llo[0]);
                    shift_split(j.h.y, j.l.y, ky * p.Lhi[1], ky * p.Llo[1]);
                    shift_split(j.h.z, j.l.z, kz * p.Lhi[2], kz * p.Llo[2]);
                }
                if (!valid) j.h.x = PAIR_FAR;
                float3 gs = make_float3(0.f, 0.f, 0.f);
                float near = INFINITY;
                // entries of the own cluster (index rule) or near half a box edge
                // (minimum image per pair) take their warp through a copy of the
                // loop with both (the same sums for the other entries)
                if (__any_sync(0xffffffffu, code == PER_PAIR || (valid && j.above < CL)))
                    group_pairs<PART, EW, CJ, true>(k, g, j, gi, gs, near, npair);
                else
                    group_pairs<PART, EW, CJ, false>(k, g, j, gi, gs, near, npair);
                if (near <= k.band) {
                    const float4 o = near_pairs<PART>(s, p, cur, I, sj, j.h, j.l, j.mol, j.above, gs);
                    gs = make_float3(o.x, o.y, o.z);
                    npair += __float_as_int(o.w);
                }
                fix_add(c.acc + sj, gs.x);
                fix_add(c.acc + ns + sj, gs.y);
                fix_add(c.acc + 2 * ns + sj, gs.z);
                if (stage < 2) advance();
            }
            // i side: lane 4 b + d adds component d of atom igroup_atom(b)
            const float mine = igroup_reduce(gi);
            const int a = igroup_atom(lane >> 2), d = lane & 3;
            if (d < 3) fix_add(c.acc + (size_t)d * ns + I * CL + a, mine);
            if (nx >= nit) break;
            w = wn;
        }
    }
    if (early) chain_wait();
    npair = warp_sum_i(npair);
    if (lane == 0 && npair) atomicAdd(&s.cnt[PART == 3 ? CNT_SHORT_PAIRS : CNT_FULL_PAIRS], (unsigned long long)npair);
    // every warp has seen the counter past the last item: the last CTA resets it
    if (cl_last_cta(&c.done_ctr[3]) && threadIdx.x == 0) c.pnitems[4 + L] = 0;
}

// The accumulated pair sums of every atom added to out (n x 3, FP64), and
// the accumulators cleared for the next evaluation.
__global__ void k_cl_collect(DevSys s, double* out) {
    const DevClu& c = s.cl;
    const size_t ns = (size_t)c.ncol * c.maxcl * CL;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.n; i += gridDim.x * blockDim.x) {
        const int sl = c.a2s[i];
        for (int d = 0; d < 3; ++d) {
            const long long v = (long long)c.acc[d * ns + sl];
            c.acc[d * ns + sl] = 0ull;
            out[3 * (size_t)i + d] += (double)v * CL_UNFIX;
        }
    }
}

}  // namespace

void launch_cluster_rebuild(const DevSys& s, const Params& p, int step_off, bool force, cudaStream_t st, bool binned) {
    const int f = force ? 1 : 0;
    if (!binned) launch_bins(s, p, step_off, force, BIN_COLUMNS, ROWS_ALL, st);
    launch_chained(k_cl_sort, std::min(s.cl.ncol, 152 * 8), SORT_NT, 0, st, s, p, step_off, f);
    const int ncl = s.cl.ncol * s.cl.maxcl;
    launch_chained(k_cl_lists, std::min(ncl, 152 * 8), NB_NT, 0, st, s, p, step_off, f);
}

// CTAs of a pair kernel that fit on the GPU at once (the warps fetch their
// work items, so one resident wave covers any number of items)
template <typename K>
static int resident_ctas(K kernel, int& blocks) {
    if (!blocks) {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, PAIRS_NT, 0);
        blocks = std::max(1, sms * std::max(per, 1));
    }
    return blocks;
}

template <int PART, bool EW, bool CJ>
static int cl_pairs_grid() {
    static int blocks = 0;
    return resident_ctas(k_cl_pairs<PART, EW, CJ>, blocks);
}

void prepare_cluster_pairs() {
    cl_pairs_grid<5, true, true>();
    cl_pairs_grid<5, false, true>();
    cl_pairs_grid<3, true, true>();
    cl_pairs_grid<3, true, false>();
    cl_pairs_grid<3, false, true>();
    cl_pairs_grid<3, false, false>();
}

template <int PART, bool CJ>
static void launch_cl_pairs(const DevSys& s, const Params& p, int step_off, int list, bool early, cudaStream_t st) {
    const PairConsts k = make_pair_consts(p);
    const int e = early ? 1 : 0;
    if (p.ebeta > 0.f)
        launch_chained(k_cl_pairs<PART, true, CJ>, cl_pairs_grid<PART, true, CJ>(), PAIRS_NT, 0, st, s, p, k, step_off, list, e);
    else
        launch_chained(k_cl_pairs<PART, false, CJ>, cl_pairs_grid<PART, false, CJ>(), PAIRS_NT, 0, st, s, p, k, step_off,
                       list, e);
}

void launch_cluster_pairs(const DevSys& s, const Params& p, int step_off, int part, int list, cudaStream_t st, bool early) {
    if (part != 3) launch_cl_pairs<5, true>(s, p, step_off, list, early, st);
    else if (p.coul_jump) launch_cl_pairs<3, true>(s, p, step_off, list, early, st);
    else launch_cl_pairs<3, false>(s, p, step_off, list, early, st);
}

void launch_cluster_collect(const DevSys& s, double* out, cudaStream_t st) {
    k_cl_collect<<<(s.n + 255) / 256, 256, 0, st>>>(s, out);
}
