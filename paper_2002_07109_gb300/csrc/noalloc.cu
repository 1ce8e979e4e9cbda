// Pair energies without any device allocation.
//
// Some callers cannot call cudaMalloc: code that lives inside an allocator
// owning the whole device pool (a caching allocator would see a foreign
// allocation it cannot account for), hosts that forbid allocation after
// start-up (embedded or real-time loops, where cudaMalloc may block and
// synchronise the device), and plug-ins that are handed device buffers but
// no allocation rights.  For them, bounce_pair_energy_noalloc computes the
// same Coulomb and Lennard-Jones pair energy totals as the energy kernel of a
// context (bounce_get_energies), but over all pairs of a caller-supplied
// state and with its scratch in a file-scope device array instead of context
// buffers.
//
// Scratch: g_noalloc_scratch below, BOUNCE_NOALLOC_MAX_ATOMS atoms
// (48 bytes per atom: split FP32 positions and FP64 partial sums, 786,432
// bytes in all), plus status bytes, held by every GPU that
// loads this library until the process exits.  Host code cannot use the
// array's name as a device address (on the host it names a shadow
// variable), so the first call on each device looks the address up with
// cudaGetSymbolAddress while that device is current and keeps it; make that
// first call before any stream capture.  Every call overwrites every slot,
// status byte and counter it reads, so nothing
// needs clearing between calls; calls whose GPU work overlaps (two streams,
// two threads) share the array and race.
#include <cmath>
#include <mutex>

#include <math_constants.h>

#include "../../include/bounce.h"
#include "common.cuh"

namespace {

constexpr int NOALLOC_MAX = BOUNCE_NOALLOC_MAX_ATOMS;
constexpr int PACK_NT = 256;  // threads of a packing CTA: one status byte each (at most 64)
constexpr int NA_NT = 128, NA_W = NA_NT / 32;  // threads and warps of a pair CTA
constexpr int NA_B = 64;                       // atoms of a block: two to a lane
static_assert(NOALLOC_MAX <= 64 * PACK_NT, "one status byte per packing CTA");
// per atom: two float4 and two doubles; then the status bytes and the CTA counter
constexpr size_t NOALLOC_BYTES = (size_t)NOALLOC_MAX * (2 * sizeof(float4) + 2 * sizeof(double)) + 256;
constexpr int MAX_DEVICES = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

std::mutex g_mu;
void* g_scratch_ptr[MAX_DEVICES] = {nullptr};

struct Layout {
    float4* hi;
    float4* lo;
    double* part;        // coulomb of each pair CTA, then (at NOALLOC_MAX) lj
    unsigned char* bad;  // [64] of each packing CTA: an atom type outside [0, n_types) seen
    unsigned int* done;  // pair CTAs that are done
};

__device__ inline Layout layout(void* base) {
    Layout l;
    l.hi = (float4*)base;
    l.lo = l.hi + NOALLOC_MAX;
    l.part = (double*)(l.lo + NOALLOC_MAX);
    l.bad = (unsigned char*)(l.part + 2 * (size_t)NOALLOC_MAX);
    l.done = (unsigned int*)(l.bad + 128);
    return l;
}

// Split FP32 copies of the positions.  A type outside [0, n_types) would
// index the LJ tables out of bounds: it is replaced by type 0 here and
// flagged, and the pair kernel then writes NaN to both totals.
__global__ void __launch_bounds__(PACK_NT) k_na_pack(void* scratch, int n, const double* q, const double* charge,
                                                     const int* type, int n_types, const __grid_constant__ Params p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    Layout l = layout(scratch);
    const int i = blockIdx.x * PACK_NT + threadIdx.x;
    int t = 0;
    bool bad = false;
    if (i < n) {
        double x = q[3 * (size_t)i], y = q[3 * (size_t)i + 1], z = q[3 * (size_t)i + 2];
        if (p.periodic) {
            x -= p.Ld[0] * floor(x / p.Ld[0]);
            y -= p.Ld[1] * floor(y / p.Ld[1]);
            z -= p.Ld[2] * floor(z / p.Ld[2]);
        }
        t = type[i];
        bad = t < 0 || t >= n_types;
        if (bad) t = 0;
        float4 h, w;
        split_double(x, h.x, w.x);
        split_double(y, h.y, w.y);
        split_double(z, h.z, w.z);
        h.w = (float)charge[i];
        w.w = __int_as_float(t);
        l.hi[i] = h;
        l.lo[i] = w;
    }
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        l.bad[blockIdx.x] = any ? 1 : 0;
        if (blockIdx.x == 0) *l.done = 0u;
    }
}

// Exact FP64 r^2 from the caller's (n, 3) positions (same operations as the
// context path).
__device__ __forceinline__ double na_exact_r2(const Params& p, const double* q, int i, int j) {
    double d[3];
    for (int c = 0; c < 3; ++c) {
        d[c] = __dsub_rn(q[3 * (size_t)i + c], q[3 * (size_t)j + c]);
        if (p.periodic) d[c] = __dsub_rn(d[c], __dmul_rn(p.Ld[c], rint(__ddiv_rn(d[c], p.Ld[c]))));
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}

// W over all pairs of different molecules inside r_c.  A warp takes a pair of
// blocks of 64 atoms, (b, b + d mod nb) for d up to nb / 2, which meets every
// pair of blocks once: two i atoms to a lane, the j atoms one by one from
// shared memory, staged by the warp.  FP32 sums of at most 64 terms per i
// atom, everything above in FP64; the CTA that ends last adds the CTAs' sums
// in their order.
//
// Bounded by the ~35 instructions of a pair.  A warp per atom, lanes over j,
// read 36 bytes a pair and looked its LJ parameters up in constant memory at
// diverging addresses: 42 us for 4,500 atoms and 12 us for the sum over the
// atoms by one CTA, where this takes 34 in all.
__global__ void __launch_bounds__(NA_NT) k_na_pairs(void* scratch, int n, const double* q, const int* mol,
                                                    const __grid_constant__ Params p, unsigned lj_types, double kfix,
                                                    double* out) {
    __shared__ float4 sh[NA_W][NA_B], sl[NA_W][NA_B];
    __shared__ int sm[NA_W][NA_B];
    __shared__ float2 tab[BOUNCE_MAXT * BOUNCE_MAXT];
    __shared__ double sum[2][NA_NT];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    if (threadIdx.x < BOUNCE_MAXT * BOUNCE_MAXT) tab[threadIdx.x] = make_float2(p.c12[threadIdx.x], p.c6[threadIdx.x]);
    chain_enter();
    Layout l = layout(scratch);
    __syncthreads();
    const int nb = (n + NA_B - 1) / NA_B, item = blockIdx.x * NA_W + wl;
    const int d = item / nb, bi = item - d * nb;
    const int bj = bi + d < nb ? bi + d : bi + d - nb;
    double acc = 0.0;  // of lanes below 16 the Coulomb sum, of the others the LJ sum
    if (d <= nb / 2 && !(d > 0 && 2 * d == nb && bi >= d)) {
        const int j0 = bj * NA_B, nj = min(NA_B, n - j0);
        for (int t = lane; t < nj; t += 32) {
            sh[wl][t] = l.hi[j0 + t];
            sl[wl][t] = l.lo[j0 + t];
            sm[wl][t] = mol[j0 + t];
        }
        int ii[2], mi[2], row[2];
        float4 hi[2], lo[2];
        float qi[2], ec[2] = {0.f, 0.f}, el[2] = {0.f, 0.f};
        // a pair's type index is that of (lower, higher) atom: the table need not be symmetric
        const bool swap = bj < bi;
        const int si = swap ? 1 : BOUNCE_MAXT, sj = swap ? BOUNCE_MAXT : 1;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            ii[a] = bi * NA_B + 32 * a + lane;
            const int i = min(ii[a], n - 1);
            hi[a] = l.hi[i];
            lo[a] = l.lo[i];
            mi[a] = mol[i];
            qi[a] = p.kcoul * hi[a].w;
            row[a] = type_of(lo[a]) * si;
        }
        __syncwarp();
#pragma unroll 2
        for (int t = 0; t < nj; ++t) {
            const float4 hj = sh[wl][t], lj = sl[wl][t];
            const int mj = sm[wl][t], j = j0 + t, tj = type_of(lj);
            const bool lj_on = lj_types >> tj & 1u;
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const float3 r = pair_disp(p, hi[a], lo[a], hj, lj);
                const float r2 = r.x * r.x + r.y * r.y + r.z * r.z;
                bool in = mj != mi[a] && ii[a] < n && (d > 0 || j > ii[a]) && r2 <= p.rc2_hi;
                if (in && !(r2 < p.rc2_lo)) in = na_exact_r2(p, q, ii[a], j) < p.rc2_d;
                if (!in) continue;
                const float ir = rsqrt_nr(r2);
                if (p.ebeta > 0.f) ec[a] += qi[a] * hj.w * erfcf(p.ebeta * (r2 * ir)) * ir;
                else ec[a] += qi[a] * hj.w * ir;
                if (lj_on) {
                    const float2 c = tab[row[a] + tj * sj];
                    const float ir2 = ir * ir, ir6 = ir2 * ir2 * ir2;
                    if (c.x != 0.f) el[a] += (c.x * ir6 - c.y) * ir6;
                }
            }
        }
        const double c = widen(ec[0]) + widen(ec[1]), v = widen(el[0]) + widen(el[1]);
        acc = lane < 16 ? c : v;
        acc += __shfl_xor_sync(0xffffffffu, lane < 16 ? v : c, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if ((lane & 15) == 0) sum[lane >> 4][wl] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double c = 0.0, v = 0.0;
        for (int w = 0; w < NA_W; ++w) {
            c += sum[0][w];
            v += sum[1][w];
        }
        l.part[blockIdx.x] = c;
        l.part[NOALLOC_MAX + blockIdx.x] = v;
        __threadfence();
        last = atomicAdd(l.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int t = 0; t < 2; ++t) {
        double a = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += NA_NT) a += __ldcg(l.part + (size_t)t * NOALLOC_MAX + i);
        sum[t][threadIdx.x] = a;
    }
    const int bad = __syncthreads_or(threadIdx.x * PACK_NT < n && l.bad[threadIdx.x]);
    for (int w = NA_NT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            sum[0][threadIdx.x] += sum[0][threadIdx.x + w];
            sum[1][threadIdx.x] += sum[1][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = bad ? CUDART_NAN : kfix * sum[0][0];
        out[1] = bad ? CUDART_NAN : sum[1][0];
    }
}

}  // namespace

extern "C" int bounce_pair_energy_noalloc(int32_t n, const double* q, const double* charge, const int32_t* type,
                                          const int32_t* molecule, int32_t n_types, const double* sigma,
                                          const double* eps, double r_cut, double ewald_beta, const double* box,
                                          double* out, void* stream) {
    if (n < 1 || n > NOALLOC_MAX || !q || !charge || !type || !molecule || !out || n_types < 1 ||
        n_types > BOUNCE_MAXT || !sigma || !eps || ewald_beta < 0)
        return BOUNCE_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return BOUNCE_ERR_CUDA;
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_scratch_ptr[dev]) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return BOUNCE_ERR_CUDA;
            g_scratch_ptr[dev] = ptr;
        }
        scratch = g_scratch_ptr[dev];
    }
    // the same scalar parameters as a context's energy kernel (no device memory)
    Params p{};
    for (int a = 0; a < n_types; ++a)
        for (int b = 0; b < n_types; ++b) {
            const double s6 = std::pow(sigma[a * n_types + b], 6);
            p.c12[a * BOUNCE_MAXT + b] = (float)(4.0 * eps[a * n_types + b] * s6 * s6);
            p.c6[a * BOUNCE_MAXT + b] = (float)(4.0 * eps[a * n_types + b] * s6);
        }
    p.kcoul = (float)KCOUL_D;
    const bool cut = std::isfinite(r_cut) && r_cut > 0;
    const double rc2 = cut ? r_cut * r_cut : INFINITY;
    p.rc2_lo = cut ? (float)(rc2 * (1.0 - 1e-5)) : INFINITY;
    p.rc2_hi = cut ? (float)(rc2 * (1.0 + 1e-5)) : INFINITY;
    p.rc2_d = rc2;
    p.ebeta = (float)ewald_beta;
    p.e2b_sqrtpi = (float)(2.0 * ewald_beta / std::sqrt(M_PI));
    p.periodic = box ? 1 : 0;
    for (int d = 0; d < 3; ++d) {
        const double Lb = box ? box[d] : 1.0;
        if (!(Lb > 0)) return BOUNCE_ERR_INVALID_ARG;
        // minimum image: beyond half an edge the sum would no longer be the pair sum
        if (box && !(cut && 2.0 * r_cut <= Lb)) return BOUNCE_ERR_INVALID_ARG;
        p.Ld[d] = Lb;
        p.iLd[d] = 1.0 / Lb;
        p.Lhi[d] = (float)Lb;
        p.Llo[d] = (float)(Lb - (double)p.Lhi[d]);
        p.invL[d] = (float)(1.0 / Lb);
    }
    cudaStream_t st = (cudaStream_t)stream;
    // an error left pending by earlier, unrelated work is not this call's:
    // refuse to launch rather than report (and clear) it as our own
    if (cudaPeekAtLastError() != cudaSuccess) return BOUNCE_ERR_CUDA;
    k_na_pack<<<(n + PACK_NT - 1) / PACK_NT, PACK_NT, 0, st>>>(scratch, n, q, charge, type, n_types, p);
    if (cudaGetLastError() != cudaSuccess) return BOUNCE_ERR_CUDA;
    unsigned lj_types = 0u;
    for (int a = 0; a < n_types; ++a)
        for (int b = 0; b < n_types; ++b)
            if (p.c12[a * BOUNCE_MAXT + b] != 0.f) lj_types |= 1u << a | 1u << b;
    const int nb = (n + NA_B - 1) / NA_B, items = nb * (nb / 2 + 1);
    launch_chained(k_na_pairs, (items + NA_W - 1) / NA_W, NA_NT, 0, st, scratch, (int)n, q, (const int*)molecule, p,
                   lj_types, KCOUL_D / (double)p.kcoul, out);
    return cudaGetLastError() == cudaSuccess ? BOUNCE_OK : BOUNCE_ERR_CUDA;
}
