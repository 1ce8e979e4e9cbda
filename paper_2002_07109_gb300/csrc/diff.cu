// Differentiable direct-space pair forces for force matching (the pair
// terms of paper Sec. IV.A / V with trainable per-type parameters).
//
// Forward: F_i = -sum_j g(r_ij) d_ij, g = W'(r)/r, d_ij = q_i - q_j, over the
// candidate rows with r^2 < r_c^2, and E = sum_{i<j} W.  W = k q_a q_b / r
// (or k q_a q_b erfc(beta r)/r) + c12/r^12 - c6/r^6, c12 = 4 eps sigma^12,
// c6 = 4 eps sigma^6, with per-type charges q_t and symmetric sigma, eps.
// Backward for L(F, E) with upstream u_i = dL/dF_i and w = dL/dE:
//   dL/dq_i = sum_j [ -H(d_ij) (u_i - u_j) + w g d_ij ],
//             H(d) = g I + (g'(r)/r) d d^T (the pair Hessian of W);
//   dL/dtheta = sum_{i<j} [ -(dg/dtheta) (u_i - u_j).d_ij + w dW/dtheta ].
// One warp per atom, FP32 pair math.  The parameters enter through (k q q,
// c12, c6) of a pair of types: the backward sums the three coefficients per
// type of j in FP32 over an atom's pairs, then in FP64 over the atoms of each
// type, in a fixed order (per CTA, then over the CTAs), and the host applies
// the chain rule to the sums of each pair of types, so the gradients do not
// depend on scheduling.
#include "common.cuh"

namespace {

constexpr int MAXT = BOUNCE_MAXT;
constexpr int NSUM = 3 * MAXT * MAXT;  // coefficient sums (q q, c12, c6) by type of i and of j
constexpr int WPB = 8;                 // atoms (warps) per CTA

struct DiffParams {
    float qt[MAXT];
    float sig[MAXT * MAXT];
    float eps[MAXT * MAXT];
    int T;
};

// Pair quantities for parameters p: g, dg/dr, W and the partial
// derivatives of g and W with respect to (q_product, c12, c6).
struct PairD {
    float g, gp, W;
    float dg_dqq, dW_dqq;   // per unit of k q_a q_b
    float dg_dc12, dg_dc6, dW_dc12, dW_dc6;
};

__device__ __forceinline__ PairD pair_terms_d(const Params& p, float r2, float qq, float c12, float c6) {
    PairD o;
    const float ir = rsqrt_nr(r2);
    const float r = r2 * ir;
    const float ir2 = ir * ir;
    float gc, gpc, wc;  // Coulomb g, g', W per unit qq
    if (p.ebeta > 0.f) {
        const float b = p.ebeta;
        const float ec = erfcf(b * r), ex = expf(-b * b * r2);
        const float c = p.e2b_sqrtpi;
        wc = ec * ir;
        const float dW = -(ec * ir2 + c * ex * ir);
        const float d2W = 2.f * ec * ir2 * ir + c * ex * (2.f * ir2 + 2.f * b * b);
        gc = dW * ir;
        gpc = d2W * ir - dW * ir2;
    } else {
        wc = ir;
        gc = -ir2 * ir;
        gpc = 3.f * ir2 * ir2;
    }
    const float ir6 = ir2 * ir2 * ir2;
    const float ir8 = ir6 * ir2;
    o.dg_dqq = gc;
    o.dW_dqq = wc;
    o.dg_dc12 = -12.f * ir6 * ir8;
    o.dg_dc6 = 6.f * ir8;
    o.dW_dc12 = ir6 * ir6;
    o.dW_dc6 = -ir6;
    o.g = qq * gc + c12 * o.dg_dc12 + c6 * o.dg_dc6;
    o.gp = qq * gpc + c12 * (168.f * ir8 * ir6 * ir) + c6 * (-48.f * ir8 * ir);
    o.W = qq * wc + c12 * o.dW_dc12 + c6 * o.dW_dc6;
    return o;
}

__device__ __forceinline__ void type_params(const DiffParams& dp, int ti, int tj, float& qq, float& c12, float& c6) {
    const float s = dp.sig[ti * MAXT + tj], e = dp.eps[ti * MAXT + tj];
    const float s2 = s * s, s6 = s2 * s2 * s2;
    qq = (float)KCOUL_D * dp.qt[ti] * dp.qt[tj];
    c12 = 4.f * e * s6 * s6;
    c6 = 4.f * e * s6;
}

// LJ and Coulomb factors of an atom of type ti with each type of j, in
// shared memory (one copy per warp).
struct TypeRow {
    float qq[MAXT], c12[MAXT], c6[MAXT];
};
__device__ __forceinline__ void set_type_row(TypeRow& t, const DiffParams& dp, int ti) {
    const int lane = threadIdx.x & 31;
    if (lane < MAXT) type_params(dp, ti, lane, t.qq[lane], t.c12[lane], t.c6[lane]);
    __syncwarp();
}

// Forward: forces per atom; the pair energies (j > i) of the CTA's atoms, in
// their order, into ecta[CTA].
__global__ void __launch_bounds__(32 * WPB) k_pair_fwd(DevSys s, Params p, DiffParams dp, int cur, double* F, double* ecta) {
    __shared__ TypeRow rows_t[WPB];
    __shared__ float se[WPB];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int i = blockIdx.x * WPB + wl;
    float e = 0.f;
    if (i < s.n) {
        const float4 hi = s.phi[cur][i], lo = s.plo[cur][i];
        set_type_row(rows_t[wl], dp, type_of(lo));
        const TypeRow& tr = rows_t[wl];
        const int n = s.nlong[i];
        const int* row = s.rows + (size_t)i * s.cap;
        float fx = 0.f, fy = 0.f, fz = 0.f;
        int jn = lane < n ? row[lane] : 0;
        for (int k = lane; k < n; k += 32) {
            const int j = jn;
            const float4 hj = s.phi[cur][j], lj = s.plo[cur][j];
            jn = k + 32 < n ? row[k + 32] : 0;
            const float3 d = pair_disp(p, hi, lo, hj, lj);
            const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
            if (!inside_cut(s, p, cur, i, j, r2)) continue;
            const int tj = type_of(lj);
            const PairD t = pair_terms_d(p, r2, tr.qq[tj], tr.c12[tj], tr.c6[tj]);
            fx -= t.g * d.x;
            fy -= t.g * d.y;
            fz -= t.g * d.z;
            if (j > i) e += t.W;
        }
        fx = warp_sum_f(fx);
        fy = warp_sum_f(fy);
        fz = warp_sum_f(fz);
        e = warp_sum_f(e);
        if (lane < 3) F[3 * (size_t)i + lane] = lane == 0 ? fx : (lane == 1 ? fy : fz);
    }
    if (lane == 0) se[wl] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < WPB; ++w) t += (double)se[w];
        ecta[blockIdx.x] = t;
    }
}

// Upstream gradients as FP32 quadruples: one 16-byte gather per pair, where
// three FP64 loads and conversions (on the FP64 pipe) bound the backward.
__global__ void k_upstream(int n, const double* U, float4* u) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) u[i] = make_float4((float)U[3 * (size_t)i], (float)U[3 * (size_t)i + 1], (float)U[3 * (size_t)i + 2], 0.f);
}

// Backward: position gradient per atom; the coefficient sums of the CTA's
// atoms (pairs j > i) by the types of i and j into part[NSUM][CTAs].
// 12,288 atoms, r_c 9 A: 91 us before (36 per-atom sums over the warp, FP64
// upstream, arrays indexed in local memory), 59 us now; the forward 47 and 38.
__global__ void __launch_bounds__(32 * WPB) k_pair_bwd(DevSys s, Params p, DiffParams dp, int cur, const float4* U, float wf,
                                                       double* gpos, double* part) {
    __shared__ TypeRow rows_t[WPB];
    __shared__ float sums[WPB][3 * MAXT];
    __shared__ int types[WPB];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int i = blockIdx.x * WPB + wl;
    float acc[3][MAXT];  // coefficients of q q, c12, c6 by type of j
#pragma unroll
    for (int b = 0; b < MAXT; ++b) acc[0][b] = acc[1][b] = acc[2][b] = 0.f;
    int ti = -1;
    if (i < s.n) {
        const float4 hi = s.phi[cur][i], lo = s.plo[cur][i], ui = U[i];
        ti = type_of(lo);
        set_type_row(rows_t[wl], dp, ti);
        const TypeRow& tr = rows_t[wl];
        const int n = s.nlong[i];
        const int* row = s.rows + (size_t)i * s.cap;
        float gx = 0.f, gy = 0.f, gz = 0.f;
        int jn = lane < n ? row[lane] : 0;
        for (int k = lane; k < n; k += 32) {
            const int j = jn;
            const float4 hj = s.phi[cur][j], lj = s.plo[cur][j], uj = U[j];
            jn = k + 32 < n ? row[k + 32] : 0;
            const float3 d = pair_disp(p, hi, lo, hj, lj);
            const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
            if (!inside_cut(s, p, cur, i, j, r2)) continue;
            const int tj = type_of(lj);
            const PairD t = pair_terms_d(p, r2, tr.qq[tj], tr.c12[tj], tr.c6[tj]);
            const float dux = ui.x - uj.x, duy = ui.y - uj.y, duz = ui.z - uj.z;
            const float ddu = d.x * dux + d.y * duy + d.z * duz;
            const float h = t.gp * rsqrt_nr(r2) * ddu;
            // -H (u_i - u_j) + w g d
            gx += -(t.g * dux + h * d.x) + wf * t.g * d.x;
            gy += -(t.g * duy + h * d.y) + wf * t.g * d.y;
            gz += -(t.g * duz + h * d.z) + wf * t.g * d.z;
            if (j > i) {
                // coefficients of -g (u_i - u_j).d + w W
                const float cq = -t.dg_dqq * ddu + wf * t.dW_dqq;
                const float c12 = -t.dg_dc12 * ddu + wf * t.dW_dc12;
                const float c6 = -t.dg_dc6 * ddu + wf * t.dW_dc6;
#pragma unroll
                for (int b = 0; b < MAXT; ++b) {
                    acc[0][b] += tj == b ? cq : 0.f;
                    acc[1][b] += tj == b ? c12 : 0.f;
                    acc[2][b] += tj == b ? c6 : 0.f;
                }
            }
        }
        gx = warp_sum_f(gx);
        gy = warp_sum_f(gy);
        gz = warp_sum_f(gz);
        if (lane < 3) gpos[3 * (size_t)i + lane] = lane == 0 ? gx : (lane == 1 ? gy : gz);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int b = 0; b < MAXT; ++b) {
            const float v = b < dp.T ? warp_sum_f(acc[c][b]) : 0.f;
            if (lane == 0) sums[wl][c * MAXT + b] = v;
        }
    if (lane == 0) types[wl] = ti;
    __syncthreads();
    const int t = threadIdx.x;
    if (t < NSUM) {  // sum (coefficient, type of i, type of j) over the CTA's atoms in order
        const int c = t / (MAXT * MAXT), a = t / MAXT % MAXT, b = t % MAXT;
        double v = 0.0;
        for (int w = 0; w < WPB; ++w)
            if (types[w] == a) v += (double)sums[w][c * MAXT + b];
        part[(size_t)t * gridDim.x + blockIdx.x] = v;
    }
}

// Fixed-order sums of `rows` arrays of length n: out[r] = sum_i x[r][i].
__global__ void k_rowsum(int n, int rows, const double* x, double* out) {
    __shared__ double red[256];
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        double acc = 0.0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) acc += x[(size_t)r * n + i];
        red[threadIdx.x] = acc;
        __syncthreads();
        for (int w = blockDim.x / 2; w > 0; w >>= 1) {
            if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) out[r] = red[0];
        __syncthreads();
    }
}

DiffParams diff_params(const float* qt, const float* sig, const float* eps, int T) {
    DiffParams dp{};
    for (int a = 0; a < MAXT; ++a) dp.qt[a] = a < T ? qt[a] : 0.f;
    for (int a = 0; a < MAXT * MAXT; ++a) dp.sig[a] = sig[a], dp.eps[a] = eps[a];
    dp.T = T;
    return dp;
}

}  // namespace

// doubles of scratch the backward needs for n atoms: the upstream quadruples,
// the CTAs' sums, the sums
size_t diff_scratch(int n) { return 2 * (size_t)n + (size_t)NSUM * ((n + WPB - 1) / WPB) + NSUM; }

void launch_pair_forward(const DevSys& s, const Params& p, const float* qt, const float* sig, const float* eps, int T,
                         int cur, double* F, double* ecta, double* esum, cudaStream_t st) {
    const int nb = (s.n + WPB - 1) / WPB;
    k_pair_fwd<<<nb, WPB * 32, 0, st>>>(s, p, diff_params(qt, sig, eps, T), cur, F, ecta);
    k_rowsum<<<1, 256, 0, st>>>(nb, 1, ecta, esum);
}

// Returns the device address of the NSUM coefficient sums (diff_chain).
const double* launch_pair_backward(const DevSys& s, const Params& p, const float* qt, const float* sig, const float* eps,
                                   int T, int cur, const double* U, double w, double* gpos, double* scratch,
                                   cudaStream_t st) {
    const int nb = (s.n + WPB - 1) / WPB;
    float4* u = reinterpret_cast<float4*>(scratch);
    double *part = scratch + 2 * (size_t)s.n, *sums = part + (size_t)NSUM * nb;
    k_upstream<<<(s.n + 255) / 256, 256, 0, st>>>(s.n, U, u);
    k_pair_bwd<<<nb, WPB * 32, 0, st>>>(s, p, diff_params(qt, sig, eps, T), cur, u, (float)w, gpos, part);
    k_rowsum<<<NSUM, 256, 0, st>>>(nb, NSUM, part, sums);
    return sums;
}

int diff_sum_count() { return NSUM; }

// Parameter gradients from the coefficient sums: dL/dq_t, and dL/dsigma_ab,
// dL/deps_ab of the shared entry (a <= b) of each pair of types.
void diff_chain(const double* sums, const float* qt, const float* sig, const float* eps, int T, double* gq, double* gs,
                double* ge) {
    for (int a = 0; a < MAXT; ++a) gq[a] = 0.0;
    for (int k = 0; k < MAXT * MAXT; ++k) gs[k] = ge[k] = 0.0;
    for (int a = 0; a < T; ++a)
        for (int b = 0; b < T; ++b) {
            const int ab = a * MAXT + b, lo = a < b ? ab : b * MAXT + a;
            const double cq = sums[ab], c12 = sums[MAXT * MAXT + ab], c6 = sums[2 * MAXT * MAXT + ab];
            gq[a] += KCOUL_D * cq * qt[b];
            gq[b] += KCOUL_D * cq * qt[a];
            const double s = sig[ab], e = eps[ab], s5 = s * s * s * s * s, s6 = s5 * s;
            gs[lo] += c12 * 48.0 * e * s6 * s5 + c6 * 24.0 * e * s5;
            ge[lo] += c12 * 4.0 * s6 * s6 + c6 * 4.0 * s6;
        }
}
