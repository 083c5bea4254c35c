// precompute.cu -- FP64 leakage-table kernels (Sec. 2.2, Sec. 2.5, Sec. 5.1).
//
// Kernel 1: phi[j] = bin mean of H(a,x) over bin j (k_ij = k0_i phi_j).  Half a
// warp sums one edge's Dawson series, a lane per term, in the series' order.
// Kernel 2, a thread per (class, bin) row; on a moving grid a block takes 127
// rows of a class, or as many whole classes of fewer bins as it has threads for
// their edges, each thread first taking one bin edge, shifted by every face's
// velocity difference in turn (faces with the same shift once), then its row:
// leakage coefficients of
//   eq. x-leakage and eq. z-leakage, the boundary / thin-neighbour form
//   2/(3 dz (k dz + 2 lambda)), probabilities p_X = k_X / sum k accumulated in
//   outcome order, 32-bit thresholds round-half-even(C 2^32) saturated at
//   2^32 - 1, the flag word (2-bit action per outcome, moving, thin) and the
//   mean dwell path 1 / sum_X k_X of the state.  Grey dust (Sec. 2.6): k_s adds
//   to every k_ij; k_a is one more outcome after the leakage ones.
// FP64 throughout: 1 - p of thick states and far-wing bin means (dcalH ~ a dx /
// (sqrt(pi) x^2) ~ 1e-8 against calH ~ 0.886) are below FP32 resolution.  This
// file is compiled without fused multiply-adds so every product and sum is
// rounded as written.
#include <algorithm>
#include <cstring>

#include "grid.h"
#include "pairs.cuh"
#include "voigt.cuh"

namespace rddmc {
namespace {

constexpr int kPhiEdges = 32;   // bin edges of a phi block (half a warp each)
constexpr int kRowEdges = 128;  // bin edges of a rows block (a thread each)

// Latency of one exponential, one division and the ordered sum of 16 terms, for
// any J: 52 us cold where a thread per bin, two series of 34 terms in a row, took
// 167-188 us.
__global__ void __launch_bounds__(kPhiEdges * 16) phi_kernel(const double* __restrict__ edges,
                                                             double* __restrict__ phi, int J, double a) {
    __shared__ VoigtEdge s_edge[kPhiEdges];
    static_assert(kDawsonTerms == 16, "a lane per term");
    const int j0 = (int)blockIdx.x * (kPhiEdges - 1), k = (int)threadIdx.x >> 4, i = (int)threadIdx.x & 15;
    const double x = edges[min(j0 + k, J)], ax = fabs(x);
    double F;
    if (ax < 0.5) {
        F = dawson_series_f64(ax);
    } else {
        F = DawsonCentre(ax).term(i);
    }
    double sum = 0.0;
    for (int q = 15; q >= 0; --q) sum += __shfl_sync(0xffffffffu, F, q, 16);
    if (ax >= 0.5) F = sum * kInvSqrtPi;
    if (i == 0) s_edge[k] = voigt_edge(x, x < 0.0 ? -F : F);
    __syncthreads();
    const int t = (int)threadIdx.x;
    if (t < kPhiEdges - 1 && j0 + t < J) phi[j0 + t] = voigt_bin_mean_f64(a, s_edge[t], s_edge[t + 1]);
}

__device__ __forceinline__ uint32_t quantise_dev(double C) {
    double t = rint(C * 4294967296.0);
    t = fmax(t, 0.0);
    t = fmin(t, 4294967295.0);
    return (uint32_t)t;
}

// Bound by FP64 issue where cells move: the neighbour's opacity over the shifted
// bin takes one Dawson series (32 exponentials and divisions) per edge and
// distinct shift.  16^3 cells x 64 bins, every cell its own shifts: 4.7 ms (12.8 ms
// with two series of 34 terms per row and face).  Classes of few bins share a
// block: 64^3 cells x 1 and x 8 bins 23 and 50 ms, 136 and 142 ms with a block each
// (29 and 129 ms with a thread per row).
template <int NDIM, bool MOVING>
__global__ void __launch_bounds__(kRowEdges)
    rows_kernel(const TableHeader h, const ClassDesc* __restrict__ cdesc, const double* __restrict__ edges,
                const double* __restrict__ phi, uint32_t* __restrict__ rows, uint2* __restrict__ fast,
                float* __restrict__ tau_row, float* __restrict__ rk, uint32_t* __restrict__ abs_thr, int dusty,
                unsigned long long* __restrict__ wq, float* __restrict__ ka_row, int weighted, int tiles,
                int per_block, int64_t nrow) {
    constexpr int K = 2 + 2 * NDIM;
    constexpr int W = NDIM == 1 ? 4 : 8;  // words per row, the last holding the flags
    __shared__ VoigtEdge s_edge[MOVING ? kRowEdges : 1];
    const int J = h.J, tid = (int)threadIdx.x;
    const int64_t lin = (int64_t)blockIdx.x * kRowEdges + tid;
    // static: rows in a line; moving: `per_block` classes, or a tile of one
    int cls, j;
    bool edge = true, row = lin < nrow;  // this thread has an edge, a row
    if (!MOVING) {
        cls = (int)(min(lin, nrow - 1) / J);
        j = (int)(lin - (int64_t)cls * J);
    } else if (per_block > 1) {
        const int64_t c = (int64_t)blockIdx.x * per_block + tid / (J + 1), last = nrow / J - 1;
        cls = (int)min(c, last);
        j = tid % (J + 1);
        edge = tid < per_block * (J + 1) && c <= last;
        row = edge && j < J;
    } else {
        cls = (int)(blockIdx.x / (unsigned)tiles);
        j = (int)(blockIdx.x % (unsigned)tiles) * (kRowEdges - 1) + tid;
        edge = j <= J;
        row = tid < kRowEdges - 1 && j < J;
    }
    const ClassDesc& D = cdesc[cls];
    // bin-mean profile over the bin shifted by each face's velocity difference
    double phi_nb[2 * NDIM];
    if (MOVING) {
#pragma unroll
        for (int f = 0; f < 2 * NDIM; ++f) {
            const double delta = D.face[f].delta;
            phi_nb[f] = 0.0;
            int same = -1;
#pragma unroll
            for (int g = 0; g < f; ++g)
                if (same < 0 && !D.face[g].exterior && D.face[g].delta == delta) same = g;
#pragma unroll
            for (int g = 0; g < f; ++g)
                if (g == same) phi_nb[f] = phi_nb[g];
            const bool shifted = !D.face[f].exterior && delta != 0.0 && same < 0;  // the same in all of a class
            if (!__syncthreads_or(shifted)) continue;  // also: the last face's readers are done
            if (shifted && edge) {
                const double x = edges[j] + delta;
                s_edge[tid] = voigt_edge(x, dawson_f64(x));
            }
            __syncthreads();
            if (shifted && row) phi_nb[f] = voigt_bin_mean_f64(h.a, s_edge[tid], s_edge[tid + 1]);
        }
    }
    if (!row) return;
    const int64_t r = (int64_t)cls * J + j;
    const bool hybrid = h.mode == RDDMC_MODE_HYBRID;
    double dzmin = h.dz[0];
    for (int ax = 1; ax < NDIM; ++ax) dzmin = fmin(dzmin, h.dz[ax]);

    const double dxj = edges[j + 1] - edges[j];
    const double k = D.k0 * phi[j] + D.ks;  // dust scattering adds to every k_ij (Sec. 2.6)
    double rate[K];
    uint32_t act[K];
    // frequency leakage, eq. x-leakage; zero flux beyond the grid ends
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
        const int jn = j + (sd ? 1 : -1);
        if (jn < 0 || jn >= J) { rate[sd] = 0.0; act[sd] = ACT_MOVE; continue; }
        const double dxn = edges[jn + 1] - edges[jn];
        const double kn = D.k0 * phi[jn] + D.ks;
        rate[sd] = 1.0 / (dxj * (dxj / k + dxn / kn));
        act[sd] = (hybrid && kn * dzmin < h.tau_ddmc) ? ACT_TO_MC : ACT_MOVE;
    }
    // spatial leakage, eq. z-leakage; exterior faces and thin neighbours use the
    // extrapolation-distance form of Sec. 5.1
#pragma unroll
    for (int ax = 0; ax < NDIM; ++ax) {
        const double dz = h.dz[ax];
#pragma unroll
        for (int sd = 0; sd < 2; ++sd) {
            const int o = 2 + 2 * ax + sd;
            const FaceDesc& F = D.face[2 * ax + sd];
            const double r_bnd = 1.0 / (3.0 * dz) * 2.0 / (k * dz + 2.0 * h.lambda);
            if (F.exterior) { rate[o] = r_bnd; act[o] = ACT_ESCAPE; continue; }
            // neighbour opacity over the Doppler-shifted bin (eq. velocity-shift)
            const double knb = F.k0_nb * (F.delta == 0.0 ? phi[j] : phi_nb[2 * ax + sd]) + F.ks_nb;
            const double dznb = dz;
            if (hybrid && knb * dznb < h.tau_ddmc) { rate[o] = r_bnd; act[o] = ACT_TO_MC; continue; }
            rate[o] = 1.0 / (3.0 * dz) * 2.0 / (k * dz + knb * dznb);
            act[o] = F.delta != 0.0 ? ACT_REBIN : ACT_MOVE;
        }
    }
    double tot = 0.0;
#pragma unroll
    for (int o = 0; o < K; ++o) tot += rate[o];
    // dust absorption: one more competing process, the last outcome; its lower
    // threshold (the end of the last leakage outcome) is stored apart
    if (dusty) tot += D.ka;
    uint32_t out[W - 1];
    double C = 0.0;
#pragma unroll
    for (int o = 0; o < K - 1; ++o) {
        C += rate[o] / tot;
        out[o] = quantise_dev(C);
    }
    abs_thr[r] = dusty ? quantise_dev(C + rate[K - 1] / tot) : 0xffffffffu;
    // weight method: -ln of the weight kept over one dwell, ln(1 + k_a / K_s),
    // in 2^-40 units (the walk sums these exactly)
    wq[r] = weighted ? (unsigned long long)llrint(log1p(D.ka / tot) * 1099511627776.0) : 0ull;
    ka_row[r] = weighted ? (float)D.ka : 0.0f;  // the time walk attenuates by exp(-k_a l)
    uint32_t fl = 0;
#pragma unroll
    for (int o = 0; o < K; ++o) fl |= (act[o] & 3u) << (2 * o);
    if (act[0] == ACT_MOVE && act[1] == ACT_MOVE) fl |= FLAG_FASTX;
    bool fastz = true;
#pragma unroll
    for (int o = 2; o < K; ++o) fastz = fastz && act[o] == ACT_MOVE;
    if (fastz) fl |= FLAG_FASTZ;
    if (D.moving) fl |= FLAG_MOVING;
    if (hybrid && k * dzmin < h.tau_ddmc) fl |= FLAG_THIN;
    // word order: thr0, thr1, thr2, flags[, thr3..thr6] so that the first 16
    // bytes carry everything a frequency move needs
    fast[r] = make_uint2(out[0], (fl & FLAG_FASTX) ? out[1] : 0u);
    tau_row[r] = (float)(k * dzmin);
    rk[r] = (float)(1.0 / tot);  // mean dwell path 1 / K_s of the state (time-dependent walk)
    if (NDIM == 1) {
        reinterpret_cast<uint4*>(rows)[r] = make_uint4(out[0], out[1], out[2], fl);
    } else {
        uint4* p = reinterpret_cast<uint4*>(rows) + 2 * r;
        p[0] = make_uint4(out[0], out[1], out[2], fl);
        p[1] = make_uint4(out[3], out[4], out[5], out[6]);
    }
}

// The walk's pair of each row (pairs.cuh) from the fast heads of the three rows
// around it in its class block.
__device__ __forceinline__ Pair pair_of(const uint2* __restrict__ fast, int J, int64_t r) {
    const int j = (int)(r % J);
    uint32_t t[3], guard = 0xffffffffu;
#pragma unroll
    for (int i = -1; i <= 1; ++i) {
        const bool in = j + i >= 0 && j + i < J;
        const uint2 f = in ? fast[r + i] : make_uint2(0u, 0xffffffffu);
        t[i + 1] = f.x;
        guard = min(guard, f.y);
    }
    return Pair{t[0], t[1], t[2], guard};
}

// Whether every cell within four moves of cell c along the axes lies in the grid and
// in its class, so that four transitions leave a packet's class as it is: up to 129
// loads per cell, of L1.
template <int NDIM>
__device__ __forceinline__ bool inside_class(const uint32_t* __restrict__ cell_class, int64_t c, int n0, int n1, int n2) {
    constexpr int M = 4, MY = NDIM == 3 ? M : 0;
    const int i0 = (int)(c % n0), i1 = (int)(c / n0 % n1), i2 = (int)(c / ((int64_t)n0 * n1));
    bool in = i0 >= M && i0 + M < n0 && (NDIM == 1 || (i1 >= M && i1 + M < n1 && i2 >= M && i2 + M < n2));
    if (!in) return false;
    const uint32_t k = cell_class[c];
    for (int z = -MY; z <= MY && in; ++z)
        for (int y = abs(z) - MY; y <= MY - abs(z) && in; ++y) {
            const int m = M - abs(z) - abs(y);
            const uint32_t* row = cell_class + c + ((int64_t)z * n1 + y) * n0;
            for (int x = -m; x <= m; ++x) in = in && row[x] == k;
        }
    return in;
}

// A thread per row's pair and, on static grids, per cell's mark, in one launch: a
// few microseconds for small grids, 1.4 ms for 256^3 cells, where a pass over the cells
// on the host took 230 ms of the 1.3 s that the grid takes.
template <int NDIM>
__global__ void pair_kernel(const uint2* __restrict__ fast, Pair* __restrict__ pair, int J, int64_t nrow,
                            const uint32_t* __restrict__ cell_class, uint8_t* __restrict__ inside, int n0, int n1,
                            int n2, int64_t nmark) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nrow) pair[i] = pair_of(fast, J, i);
    if (i < nmark) inside[i] = inside_class<NDIM>(cell_class, i, n0, n1, n2) ? 1 : 0;
}

// Split points (u1, u0) of the three-part rejection envelope of the parallel
// atom velocity, f(u) = e^{-u^2} / (a^2 + (x-u)^2) (Sec. 5.2), for |x| = i/16:
//   u < u1: e^{-u^2} g(u1);  u1 <= u <= u0: c g(u), c = max e^{-u^2} on [u1,u0];
//   u > u0: e^{-u0^2} g(u),  g(u) = 1/(a^2 + (x-u)^2),  u1 <= u0 <= x, u0 >= 0.
// Each piece bounds f, so any such pair samples f exactly; the pair with the
// smallest envelope mass on a grid of candidates gives the best acceptance.
// A block per |x|: a thread takes every 128th candidate, and the block keeps the
// first of the smallest (as one pass in order would).  0.34 ms (5.4 ms with a
// thread per |x|).
__global__ void __launch_bounds__(128) upar_kernel(float2* __restrict__ tab, double a) {
    constexpr int NP = 33, NQ = 34;
    __shared__ double s_m[128], s_th0[NP], s_m3[NP];
    __shared__ int s_c[128];
    const int i = (int)blockIdx.x, tid = (int)threadIdx.x;
    const double x = (double)i / 16.0;
    if (tid < NP) {
        const double u0 = x * tid / 32.0;
        const double th0 = atan((u0 - x) / a);
        s_th0[tid] = th0;
        s_m3[tid] = exp(-u0 * u0) * (1.5707963267948966 - th0) / a;
    }
    __syncthreads();
    auto split = [&](int c, double& u0, double& u1) {
        const int p = c / NQ, q = c % NQ;
        u0 = x * p / 32.0;
        u1 = (q == 33) ? -30.0 : -4.0 + (u0 + 4.0) * q / 32.0;
    };
    double best = 1e300;
    int bc = 0x7fffffff;
    for (int c = tid; c < NP * NQ; c += 128) {
        double u0, u1;
        split(c, u0, u1);
        const double g1 = 1.0 / (a * a + (x - u1) * (x - u1));
        const double m1 = g1 * 0.88622692545275801365 * (1.0 + erf(u1));
        const double cc = u1 <= 0.0 ? 1.0 : exp(-u1 * u1);
        const double m2 = cc * (s_th0[c / NQ] - atan((u1 - x) / a)) / a;
        const double m = m1 + m2 + s_m3[c / NQ];
        if (m < best) { best = m; bc = c; }
    }
    s_m[tid] = best;
    s_c[tid] = bc;
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if (tid < w) {
            const double m = s_m[tid + w];
            const int c = s_c[tid + w];
            if (m < s_m[tid] || (m == s_m[tid] && c < s_c[tid])) {
                s_m[tid] = m;
                s_c[tid] = c;
            }
        }
        __syncthreads();
    }
    if (tid == 0) {
        double u0 = 0.0, u1 = -30.0;
        if (s_m[0] < 1e300) split(s_c[0], u0, u1);
        tab[i] = make_float2((float)u1, (float)fmin(u0, x));
    }
}

}  // namespace

cudaError_t launch_precompute(const rddmc_grid& g, void* d_table, cudaStream_t s) {
    char* base = (char*)d_table;
    const double* edges = (const double*)(base + g.off_edges);
    double* phi = (double*)(base + g.off_phi);
    phi_kernel<<<(g.J + kPhiEdges - 2) / (kPhiEdges - 1), kPhiEdges * 16, 0, s>>>(edges, phi, g.J, g.a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    TableHeader h;
    std::memset(&h, 0, sizeof(h));
    h.J = g.J;
    h.mode = g.params.mode;
    h.tau_ddmc = g.params.tau_ddmc;
    h.lambda = g.params.lambda;
    h.f_mu = g.params.f_mu;
    h.a = g.a;
    for (int a = 0; a < 3; ++a) h.dz[a] = 2.0 * g.R / g.n[a];
    const int64_t nrow = (int64_t)g.n_class * g.J;
    const int tiles = (g.J + kRowEdges - 2) / (kRowEdges - 1);
    // Whole classes of a block's edges, once every SM has two blocks: one warp keeps
    // an SM's FP64 units busy, so few classes are spread first (270 classes x 16 bins:
    // 0.34 ms from grid to table, 0.40 with seven to a block), and many more where
    // that saves no warps (1000 classes x 62 bins: 1.0 ms, 1.1 with two to a block).
    int dev = 0, nsm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    const int whole = kRowEdges / (g.J + 1), alone = (g.J + 32) / 32 * 32;  // threads of a class's own warps
    const int per_block = std::min(whole, g.n_class / ((whole * alone > kRowEdges ? 2 : 16) * nsm));
    const int64_t blocks = !g.moving ? (nrow + kRowEdges - 1) / kRowEdges
                           : per_block > 1 ? (g.n_class + per_block - 1) / per_block
                                           : (int64_t)g.n_class * tiles;
    const ClassDesc* cd = (const ClassDesc*)(base + g.off_cdesc);
    uint32_t* rows = (uint32_t*)(base + g.off_rows);
    uint2* fast = (uint2*)(base + g.off_fast);
    float* tau_row = (float*)(base + g.off_tau);
    float* rk = (float*)(base + g.off_rk);
    uint32_t* abs_thr = (uint32_t*)(base + g.off_abs);
    const int dusty = g.dusty() ? 1 : 0;
    unsigned long long* wq = (unsigned long long*)(base + g.off_wq);
    const int weighted = g.weighted() ? 1 : 0;
    float* ka_row = (float*)(base + g.off_ka);
    auto rows_k = g.ndim == 1 ? (g.moving ? rows_kernel<1, true> : rows_kernel<1, false>)
                              : (g.moving ? rows_kernel<3, true> : rows_kernel<3, false>);
    rows_k<<<(unsigned)blocks, kRowEdges, 0, s>>>(h, cd, edges, phi, rows, fast, tau_row, rk, abs_thr, dusty, wq,
                                                  ka_row, weighted, tiles, per_block, nrow);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (g.pairs()) {
        const int64_t nmark = g.inside() ? g.ncell : 0;
        const auto pair_k = g.ndim == 1 ? pair_kernel<1> : pair_kernel<3>;
        pair_k<<<(unsigned)((std::max(nrow, nmark) + 255) / 256), 256, 0, s>>>(
            fast, (Pair*)(base + g.off_pair), g.J, nrow, (const uint32_t*)(base + g.off_class),
            (uint8_t*)(base + g.off_inside), g.n[0], g.n[1], g.n[2], nmark);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // the u_par envelope table serves only the continuous MC of the hybrid scheme
    if (g.params.mode == RDDMC_MODE_HYBRID)
        upar_kernel<<<kUparN, 128, 0, s>>>((float2*)(base + g.off_upar), g.a);
    return cudaGetLastError();
}

}  // namespace rddmc
