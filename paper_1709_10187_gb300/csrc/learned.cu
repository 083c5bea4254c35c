// learned.cu -- the learned exit proposal: first-passage data generation, the
// BF16 MLP (forward, backward, softmax cross-entropy, Adam) on tensor cores,
// and batched inference that samples exits for parked packets.
//
// First passages: sample i picks a density level, a start bin and a cell of a
// b^3 brick of uniform medium from its event stream, folds the cell into the
// fundamental domain of the cube's symmetry group and walks from it with the
// rows of an interior cell of that medium (the same rows and transition
// stream as the walk) until a spatial move leaves the brick.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "grid.h"
#include "learned_common.cuh"
#include "umma.cuh"

namespace rddmc {
namespace {

constexpr int kMaxLevels = 64;

struct FpParams {
    const uint4* rows[kMaxLevels];  // 3D rows (two uint4) of the interior class, J per level
    const uint2* fast[kMaxLevels];
    int jlo[kMaxLevels], jhi[kMaxLevels];
    int L, J, b;
    uint32_t k0, k1;
    unsigned long long p0, n, cap;
    int* out;                    // 8 ints per sample (rddmc_fp_generate)
    unsigned long long* steps;   // transitions per sample
    // optional training tensors: inputs (bf16, 16 per sample), targets
    __nv_bfloat16* X;
    int* tA;                     // exit face * J + exit bin, -1 when the step cap was reached
    int* tB;                     // log2 step bucket
    int* tC;                     // exit face * b^2 + exit position, -1 when the step cap was reached
    const float* lk;             // per level: log10(k0 dz)
    const float* lp;             // per bin: log10 of the bin-mean profile
    const float* xc;             // per bin: centre frequency
    FeatConst fc;
};

__device__ __forceinline__ uint4 fp_philox(uint4 c, uint32_t k0, uint32_t k1) { return philox4x32_10(c, k0, k1); }

__global__ void __launch_bounds__(256) fp_kernel(const FpParams P) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += stride) {
        const unsigned long long pk = P.p0 + i;
        const uint32_t pl = (uint32_t)pk, ph = (uint32_t)(pk >> 32);
        const uint4 ew = fp_philox(make_uint4(0u, 0u, pl, ph | 0x80000000u), P.k0, P.k1);  // event words 0..3
        const int l = min((int)(((unsigned long long)ew.x * (unsigned long long)P.L) >> 32), P.L - 1);
        const int nb = P.jhi[l] - P.jlo[l] + 1;
        int j = P.jlo[l] + (int)(((unsigned long long)ew.y * (unsigned long long)nb) >> 32);
        const int m = (int)(((unsigned long long)ew.z * (unsigned long long)(P.b * P.b * P.b)) >> 32);
        const int lw[3] = {m % P.b, (m / P.b) % P.b, m / (P.b * P.b)};
        int idx[3], perm[3];
        bool flip[3];
        fold_cell(lw, P.b, idx, perm, flip);
        const uint4* rows = P.rows[l];
        const uint2* fast = P.fast[l];
        const int j0 = j;
        const int start = idx[0] + P.b * (idx[1] + P.b * idx[2]);
        const int c0[3] = {idx[0], idx[1], idx[2]};
        int face = 6, pos = -1;
        unsigned long long t = 0;
        const unsigned J1 = (unsigned)P.J - 1u;
        while (t < P.cap && face == 6) {
            const unsigned long long blk = t >> 2;
            const uint4 r = fp_philox(make_uint4((uint32_t)blk, (uint32_t)(blk >> 32), pl, ph), P.k0, P.k1);
            for (unsigned q = (unsigned)(t & 3u); q < 4u && t < P.cap; ++q) {
                const unsigned w = q == 0 ? r.x : (q == 1 ? r.y : (q == 2 ? r.z : r.w));
                ++t;
                const unsigned jj = min((unsigned)j, J1);
                const uint2 f = __ldg(&fast[jj]);
                if (w < f.y) { j += (w >= f.x) ? 1 : -1; continue; }
                const uint4 a = __ldg(&rows[2 * jj]), c = __ldg(&rows[2 * jj + 1]);
                const unsigned o = (unsigned)(w >= a.x) + (unsigned)(w >= a.y) + (unsigned)(w >= a.z) +
                                   (unsigned)(w >= c.x) + (unsigned)(w >= c.y) + (unsigned)(w >= c.z) +
                                   (unsigned)(w >= c.w);
                if (o < 2u) { j += o ? 1 : -1; continue; }
                const int fc = (int)o - 2, ax = fc >> 1, side = (fc & 1) ? 1 : -1;
                if (idx[ax] + side < 0 || idx[ax] + side >= P.b) {
                    face = fc;
                    const int u = ax == 0 ? 1 : 0, v = ax == 2 ? 1 : 2;  // the other two axes, lower first
                    pos = idx[u] + P.b * idx[v];
                    break;
                }
                idx[ax] += side;
            }
        }
        int* o8 = P.out + 8 * i;
        o8[0] = l;
        o8[1] = j0;
        o8[2] = start;
        o8[3] = face;
        o8[4] = j;
        o8[5] = pos;
        o8[6] = 0;
        o8[7] = 0;
        P.steps[i] = t;
        if (P.X) {
            features(P.lk[l], P.lp[j0], P.xc[j0], c0, P.b, P.fc, P.X + kFeat * i);
            P.tA[i] = face < 6 ? face * P.J + min(max(j, 0), P.J - 1) : -1;
            P.tB[i] = step_bucket(t);
            if (P.tC) P.tC[i] = face < 6 ? face * P.b * P.b + pos : -1;
        }
    }
}

}  // namespace
}  // namespace rddmc

using namespace rddmc;

extern "C" {

int rddmc_cell_tau(const rddmc_grid* g, const void* d_table, int64_t cell, float* tau, void* stream) {
    if (!g || !d_table || !tau || cell < 0 || cell >= g->ncell) return RDDMC_ERR_ARG;
    if (!g->precomputed) return RDDMC_ERR_TABLE;
    const uint32_t cls = g->cell_class[cell];
    if (cls == UINT32_MAX) return RDDMC_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const char* src = (const char*)d_table + g->off_tau + (uint64_t)cls * g->J * 4;
    if (cudaMemcpyAsync(tau, src, (size_t)g->J * 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) return RDDMC_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? RDDMC_OK : RDDMC_ERR_CUDA;
}

int rddmc_fp_generate(const rddmc_grid* const* grids, const void* const* d_tables, int L, int b, const int32_t* jlo,
                      const int32_t* jhi, uint64_t seed, uint64_t p0, uint64_t n, uint64_t cap, int32_t* d_out,
                      uint64_t* d_steps, const rddmc_fp_train* train, void* stream) {
    if (!grids || !d_tables || !jlo || !jhi || !d_out || !d_steps) return RDDMC_ERR_ARG;
    if (L < 1 || L > kMaxLevels || b < 1 || b > 64 || n == 0 || cap == 0) return RDDMC_ERR_ARG;
    FpParams P;
    std::memset(&P, 0, sizeof(P));
    int J = -1;
    for (int l = 0; l < L; ++l) {
        const rddmc_grid* g = grids[l];
        if (!g || !d_tables[l]) return RDDMC_ERR_ARG;
        if (!g->precomputed) return RDDMC_ERR_TABLE;
        if (g->ndim != 3 || g->params.mode != RDDMC_MODE_DDMC || g->dusty() || g->weighted())
            return RDDMC_ERR_UNSUPPORTED;
        if (J < 0) J = g->J;
        if (g->J != J) return RDDMC_ERR_ARG;
        int idx[3] = {g->n[0] / 2, g->n[1] / 2, g->n[2] / 2};
        for (int a = 0; a < 3; ++a)
            for (int sd = -1; sd <= 1; sd += 2) {
                int nidx[3] = {idx[0], idx[1], idx[2]};
                nidx[a] += sd;
                if (!g->in_medium(nidx)) return RDDMC_ERR_ARG;  // the centre cell must be interior
            }
        const uint32_t cls = g->cell_class[g->cell_of(idx)];
        const char* tb = (const char*)d_tables[l];
        P.rows[l] = (const uint4*)(tb + g->off_rows) + (uint64_t)cls * J * 2;
        P.fast[l] = (const uint2*)(tb + g->off_fast) + (uint64_t)cls * J;
        if (jlo[l] < 0 || jhi[l] >= J || jlo[l] > jhi[l]) return RDDMC_ERR_ARG;
        P.jlo[l] = jlo[l];
        P.jhi[l] = jhi[l];
    }
    P.L = L; P.J = J; P.b = b;
    P.k0 = (uint32_t)seed; P.k1 = (uint32_t)(seed >> 32);
    P.p0 = p0; P.n = n; P.cap = cap;
    P.out = d_out;
    P.steps = (unsigned long long*)d_steps;
    if (train) {
        if (!train->d_x || !train->d_ta || !train->d_tb || !train->d_lk || !train->d_lp || !train->d_xc)
            return RDDMC_ERR_ARG;
        P.X = (__nv_bfloat16*)train->d_x;
        P.tA = train->d_ta;
        P.tB = train->d_tb;
        P.tC = train->d_tc;
        P.lk = train->d_lk;
        P.lp = train->d_lp;
        P.xc = train->d_xc;
        P.fc.log_b = log10f((float)b);
        P.fc.log_a = (float)log10(grids[0]->a);
        P.fc.inv_xs = (float)(1.0 / std::max(std::fabs(grids[0]->edges.front()), std::fabs(grids[0]->edges.back())));
    }
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return RDDMC_ERR_CUDA;
    const unsigned long long want = (n + 255) / 256;
    const unsigned blocks = (unsigned)(want < (unsigned long long)nsm * 8 ? want : (unsigned long long)nsm * 8);
    fp_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(P);
    return cudaGetLastError() == cudaSuccess ? RDDMC_OK : RDDMC_ERR_CUDA;
}

}  // extern "C"

// ===================================================================== MLP
// Architecture: n_in = 16 inputs -> 3 hidden layers of 128 (ReLU) -> n_out
// logits (a multiple of 16): head A over [0, nA) (exit face x exit bin),
// head B over [nA, nA + nB) (log2 step bucket) and head C over
// [nA + nB, nA + nB + 6 S) (exit cell on each face, S = b^2 per face, used
// one slice at a time); columns past the heads are padding.  Parameters, FP32 master copy and BF16 copy in the same order:
// W1[128x16] b1[128] W2[128x128] b2[128] W3[128x128] b3[128] W4[n_out x 128]
// b4[n_out].  Every matrix product runs on the tcgen05 tensor cores
// (umma.cuh: BF16 operands, FP32 accumulators in tensor memory), the backward
// ones on the activations and weights as they lie in memory; softmax,
// cross-entropy, bias sums and Adam in FP32.
namespace rddmc {
namespace {

constexpr int kIn = 16, kHid = 128;

struct MlpOffsets {
    uint64_t W[4], b[4], total;
};

MlpOffsets mlp_offsets(int n_out) {
    MlpOffsets o;
    const int fan_in[4] = {kIn, kHid, kHid, kHid}, fan_out[4] = {kHid, kHid, kHid, n_out};
    uint64_t off = 0;
    for (int l = 0; l < 4; ++l) {
        o.W[l] = off; off += (uint64_t)fan_in[l] * fan_out[l];
        o.b[l] = off; off += (uint64_t)fan_out[l];
    }
    o.total = off;
    return o;
}

// Softmax cross-entropy of the heads, a warp per row: loss += CE_A + CE_B (+ CE_C
// over the S logits of the target's slice when head C is present and its target
// is >= 0), summed over the batch; dlogits = (softmax - onehot) / B on the logits
// a head used, zero elsewhere, in BF16 for the products, and its FP32 column sums
// added to db.  ACC: every warp sums its rows' columns in shared memory (n_out
// floats a warp) before the block adds them to db; otherwise (an n_out past
// shared memory) each goes straight to db.
//
// One pass over the FP32 logits (the second and third read them back through L1)
// and one over the BF16 gradients; the FP32 gradients are not stored.
template <bool ACC>
__global__ void softmax_ce_kernel(const float* __restrict__ logits, int n_out, int nA, int nB, int nC, int S,
                                  const int* __restrict__ tA, const int* __restrict__ tB, const int* __restrict__ tC,
                                  int Bsz, __nv_bfloat16* __restrict__ dlogb, float* __restrict__ db, float* loss) {
    extern __shared__ float s_acc[];
    const int warps = (int)blockDim.x >> 5, warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    float* acc = s_acc + (size_t)warp * n_out;
    if (ACC)
        for (int k = lane; k < n_out; k += 32) acc[k] = 0.0f;
    float total = 0.0f;
    for (int row = (int)blockIdx.x * warps + warp; row < Bsz; row += (int)gridDim.x * warps) {
        const float* z = logits + (size_t)row * n_out;
        __nv_bfloat16* gb = dlogb + (size_t)row * n_out;
        const bool skip = tA[row] < 0;  // ignored sample: no loss, no gradient
        // zero everything past heads A and B (head C's unused slices, padding)
        for (int k = (skip ? 0 : nA + nB) + lane; k < n_out; k += 32) gb[k] = __float2bfloat16(0.0f);
        if (skip) continue;
        int tc = (nC > 0 && tC) ? tC[row] : -1;
        if (tc >= nC) tc = -1;
        const int nh = tc >= 0 ? 3 : 2;
        for (int h = 0; h < nh; ++h) {
            int lo, hi, tgt;
            if (h == 0) { lo = 0; hi = nA; tgt = tA[row]; }
            else if (h == 1) { lo = nA; hi = nA + nB; tgt = nA + tB[row]; }
            else { lo = nA + nB + (tc / S) * S; hi = lo + S; tgt = nA + nB + tc; }
            float mx = -3.0e38f;
#pragma unroll 8
            for (int k = lo + lane; k < hi; k += 32) mx = fmaxf(mx, z[k]);
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            float se = 0.0f;
#pragma unroll 8
            for (int k = lo + lane; k < hi; k += 32) se += __expf(z[k] - mx);
            for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
            const float lse = mx + __logf(se);
            total += lse - z[tgt];
            __syncwarp();  // the zeros above and the columns of the last head come from other lanes
#pragma unroll 8
            for (int k = lo + lane; k < hi; k += 32) {
                const float g = (__expf(z[k] - lse) - (k == tgt ? 1.0f : 0.0f)) / (float)Bsz;
                gb[k] = __float2bfloat16(g);
                if (ACC) acc[k] += g;
                else atomicAdd(&db[k], g);
            }
        }
        __syncwarp();
    }
    if (lane == 0 && total != 0.0f) atomicAdd(loss, total);
    if (ACC) {
        __syncthreads();
        for (int k = (int)threadIdx.x; k < n_out; k += (int)blockDim.x) {
            float t = 0.0f;
            for (int w = 0; w < warps; ++w) t += s_acc[(size_t)w * n_out + k];
            if (t != 0.0f) atomicAdd(&db[k], t);
        }
    }
}

// The same with a row of head A in registers, a warp per row: V 16-byte pieces
// a lane hold its logits from one read to the gradients, V more its columns'
// sums over the warp's rows; only heads B and C (the columns past nA) sum in
// shared memory.  nA and n_out are multiples of 4, nA <= 128 V.  Bound by the
// logits' read and the gradients' write, and before by reading each logit three
// times, by a shared-memory sum per column and by 608 blocks' atomics on every
// column: a training step of 8192 rows, 1536 + 32 + 216 logits, 277 -> 195 us.
template <int V>
__global__ void __launch_bounds__(V <= 12 ? 512 : 384, 1)
softmax_ce_rows_kernel(const float* __restrict__ logits, int n_out, int nA, int nB, int nC, int S,
                       const int* __restrict__ tA, const int* __restrict__ tB, const int* __restrict__ tC, int Bsz,
                       __nv_bfloat16* __restrict__ dlogb, float* __restrict__ db, float* loss) {
    extern __shared__ __align__(16) float s_sum[];  // warps x n_out
    const int warps = (int)blockDim.x >> 5, warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    float* acc = s_sum + (size_t)warp * n_out;
    for (int k = nA + lane; k < n_out; k += 32) acc[k] = 0.0f;
    float4 sum[V];
#pragma unroll
    for (int i = 0; i < V; ++i) sum[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const int n4 = nA >> 2;
    // x / Bsz: a product where it is exact
    const bool pow2 = (Bsz & (Bsz - 1)) == 0;
    const float inv = 1.0f / (float)Bsz;
    auto mean = [&](float x) { return pow2 ? x * inv : x / (float)Bsz; };
    float total = 0.0f;
    for (int row = (int)blockIdx.x * warps + warp; row < Bsz; row += (int)gridDim.x * warps) {
        const float* z = logits + (size_t)row * n_out;
        __nv_bfloat16* gb = dlogb + (size_t)row * n_out;
        const int ta = tA[row];
        const bool skip = ta < 0;  // ignored sample: no loss, no gradient
        for (int k = (skip ? 0 : nA + nB) + lane; k < n_out; k += 32) gb[k] = __float2bfloat16(0.0f);
        if (skip) continue;
        int tc = (nC > 0 && tC) ? tC[row] : -1;
        if (tc >= nC) tc = -1;
        {
            float4 v[V];
            float mx = -3.0e38f;
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (lane + 32 * i < n4) v[i] = __ldcs(reinterpret_cast<const float4*>(z) + lane + 32 * i);
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (lane + 32 * i < n4) mx = fmaxf(mx, fmaxf(fmaxf(v[i].x, v[i].y), fmaxf(v[i].z, v[i].w)));
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            float se = 0.0f;
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (lane + 32 * i < n4)
                    se += (__expf(v[i].x - mx) + __expf(v[i].y - mx)) + (__expf(v[i].z - mx) + __expf(v[i].w - mx));
            for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
            const float lse = mx + __logf(se);
            total += lse - z[ta];
#pragma unroll
            for (int i = 0; i < V; ++i) {
                if (lane + 32 * i >= n4) continue;
                const int k = 4 * (lane + 32 * i);
                float4 g;
                g.x = mean(__expf(v[i].x - lse) - (k == ta ? 1.0f : 0.0f));
                g.y = mean(__expf(v[i].y - lse) - (k + 1 == ta ? 1.0f : 0.0f));
                g.z = mean(__expf(v[i].z - lse) - (k + 2 == ta ? 1.0f : 0.0f));
                g.w = mean(__expf(v[i].w - lse) - (k + 3 == ta ? 1.0f : 0.0f));
                const __nv_bfloat162 lo = __floats2bfloat162_rn(g.x, g.y), hi = __floats2bfloat162_rn(g.z, g.w);
                *reinterpret_cast<uint2*>(gb + k) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                                                               *reinterpret_cast<const uint32_t*>(&hi));
                sum[i].x += g.x;
                sum[i].y += g.y;
                sum[i].z += g.z;
                sum[i].w += g.w;
            }
        }
        for (int h = 1; h < (tc >= 0 ? 3 : 2); ++h) {
            const int lo = h == 1 ? nA : nA + nB + (tc / S) * S, hi = h == 1 ? nA + nB : lo + S;
            const int tgt = h == 1 ? nA + tB[row] : nA + nB + tc;
            float mx = -3.0e38f;
            for (int k = lo + lane; k < hi; k += 32) mx = fmaxf(mx, z[k]);
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            float se = 0.0f;
            for (int k = lo + lane; k < hi; k += 32) se += __expf(z[k] - mx);
            for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
            const float lse = mx + __logf(se);
            total += lse - z[tgt];
            __syncwarp();  // the zeros above and the columns of the last head come from other lanes
            for (int k = lo + lane; k < hi; k += 32) {
                const float g = (__expf(z[k] - lse) - (k == tgt ? 1.0f : 0.0f)) / (float)Bsz;
                gb[k] = __float2bfloat16(g);
                acc[k] += g;
            }
        }
        __syncwarp();
    }
    if (lane == 0 && total != 0.0f) atomicAdd(loss, total);
#pragma unroll
    for (int i = 0; i < V; ++i)
        if (lane + 32 * i < n4) reinterpret_cast<float4*>(acc)[lane + 32 * i] = sum[i];
    __syncthreads();
    for (int k = (int)threadIdx.x; k < n_out; k += (int)blockDim.x) {
        float t = 0.0f;
        for (int w = 0; w < warps; ++w) t += s_sum[(size_t)w * n_out + k];
        if (t != 0.0f) atomicAdd(&db[k], t);
    }
}

template <int V>
cudaError_t softmax_ce_rows(const float* logits, int n_out, int nA, int nB, int nC, int S, const int* tA, const int* tB,
                            const int* tC, int Bsz, __nv_bfloat16* dlogb, float* db, float* loss, cudaStream_t s) {
    const int warps = V <= 12 ? 16 : 12;
    const size_t smem = (size_t)warps * n_out * sizeof(float);
    int dev = 0, nsm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = allow_smem(softmax_ce_rows_kernel<V>, kSmemMost)) != cudaSuccess)
        return e;
    softmax_ce_rows_kernel<V><<<std::min((Bsz + warps - 1) / warps, nsm), warps * 32, smem, s>>>(
        logits, n_out, nA, nB, nC, S, tA, tB, tC, Bsz, dlogb, db, loss);
    return cudaGetLastError();
}

cudaError_t softmax_ce(const float* logits, int n_out, int nA, int nB, int nC, int S, const int* tA, const int* tB,
                       const int* tC, int Bsz, __nv_bfloat16* dlogb, float* db, float* loss, cudaStream_t s) {
    // rows that fit a warp's registers and, 16 at a time, a block's shared memory
    // (grids of up to 341 bins); the heads' columns one by one otherwise
    if (nA % 4 == 0 && n_out % 4 == 0 && nA <= 2048 && n_out <= 3200) {
        const auto rows = nA <= 512 ? softmax_ce_rows<4>
                                    : (nA <= 1024 ? softmax_ce_rows<8> : (nA <= 1536 ? softmax_ce_rows<12> : softmax_ce_rows<16>));
        return rows(logits, n_out, nA, nB, nC, S, tA, tB, tC, Bsz, dlogb, db, loss, s);
    }
    // at most 64 KiB of column sums a block (three blocks per SM), 8 warps while they fit
    const size_t row = (size_t)n_out * sizeof(float);
    const int warps = (int)std::max<size_t>(1, std::min<size_t>(8, (64u * 1024u) / row));
    if (row > kSmemMost) {
        softmax_ce_kernel<false><<<(Bsz + 7) / 8, 256, 0, s>>>(logits, n_out, nA, nB, nC, S, tA, tB, tC, Bsz, dlogb,
                                                              db, loss);
        return cudaGetLastError();
    }
    const size_t smem = row * warps;
    cudaError_t e = allow_smem(softmax_ce_kernel<true>, kSmemMost);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, softmax_ce_kernel<true>, warps * 32, smem)) !=
            cudaSuccess)
        return e;
    const int blocks = std::min((Bsz + warps - 1) / warps, nsm * std::max(1, per_sm));
    softmax_ce_kernel<true><<<blocks, warps * 32, smem, s>>>(logits, n_out, nA, nB, nC, S, tA, tB, tC, Bsz, dlogb, db,
                                                            loss);
    return cudaGetLastError();
}

// K splits for a weight-gradient product (K = batch rows) on 128 x min(N, 256)
// tensor-core tiles: about two waves of CTAs over the GPU, at most one split
// per 64-column panel of K.
int ksplit_for(int M, int N, int K) {
    const int nt = std::min(256, N);
    const int tiles = ((M + 127) / 128) * ((N + nt - 1) / nt);
    return std::max(1, std::min((K + 63) / 64, (304 + tiles - 1) / tiles));
}

__global__ void adam_kernel(uint64_t n, float* __restrict__ w, __nv_bfloat16* __restrict__ wb,
                            const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi, vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    wb[i] = __float2bfloat16(wi);
}

__global__ void to_bf16_kernel(uint64_t n, const float* __restrict__ w, __nv_bfloat16* __restrict__ wb) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) wb[i] = __float2bfloat16(w[i]);
}

// Work buffer (rows B a multiple of 64): H1 H2 H3 bf16 [B x 128] each, dHb bf16
// [B x 128] x2, logits f32 [B x n_out], dlogb bf16 [B x n_out], XT bf16 [16 x B].
struct MlpWork {
    __nv_bfloat16 *H[3], *dHb[2], *dlogb, *XT;
    float* logits;
};

uint64_t mlp_work_bytes(int Bsz, int n_out) {
    return align256((uint64_t)Bsz * kHid * 2) * 5 + align256((uint64_t)Bsz * n_out * 4) +
           align256((uint64_t)Bsz * n_out * 2) + align256((uint64_t)Bsz * kIn * 2);
}

MlpWork mlp_work(void* d_work, int Bsz, int n_out) {
    char* p = (char*)d_work;
    const uint64_t bh = (uint64_t)Bsz * kHid;
    MlpWork w;
    for (int i = 0; i < 3; ++i) { w.H[i] = (__nv_bfloat16*)p; p += align256(bh * 2); }
    for (int i = 0; i < 2; ++i) { w.dHb[i] = (__nv_bfloat16*)p; p += align256(bh * 2); }
    w.logits = (float*)p; p += align256((uint64_t)Bsz * n_out * 4);
    w.dlogb = (__nv_bfloat16*)p; p += align256((uint64_t)Bsz * n_out * 2);
    w.XT = (__nv_bfloat16*)p;
    return w;
}

// Device status of the tensor-core products (set when a bounded wait runs out).
__device__ unsigned g_tc_err = 0;

// The status word's device address, looked up on every call (a cheap host
// call; a cached address would go stale when the device is reset and the
// module loaded again).
unsigned* tc_err_ptr() {
    void* a = nullptr;
    if (cudaGetSymbolAddress(&a, g_tc_err) != cudaSuccess) return nullptr;
    return (unsigned*)a;
}

// C = epi(A W^T (+ bias)) on tcgen05 (umma.cuh): A [M x K], W [N x K]; an operand
// given MN-major lies as [K x M] (or [K x N]) row-major.  ksplit > 1 only with
// F32_ADD.  K <= 128 and not a multiple of 64 is staged by the threads (K-major),
// everything else by TMA.
template <int EPI, bool MNA = false, bool MNB = false>
cudaError_t gemm_tc(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* W, int ldw,
                    const float* bias, const __nv_bfloat16* mask, int ldmask, __nv_bfloat16* outb, float* outf,
                    int ldc, cudaStream_t s, int ksplit = 1, float* colsum = nullptr) {
    unsigned* err = tc_err_ptr();
    if (!err || K % 16 || N % 16 || ksplit < 1 || (ksplit > 1 && EPI != umma::F32_ADD)) return cudaErrorInvalidValue;
    const int NT = std::min(256, N);
    if (MNB && NT % 64) return cudaErrorInvalidValue;
    if ((EPI == umma::RELU_BF16 || EPI == umma::MASK_BF16) && N != kHid) return cudaErrorInvalidValue;
    const bool staged = !MNA && !MNB && K <= 128 && K % umma::kPanel != 0;
    if (staged && ksplit != 1) return cudaErrorInvalidValue;
    // panels in flight: three of a split (two CTAs per SM), up to six where one
    // CTA runs the whole of a long K
    const int kpanels = (K + umma::kPanel - 1) / umma::kPanel;
    const int per_split = (kpanels + ksplit - 1) / ksplit;
    int nstage = staged ? 2 : std::min(per_split, ksplit > 1 ? 3 : umma::kMaxStages);
    while (nstage > 2 && umma::smem_bytes(NT, nstage, MNB) > kSmemMost) --nstage;
    // at least 80 KiB of shared memory: at most two CTAs per SM, so their TMEM
    // accumulators (<= 256 columns each) always fit the SM's 512 columns
    const size_t smem = std::max<size_t>(umma::smem_bytes(NT, nstage, MNB), 80 * 1024);
    dim3 grid((N + NT - 1) / NT, (M + umma::kTileM - 1) / umma::kTileM, ksplit);
    CUtensorMap mapA, mapW;
    std::memset(&mapA, 0, sizeof(mapA));
    std::memset(&mapW, 0, sizeof(mapW));
    if (!staged && !((MNA ? umma::make_map(&mapA, A, K, M, lda, umma::kPanel)
                          : umma::make_map(&mapA, A, M, K, lda, umma::kTileM)) &&
                     (MNB ? umma::make_map(&mapW, W, K, N, ldw, umma::kPanel)
                          : umma::make_map(&mapW, W, N, K, ldw, NT))))
        return cudaErrorInvalidValue;
    auto kern = umma::gemm_tc_kernel<EPI, true, MNA, MNB>;
    if constexpr (!MNA && !MNB)
        if (staged) kern = umma::gemm_tc_kernel<EPI, false, false, false>;
    cudaError_t e = allow_smem(kern, kSmemMost);
    if (e != cudaSuccess) return e;
    kern<<<grid, umma::kThreads, smem, s>>>(M, N, K, NT, A, lda, W, ldw, mapA, mapW, bias, mask, ldmask, outb, outf,
                                            ldc, colsum, nstage, err);
    return cudaGetLastError();
}

cudaError_t transpose(const __nv_bfloat16* in, int rows, int cols, int ld_in, __nv_bfloat16* out, int ld_out,
                      cudaStream_t s) {
    dim3 grid((cols + 31) / 32, (rows + 31) / 32);
    umma::transpose_bf16_kernel<<<grid, dim3(32, 8), 0, s>>>(in, rows, cols, ld_in, out, ld_out);
    return cudaGetLastError();
}

cudaError_t mlp_forward(int n_out, const float* wf, const __nv_bfloat16* wb, const __nv_bfloat16* X, int Bsz,
                        const MlpWork& w, float* logits, cudaStream_t s) {
    const MlpOffsets o = mlp_offsets(n_out);
    cudaError_t e;
    if ((e = gemm_tc<umma::RELU_BF16>(Bsz, kHid, kIn, X, kIn, wb + o.W[0], kIn, wf + o.b[0], nullptr, 0, w.H[0],
                                      nullptr, kHid, s)) != cudaSuccess)
        return e;
    for (int l = 1; l < 3; ++l)
        if ((e = gemm_tc<umma::RELU_BF16>(Bsz, kHid, kHid, w.H[l - 1], kHid, wb + o.W[l], kHid, wf + o.b[l],
                                          nullptr, 0, w.H[l], nullptr, kHid, s)) != cudaSuccess)
            return e;
    return gemm_tc<umma::LINEAR_F32>(Bsz, n_out, kHid, w.H[2], kHid, wb + o.W[3], kHid, wf + o.b[3], nullptr, 0,
                                     nullptr, logits, n_out, s);
}

}  // namespace
}  // namespace rddmc

extern "C" {

uint64_t rddmc_mlp_param_count(int n_out) { return (n_out > 0 && n_out % 16 == 0) ? mlp_offsets(n_out).total : 0; }

uint64_t rddmc_mlp_work_bytes(int batch, int n_out) {
    return (batch > 0 && batch % 64 == 0 && n_out > 0 && n_out % 16 == 0) ? mlp_work_bytes(batch, n_out) : 0;
}

int rddmc_mlp_to_bf16(int n_out, const float* d_wf, void* d_wb, void* stream) {
    const uint64_t n = rddmc_mlp_param_count(n_out);
    if (!n || !d_wf || !d_wb) return RDDMC_ERR_ARG;
    to_bf16_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(n, d_wf, (__nv_bfloat16*)d_wb);
    return cudaGetLastError() == cudaSuccess ? RDDMC_OK : RDDMC_ERR_CUDA;
}

int rddmc_mlp_forward(int n_out, const float* d_wf, const void* d_wb, const void* d_x, int batch, void* d_work,
                      float* d_logits, void* stream) {
    if (!rddmc_mlp_param_count(n_out) || !rddmc_mlp_work_bytes(batch, n_out) || !d_wf || !d_wb || !d_x || !d_work)
        return RDDMC_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const MlpWork w = mlp_work(d_work, batch, n_out);
    return mlp_forward(n_out, d_wf, (const __nv_bfloat16*)d_wb, (const __nv_bfloat16*)d_x, batch, w,
                       d_logits ? d_logits : w.logits, s) == cudaSuccess
               ? RDDMC_OK
               : RDDMC_ERR_CUDA;
}

int rddmc_mlp_loss_grad(int n_out, int nA, int nB, int nC, int S, const float* d_wf, const void* d_wb,
                        const void* d_x, const int32_t* d_ta, const int32_t* d_tb, const int32_t* d_tc, int batch,
                        void* d_work, float* d_grad, float* d_loss, void* stream) {
    if (!rddmc_mlp_param_count(n_out) || !rddmc_mlp_work_bytes(batch, n_out) || nA < 1 || nB < 1 || nC < 0 ||
        nA + nB + nC > n_out || !d_wf || !d_wb || !d_x || !d_ta || !d_tb || !d_work || !d_grad || !d_loss)
        return RDDMC_ERR_ARG;
    if (nC > 0 && (S < 1 || nC != 6 * S || !d_tc)) return RDDMC_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const MlpOffsets o = mlp_offsets(n_out);
    const __nv_bfloat16* wb = (const __nv_bfloat16*)d_wb;
    const __nv_bfloat16* X = (const __nv_bfloat16*)d_x;
    const MlpWork w = mlp_work(d_work, batch, n_out);
    if (mlp_forward(n_out, d_wf, wb, X, batch, w, w.logits, s) != cudaSuccess) return RDDMC_ERR_CUDA;
    if (cudaMemsetAsync(d_loss, 0, 4, s) != cudaSuccess) return RDDMC_ERR_CUDA;
    // gradients accumulate (split-K products, column sums) into a zeroed buffer
    if (cudaMemsetAsync(d_grad, 0, o.total * sizeof(float), s) != cudaSuccess) return RDDMC_ERR_CUDA;
    // Every product runs on tcgen05 with the operands as they lie in memory:
    //   dW = dZ^T H             A = dZ [B x out] and W = H [B x in], both MN-major, K = batch, split over K
    //   dH = (dZ W) .* [H > 0]  A = dZ [B x out], W = W [out x in] MN-major, K = out
    // and the masked epilogue adds the columns of dH to the next bias gradient.
    cudaError_t e = cudaSuccess;
    auto chk = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    chk(softmax_ce(w.logits, n_out, nA, nB, nC, S, d_ta, d_tb, nC > 0 ? d_tc : nullptr, batch, w.dlogb,
                   d_grad + o.b[3], d_loss, s));
    // output layer
    chk(gemm_tc<umma::F32_ADD, true, true>(n_out, kHid, batch, w.dlogb, n_out, w.H[2], kHid, nullptr, nullptr, 0,
                                           nullptr, d_grad + o.W[3], kHid, s, ksplit_for(n_out, kHid, batch)));
    chk(gemm_tc<umma::MASK_BF16, false, true>(batch, kHid, n_out, w.dlogb, n_out, wb + o.W[3], kHid, nullptr, w.H[2],
                                              kHid, w.dHb[0], nullptr, kHid, s, 1, d_grad + o.b[2]));
    int cur = 0;
    for (int l = 2; l >= 1; --l) {
        // layer l (W[l]: H[l-1] -> H[l]); dHb[cur] holds dL/d(pre-activation of H[l])
        chk(gemm_tc<umma::F32_ADD, true, true>(kHid, kHid, batch, w.dHb[cur], kHid, w.H[l - 1], kHid, nullptr, nullptr,
                                               0, nullptr, d_grad + o.W[l], kHid, s, ksplit_for(kHid, kHid, batch)));
        chk(gemm_tc<umma::MASK_BF16, false, true>(batch, kHid, kHid, w.dHb[cur], kHid, wb + o.W[l], kHid, nullptr,
                                                  w.H[l - 1], kHid, w.dHb[cur ^ 1], nullptr, kHid, s, 1,
                                                  d_grad + o.b[l - 1]));
        cur ^= 1;
    }
    // input layer: dW1 = dZ1^T X (16 columns, short of a box: a K-major copy)
    chk(transpose(X, batch, kIn, kIn, w.XT, batch, s));
    chk(gemm_tc<umma::F32_ADD, true, false>(kHid, kIn, batch, w.dHb[cur], kHid, w.XT, batch, nullptr, nullptr, 0,
                                            nullptr, d_grad + o.W[0], kIn, s, ksplit_for(kHid, kIn, batch)));
    if (e != cudaSuccess) return RDDMC_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? RDDMC_OK : RDDMC_ERR_CUDA;
}

int rddmc_mlp_status(void* stream) {
    unsigned* p = tc_err_ptr();
    if (!p) return RDDMC_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    unsigned v = 0;
    if (cudaStreamSynchronize(s) != cudaSuccess || cudaMemcpy(&v, p, 4, cudaMemcpyDeviceToHost) != cudaSuccess)
        return RDDMC_ERR_CUDA;
    if (v && cudaMemset(p, 0, 4) != cudaSuccess) return RDDMC_ERR_CUDA;
    return v ? RDDMC_ERR_TIMEOUT : RDDMC_OK;
}

int rddmc_mlp_adam(int n_out, float* d_wf, void* d_wb, const float* d_grad, float* d_m, float* d_v, int step, float lr,
                   float beta1, float beta2, float eps, void* stream) {
    const uint64_t n = rddmc_mlp_param_count(n_out);
    if (!n || !d_wf || !d_wb || !d_grad || !d_m || !d_v || step < 1) return RDDMC_ERR_ARG;
    const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
    adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        n, d_wf, (__nv_bfloat16*)d_wb, d_grad, d_m, d_v, lr, beta1, beta2, eps, c1, c2);
    return cudaGetLastError() == cudaSuccess ? RDDMC_OK : RDDMC_ERR_CUDA;
}

}  // extern "C"
