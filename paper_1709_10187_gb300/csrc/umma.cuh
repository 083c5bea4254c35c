// umma.cuh -- dense BF16 products on the 5th-generation tensor cores
// (tcgen05.mma, FP32 accumulators in tensor memory) for the learned proposal's
// network: C[M x N] = A[M x K] W[N x K]^T (+ bias, epilogue).  Each operand is
// read as it lies in memory: K contiguous ("K-major", a row per M or N index) or
// M or N contiguous ("MN-major", a row per K index), so that the backward
// products need no transposed copies.
//
// One CTA of 128 threads computes a 128 x NT tile (NT <= 256, a multiple of
// 16; of 64 when W is MN-major), over K in panels of 64, optionally a range of
// them per blockIdx.z (split-K).  A panel of A and W is staged in shared memory
// by TMA (cp.async.bulk.tensor with 128-byte swizzle, elements past the matrix
// filled with zeros by the copy engine), or by the threads for a single K-major
// block of K <= 128 that is not a multiple of 64:
//   K-major:  rows of 64 BF16 = 128 B, eight-row atoms of 1 KiB, 16-byte chunk c
//             of row r at chunk c ^ (r mod 8); one box of all rows;
//   MN-major: boxes of 64 M (or N) indices x 64 K rows, 8 KiB each, in the same
//             atoms of eight K rows.
// One elected thread keeps nstage panels in flight, issues each panel's four
// tcgen05.mma into a TMEM accumulator of 128 lanes x NT columns and commits them
// to the mbarrier that frees the stage.  After the last panel every warp reads
// its 32 lanes back with tcgen05.ld; FP32 outputs are turned around in shared
// memory, 32 x 32 at a time, so that their stores run along rows.  Waits are bounded: a
// wait that runs out sets the error word and the tile's outputs are left
// unwritten.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rddmc {
namespace umma {

constexpr int kTileM = 128;
constexpr int kThreads = 128;
constexpr int kPanel = 64;  // BF16 per 128-byte swizzled row
constexpr int kMaxStages = 6;
constexpr uint32_t kBoxBytes = 8192;  // an MN-major box: 64 K rows of 128 B

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: start address, leading byte offset (between
// boxes of 64 M or N indices of an MN-major operand; unused by swizzled K-major
// layouts, set to 16 B), stride byte offset between eight-row atoms (1 KiB),
// descriptor version 1, 128-byte swizzle.
template <bool MN>
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((MN ? kBoxBytes : 16u) >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1u << 46;
    d |= (uint64_t)2u << 61;
    return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, each
// K-major or MN-major (transpose bits 15 and 16), N >> 3 and M >> 4.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n, bool mn_a, bool mn_b) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((mn_a ? 1u : 0u) << 15) | ((mn_b ? 1u : 0u) << 16) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__host__ __device__ constexpr int tmem_cols(int nt) {
    return nt <= 32 ? 32 : (nt <= 64 ? 64 : (nt <= 128 ? 128 : 256));
}

// Copy rows [row0, row0 + rows) x K of a row-major BF16 matrix into the
// swizzled K-major layout at dst (1 KiB aligned; rows a multiple of 8); rows
// past `valid` are zero.
__device__ __forceinline__ void stage(const __nv_bfloat16* __restrict__ src, int ld, int row0, int rows, int valid,
                                      int K, unsigned char* dst) {
    const int chunks_per_row = K / 8;  // 16-byte chunks of K
    const int total = rows * chunks_per_row;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int r = i / chunks_per_row, q = i % chunks_per_row;
        const int p = q >> 3, c = q & 7;  // panel, chunk in the 128-byte row
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < valid) v = *reinterpret_cast<const uint4*>(src + (size_t)(row0 + r) * ld + q * 8);
        unsigned char* d = dst + (size_t)p * rows * 128 + (size_t)(r >> 3) * 1024 + (r & 7) * 128 +
                           ((c ^ (r & 7)) << 4);
        *reinterpret_cast<uint4*>(d) = v;
    }
}

enum Epi { RELU_BF16 = 0, LINEAR_F32 = 1, MASK_BF16 = 2, F32_ADD = 3 };

// Bounded wait for the given phase parity of an mbarrier; false when it ran out.
__device__ __forceinline__ bool wait_parity(uint64_t* mbar, uint32_t parity) {
    uint32_t done = 0;
    for (int it = 0; it < (1 << 22) && !done; ++it) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(smem_u32(mbar)), "r"(parity));
    }
    return done != 0;
}

// TMA copy of the box at element coordinates (x, y) of a 2D tensor map into
// shared memory, counted on the mbarrier's transaction bytes.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* mbar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(mbar))
        : "memory");
}

// Issue the tcgen05.mma instructions of `slices` K-slices of 16 (four per panel;
// panels panel_a and panel_b bytes apart, for the thread-staged block), the
// first of them overwriting the accumulator when `first`.
template <bool MNA, bool MNB>
__device__ __forceinline__ void mma_panel(uint32_t tmem, unsigned char* sA, unsigned char* sB, int NT, int slices,
                                          bool first, uint32_t panel_a, uint32_t panel_b) {
    const uint32_t idesc = instr_desc(kTileM, NT, MNA, MNB);
    for (int s = 0; s < slices; ++s) {
        // 16 K indices further: 32 bytes along a K-major row, 16 rows of an MN-major box
        const uint32_t p = (uint32_t)(s >> 2), k = (uint32_t)(s & 3);
        const uint64_t ad = smem_desc<MNA>(smem_u32(sA) + p * panel_a + k * (MNA ? 2048u : 32u));
        const uint64_t bd = smem_desc<MNB>(smem_u32(sB) + p * panel_b + k * (MNB ? 2048u : 32u));
        const uint32_t acc = (first && s == 0) ? 0u : 1u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            :: "r"(tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
    }
}

__device__ __forceinline__ void commit_to(uint64_t* mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(smem_u32(mbar)));
}

// 32 accumulator columns of this warp's 32 TMEM lanes: thread t's row.
__device__ __forceinline__ void load_acc32(uint32_t ta, float* v) {
    uint32_t u[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
          "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]),
          "=r"(u[15]), "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]),
          "=r"(u[22]), "=r"(u[23]), "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]),
          "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
        : "r"(ta));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(u[j]);
}

// Bytes of a stage's W panel.
__host__ __device__ constexpr uint32_t w_bytes(int NT, bool mn_b) {
    return mn_b ? (uint32_t)((NT + 63) / 64) * kBoxBytes : (uint32_t)NT * 128u;
}

// C = epi(A W^T (+ bias)).  Grid: (ceil(N / NT), ceil(M / 128), ksplit);
// blockIdx.z takes a range of K in 64-wide panels.  TMA path: tensor maps mapA
// and mapW (boxes of 64 columns x all tile rows when K-major, x 64 rows when
// MN-major); thread-staged path: K <= 128, both K-major.  Epilogues: RELU_BF16
// and LINEAR_F32 add the bias; MASK_BF16 keeps entries where mask > 0, writes
// them to outb (BF16) and adds their FP32 column sums to colsum; F32_ADD adds
// into outf (split-K partial sums).  err: set to 1 when a wait ran out (the
// tile's outputs are then left unwritten).
template <int EPI, bool TMA, bool MNA, bool MNB>
__global__ void __launch_bounds__(kThreads) gemm_tc_kernel(int M, int N, int K, int NT,
                                                           const __nv_bfloat16* __restrict__ A, int lda,
                                                           const __nv_bfloat16* __restrict__ W, int ldw,
                                                           const __grid_constant__ CUtensorMap mapA,
                                                           const __grid_constant__ CUtensorMap mapW,
                                                           const float* __restrict__ bias,
                                                           const __nv_bfloat16* __restrict__ mask, int ldmask,
                                                           __nv_bfloat16* __restrict__ outb, float* __restrict__ outf,
                                                           int ldc, float* __restrict__ colsum, int nstage,
                                                           unsigned* err) {
    static_assert(TMA || (!MNA && !MNB), "the thread-staged block is K-major");
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    // nstage staging areas of one panel each: A, then W
    constexpr uint32_t a_bytes = kTileM * 128;
    const uint32_t b_bytes = w_bytes(NT, MNB);
    unsigned char* sA = base;  // also the epilogue's scratch
    auto stage_a = [&](int st) { return base + (size_t)st * (a_bytes + b_bytes); };
    auto stage_b = [&](int st) { return base + (size_t)st * (a_bytes + b_bytes) + a_bytes; };
    // per stage: full (its copies landed) and empty (its products completed);
    // then the barrier of the last products
    uint64_t* full = reinterpret_cast<uint64_t*>(base + (size_t)nstage * (a_bytes + b_bytes));
    uint64_t* empty = full + kMaxStages;
    uint64_t* last = empty + kMaxStages;
    uint32_t* taddr_s = reinterpret_cast<uint32_t*>(last + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * kTileM, n0 = blockIdx.x * NT;
    const int ncols = tmem_cols(NT);
    // this split's range of K, in whole 64-column panels
    const int kpanels = (K + kPanel - 1) / kPanel;
    const int per = (kpanels + (int)gridDim.z - 1) / (int)gridDim.z;
    const int p_begin = (int)blockIdx.z * per, p_end = min(kpanels, p_begin + per);
    if (p_begin >= p_end) return;  // an empty split adds nothing

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(taddr_s)), "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kMaxStages + 1; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(full + i)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (!TMA) {  // one block: K <= 128
        stage(A, lda, m0, kTileM, min(kTileM, M - m0), K, stage_a(0));
        stage(W, ldw, n0, NT, min(NT, N - n0), K, base + 2 * a_bytes);
        asm volatile("fence.proxy.async.shared::cta;");  // generic-proxy stores -> tensor-core reads
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *taddr_s;

    // One thread copies (TMA), issues and waits.  Panel p uses stage p mod
    // nstage; its copy is issued once the products of panel p - nstage have
    // completed, nstage panels ahead of the products at most.  Use k of a stage
    // completes phase k of its two barriers (parity k & 1), and a stage is
    // rewritten only after its previous use was waited for, so no barrier runs
    // two phases ahead of its wait.
    __shared__ int ok_s;
    if (threadIdx.x == 0) {
        bool ok = true;
        if (TMA) {
            const int np = p_end - p_begin;
            int issued = 0, landed = 0;
            for (int p = 0; p < np && ok; ++p) {
                while (issued < np && issued < p + nstage) {
                    const int st = issued % nstage, use = issued / nstage;
                    if (use > 0 && !(ok = wait_parity(empty + st, (uint32_t)(use - 1) & 1u))) break;
                    const int k = (p_begin + issued) * kPanel;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                 :: "r"(smem_u32(full + st)), "r"(a_bytes + b_bytes) : "memory");
                    if (MNA) {
                        for (int c = 0; c < kTileM / 64; ++c)
                            tma_load_2d(stage_a(st) + c * kBoxBytes, &mapA, m0 + 64 * c, k, full + st);
                    } else {
                        tma_load_2d(stage_a(st), &mapA, k, m0, full + st);
                    }
                    if (MNB) {
                        for (int c = 0; c < (NT + 63) / 64; ++c)
                            tma_load_2d(stage_b(st) + c * kBoxBytes, &mapW, n0 + 64 * c, k, full + st);
                    } else {
                        tma_load_2d(stage_b(st), &mapW, k, n0, full + st);
                    }
                    ++issued;
                }
                if (!ok) break;
                const int st = p % nstage;
                if (!(ok = wait_parity(full + st, (uint32_t)(p / nstage) & 1u))) break;
                ++landed;
                asm volatile("tcgen05.fence::after_thread_sync;");
                mma_panel<MNA, MNB>(tmem, stage_a(st), stage_b(st), NT, 4, p == 0, 0u, 0u);
                commit_to(empty + st);
            }
            if (ok) {
                commit_to(last);  // covers every product issued before it
                ok = wait_parity(last, 0);
            }
            // a wait ran out: give the copies still in flight another bounded wait
            // before the CTA leaves
            for (int p = landed; !ok && p < issued; ++p) wait_parity(full + p % nstage, (uint32_t)(p / nstage) & 1u);
        } else {
            // only the staged K columns
            mma_panel<false, false>(tmem, stage_a(0), base + 2 * a_bytes, NT, K / 16, true, a_bytes, (uint32_t)NT * 128u);
            commit_to(last);
            ok = wait_parity(last, 0);
        }
        if (!ok) atomicOr(err, 1u);
        ok_s = ok ? 1 : 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok_s && (EPI == RELU_BF16 || EPI == MASK_BF16)) {
        // thread t of warp w holds row m0 + 32 w + t: its BF16 outputs are 64
        // contiguous bytes per 32 columns, so it stores (and reads the mask) in
        // 16-byte pieces.  N is 128 here: a tile's columns are all there.
        const int row = m0 + warp * 32 + lane;
        const bool row_ok = row < M;
        uint4 mk[4][4];
        if (EPI == MASK_BF16) {  // all of the row's mask in flight together
            const uint4* mrow = reinterpret_cast<const uint4*>(mask + (size_t)min(row, M - 1) * ldmask + n0);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) mk[c][i] = mrow[4 * c + i];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float v[32];
            load_acc32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(32 * c), v);
            uint32_t packed[16];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                if (EPI == RELU_BF16) {
                    v[j] = fmaxf(v[j] + bias[n0 + 32 * c + j], 0.0f);
                } else {
                    const uint32_t w = (&mk[c][j >> 3].x)[(j >> 1) & 3];
                    const float h = __uint_as_float((j & 1) ? (w & 0xffff0000u) : (w << 16));
                    v[j] = (h > 0.0f && row_ok) ? v[j] : 0.0f;
                }
                if (j & 1) {
                    const __nv_bfloat162 b2 = __floats2bfloat162_rn(v[j - 1], v[j]);
                    packed[j >> 1] = *reinterpret_cast<const uint32_t*>(&b2);
                }
            }
            if (row_ok) {
                uint4* o = reinterpret_cast<uint4*>(outb + (size_t)row * ldc + n0 + 32 * c);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    o[i] = make_uint4(packed[4 * i], packed[4 * i + 1], packed[4 * i + 2], packed[4 * i + 3]);
            }
            if (EPI == MASK_BF16) {
                // column sums over the warp's 32 rows: halve the columns a lane holds
                // at every exchange, until lane l holds the sum of column l
#pragma unroll
                for (int w = 16; w > 0; w >>= 1) {
                    const bool up = (lane & w) != 0;
#pragma unroll
                    for (int j = 0; j < w; ++j) {
                        const float keep = up ? v[j + w] : v[j], send = up ? v[j] : v[j + w];
                        v[j] = keep + __shfl_xor_sync(0xffffffffu, send, w);
                    }
                }
                atomicAdd(&colsum[n0 + 32 * c + lane], v[0]);
            }
        }
    } else if (ok_s) {
        // warp w reads TMEM lanes 32w..32w+31 (thread t holds row m0 + 32w + t,
        // 32 columns at a time), then turns each 32 x 32 block around through
        // shared memory (the operand staging area, free now that the products
        // completed; 33-float rows keep both passes free of bank conflicts) so
        // that lane l writes column c0 + l: every store covers consecutive
        // columns of one row
        float* st = reinterpret_cast<float*>(sA) + warp * (32 * 33);
        for (int c0 = 0; c0 < NT; c0 += 32) {
            float v[32];
            load_acc32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) st[lane * 33 + j] = v[j];
            __syncwarp();
            const int n = n0 + c0 + lane;
            const bool col_ok = c0 + lane < NT && n < N;
            const float b = (col_ok && EPI == LINEAR_F32) ? bias[n] : 0.0f;
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                const int row = m0 + warp * 32 + r;
                if (row >= M || !col_ok) continue;
                const float x = st[r * 33 + lane];
                const size_t o = (size_t)row * ldc + n;
                if (EPI == LINEAR_F32) outf[o] = x + b;
                else atomicAdd(&outf[o], x);
            }
            __syncwarp();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(ncols));
    }
}

// BF16 transpose: out[c][r] = in[r][c] for in [rows x cols] (leading dims
// ld_in, ld_out), 32 x 32 tiles through shared memory.
__global__ void transpose_bf16_kernel(const __nv_bfloat16* __restrict__ in, int rows, int cols, int ld_in,
                                      __nv_bfloat16* __restrict__ out, int ld_out) {
    __shared__ __nv_bfloat16 t[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        t[i][threadIdx.x] = (r < rows && c < cols) ? in[(size_t)r * ld_in + c] : __float2bfloat16(0.0f);
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (c < cols && r < rows) out[(size_t)c * ld_out + r] = t[threadIdx.x][i];
    }
}

// Dynamic shared memory of a 128 x NT tile with `stages` panels of A and W (+1 KiB
// alignment slack, the barriers and the TMEM address); the thread-staged block
// takes two panels of each.
__host__ __device__ constexpr size_t smem_bytes(int nt, int stages, bool mn_b) {
    return 1024 + (size_t)stages * (kTileM * 128 + w_bytes(nt, mn_b)) + (2 * kMaxStages + 2) * 8;
}

// 2D BF16 tensor map of a row-major [rows x cols] matrix with leading
// dimension ld, box of box_rows x 64 columns, 128-byte swizzle, zero fill.
inline bool make_map(CUtensorMap* map, const void* ptr, int rows, int cols, int ld, int box_rows) {
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Encode encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
            return false;
        encode = (Encode)fn;
    }
    if (((uintptr_t)ptr & 15u) || ((size_t)ld * 2) % 16) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kPanel, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace umma
}  // namespace rddmc
