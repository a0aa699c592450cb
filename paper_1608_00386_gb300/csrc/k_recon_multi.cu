// Reconstructor product for up to 16 realizations sharing a float32 R ("The closed loop": slopes times
// the control matrix, here for a batch of independent realizations): D[r][i] = sum_j R[i][j] s_r[j].
//
// R is streamed once per pass.  It is held in blocks of 128 rows, column by column ([row block][column]
// [128 rows]), so that 16 columns of a block are 8 KB of consecutive memory.  A warp item is one block of
// rows x 1024 columns: lane 0 keeps a two-stage ring of the warp's shared memory filled with bulk copies
// (16 columns of R, and their slopes of every realization from a transposed copy S_t[j][r], zero past
// n_real), the lanes take 4 rows each and accumulate 4 rows x 16 realizations in float32 with packed
// multiply-adds, columns in ascending order.  Items write split-K partials [chunk][16][n_cmd]; a second
// kernel sums them in a fixed order, so the result does not depend on which warp took which item.
//
// Bound by the float32 multiply-adds (14.3 GFLOP at 16 realizations and the 39 m size: 180 us at two
// packed operations per four cycles and scheduler) and by R's bytes (1.79 GB: 264 us); the whole
// call takes 349 us at 39 m (579 before).  With R column-major and every lane copying its own 16 bytes of each column the address
// arithmetic and copies took a third of the instructions (66 per column and warp, 32 of them
// multiply-adds): 460 us.  Six warps a block and two blocks per SM leave 110 KB of ring each.
// Every wait is bounded; on expiry the warp records kErrReconTimeout, waits (bounded) for its copies in
// flight and leaves.
#include "bulk_copy.cuh"
#include "mcao_internal.h"

namespace mcao {

namespace {

constexpr int kMRows = 128;    // rows per item (4 per lane)
constexpr int kMCols = 1024;   // columns per item
constexpr int kMGroup = 16;    // columns per stage
constexpr int kMB = kMultiRhs; // realizations per pass
constexpr int kMStages = 2;
constexpr int kMWarps = 6;

// packed float32 pairs held in 64-bit registers: packing once per operand and accumulating in
// place keeps the packed multiply-adds free of per-call register moves
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ void ffma2_acc(unsigned long long& acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

struct MultiRing {
    float4 v[kMWarps][kMStages][kMGroup][kMRows / 4];   // columns of the row block
    float4 s[kMWarps][kMStages][kMGroup][kMB / 4];      // S_t of those columns
    unsigned long long bar[kMWarps][kMStages];
};

__global__ void __launch_bounds__(kMWarps * 32) recon_multi_kernel(MultiLaunch L) {
    extern __shared__ __align__(128) unsigned char multi_raw[];
    MultiRing& ring = *reinterpret_cast<MultiRing*>(multi_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int st = 0; st < kMStages; ++st) mbar_init(&ring.bar[warp][st], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    const uint64_t pol = evict_first_policy();
    const int n_warps = gridDim.x * kMWarps;
    const int n_rb = (L.n_cmd + kMRows - 1) / kMRows, n_kc = multi_chunks(L.K), n_items = n_rb * n_kc;
    const int first = blockIdx.x * kMWarps + warp;
    // producer position (lane 0): the stages of this warp's items, one after another
    int p_item = first, p_col = 0;
    uint32_t issued = 0;
    auto issue = [&]() {
        if (p_item >= n_items) return;
        const int kc = p_item / n_rb, rb = p_item - kc * n_rb, c0 = kc * kMCols + p_col;
        const int left = min(L.K, (kc + 1) * kMCols) - c0, n = min(kMGroup, left);
        const int st = issued % kMStages;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(&ring.bar[warp][st], (uint32_t)(n * (kMRows + kMB)) * 4u);
        bulk_g2s(ring.v[warp][st], L.R + ((long long)rb * L.K + c0) * kMRows, (uint32_t)(n * kMRows) * 4u, &ring.bar[warp][st], pol);
        bulk_g2s(ring.s[warp][st], L.s_t + (long long)c0 * kMB, (uint32_t)(n * kMB) * 4u, &ring.bar[warp][st], pol);
        ++issued;
        p_col += n;
        if (left <= kMGroup) {
            p_item += n_warps;
            p_col = 0;
        }
    };
    if (lane == 0)
        for (int i = 0; i < kMStages; ++i) issue();
    uint32_t taken = 0;   // stages consumed so far
    for (int item = first; item < n_items; item += n_warps) {
        const int kc = item / n_rb, rb = item - kc * n_rb;
        const int n_cols = min(L.K - kc * kMCols, kMCols);
        unsigned long long acc[4][kMB / 2];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int b = 0; b < kMB / 2; ++b) acc[q][b] = 0ull;   // (+0.0f, +0.0f)
        for (int g = 0; g < n_cols; g += kMGroup, ++taken) {
            const int st = taken % kMStages;
            if (!mbar_wait_bounded(&ring.bar[warp][st], (taken / kMStages) & 1u)) {
                if (lane == 0) {
                    atomicExch(L.err, kErrReconTimeout);
                    for (uint32_t k = taken + 1; k < issued; ++k)
                        mbar_wait_bounded(&ring.bar[warp][k % kMStages], (k / kMStages) & 1u);
                }
                __syncwarp();
                return;
            }
            auto column = [&](int u) {
                const float4 r = ring.v[warp][st][u][lane];
                const unsigned long long rp[4] = {pack2(r.x, r.x), pack2(r.y, r.y), pack2(r.z, r.z), pack2(r.w, r.w)};
#pragma unroll
                for (int b4 = 0; b4 < kMB / 4; ++b4) {
                    const float4 sv = ring.s[warp][st][u][b4];
                    const unsigned long long s01 = pack2(sv.x, sv.y), s23 = pack2(sv.z, sv.w);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        ffma2_acc(acc[q][2 * b4], rp[q], s01);
                        ffma2_acc(acc[q][2 * b4 + 1], rp[q], s23);
                    }
                }
            };
            if (n_cols - g >= kMGroup) {
#pragma unroll
                for (int u = 0; u < kMGroup; ++u) column(u);
            } else {
                for (int u = 0; u < n_cols - g; ++u) column(u);
            }
            __syncwarp();   // every lane has read the slot before it is refilled
            if (lane == 0) issue();
        }
        const int row0 = rb * kMRows + 4 * lane;
        float* out = L.partial + (long long)kc * kMB * L.n_cmd;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = row0 + q;
            if (row >= L.n_cmd) continue;
#pragma unroll
            for (int b = 0; b < kMB / 2; ++b) {
                const float2 v = unpack2(acc[q][b]);
                out[(long long)(2 * b) * L.n_cmd + row] = v.x;
                out[(long long)(2 * b + 1) * L.n_cmd + row] = v.y;
            }
        }
    }
}

// S_t[j][r] = slopes of realization r at padded column j (zero for r >= n_real), 64 columns per block
// through shared memory
__global__ void __launch_bounds__(256) slopes_t_kernel(const float* __restrict__ slopes_pad, int n_real, int K, int pad_stride,
                                                       float* __restrict__ s_t) {
    __shared__ float tile[kMB][65];
    const int j0 = blockIdx.x * 64;
    for (int q = threadIdx.x; q < kMB * 64; q += 256) {
        const int r = q >> 6, j = j0 + (q & 63);
        tile[r][q & 63] = (r < n_real && j < K) ? slopes_pad[(long long)r * pad_stride + j] : 0.0f;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < kMB * 64; q += 256) {
        const int j = j0 + q / kMB;
        if (j < K) s_t[(long long)j * kMB + q % kMB] = tile[q % kMB][q / kMB];
    }
}

// out[r][i] = alpha sum_kc partial[kc][r][i] + beta out[r][i] (beta = 0: out not read)
__global__ void multi_reduce_kernel(const float* __restrict__ partial, int n_kc, int n_real, int n_cmd, float alpha, float beta,
                                    float* __restrict__ out) {
    const long long total = (long long)n_real * n_cmd;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(i / n_cmd), row = (int)(i - (long long)r * n_cmd);
        float s = 0.0f;
#pragma unroll 8
        for (int kc = 0; kc < n_kc; ++kc) s += partial[((long long)kc * kMB + r) * n_cmd + row];
        out[i] = beta == 0.0f ? alpha * s : fmaf(alpha, s, beta * out[i]);
    }
}

// row-major [rows][ld] -> [row block][ld][128] (rows at or beyond `rows`: zeros), 32 x 32 tiles
__global__ void multi_tile_kernel(const float* __restrict__ src, int rows, int ld, float* __restrict__ out) {
    __shared__ float tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        tile[i][threadIdx.x] = (r < rows && c < ld) ? src[(long long)r * ld + c] : 0.0f;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (c < ld) out[((long long)(r / kMRows) * ld + c) * kMRows + r % kMRows] = tile[threadIdx.x][i];
    }
}

// one sensor's block of slopes per block y, one vector per block z
__global__ void __launch_bounds__(256) pad_slopes_kernel(const float* __restrict__ slopes, int n_slopes, const WfsDev* wfs,
                                                         float* __restrict__ pad, int pad_stride) {
    const WfsDev& w = wfs[blockIdx.y];
    const int n = 2 * w.n_valid;
    const float* src = slopes + (long long)blockIdx.z * n_slopes + w.slope0;
    float* dst = pad + (long long)blockIdx.z * pad_stride + w.rcol0;
    for (int j = blockIdx.x * 256 + threadIdx.x; j < n; j += gridDim.x * 256) dst[j] = src[j];
}

}  // namespace

cudaError_t launch_pad_slopes(const float* slopes, int n_slopes, int n_rhs, const WfsDev* wfs, int n_wfs, float* pad,
                              int pad_stride, cudaStream_t s) {
    pad_slopes_kernel<<<dim3(8, (unsigned)n_wfs, (unsigned)n_rhs), 256, 0, s>>>(slopes, n_slopes, wfs, pad, pad_stride);
    return cudaGetLastError();
}

__host__ __device__ int multi_chunks(int K) { return (K + kMCols - 1) / kMCols; }

size_t multi_tiled_floats(int n_cmd, int K) { return (size_t)((n_cmd + kMRows - 1) / kMRows) * kMRows * (size_t)K; }

cudaError_t launch_multi_tile(const float* src, int rows, int n_cmd, int ld, float* out, cudaStream_t s) {
    const int n_rb = (n_cmd + kMRows - 1) / kMRows;
    if (n_rb == 0) return cudaSuccess;
    multi_tile_kernel<<<dim3((unsigned)((ld + 31) / 32), (unsigned)(n_rb * kMRows / 32)), dim3(32, 8), 0, s>>>(src, rows, ld, out);
    return cudaGetLastError();
}

cudaError_t multi_prepare() {
    return cudaFuncSetAttribute(recon_multi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MultiRing));
}

cudaError_t launch_recon_multi(const MultiLaunch& L, int n_real, int pad_stride, const float* slopes_pad, float alpha,
                               float beta, float* out, int sm_count, int blocks_per_sm, cudaStream_t s) {
    if (n_real < 1 || n_real > kMB) return cudaErrorInvalidValue;
    slopes_t_kernel<<<(L.K + 63) / 64, 256, 0, s>>>(slopes_pad, n_real, L.K, pad_stride, L.s_t);
    const int items = ((L.n_cmd + kMRows - 1) / kMRows) * multi_chunks(L.K);
    int blocks = (items + kMWarps - 1) / kMWarps;
    const int cap = (blocks_per_sm > 0 ? blocks_per_sm : 2) * sm_count;   // at most two resident per SM
    if (blocks > cap) blocks = cap;
    if (blocks > 0) recon_multi_kernel<<<blocks, kMWarps * 32, sizeof(MultiRing), s>>>(L);
    multi_reduce_kernel<<<(n_real * L.n_cmd + 255) / 256, 256, 0, s>>>(L.partial, multi_chunks(L.K), n_real, L.n_cmd,
                                                                       alpha, beta, out);
    return cudaGetLastError();
}

}  // namespace mcao
