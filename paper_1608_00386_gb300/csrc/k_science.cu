// Science path ("The Point Spread Functions (PSFs)" of arXiv:1608.00386: PSF at a user
// wavelength and pixel scale computed on the GPU; Strehl ratio from the PSF or the residual):
//   field E = A exp(i (lambda_ref / lambda) phi) along the science direction (source at
//   infinity), on-axis Strehl |sum E|^2 / (sum A)^2 every step, and every psf_every steps the
//   long-exposure PSF += |FFT2(E zero-padded to M x M)|^2 accumulated in double.
// The 2-D FFT runs as two passes of batched radix-4/5/2 Stockham FFTs in shared memory: rows of
// the field (zero-padded) written transposed, then rows of the transposed array; the PSF
// accumulator is therefore held transposed and unshifted, [kx][ky] (psf_out_kernel reorders it).
#include <algorithm>
#include <cmath>
#include <vector>

#include "device_common.cuh"
#include "mcao_internal.h"

namespace mcao {

namespace {

constexpr int kRowsPerBlock = 4;

// per-realization views of the launch (grid y = realization)
__device__ __forceinline__ SciLaunch sci_for_real(const SciLaunch& L0, int r) {
    SciLaunch L = L0;
    L.field += (long long)r * L.N * L.N;
    L.ft += (long long)r * L.M * L.N;
    L.psf_t += (long long)r * L.M * L.M;
    L.sr_part += (long long)r * L.n_tiles;
    L.acc += (long long)r * L.acc_stride;
    L.ctx.views += r * L.ctx.view_stride;
    return L;
}

struct SciGrid {
    const float* data;
    int n;
    float sign;
};

__global__ void __launch_bounds__(256, 6) sci_field_kernel(SciLaunch L0) {
    __shared__ SciGrid s_gm[8][kMaxEntries];
    __shared__ AxisEnt s_ex[8][kMaxEntries * 8];
    __shared__ AxisEnt s_ey[8][kMaxEntries * 8];
    const SciLaunch L = sci_for_real(L0, blockIdx.y);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles_x = L.N / 8;
    const int tile = blockIdx.x * 8 + warp;
    if (tile >= tiles_x * tiles_x) return;
    const int i0 = (tile % tiles_x) * 8, j0 = (tile / tiles_x) * 8;
    const int n_grids = L.ctx.n_grids;
    const GridView* V = L.ctx.views + (long long)L.view * n_grids;
    tile_entries<8>(V, n_grids, L.ctx.st->k, i0, j0, s_ex[warp], s_ey[warp], lane, 32);
    __syncwarp();
    // phase of samples (x, 2h) and (x, 2h + 1), h = lane / 8: where samples lie at most one grid sample
    // apart (rows_overlap, here for every grid) the second row's cell is the first's or the next one, so
    // that three grid rows serve both: 6 loads instead of 8, two grids' loads in flight together.
    // The kernel waits for these gathers: 32.7 us before, 22.8 us now at 640 x 640 samples and 13 grids.
    // (Four grids in flight and 80 registers: 2.4 us less a step at 20 m, but 6 us more at 39 m, where the
    // blocks take the laser stars' places.)
    if (lane < n_grids) s_gm[warp][lane] = SciGrid{V[lane].data, V[lane].n, V[lane].sign};
    const bool near = __all_sync(0xffffffffu, lane >= n_grids || rows_overlap(V[lane].bp));
    __syncwarp();
    const int x = lane & 7, yy = (lane >> 3) * 2;
    float p0 = 0.0f, p1 = 0.0f;
    if (near) {
#pragma unroll 2
        for (int g = 0; g < n_grids; ++g) {
            const SciGrid gm = s_gm[warp][g];
            const AxisEnt ex = s_ex[warp][g * 8 + x], e0 = s_ey[warp][g * 8 + yy], e1 = s_ey[warp][g * 8 + yy + 1];
            const float2 p = bilinear_rows(gm.data, gm.n, ex, e0, e1);
            p0 = fmaf(gm.sign, p.x, p0);
            p1 = fmaf(gm.sign, p.y, p1);
        }
    } else {
#pragma unroll 2
        for (int g = 0; g < n_grids; ++g) {
            const SciGrid gm = s_gm[warp][g];
            const AxisEnt ex = s_ex[warp][g * 8 + x];
            p0 = fmaf(gm.sign, bilinear(gm.data, gm.n, ex, s_ey[warp][g * 8 + yy]), p0);
            p1 = fmaf(gm.sign, bilinear(gm.data, gm.n, ex, s_ey[warp][g * 8 + yy + 1]), p1);
        }
    }
    // the lane sums rows lane / 8 and lane / 8 + 4, as the Strehl partials have always been summed
    float sr = 0.0f, si = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int y = (lane >> 3) + 4 * hh;
        const int from = (y >> 1) * 8 + x;
        const float q0 = __shfl_sync(0xffffffffu, p0, from), q1 = __shfl_sync(0xffffffffu, p1, from);
        const float phi = (y & 1) ? q1 : q0;
        float a = __ldg(L.amp + (long long)(j0 + y) * L.N + i0 + x);
        const float ph = L.scale * phi;
        float sn, cs;
        sincosf(ph, &sn, &cs);
        float2 e = make_float2(a * cs, a * sn);
        L.field[(long long)(j0 + y) * L.N + i0 + x] = e;
        sr += e.x;
        si += e.y;
        s1 = fmaf(a, ph, s1);
        s2 = fmaf(a * ph, ph, s2);
    }
    sr = warp_sum(sr);
    si = warp_sum(si);
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0) L.sr_part[tile] = make_float4(sr, si, s1, s2);
}

// Strehl of this step from the field partial sums, and the Marechal residual variance (piston removed,
// amplitude-weighted, science band) from the phase sums; fixed order, double.  The first block of the
// column pass forms them, beside the transforms' blocks.  As the last block of the row pass it was that
// pass's longest and the column pass waited for it (8 m: 20.5 us a step); as a kernel of its own beside
// the passes a single loop is faster (8 m 18.3, here 20.0) but 63 loops advanced together take 1.86 ms
// a step instead of 1.34.
__device__ void strehl_sums(const SciLaunch& L) {
    __shared__ double red[8][4];
    const int tid = threadIdx.x, nthr = blockDim.x;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    // the thread's partials q = tid, tid + nthr, ... in that order, loaded eight at a time (the
    // loads of a batch in flight together)
    constexpr int kBatch = 8;
    for (int q0 = tid; q0 < L.n_tiles; q0 += kBatch * nthr) {
        float4 p[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const int q = q0 + i * nthr;
            p[i] = q < L.n_tiles ? L.sr_part[q] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (q0 + i * nthr >= L.n_tiles) break;
            v[0] += p[i].x;
            v[1] += p[i].y;
            v[2] += p[i].z;
            v[3] += p[i].w;
        }
    }
    const SciAcc old = *L.acc;   // read while the sums are formed
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if ((tid & 31) == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) red[tid >> 5][i] = v[i];
    __syncthreads();
    if (tid < 4) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][tid];
        red[0][tid] = t;
    }
    __syncwarp();
    if (tid == 0) {
        const double s = (red[0][0] * red[0][0] + red[0][1] * red[0][1]) / (L.sum_amp * L.sum_amp);
        L.acc->sr_sum = old.sr_sum + s;
        L.acc->sr_last = s;
        L.acc->n_sr = old.n_sr + 1;
        const double mean = red[0][2] / L.sum_amp;
        const double var = red[0][3] / L.sum_amp - mean * mean;
        L.acc->var_sum = old.var_sum + var;
        L.acc->var_last = var;
    }
}

__device__ __forceinline__ bool psf_step(const SciLaunch& L) {
    return L.psf_every > 0 && (L.ctx.st->k % L.psf_every) == 0;
}

__global__ void __launch_bounds__(256) sci_rows_kernel(SciLaunch L0) {
    const SciLaunch L = sci_for_real(L0, blockIdx.y);
    extern __shared__ float4 smem_raw[];
    float2* A = reinterpret_cast<float2*>(smem_raw);
    float2* B = A + kRowsPerBlock * L.M;
    float2* W = B + kRowsPerBlock * L.M;
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (!psf_step(L)) return;

    const int row0 = blockIdx.x * kRowsPerBlock;
    for (int q = tid; q < L.M; q += nthr) W[q] = L.w[q];
    for (int q = tid; q < kRowsPerBlock * L.M; q += nthr) {
        int r = q / L.M, c = q - r * L.M;
        int row = row0 + r;
        A[q] = (row < L.N && c < L.N) ? L.field[(long long)row * L.N + c] : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    float2* R = stockham_fft(A, B, L.M, L.radices, L.n_radices, kRowsPerBlock, L.M, 1, W, tid, nthr);
    // transposed store: ft[c][row], four consecutive rows per column
    for (int q = tid; q < kRowsPerBlock * L.M; q += nthr) {
        int c = q / kRowsPerBlock, r = q - c * kRowsPerBlock;
        int row = row0 + r;
        if (row < L.N) L.ft[(long long)c * L.N + row] = R[r * L.M + c];
    }
}

__global__ void __launch_bounds__(256) sci_cols_kernel(SciLaunch L0) {
    const SciLaunch L = sci_for_real(L0, blockIdx.y);
    if (blockIdx.x == 0) {
        strehl_sums(L);
        return;
    }
    if (!psf_step(L)) return;
    extern __shared__ float4 smem_raw[];
    float2* A = reinterpret_cast<float2*>(smem_raw);
    float2* B = A + kRowsPerBlock * L.M;
    float2* W = B + kRowsPerBlock * L.M;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int c0 = (blockIdx.x - 1) * kRowsPerBlock;
    for (int q = tid; q < L.M; q += nthr) W[q] = L.w[q];
    for (int q = tid; q < kRowsPerBlock * L.M; q += nthr) {
        int r = q / L.M, j = q - r * L.M;
        A[q] = (j < L.N) ? L.ft[(long long)(c0 + r) * L.N + j] : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    float2* R = stockham_fft(A, B, L.M, L.radices, L.n_radices, kRowsPerBlock, L.M, 1, W, tid, nthr);
    for (int q = tid; q < kRowsPerBlock * L.M; q += nthr) {
        int r = q / L.M, j = q - r * L.M;
        float2 v = R[q];
        float p = fmaf(v.x, v.x, v.y * v.y);   // frame intensity in float, accumulated in double
        L.psf_t[(long long)(c0 + r) * L.M + j] += (double)p;
    }
    if (c0 == 0 && tid == 0) L.acc->n_psf += 1;
}

// Compile-time-size versions of the two FFT passes (2 rows / columns per block, 256 threads);
// their twiddle table is stage-major (sci_twiddles).  Global loads are issued a whole pass at a
// time into registers before anything is stored, so that a block waits for about one memory
// round trip per pass rather than one per element.
constexpr int kCtRows = 2;
constexpr int kCtThreads = 256;

template <int M>
__global__ void __launch_bounds__(256) sci_rows_ct(SciLaunch L0) {
    const SciLaunch L = sci_for_real(L0, blockIdx.y);
    extern __shared__ float4 smem_raw[];
    float2* A = reinterpret_cast<float2*>(smem_raw);
    float2* B = A + kCtRows * M;
    float2* W = B + kCtRows * M;
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (!psf_step(L)) return;
    static_assert((kCtRows * M) % kCtThreads == 0, "whole passes per thread");
    constexpr int PER = kCtRows * M / kCtThreads, PW = (M + kCtThreads - 1) / kCtThreads;
    const int row0 = blockIdx.x * kCtRows;
    {
        float2 w[PW], v[PER];
#pragma unroll
        for (int i = 0; i < PW; ++i) w[i] = tid + i * kCtThreads < M ? L.w[tid + i * kCtThreads] : make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int q = tid + i * kCtThreads, r = q / M, c = q - r * M, row = row0 + r;
            v[i] = (row < L.N && c < L.N) ? L.field[(long long)row * L.N + c] : make_float2(0.0f, 0.0f);
        }
#pragma unroll
        for (int i = 0; i < PW; ++i)
            if (tid + i * kCtThreads < M) W[tid + i * kCtThreads] = w[i];
#pragma unroll
        for (int i = 0; i < PER; ++i) A[tid + i * kCtThreads] = v[i];
    }
    __syncthreads();
    float2* R = fft_tab<M>(A, B, kCtRows, W, tid, nthr);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = tid + i * kCtThreads, c = q / kCtRows, r = q - c * kCtRows, row = row0 + r;
        if (row < L.N) L.ft[(long long)c * L.N + row] = R[r * M + c];
    }
}

template <int M>
__global__ void __launch_bounds__(256) sci_cols_ct(SciLaunch L0) {
    const SciLaunch L = sci_for_real(L0, blockIdx.y);
    if (blockIdx.x == 0) {
        strehl_sums(L);
        return;
    }
    if (!psf_step(L)) return;
    extern __shared__ float4 smem_raw[];
    float2* A = reinterpret_cast<float2*>(smem_raw);
    float2* B = A + kCtRows * M;
    float2* W = B + kCtRows * M;
    const int tid = threadIdx.x, nthr = blockDim.x;
    static_assert((kCtRows * M) % kCtThreads == 0, "whole passes per thread");
    constexpr int PER = kCtRows * M / kCtThreads, PW = (M + kCtThreads - 1) / kCtThreads;
    const int c0 = (blockIdx.x - 1) * kCtRows;
    {
        float2 w[PW], v[PER];
#pragma unroll
        for (int i = 0; i < PW; ++i) w[i] = tid + i * kCtThreads < M ? L.w[tid + i * kCtThreads] : make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int q = tid + i * kCtThreads, r = q / M, j = q - r * M;
            v[i] = (j < L.N) ? L.ft[(long long)(c0 + r) * L.N + j] : make_float2(0.0f, 0.0f);
        }
#pragma unroll
        for (int i = 0; i < PW; ++i)
            if (tid + i * kCtThreads < M) W[tid + i * kCtThreads] = w[i];
#pragma unroll
        for (int i = 0; i < PER; ++i) A[tid + i * kCtThreads] = v[i];
    }
    // this block's PSF accumulator entries, read while the transform runs
    double acc[PER];
    double* psf = L.psf_t + (long long)c0 * M;
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = psf[tid + i * kCtThreads];
    __syncthreads();
    float2* R = fft_tab<M>(A, B, kCtRows, W, tid, nthr);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = tid + i * kCtThreads;
        const float2 v = R[q];
        const float p = fmaf(v.x, v.x, v.y * v.y);   // frame intensity in float, accumulated in double
        psf[q] = acc[i] + (double)p;
    }
    if (c0 == 0 && tid == 0) L.acc->n_psf += 1;
}

template <int M>
size_t ct_smem() {
    return sizeof(float2) * (2 * kCtRows * (size_t)M + M);
}

template <int M>
cudaError_t ct_prepare() {
    cudaError_t e = cudaFuncSetAttribute((const void*)sci_rows_ct<M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)ct_smem<M>());
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute((const void*)sci_cols_ct<M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)ct_smem<M>());
}

template <int M>
cudaError_t ct_rows(const SciLaunch& L, cudaStream_t s) {
    sci_rows_ct<M><<<dim3((unsigned)((L.N + kCtRows - 1) / kCtRows), (unsigned)L.ctx.n_real), 256, ct_smem<M>(), s>>>(L);
    return cudaGetLastError();
}

template <int M>
cudaError_t ct_cols(const SciLaunch& L, cudaStream_t s) {
    sci_cols_ct<M><<<dim3((unsigned)(M / kCtRows + 1), (unsigned)L.ctx.n_real), 256, ct_smem<M>(), s>>>(L);
    return cudaGetLastError();
}

// sizes with a compile-time kernel; other sizes use the generic one
#define MCAO_SCI_CT_SIZES(X) X(128) X(256) X(512) X(640) X(1024) X(1280) X(2048)

size_t fft_smem_bytes(int M) {
    return sizeof(float2) * (2 * kRowsPerBlock * (size_t)M + M);
}

cudaError_t set_smem(const void* fn, size_t bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

cudaError_t launch_sci_field(const SciLaunch& L, cudaStream_t s) {
    int tiles = (L.N / 8) * (L.N / 8);
    sci_field_kernel<<<dim3((unsigned)((tiles + 7) / 8), (unsigned)L.ctx.n_real), 256, 0, s>>>(L);
    return cudaGetLastError();
}

bool sci_ct_size(int M) {
#define MCAO_CT_IS(n) \
    if (M == n) return true;
    MCAO_SCI_CT_SIZES(MCAO_CT_IS)
#undef MCAO_CT_IS
    return false;
}

std::vector<float2> sci_twiddles(int M) {
    auto w = [M](long long m) {
        const double a = -2.0 * M_PI * (double)m / (double)M;
        return make_float2((float)std::cos(a), (float)std::sin(a));
    };
    std::vector<float2> W(M);
    if (!sci_ct_size(M)) {
        for (int m = 0; m < M; ++m) W[m] = w(m);
        return W;
    }
    int off = 0;
    for (int ns = 1; ns < M; ns *= ct_radix(M / ns)) {
        const int R = ct_radix(M / ns);
        for (int r = 1; r < R; ++r)
            for (int k = 0; k < ns; ++k) W[off + (r - 1) * ns + k] = w(((long long)r * k * (M / (ns * R))) % M);
        off += ns * (R - 1);
    }
    return W;
}

cudaError_t sci_prepare(int M) {
    // the limit is the kernel's, not one simulation's: always that of the largest size that fits, so that
    // simulations of different sizes coexist
    const size_t sm = std::max(fft_smem_bytes(3200), fft_smem_bytes(M));
    cudaError_t e = set_smem((const void*)sci_rows_kernel, sm);
    if (e != cudaSuccess) return e;
    e = set_smem((const void*)sci_cols_kernel, sm);
    if (e != cudaSuccess) return e;
#define MCAO_CT_PREP(n) \
    if (M >= n) {       \
        e = ct_prepare<n>(); \
        if (e != cudaSuccess) return e; \
    }
    MCAO_SCI_CT_SIZES(MCAO_CT_PREP)
#undef MCAO_CT_PREP
    return cudaSuccess;
}

size_t sci_smem_bytes(int M) { return fft_smem_bytes(M); }

cudaError_t launch_sci_rows(const SciLaunch& L, cudaStream_t s) {
#define MCAO_CT_ROWS(n) \
    if (L.M == n) return ct_rows<n>(L, s);
    MCAO_SCI_CT_SIZES(MCAO_CT_ROWS)
#undef MCAO_CT_ROWS
    size_t sm = fft_smem_bytes(L.M);
    sci_rows_kernel<<<dim3((unsigned)((L.N + kRowsPerBlock - 1) / kRowsPerBlock), (unsigned)L.ctx.n_real), 256, sm, s>>>(L);
    return cudaGetLastError();
}

cudaError_t launch_sci_cols(const SciLaunch& L, cudaStream_t s) {
#define MCAO_CT_COLS(n) \
    if (L.M == n) return ct_cols<n>(L, s);
    MCAO_SCI_CT_SIZES(MCAO_CT_COLS)
#undef MCAO_CT_COLS
    size_t sm = fft_smem_bytes(L.M);
    sci_cols_kernel<<<dim3((unsigned)(L.M / kRowsPerBlock + 1), (unsigned)L.ctx.n_real), 256, sm, s>>>(L);
    return cudaGetLastError();
}

namespace {

// out[j][i] = psf_t[(i + M/2) mod M][(j + M/2) mod M] norm, 32 x 32 tiles through shared memory.  (The host
// did this over the copied accumulator, one strided read and two remainders per pixel: reading a
// 1280 x 1280 image took 4.9 ms; under half a millisecond now, most of it the copy.)
__global__ void __launch_bounds__(256) psf_out_kernel(const double* __restrict__ psf_t, int M, double norm,
                                                      double* __restrict__ out) {
    __shared__ double tile[32][33];
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32, x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (i0 + y < M && j0 + x < M) tile[y][x] = psf_t[(size_t)((i0 + y + M / 2) % M) * M + (j0 + x + M / 2) % M];
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (j0 + y < M && i0 + x < M) out[(size_t)(j0 + y) * M + i0 + x] = tile[x][y] * norm;
}

// a step's readout into one slot of the device ring (or into page-locked host buffers): the commands copied, the
// (long-exposure, instantaneous) Strehl ratios of each science direction from its accumulators
__global__ void readout_kernel(const float* __restrict__ c, int n_cmd, const SciAcc* __restrict__ acc, int n_sci,
                               float* __restrict__ ring_c, double* __restrict__ ring_s) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_cmd) ring_c[i] = c[i];
    if (i < n_sci) {
        const SciAcc a = acc[i];
        ring_s[2 * i] = a.n_sr ? a.sr_sum / (double)a.n_sr : 0.0;
        ring_s[2 * i + 1] = a.sr_last;
    }
}

}  // namespace

cudaError_t launch_psf_out(const double* psf_t, int M, double norm, double* out, cudaStream_t s) {
    const unsigned t = (unsigned)((M + 31) / 32);
    psf_out_kernel<<<dim3(t, t), 256, 0, s>>>(psf_t, M, norm, out);
    return cudaGetLastError();
}

cudaError_t launch_readout(const float* c, int n_cmd, const SciAcc* acc, int n_sci, float* ring_c, double* ring_s,
                           cudaStream_t s) {
    const int n = std::max(n_cmd, n_sci);
    if (n > 0) readout_kernel<<<(n + 255) / 256, 256, 0, s>>>(c, n_cmd, acc, n_sci, ring_c, ring_s);
    return cudaGetLastError();
}

}  // namespace mcao
