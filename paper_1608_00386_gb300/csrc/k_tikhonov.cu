// Tikhonov-regularised least-squares control matrix in FP64 on the GPU ("Control Matrix": the
// reconstructor is a pseudo-inverse of the interaction matrix, and MCAO least squares is
// ill-posed, hence a regularisation coefficient):
//   R = -(D^T D + lambda I)^(-1) D^T,   lambda = alpha tr(D^T D) / n_cmd,
// D [n_slopes][n_cmd] the interaction matrix (float32), R [n_cmd][n_slopes].  The minus sign: D is
// measured with the DM subtracted from the wavefront, and the loop applies c <- c + g R s.
//
// Every step runs in double precision in the kernels below:
//   1. D compressed by rows and by columns (a subaperture sees only the actuators within the
//      influence functions' reach: 6 % of D at 20 m, less at 39 m);
//   2. Gram matrix G = D^T D over the nonzero pairs;
//   3. lambda from the trace, G + lambda I (padding rows past n_cmd get a unit diagonal);
//   4. blocked right-looking Cholesky G = L L^T on 64 x 64 tiles together with X = L^(-1): per block
//      column k, the diagonal block is factored and inverted in one block's registers (potrf); the
//      panel L[i][k] and the block row X[k][j] are multiplied by that inverse (panel); the
//      trailing tiles of L and the rows of X below are updated (update);
//   5. M^(-1) = X^T X (lower tiles, mirrored), written over L;
//   6. R = -M^(-1) D^T over the nonzeros of D's rows; rounded to float32 once, at the store (or
//      stored in double).
// The GB300 issues two double FMAs per cycle and SM, 1/64 of the float32 rate, so operations are all
// that counts: the tile products run at that rate with operands straight from L2 and shared memory,
// and what is worth doing is to leave out multiplications by zeros and to keep every SM's pipe busy.
// Hence the compressed D (64 x 64 tiles of D that hold a nonzero cover six times the nonzeros: Gram
// 8.2 ms and product 16.4 ms at 20 m before), the lower halves of triangular blocks only, and 32 x 32
// outputs per block, four of which share an SM's pipe: the last wave of a launch costs a quarter of
// what 64 x 64 outputs cost.  A dense D (more than a third nonzero) takes the tile products, where
// each operand read serves 32 outputs.
// 20 m (7280 x 1870): 46.6 ms before, 12.3 ms now; 39 m (55608 x 8051): 2.2 s before.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>

#include "../../include/mcao.h"

namespace {

constexpr int kT = 64;          // tile side
constexpr int kS = 32;          // output side and k depth of one block's product
constexpr int kThreads = 128;   // 16 x 8 threads, 2 x 4 outputs each
constexpr int kGramMaxCmd = 28000;   // commands whose row of G fits in shared memory

// One chunk of a product: a[k][r], b[k][c] for k < kS (rows padded by one double).
struct Chunk {
    double a[kS][kS + 1];
    double b[kS][kS + 1];
};

__device__ __forceinline__ void chunk_fma(const Chunk& ch, double (&c)[2][4]) {
    const int r = threadIdx.x / 8 * 2, q = threadIdx.x % 8;
#pragma unroll 8
    for (int k = 0; k < kS; ++k) {
        double av[2], bv[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) av[i] = ch.a[k][r + i];
#pragma unroll
        for (int j = 0; j < 4; ++j) bv[j] = ch.b[k][q + 8 * j];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) c[i][j] = fma(av[i], bv[j], c[i][j]);
    }
}
// output (i, j) of this thread: row and column within the 32 x 32 block
__device__ __forceinline__ int out_row(int i) { return threadIdx.x / 8 * 2 + i; }
__device__ __forceinline__ int out_col(int j) { return threadIdx.x % 8 + 8 * j; }

// T[k][i] = src[(r0 + k) ld + c0 + i] for k, i < 32 (the source block as it is), zero past (nr, nc);
// float or double source
template <typename S>
__device__ __forceinline__ void load_direct(double (*T)[kS + 1], const S* src, long long ld, long long r0, long long c0,
                                            long long nr, long long nc) {
#pragma unroll
    for (int q = threadIdx.x; q < kS * kS; q += kThreads) {
        const int k = q / kS, i = q % kS;
        const long long r = r0 + k, c = c0 + i;
        T[k][i] = (r < nr && c < nc) ? (double)src[r * ld + c] : 0.0;
    }
}

// T[k][i] = src[(r0 + i) ld + c0 + k] (the source block transposed), zero past (nr, nc)
template <typename S>
__device__ __forceinline__ void load_trans(double (*T)[kS + 1], const S* src, long long ld, long long r0, long long c0,
                                           long long nr, long long nc) {
#pragma unroll
    for (int q = threadIdx.x; q < kS * kS; q += kThreads) {
        const int i = q / kS, k = q % kS;   // consecutive threads walk along a source row
        const long long r = r0 + i, c = c0 + k;
        T[k][i] = (r < nr && c < nc) ? (double)src[r * ld + c] : 0.0;
    }
}

// lower-triangle tile index t -> (i, j), i >= j
__device__ __forceinline__ void tri_index(long long t, int& i, int& j) {
    int ii = (int)floorf((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((long long)(ii + 1) * (ii + 2) / 2 <= t) ++ii;
    while ((long long)ii * (ii + 1) / 2 > t) --ii;
    i = ii;
    j = (int)(t - (long long)ii * (ii + 1) / 2);
}

// ------------------------------------------------------------------------------------------
// 1. compressed D
// ------------------------------------------------------------------------------------------
constexpr int kCscWarps = 32;   // warps of a column block, each a slab of consecutive rows

// nonzeros of each row (one warp per row)
__global__ void __launch_bounds__(256) tik_row_count_kernel(const float* __restrict__ D, long long ld, int n_slopes,
                                                            int n_cmd, int* __restrict__ count) {
    const int r = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x & 31;
    if (r >= n_slopes) return;
    int n = 0;
#pragma unroll 8
    for (int c = lane; c < n_cmd; c += 32) n += D[r * ld + c] != 0.0f;
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) count[r] = n;
}

// nonzeros of the 32 columns of this block in each warp's slab of rows
__device__ __forceinline__ int slab_count(const float* D, long long ld, int r0, int r1, int c, int n_cmd) {
    int n = 0;
    if (c < n_cmd)
#pragma unroll 8
        for (int r = r0; r < r1; ++r) n += D[r * ld + c] != 0.0f;
    return n;
}

__global__ void __launch_bounds__(32 * kCscWarps) tik_col_count_kernel(const float* __restrict__ D, long long ld, int n_slopes,
                                                                       int n_cmd, int* __restrict__ count) {
    __shared__ int s_n[kCscWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32, c = blockIdx.x * 32 + lane;
    const int slab = (n_slopes + kCscWarps - 1) / kCscWarps, r0 = w * slab, r1 = min(n_slopes, r0 + slab);
    s_n[w][lane] = slab_count(D, ld, r0, r1, c, n_cmd);
    __syncthreads();
    if (w == 0 && c < n_cmd) {
        int n = 0;
        for (int q = 0; q < kCscWarps; ++q) n += s_n[q][lane];
        count[c] = n;
    }
}

// exclusive prefix sums in place, count[n] = total (one block)
__global__ void __launch_bounds__(1024) tik_scan_kernel(int* __restrict__ count, int n) {
    __shared__ int s_w[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32;
    int base = 0;
    for (int i0 = 0; i0 < n; i0 += 1024) {
        const int i = i0 + threadIdx.x, v = i < n ? count[i] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_w[w] = x;
        __syncthreads();
        int before = 0, total = 0;
        for (int q = 0; q < 32; ++q) {
            before += q < w ? s_w[q] : 0;
            total += s_w[q];
        }
        if (i < n) count[i] = base + before + x - v;
        base += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) count[n] = base;
}

// columns and values of each row's nonzeros, ascending; the values as doubles, since each of them meets
// thousands of products and a conversion takes the double pipe half as long as a multiply-add (20 m,
// Gram 885 -> 765 us and product 4400 -> 2700; 2660 is the double pipes' time)
__global__ void __launch_bounds__(256) tik_row_fill_kernel(const float* __restrict__ D, long long ld, int n_slopes, int n_cmd,
                                                           const int* __restrict__ row, int* __restrict__ col,
                                                           double* __restrict__ val) {
    const int r = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x & 31;
    if (r >= n_slopes) return;
    int at = row[r];
    for (int c0 = 0; c0 < n_cmd; c0 += 32) {
        const int c = c0 + lane;
        const float v = c < n_cmd ? D[r * ld + c] : 0.0f;
        const unsigned m = __ballot_sync(0xffffffffu, v != 0.0f);
        if (v != 0.0f) {
            const int p = at + __popc(m & ((1u << lane) - 1u));
            col[p] = c;
            val[p] = (double)v;
        }
        at += __popc(m);
    }
}

// rows and values of each column's nonzeros, ascending
__global__ void __launch_bounds__(32 * kCscWarps) tik_col_fill_kernel(const float* __restrict__ D, long long ld, int n_slopes,
                                                                      int n_cmd, const int* __restrict__ col_at,
                                                                      int* __restrict__ row, float* __restrict__ val) {
    __shared__ int s_n[kCscWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32, c = blockIdx.x * 32 + lane;
    const int slab = (n_slopes + kCscWarps - 1) / kCscWarps, r0 = w * slab, r1 = min(n_slopes, r0 + slab);
    s_n[w][lane] = slab_count(D, ld, r0, r1, c, n_cmd);
    __syncthreads();
    if (c >= n_cmd) return;
    int at = col_at[c];
    for (int q = 0; q < w; ++q) at += s_n[q][lane];
#pragma unroll 8
    for (int r = r0; r < r1; ++r) {
        const float v = D[r * ld + c];
        if (v != 0.0f) {
            row[at] = r;
            val[at++] = v;
        }
    }
}

// ------------------------------------------------------------------------------------------
// 2. Gram matrix
// ------------------------------------------------------------------------------------------
// One block per actuator a: G[a][b] for b <= a, summed in shared memory over the rows s where D[s][a]
// is nonzero, in ascending order; the threads take the row's nonzeros side by side (the next row's
// are read while this one is added).
__global__ void __launch_bounds__(128) tik_gram_sparse_kernel(const int* __restrict__ col_at, const int* __restrict__ col_row,
                                                              const float* __restrict__ col_val, const int* __restrict__ row,
                                                              const int* __restrict__ col, const double* __restrict__ val,
                                                              double* __restrict__ G, long long ldg) {
    extern __shared__ double gram_acc[];
    const int a = gridDim.x - 1 - blockIdx.x;   // the longest rows of G first
    const int tid = threadIdx.x;
    for (int b = tid; b <= a; b += 128) gram_acc[b] = 0.0;
    const int p0 = col_at[a], p1 = col_at[a + 1];
    __syncthreads();
    int q0 = 0, q1 = 0, b = 0;
    float dsa = 0.0f;
    double v = 0.0;
    auto fetch = [&](int p) {
        const int s = col_row[p];
        dsa = col_val[p];
        q0 = row[s];
        q1 = row[s + 1];
        b = q0 + tid < q1 ? col[q0 + tid] : a + 1;
        v = q0 + tid < q1 ? val[q0 + tid] : 0.0;
    };
    if (p0 < p1) fetch(p0);
    for (int p = p0; p < p1; ++p) {
        const int bb = b, n = q1, first = q0;
        const double vv = v, d = (double)dsa;
        if (p + 1 < p1) fetch(p + 1);
        if (bb <= a) gram_acc[bb] = fma(d, vv, gram_acc[bb]);
        for (int q = first + 128 + tid; q < n; q += 128) {
            const int e = col[q];
            if (e <= a) gram_acc[e] = fma(d, val[q], gram_acc[e]);
        }
        __syncthreads();
    }
    for (int e = tid; e <= a; e += 128) {
        G[(long long)a * ldg + e] = gram_acc[e];
        if (e < a) G[(long long)e * ldg + a] = gram_acc[e];
    }
}

// dense D: mask[S][J] = 1 if the tile (slopes 64 S.., commands 64 J..) of D holds a nonzero
__global__ void __launch_bounds__(kThreads) tik_mask_kernel(const float* __restrict__ D, long long ld, int n_slopes,
                                                            int n_cmd, int nJ, unsigned char* __restrict__ mask) {
    const int J = blockIdx.x, S = blockIdx.y;
    int any = 0;
    for (int q = threadIdx.x; q < kT * kT; q += kThreads) {
        const int r = S * kT + q / kT, c = J * kT + (q % kT);
        if (r < n_slopes && c < n_cmd && D[(long long)r * ld + c] != 0.0f) any = 1;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) mask[(long long)S * nJ + J] = (unsigned char)any;
}

// dense D: 32 x 32 block (I, J) of G, I >= J, over the slope tiles where both tiles of D hold a
// nonzero; mirrored
__global__ void __launch_bounds__(kThreads) tik_gram_kernel(const float* __restrict__ D, long long ld, int n_slopes,
                                                            int n_cmd, int nS, int nt,
                                                            const unsigned char* __restrict__ mask,
                                                            double* __restrict__ G, long long ldg) {
    __shared__ Chunk ch;
    int I, J;
    tri_index(blockIdx.x, I, J);
    double c[2][4] = {};
    for (int S = 0; S < nS; ++S) {
        if (!mask[(long long)S * nt + I / 2] || !mask[(long long)S * nt + J / 2]) continue;
        for (int k0 = 0; k0 < kT; k0 += kS) {
            load_direct(ch.a, D, ld, (long long)S * kT + k0, (long long)I * kS, n_slopes, n_cmd);
            load_direct(ch.b, D, ld, (long long)S * kT + k0, (long long)J * kS, n_slopes, n_cmd);
            __syncthreads();
            chunk_fma(ch, c);
            __syncthreads();
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long r = (long long)I * kS + out_row(i), q = (long long)J * kS + out_col(j);
            G[r * ldg + q] = c[i][j];
            if (I != J) G[q * ldg + r] = c[i][j];
        }
}

// 3. lambda = alpha tr(G) / n_cmd; G + lambda I on the first n_cmd rows, unit diagonal on the
// padding rows (their rows and columns of G are zero)
__global__ void tik_regularize_kernel(double* __restrict__ G, long long ldg, int n_cmd, int npad, double alpha,
                                      double* __restrict__ lambda_out) {
    __shared__ double part[1024];
    double s = 0.0;
    for (int i = threadIdx.x; i < n_cmd; i += blockDim.x) s += G[(long long)i * ldg + i];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    const double lam = alpha * part[0] / (double)n_cmd;
    for (int i = threadIdx.x; i < npad; i += blockDim.x) {
        if (i < n_cmd)
            G[(long long)i * ldg + i] += lam;
        else
            G[(long long)i * ldg + i] = 1.0;
    }
    if (threadIdx.x == 0) *lambda_out = lam;
}

// ------------------------------------------------------------------------------------------
// 4. Cholesky factor and its inverse
// ------------------------------------------------------------------------------------------
// 1 / d: float reciprocal of the significand (2^-23) and two Newton steps y + y (1 - m y), the exponent
// put back in the high word; zeros, subnormals and infinities take the division
__device__ __forceinline__ double reciprocal(double d) {
    const int hi = __double2hiint(d), ex = (hi >> 20) & 0x7ff;
    if (ex == 0 || ex >= 2045) return 1.0 / d;
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(d));   // [1, 2)
    double y = (double)(1.0f / (float)m);
    y = fma(y, fma(-m, y, 1.0), y);
    y = fma(y, fma(-m, y, 1.0), y);
    return __hiloint2double(__double2hiint(y) + ((1023 - ex) << 20), __double2loint(y));
}

// 4a. Linv = L^(-1) of the diagonal block S = L L^T, in one block: the lower triangle of a 64 x 64
// array W, 8 or 9 entries (m, c) per thread in registers, starts as S and ends as the inverse of the
// unit factor of S = U D U^T.  Before step j the columns c >= j of the rows m >= j hold the trailing
// matrix S, the columns c < j the rows of X = U^(-1) so far.  Step j takes v_m = S_mj / S_jj and u_c =
// X_jc (c < j), 1 (c = j), S_cj (c > j), then W_mc -= v_m u_c on every row below (W_mj counts as 0
// there: column j of X begins).  At the end row m is scaled by 1 / sqrt(D_m).  So factor and inverse cost
// one pass of 64^3 / 3 multiply-adds with two barriers a step, and no square root is in the chain from
// one pivot to the next.  Entries are dealt row by row, so finished rows leave whole warps idle.
// Bound by the latency of the double operations of that chain (the 87 k multiply-adds alone are 22 us
// of one SM's pipe).  Factor and inverse one after the other in shared memory took 228 us a block, 6.9
// of 46.6 ms at 20 m; in one pass with L and its square roots 114 us; 75 us now.  A pivot <= 0
// (or NaN) sets *err and is replaced by 1 so that the remaining steps stay finite.
// For k > 0 the block first takes panel k - 1 out of its tile (4c leaves that tile to it), and the
// update of the other tiles runs at the same time as a programmatic dependent: 114 us on one SM beside
// the 205 us of an update at 20 m (14.1 -> 12.3 ms a call).  The block asks for more shared memory than it uses, so that no
// update block shares its SM's double pipe (sharing it, the chain took longer than the update).
constexpr int kPotrfSmem = 210 * 1024;
static_assert(kT * (kT + 1) * sizeof(double) <= kPotrfSmem);
__global__ void __launch_bounds__(256) tik_potrf_kernel(const double* __restrict__ A, long long lda, int k,
                                                        double* __restrict__ Linv, int* __restrict__ err) {
    extern __shared__ double s_pan[];   // [64][65]: L[k][k - 1]
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int kEnt = kT * (kT + 1) / 2, kPer = (kEnt + 255) / 256;
    __shared__ double s_col[2][kT], s_u[2][kT], s_v[2][kT], s_diag[kT];
    const int tid = threadIdx.x;
    const long long o = (long long)k * kT;
    double w[kPer];
    int mc[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int p = i * 256 + tid;
        int m = kT, c = 0;   // past the triangle: never touched
        if (p < kEnt) tri_index(p, m, c);
        mc[i] = m << 8 | c;
        w[i] = p < kEnt ? A[(o + m) * lda + o + c] : 0.0;
    }
    if (k > 0) {
        for (int q = tid; q < kT * kT; q += 256) s_pan[q / kT * (kT + 1) + q % kT] = A[(o + q / kT) * lda + o - kT + q % kT];
        __syncthreads();
        double acc[kPer] = {};
#pragma unroll 2
        for (int q = 0; q < kT; ++q)
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int m = min(mc[i] >> 8, kT - 1), c = mc[i] & 255;
                acc[i] = fma(s_pan[m * (kT + 1) + q], s_pan[c * (kT + 1) + q], acc[i]);
            }
#pragma unroll
        for (int i = 0; i < kPer; ++i) w[i] -= acc[i];
    }
    for (int j = 0; j < kT; ++j) {
        double *col = s_col[j & 1], *u = s_u[j & 1], *v = s_v[j & 1];   // the other pair may still be read
        // column j from the diagonal down, and row j of X
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int m = mc[i] >> 8, c = mc[i] & 255;
            if (m < kT && c == j) col[m] = w[i];
            if (m == j && c < j) u[c] = w[i];
        }
        __syncthreads();
        if (tid < kT) {
            double d = col[j];
            if (!(d > 0.0)) {
                if (tid == 0) atomicExch(err, 1);
                d = 1.0;
            }
            if (tid == j) {
                s_diag[j] = d;
                u[j] = 1.0;
            } else if (tid > j) {
                u[tid] = col[tid];
                v[tid] = col[tid] * reciprocal(d);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int m = mc[i] >> 8, c = mc[i] & 255;
            if (m > j && m < kT) w[i] = fma(-v[m], u[c], c == j ? 0.0 : w[i]);
            else if (m == j && c == j) w[i] = 1.0;
        }
    }
    __syncthreads();
    if (tid < kT) s_v[0][tid] = 1.0 / sqrt(s_diag[tid]);
    double* Lk = Linv + (long long)k * kT * kT;
    for (int q = tid; q < kT * kT; q += 256)
        if (q % kT > q / kT) Lk[q] = 0.0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int m = mc[i] >> 8, c = mc[i] & 255;
        if (m < kT) Lk[m * kT + c] = w[i] * s_v[0][m];
    }
}

// 4b. block column k of L below the diagonal, A[i][k] <- A[i][k] Linv_kk^T, and block row k of X,
// X[k][j] <- Linv_kk X[k][j] for j < k, X[k][k] = Linv_kk, both in place.  One block per strip of 16
// rows (A) or columns (X), read whole before it is written; Linv is lower triangular, so its first 32
// rows need half the depth.  (Strips of 32: 41 us a launch at 20 m, 60 blocks on 152 SMs; 26
// us with 120.)
constexpr int kStrip = 16;
__global__ void __launch_bounds__(kThreads) tik_panel_kernel(double* __restrict__ A, double* __restrict__ X, long long ld, int k,
                                                             int nt, const double* __restrict__ Linv) {
    __shared__ double s_l[kT][kT + 1];         // Linv
    __shared__ double s_p[kT][kStrip + 1];     // the strip, [depth][row or column]
    constexpr int kPerTile = kT / kStrip;
    const int n_a = kPerTile * (nt - k - 1), t = threadIdx.x;
    const bool is_a = (int)blockIdx.x < n_a;
    const double* Lk = Linv + (long long)k * kT * kT;
    const int q0 = is_a ? 0 : ((int)blockIdx.x - n_a) * kStrip;   // first column of a strip of X
    double* P = is_a ? A + ((long long)(k + 1) * kT + blockIdx.x * kStrip) * ld + (long long)k * kT : X + (long long)k * kT * ld + q0;
    if (!is_a && q0 >= k * kT) {
        for (int q = t; q < kT * kStrip; q += kThreads)
            P[q / kStrip * ld + q % kStrip] = Lk[q / kStrip * kT + q0 - k * kT + q % kStrip];
        return;
    }
    for (int q = t; q < kT * kT; q += kThreads) s_l[q / kT][q % kT] = Lk[q];
    for (int q = t; q < kT * kStrip; q += kThreads) {
        if (is_a) s_p[q % kT][q / kT] = P[q / kT * ld + q % kT];
        else s_p[q / kStrip][q % kStrip] = P[q / kStrip * ld + q % kStrip];
    }
    __syncthreads();
    // this thread: strip entry e, Linv rows g, g + 8, ..
    const int e = t % kStrip, g = t / kStrip;
    double c[8] = {};
#pragma unroll 4
    for (int m = 0; m < kT / 2; ++m) {
        const double p = s_p[m][e];
#pragma unroll
        for (int i = 0; i < 8; ++i) c[i] = fma(p, s_l[g + 8 * i][m], c[i]);
    }
#pragma unroll 4
    for (int m = kT / 2; m < kT; ++m) {
        const double p = s_p[m][e];
#pragma unroll
        for (int i = 4; i < 8; ++i) c[i] = fma(p, s_l[g + 8 * i][m], c[i]);
    }
    if (is_a) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) s_p[g + 8 * i][e] = c[i];
        __syncthreads();
        for (int q = t; q < kT * kStrip; q += kThreads) P[q / kT * ld + q % kT] = s_p[q % kT][q / kT];
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) P[(g + 8 * i) * ld + e] = c[i];
    }
}

// 4c. with L[.][k] and X[k][.] final: A[i][j] -= L[i][k] L[j][k]^T for the lower tiles i >= j > k but the
// first (the next diagonal block's launch takes that one), and X[m][j] -= L[m][k] X[k][j] for m > k,
// j <= k, in 32 x 32 blocks of one launch (blocks of the trailing matrix first, in order of rows).  It
// starts beside that launch, whose end the last block waits for: what follows needs both.
__global__ void __launch_bounds__(kThreads) tik_update_kernel(double* __restrict__ A, double* __restrict__ X, long long ld, int k,
                                                              int nt) {
    __shared__ Chunk ch;
    const int rest = 2 * (nt - k - 1);   // 32-row blocks below
    const long long n_a = (long long)rest * (rest + 1) / 2;
    const long long L0 = (long long)(k + 1) * kT, kc = (long long)k * kT, npad = (long long)nt * kT;
    const long long b0 = (long long)blockIdx.x + 3;   // three 32 x 32 blocks of the first tile
    double c[2][4] = {};
    if (b0 < n_a) {
        int i, j;
        tri_index(b0, i, j);
        for (int k0 = 0; k0 < kT; k0 += kS) {
            load_trans(ch.a, A, ld, L0 + i * kS, kc + k0, npad, npad);
            load_trans(ch.b, A, ld, L0 + j * kS, kc + k0, npad, npad);
            __syncthreads();
            chunk_fma(ch, c);
            __syncthreads();
        }
        double* P = A + (L0 + i * kS) * ld + L0 + j * kS;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) P[out_row(a) * ld + out_col(b)] -= c[a][b];
        return;
    }
    const int t = (int)(b0 - n_a), cols = 2 * (k + 1);
    const long long r0 = L0 + (long long)(t / cols) * kS, c0 = (long long)(t % cols) * kS;
    for (int k0 = 0; k0 < kT; k0 += kS) {
        load_trans(ch.a, A, ld, r0, kc + k0, npad, npad);
        load_direct(ch.b, X, ld, kc + k0, c0, npad, npad);
        __syncthreads();
        chunk_fma(ch, c);
        __syncthreads();
    }
    double* P = X + r0 * ld + c0;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) P[out_row(a) * ld + out_col(b)] -= c[a][b];
    if (blockIdx.x == gridDim.x - 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// 5. Minv[I][J] = sum_m X[m][I]^T X[m][J] over the 32-row blocks m >= I (X lower triangular) for the
// lower blocks, mirrored; the longest sums first
__global__ void __launch_bounds__(kThreads) tik_xtx_kernel(const double* __restrict__ X, long long ldx, int nb,
                                                           double* __restrict__ Minv, long long ldm) {
    __shared__ Chunk ch;
    int I, J;
    tri_index(blockIdx.x, I, J);
    const long long npad = (long long)nb * kS;
    double c[2][4] = {};
    for (int m = I; m < nb; ++m) {
        load_direct(ch.a, X, ldx, (long long)m * kS, (long long)I * kS, npad, npad);
        load_direct(ch.b, X, ldx, (long long)m * kS, (long long)J * kS, npad, npad);
        __syncthreads();
        chunk_fma(ch, c);
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const long long r = (long long)I * kS + out_row(a), q = (long long)J * kS + out_col(b);
            Minv[r * ldm + q] = c[a][b];
            if (I != J) Minv[q * ldm + r] = c[a][b];
        }
}

// ------------------------------------------------------------------------------------------
// 6. R = -M^(-1) D^T
// ------------------------------------------------------------------------------------------
// 64 commands x 32 slopes per block: a warp takes 4 slopes one after another, each lane 2 commands
// (Minv is symmetric: the row of each nonzero's actuator is read, 512 bytes per warp, mostly from L1
// since neighbouring slopes share actuators); transposed through shared memory for the store.
template <typename Out>
__global__ void __launch_bounds__(256) tik_apply_sparse_kernel(const double* __restrict__ Minv, long long ldm,
                                                               const int* __restrict__ row, const int* __restrict__ col,
                                                               const double* __restrict__ val, int n_slopes, int n_cmd,
                                                               Out* __restrict__ R, long long ldr) {
    __shared__ Out s_r[kT][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32;
    const int s0 = blockIdx.x * 32, i0 = blockIdx.y * kT;   // slopes run fastest: the blocks in flight share Minv's columns
    const double* M = Minv + i0 + 2 * lane;
    for (int q = 0; q < 4; ++q) {
        const int s = s0 + 4 * w + q;
        double x = 0.0, y = 0.0;
        if (s < n_slopes) {
            const int p1 = row[s + 1];
#pragma unroll 4
            for (int p = row[s]; p < p1; ++p) {
                const double2 m = *reinterpret_cast<const double2*>(M + (long long)__ldg(col + p) * ldm);
                const double d = __ldg(val + p);
                x = fma(m.x, d, x);
                y = fma(m.y, d, y);
            }
        }
        s_r[2 * lane][4 * w + q] = (Out)(-x);
        s_r[2 * lane + 1][4 * w + q] = (Out)(-y);
    }
    __syncthreads();
    for (int i = w; i < kT; i += 8)
        if (i0 + i < n_cmd && s0 + lane < n_slopes) R[(long long)(i0 + i) * ldr + s0 + lane] = s_r[i][lane];
}

// dense D: 32 x 32 block (commands I, slopes S) over the nonzero tiles of D
template <typename Out>
__global__ void __launch_bounds__(kThreads) tik_apply_kernel(const double* __restrict__ Minv, long long ldm, int nt,
                                                             const float* __restrict__ D, long long ld, int n_slopes,
                                                             int n_cmd, const unsigned char* __restrict__ mask,
                                                             Out* __restrict__ R, long long ldr) {
    __shared__ Chunk ch;
    const int I = blockIdx.y, S = blockIdx.x;
    const long long npad = (long long)nt * kT;
    double c[2][4] = {};
    for (int J = 0; J < nt; ++J) {
        if (!mask[(long long)(S / 2) * nt + J]) continue;
        for (int k0 = 0; k0 < kT; k0 += kS) {
            // C[r][q] = sum_m Minv[J0 + m][I0 + r] D[S0 + q][J0 + m]
            load_direct(ch.a, Minv, ldm, (long long)J * kT + k0, (long long)I * kS, npad, npad);
            load_trans(ch.b, D, ld, (long long)S * kS, (long long)J * kT + k0, n_slopes, n_cmd);
            __syncthreads();
            chunk_fma(ch, c);
            __syncthreads();
        }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const long long r = (long long)I * kS + out_row(a), q = (long long)S * kS + out_col(b);
            if (r < n_cmd && q < n_slopes) R[r * ldr + q] = (Out)(-c[a][b]);
        }
}

mcao_status report(char* err, size_t err_len, mcao_status st, const char* fmt, ...) {
    if (err && err_len) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(err, err_len, fmt, ap);
        va_end(ap);
    }
    return st;
}

}  // namespace

extern "C" mcao_status mcao_tikhonov_reconstructor(const float* D, int n_slopes, int n_cmd, size_t ld_d, double alpha,
                                                   void* R, size_t ld_r, int r_fp64, void* stream, double* lambda,
                                                   char* err, size_t err_len) {
    if (err && err_len) err[0] = '\0';
    if (!D || !R) return report(err, err_len, MCAO_E_INVALID_ARG, "D and R must be device pointers");
    if (n_slopes < 1 || n_cmd < 1) return report(err, err_len, MCAO_E_SHAPE, "n_slopes and n_cmd must be >= 1");
    if (ld_d < (size_t)n_cmd || ld_r < (size_t)n_slopes)
        return report(err, err_len, MCAO_E_SHAPE, "need ld_d >= n_cmd and ld_r >= n_slopes");
    if (!std::isfinite(alpha) || alpha < 0.0) return report(err, err_len, MCAO_E_INVALID_ARG, "alpha must be >= 0");
    if (r_fp64 != 0 && r_fp64 != 1) return report(err, err_len, MCAO_E_INVALID_ARG, "r_fp64 must be 0 or 1");
    const int nt = (n_cmd + kT - 1) / kT, nS = (n_slopes + kT - 1) / kT;
    const long long npad = (long long)nt * kT, ld = (long long)ld_d;
    cudaStream_t st = (cudaStream_t)stream;
    double *G = nullptr, *X = nullptr, *Linv = nullptr, *d_lam = nullptr;
    int *at = nullptr, *idx = nullptr, *d_err = nullptr;
    double* val = nullptr;       // of the rows
    float* col_val = nullptr;
    unsigned char* mask = nullptr;
    cudaError_t e = cudaMalloc(&G, sizeof(double) * npad * npad);
    if (e == cudaSuccess) e = cudaMalloc(&X, sizeof(double) * npad * npad);
    if (e == cudaSuccess) e = cudaMalloc(&Linv, sizeof(double) * nt * kT * kT);
    if (e == cudaSuccess) e = cudaMalloc(&at, sizeof(int) * ((size_t)n_slopes + n_cmd + 2));
    if (e == cudaSuccess) e = cudaMalloc(&d_err, 2 * sizeof(double));   // error flag, then lambda
    // nonzeros: row starts at at[0 .. n_slopes], column starts at at[n_slopes + 1 ..]
    int* col_at = at + n_slopes + 1;
    int nnz = 0;
    if (e == cudaSuccess) {
        tik_row_count_kernel<<<(n_slopes + 7) / 8, 256, 0, st>>>(D, ld, n_slopes, n_cmd, at);
        tik_col_count_kernel<<<(n_cmd + 31) / 32, 32 * kCscWarps, 0, st>>>(D, ld, n_slopes, n_cmd, col_at);
        tik_scan_kernel<<<1, 1024, 0, st>>>(at, n_slopes);
        tik_scan_kernel<<<1, 1024, 0, st>>>(col_at, n_cmd);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&nnz, at + n_slopes, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    // compressed products up to a third of nonzeros (more than 2^31 of them wrap to a negative count),
    // as long as a row of G fits in shared memory and the device has room for the nonzeros; else tile products
    const int gram_smem = n_cmd * (int)sizeof(double);
    bool sparse = (long long)n_slopes * n_cmd < (1LL << 31) && (long long)nnz * 3 <= (long long)n_slopes * n_cmd &&
                  n_cmd <= kGramMaxCmd;
    if (e == cudaSuccess && sparse) {
        e = cudaMalloc(&idx, sizeof(int) * 2 * (size_t)(nnz > 0 ? nnz : 1));
        if (e == cudaSuccess) e = cudaMalloc(&val, sizeof(double) * (size_t)(nnz > 0 ? nnz : 1));
        if (e == cudaSuccess) e = cudaMalloc(&col_val, sizeof(float) * (size_t)(nnz > 0 ? nnz : 1));
        if (e == cudaErrorMemoryAllocation) {   // no room beside the factors: the tiles need none
            cudaGetLastError();
            for (void* p : {(void*)idx, (void*)val, (void*)col_val}) cudaFree(p);
            idx = nullptr;
            val = nullptr;
            col_val = nullptr;
            sparse = false;
            e = cudaSuccess;
        }
    }
    if (e == cudaSuccess && !sparse) e = cudaMalloc(&mask, (size_t)nS * nt);
    auto cleanup = [&]() {
        for (void* p : {(void*)G, (void*)X, (void*)Linv, (void*)at, (void*)idx, (void*)val, (void*)col_val, (void*)mask, (void*)d_err}) cudaFree(p);
    };
    if (e != cudaSuccess) {
        cleanup();
        cudaGetLastError();
        return report(err, err_len, e == cudaErrorMemoryAllocation ? MCAO_E_OOM : MCAO_E_CUDA,
                      "allocation of the FP64 work arrays (%lld x %lld doubles, twice): %s", npad, npad,
                      cudaGetErrorString(e));
    }
    d_lam = reinterpret_cast<double*>(d_err) + 1;
    e = cudaMemsetAsync(d_err, 0, sizeof(int), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(G, 0, sizeof(double) * npad * npad, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(X, 0, sizeof(double) * npad * npad, st);
    // the limit is the kernel's, for calls of every size from every thread
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tik_gram_sparse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramMaxCmd * (int)sizeof(double));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(tik_potrf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPotrfSmem);
    if (e == cudaSuccess) {
        if (sparse) {
            tik_row_fill_kernel<<<(n_slopes + 7) / 8, 256, 0, st>>>(D, ld, n_slopes, n_cmd, at, idx, val);
            tik_col_fill_kernel<<<(n_cmd + 31) / 32, 32 * kCscWarps, 0, st>>>(D, ld, n_slopes, n_cmd, col_at, idx + nnz, col_val);
            tik_gram_sparse_kernel<<<n_cmd, 128, gram_smem, st>>>(col_at, idx + nnz, col_val, at, idx, val, G, npad);
        } else {
            tik_mask_kernel<<<dim3(nt, nS), kThreads, 0, st>>>(D, ld, n_slopes, n_cmd, nt, mask);
            tik_gram_kernel<<<(unsigned)((long long)2 * nt * (2 * nt + 1) / 2), kThreads, 0, st>>>(D, ld, n_slopes, n_cmd, nS, nt,
                                                                                                 mask, G, npad);
        }
        tik_regularize_kernel<<<1, 1024, 0, st>>>(G, npad, n_cmd, (int)npad, alpha, d_lam);
        tik_potrf_kernel<<<1, 256, kPotrfSmem, st>>>(G, npad, 0, Linv, d_err);
        for (int k = 0; k < nt; ++k) {
            const long long below = nt - k - 1, rest = 2 * below;
            tik_panel_kernel<<<(unsigned)(kT / kStrip * nt), kThreads, 0, st>>>(G, X, npad, k, nt, Linv);
            if (below == 0) break;
            tik_potrf_kernel<<<1, 256, kPotrfSmem, st>>>(G, npad, k + 1, Linv, d_err);
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)(rest * (rest + 1) / 2 - 3 + rest * 2 * (k + 1)));
            cfg.blockDim = dim3(kThreads);
            cfg.stream = st;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            cudaLaunchKernelEx(&cfg, tik_update_kernel, G, X, npad, k, nt);
        }
        // M^-1 over the factor
        tik_xtx_kernel<<<(unsigned)((long long)2 * nt * (2 * nt + 1) / 2), kThreads, 0, st>>>(X, npad, 2 * nt, G, npad);
        const dim3 gs((unsigned)((n_slopes + 31) / 32), (unsigned)nt), gd((unsigned)((n_slopes + kS - 1) / kS), (unsigned)(2 * nt));
        if (sparse && r_fp64)
            tik_apply_sparse_kernel<double><<<gs, 256, 0, st>>>(G, npad, at, idx, val, n_slopes, n_cmd, (double*)R, (long long)ld_r);
        else if (sparse)
            tik_apply_sparse_kernel<float><<<gs, 256, 0, st>>>(G, npad, at, idx, val, n_slopes, n_cmd, (float*)R, (long long)ld_r);
        else if (r_fp64)
            tik_apply_kernel<double><<<gd, kThreads, 0, st>>>(G, npad, nt, D, ld, n_slopes, n_cmd, mask, (double*)R, (long long)ld_r);
        else
            tik_apply_kernel<float><<<gd, kThreads, 0, st>>>(G, npad, nt, D, ld, n_slopes, n_cmd, mask, (float*)R, (long long)ld_r);
        e = cudaGetLastError();
    }
    int h_err = 0;
    double h_lam = 0.0;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = cudaMemcpy(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&h_lam, d_lam, sizeof(double), cudaMemcpyDeviceToHost);
    cleanup();
    if (e != cudaSuccess) return report(err, err_len, MCAO_E_CUDA, "Tikhonov reconstructor: %s", cudaGetErrorString(e));
    if (lambda) *lambda = h_lam;
    if (h_err)
        return report(err, err_len, MCAO_E_UNSUPPORTED,
                      "D^T D + lambda I is not positive definite in double precision (lambda = %g): raise alpha", h_lam);
    return MCAO_OK;
}
