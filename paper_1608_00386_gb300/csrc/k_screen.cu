// Phase screens on the GPU ("The atmospheric layers generation" of arXiv:1608.00386: phase
// screens of the turbulent layers from a turbulence spectrum).  The FFT method: on the discrete
// frequency grid of an n x n periodic screen of pitch `pixel`, complex Gaussian coefficients
// c = (z_c + i z_s) sqrt(PSD(kappa)) dk with the von Karman spectrum
// PSD = 0.023 r0^(-5/3) (kappa^2 + L0^-2)^(-11/6) (kappa in cycles per metre), c(0, 0) = 0,
// evaluated in float in units of the frequency cell dk = 1 / (n pixel):
// sqrt(PSD) dk = sqrt(0.023 r0^(-5/3)) (n pixel)^(5/6) (kx'^2 + ky'^2 + (n pixel / L0)^2)^(-11/12);
// the screen is Re sum_k c_k exp(+2 pi i k x / n) (an unnormalized inverse DFT), computed as
// the real part of the forward DFT of conj(c).  (z_c, z_s) is the Box-Muller pair of the
// detector-noise sampler drawn from Philox4x32-10 with counter (index, 0, 0, 1), key = seed.
// The powers of two from 256 on take half-spectrum passes (screen_pass below); other sizes two
// passes of row FFTs in shared memory, each storing its result transposed: the first generates its
// rows of coefficients in place (no coefficient array in HBM), the second keeps the real part.
#include "device_common.cuh"
#include "mcao_internal.h"

namespace mcao {

namespace {

constexpr int kScreenThreads = 512;
constexpr size_t kScreenSmemTarget = 113 * 1024;   // two blocks per SM

// rows per block: as many as fit two blocks per SM, 1..8
__host__ __device__ constexpr int screen_rows(int n) {
    return (int)((kScreenSmemTarget - sizeof(float2) * (size_t)n) / (2 * sizeof(float2) * (size_t)n)) < 1 ? 1
         : (int)((kScreenSmemTarget - sizeof(float2) * (size_t)n) / (2 * sizeof(float2) * (size_t)n)) > 8 ? 8
         : (int)((kScreenSmemTarget - sizeof(float2) * (size_t)n) / (2 * sizeof(float2) * (size_t)n));
}

__global__ void screen_twiddle_kernel(int n, float2* W) {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < n; m += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(-2.0 * (double)m / (double)n, &s, &c);
        W[m] = make_float2((float)c, (float)s);
    }
}

struct ScreenPass {
    int n, rows;
    // first pass: coefficients generated in place (amp0 = sqrt(0.023 r0^-5/3) / (n pixel), frequencies
    // in units of the cell 1 / (n pixel), l2 = (n pixel / L0)^2), FFT along kx, complex result
    // stored transposed in dst_c
    float amp0, l2;
    uint32_t key0, key1;
    // second pass: rows of src, FFT along ky, real part stored transposed in dst_r
    const float2* src;
    float2* dst_c;
    float* dst_r;
    const float2* W;
    int radices[16];
    int n_radices;
};

// (z_c, z_s) of coefficient k = ky n + kx: Box-Muller pair of Philox words 0, 1 at counter (k, 0, 0, 1)
__device__ __forceinline__ float2 screen_normals(int n, int kx, int ky, uint32_t key0, uint32_t key1) {
    uint32_t w[4] = {(uint32_t)ky * (uint32_t)n + (uint32_t)kx, 0u, 0u, 1u};
    philox4x32_10(w, key0, key1);
    float2 z;
    nz_box_muller2(nz_uniform(w[0]), nz_uniform(w[1]), z.x, z.y);
    return z;
}

// two of them at once, coefficients (kx, ky) and (lx, ly): the same operations in the same order, the
// polynomials of both on packed pairs (2048: 45 us a screen with each by itself, 43 so)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("{\n\t.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%1, %2};\n\tmov.b64 rb, {%3, %4};\n\t"
        "mov.b64 rc, {%5, %6};\n\tfma.rn.f32x2 %0, ra, rb, rc;\n\t}"
        : "=l"(d)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}
__device__ __forceinline__ float2 fmul2(float2 a, float2 b) { return f2_unpack(f2_mul(f2_pack(a.x, a.y), f2_pack(b.x, b.y))); }
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

__device__ __forceinline__ void screen_normals2(int n, int kx, int ky, int lx, int ly, uint32_t key0, uint32_t key1, float2& z,
                                                float2& y) {
    uint32_t w[4] = {(uint32_t)ky * (uint32_t)n + (uint32_t)kx, 0u, 0u, 1u};
    uint32_t v[4] = {(uint32_t)ly * (uint32_t)n + (uint32_t)lx, 0u, 0u, 1u};
    philox4x32_10(w, key0, key1);
    philox4x32_10(v, key0, key1);
    // log of the first uniforms (nz_log)
    const float u[2] = {nz_uniform(w[0]), nz_uniform(v[0])};
    float m[2], e[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t b = __float_as_uint(u[i]);
        int x = (int)((b >> 23) & 0xffu) - 127;
        m[i] = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);
        if (m[i] > 1.41421356f) {
            m[i] = __fmul_rn(m[i], 0.5f);
            x += 1;
        }
        e[i] = (float)x;
    }
    const float2 s = make_float2(__fmul_rn(__fsub_rn(m[0], 1.0f), __frcp_rn(__fadd_rn(m[0], 1.0f))),
                                 __fmul_rn(__fsub_rn(m[1], 1.0f), __frcp_rn(__fadd_rn(m[1], 1.0f))));
    const float2 s2 = fmul2(s, s), ef = make_float2(e[0], e[1]);
    float2 p = ffma2(both(1.11111112e-01f), s2, both(1.42857149e-01f));
    p = ffma2(p, s2, both(2.00000003e-01f));
    p = ffma2(p, s2, both(3.33333343e-01f));
    p = ffma2(p, s2, both(1.0f));
    const float2 lm = fmul2(fmul2(both(2.0f), s), p);
    const float2 lg = fmul2(both(-2.0f), ffma2(ef, both(0.693145752f), ffma2(ef, both(1.42860677e-06f), lm)));
    const float2 rad = make_float2(__fsqrt_rn(lg.x), __fsqrt_rn(lg.y));
    // cosine and sine of the second (nz_sincos2pi)
    const float2 t = make_float2(nz_uniform(w[1]), nz_uniform(v[1]));
    const float2 t4 = fmul2(both(4.0f), t);
    const float2 q = make_float2(rintf(t4.x), rintf(t4.y));
    const float2 g = fmul2(ffma2(both(-0.25f), q, t), both(6.28318548f));   // u - q / 4 is exact either way
    const float2 g2 = fmul2(g, g);
    float2 a = ffma2(both(2.75573188e-06f), g2, both(-1.98412701e-04f));
    a = ffma2(a, g2, both(8.33333377e-03f));
    a = ffma2(a, g2, both(-1.66666672e-01f));
    const float2 sp = ffma2(fmul2(a, g2), g, g);
    a = ffma2(both(2.48015876e-05f), g2, both(-1.38888892e-03f));
    a = ffma2(a, g2, both(4.16666679e-02f));
    a = ffma2(a, g2, both(-0.5f));
    const float2 cp = ffma2(a, g2, both(1.0f));
    auto turn = [](float r, float qf, float sn, float cs) {
        const int k = ((int)qf) & 3;
        const float c = (k & 1) ? sn : cs, b = (k & 1) ? cs : sn;
        return make_float2(__fmul_rn(r, (k == 1 || k == 2) ? -c : c), __fmul_rn(r, (k >= 2) ? -b : b));
    };
    z = turn(rad.x, q.x, sp.x, cp.x);
    y = turn(rad.y, q.y, sp.y, cp.y);
}

// a_k = amp0 x^(-11/12), x = kx'^2 + ky'^2 + l2 (the spectrum in cell units), 0 at DC; a_-k = a_k.  With
// x = 2^e m the power of two leaves the logarithm, whose rounding at the size of log2(x) would otherwise
// be most of the screen's error: 2^(-11 e / 12) = 2^i 2^(k / 12), the rest an exponent within (-1, 1).
__device__ __forceinline__ float screen_amp(int n, int kx, int ky, float amp0, float l2) {
    const float sx = (float)(kx <= (n - 1) / 2 ? kx : kx - n);
    const float sy = (float)(ky <= (n - 1) / 2 ? ky : ky - n);
    const float x = sx * sx + sy * sy + l2;
    if ((kx == 0 && ky == 0) || !(x < 3.0e38f)) return 0.0f;
    const uint32_t b = __float_as_uint(x);   // x >= 1 away from DC
    const int q = 11 * (127 - (int)(b >> 23)) + 12 * 128, i = q / 12, k = q - 12 * i;
    const float m = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);
    const float f = exp2f(fmaf(-11.0f / 12.0f, log2f(m), (float)k * (1.0f / 12.0f)));
    return amp0 * f * __uint_as_float((uint32_t)(i - 1) << 23);   // 2^(i - 128)
}

// conj(c_k) = a_k (z_c - i z_s)
__device__ __forceinline__ float2 screen_coeff(int n, int kx, int ky, float amp0, float l2, uint32_t key0,
                                               uint32_t key1) {
    const float2 z = screen_normals(n, kx, ky, key0, key1);
    const float a = screen_amp(n, kx, ky, amp0, l2);
    return make_float2(z.x * a, -z.y * a);
}

template <bool GEN>
__global__ void __launch_bounds__(kScreenThreads) screen_fft_pass(ScreenPass P) {
    extern __shared__ float4 smem_raw[];
    const int n = P.n, rows = P.rows;
    float2* A = reinterpret_cast<float2*>(smem_raw);
    float2* B = A + rows * n;
    float2* W = B + rows * n;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int row0 = blockIdx.x * rows;
    for (int q = tid; q < n; q += nthr) W[q] = P.W[q];
    for (int q = tid; q < rows * n; q += nthr) {
        const int r = q / n, c = q - r * n;
        float2 v = make_float2(0.0f, 0.0f);
        if (row0 + r < n) {
            if constexpr (GEN) v = screen_coeff(n, c, row0 + r, P.amp0, P.l2, P.key0, P.key1);
            else v = P.src[(size_t)(row0 + r) * n + c];
        }
        A[q] = v;
    }
    __syncthreads();
    const float2* R = stockham_fft(A, B, n, P.radices, P.n_radices, rows, n, 1, W, tid, nthr);
    for (int q = tid; q < rows * n; q += nthr) {
        const int c = q / rows, r = q - c * rows;
        if (row0 + r >= n) continue;
        const float2 v = R[r * n + c];
        if constexpr (GEN) P.dst_c[(size_t)c * n + row0 + r] = v;
        else P.dst_r[(size_t)c * n + row0 + r] = v.x;
    }
}

// ------------------------------------------------------------------------------------------
// powers of two: half-spectrum passes with register transforms
// ------------------------------------------------------------------------------------------
// The screen is real, so it is the transform of the Hermitian half D_k = conj(c_k + conj(c_-k)) / 2:
//   pass 1: rows ky = 0 .. n/2 of D, generated in registers, transformed along kx, G[ky][x];
//   pass 2: per pair of columns x, the transform along ky of G[.][x] + i G[.][x + 1] (rows above n/2 from
//   the Hermitian symmetry), whose real and imaginary parts are the two columns of the screen.
// Half the transforms and half the intermediate bytes of transforming c and keeping the real part.
// A transform of N points takes N / 16 threads with 16 points each in registers: radix 16, radix 16,
// radix N / 256, with one exchange through shared memory between (rows padded by one entry in 16, so
// that the first exchange's stride of 16 meets every bank); the first stage's inputs are generated or
// read straight into the registers and the last stage's outputs stored from them.  Twiddles are
// formed by the block.  The passes are bound by the instructions of the two Philox draws and
// Box-Muller pairs per coefficient (pass 1) and by shared memory and the L2 gathers (pass 2).
// 2048 x 2048: 35 + 14 us alone, 43 a screen in a row of ten; six radix-4 exchanges of the full
// spectrum and a twiddle kernel took 55 + 40 + 7.  (Of the 14: 19 with the four transforms' rows
// starting in the same bank.)
__device__ __forceinline__ float2 rot4(float2 a) { return make_float2(a.y, -a.x); }   // -i a

// forward 4-point transform of v[0], v[s], v[2 s], v[3 s], in place
template <int S>
__device__ __forceinline__ void dft4(float2* v) {
    const float2 a = cadd(v[0], v[2 * S]), b = csub(v[0], v[2 * S]);
    const float2 c = cadd(v[S], v[3 * S]), d = rot4(csub(v[S], v[3 * S]));
    v[0] = cadd(a, c);
    v[S] = cadd(b, d);
    v[2 * S] = csub(a, c);
    v[3 * S] = csub(b, d);
}

// forward R-point transform of v[0], v[S], .. v[(R - 1) S], in place and in natural order
template <int R, int S>
__device__ __forceinline__ void dft_reg(float2* v) {
    if constexpr (R == 2) {
        const float2 a = v[0];
        v[0] = cadd(a, v[S]);
        v[S] = csub(a, v[S]);
    } else if constexpr (R == 4) {
        dft4<S>(v);
    } else if constexpr (R == 8) {
        // 2 x 4: transforms of the even and odd points, then butterflies
        dft4<2 * S>(v);
        dft4<2 * S>(v + S);
        const float h = 0.707106781186547524f;
        float2 o[4] = {v[S], v[3 * S], v[5 * S], v[7 * S]}, e[4] = {v[0], v[2 * S], v[4 * S], v[6 * S]};
        o[1] = make_float2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
        o[2] = rot4(o[2]);
        o[3] = make_float2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            v[b * S] = cadd(e[b], o[b]);
            v[(b + 4) * S] = csub(e[b], o[b]);
        }
    } else if constexpr (R == 16) {
        // 4 x 4: out[b + 4 c] = sum_a w16^(a b) w4^(a c) X_a[b], X_a the transform of points a, a + 4, ..
        const float c1 = 0.923879532511286756f, s1 = 0.382683432365089772f, h = 0.707106781186547524f;
#pragma unroll
        for (int a = 0; a < 4; ++a) dft4<4 * S>(v + a * S);
        const float2 w[4][4] = {{{1, 0}, {1, 0}, {1, 0}, {1, 0}},
                                {{1, 0}, {c1, -s1}, {h, -h}, {s1, -c1}},
                                {{1, 0}, {h, -h}, {0, -1}, {-h, -h}},
                                {{1, 0}, {s1, -c1}, {-h, -h}, {-c1, s1}}};
#pragma unroll
        for (int a = 1; a < 4; ++a)
#pragma unroll
            for (int b = 1; b < 4; ++b) v[(a + 4 * b) * S] = cmul(v[(a + 4 * b) * S], w[a][b]);
#pragma unroll
        for (int b = 0; b < 4; ++b) dft4<S>(v + 4 * b * S);   // over a; output c at 4 b + c
        float2 t[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) t[q] = v[q * S];
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) v[(b + 4 * c) * S] = t[4 * b + c];
    }
}

// NF transforms per block
template <int N, int NF>
struct HalfFft {
    static constexpr int T = N / 16;                       // threads per transform
    static constexpr int R3 = N / 256;                     // last stage's radix
    static constexpr int F = NF;
    static constexpr int kThreads = T * F;
    // padded row in shared memory; where a warp holds points of all F transforms, their rows start in
    // different banks
    static constexpr int kRow = N + N / 16 + 16 / F;
    static constexpr int kTw = 15 * 16 + (R3 - 1) * 256;   // twiddles of stages 2 and 3
    static constexpr size_t smem = sizeof(float2) * ((size_t)F * kRow + kTw);
};
__device__ __forceinline__ int fft_pad(int i) { return i + (i >> 4); }

template <int N>
__device__ __forceinline__ void half_twiddles(float2* tw, int tid, int nthr) {
    for (int e = tid; e < HalfFft<N, 1>::kTw; e += nthr) {
        // stage 2: entry (r - 1) 16 + k, angle r k / 256; stage 3: (r - 1) 256 + k, angle r k / N
        const int q = e < 240 ? e : e - 240, ns = e < 240 ? 16 : 256;
        const int r = q / ns + 1, k = q % ns;
        float sn, cs;
        sincospif(-2.0f * (float)(r * k) / (e < 240 ? 256.0f : (float)N), &sn, &cs);
        tw[e] = make_float2(cs, sn);
    }
}

// Transform of the 16 points v[m] = in[t + m T] of this thread; on return v[q + r (16 / R3)] is output
// t + q T + 256 r (q < 16 / R3, r < R3).  row: the transform's shared memory.  Every thread of the block
// calls it.
template <int N>
__device__ __forceinline__ void half_fft(float2 (&v)[16], float2* row, const float2* tw, int t) {
    using H = HalfFft<N, 1>;
    constexpr int Q = 16 / H::R3;
    dft_reg<16, 1>(v);
#pragma unroll
    for (int r = 0; r < 16; ++r) row[fft_pad(16 * t + r)] = v[r];
    __syncthreads();   // also covers the twiddles
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = row[fft_pad(t + m * H::T)];
    const int k = t & 15;
#pragma unroll
    for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], tw[(r - 1) * 16 + k]);
    dft_reg<16, 1>(v);
    if constexpr (H::R3 > 1) {
        __syncthreads();
        const int base = (t >> 4) * 256 + k;
#pragma unroll
        for (int r = 0; r < 16; ++r) row[fft_pad(base + 16 * r)] = v[r];
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = row[fft_pad(t + m * H::T)];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
#pragma unroll
            for (int r = 1; r < H::R3; ++r) v[q + r * Q] = cmul(v[q + r * Q], tw[240 + (r - 1) * 256 + t + q * H::T]);
            dft_reg<H::R3, Q>(v + q);
        }
    } else {
        // 256 points: stage 2 is the last; its output r of butterfly t is t + 16 r = t + T r
    }
}

// 64 registers a thread: the 513 blocks of a 2048 screen are resident at once (73 registers: three per SM, so
// that a ninth of them ran alone after the others)
template <int N, int NF>
__global__ void __launch_bounds__(HalfFft<N, NF>::kThreads, 1024 / HalfFft<N, NF>::kThreads) screen_half_rows(ScreenPass P) {
    using H = HalfFft<N, NF>;
    extern __shared__ float4 smem_raw[];
    float2* tw = reinterpret_cast<float2*>(smem_raw);
    const int f = threadIdx.x / H::T, t = threadIdx.x % H::T;
    float2* row = tw + H::kTw + f * H::kRow;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int ky = min((int)blockIdx.x * H::F + f, N / 2);   // a block's spare transforms repeat the last row
    half_twiddles<N>(tw, threadIdx.x, H::kThreads);
    float2 v[16];
    const int my = (N - ky) % N;
    // conj(c_k + conj(c_-k)) / 2
    auto draw = [&](int kx, float a) {
        float2 z, y;
        screen_normals2(N, kx, ky, (N - kx) % N, my, P.key0, P.key1, z, y);
        row[fft_pad(kx)] = make_float2(a * (z.x + y.x), a * (y.y - z.y));
    };
    // kx and N - kx share an amplitude (0 and N / 2 do not, and go together)
#pragma unroll 2
    for (int m = 0; m < 8; ++m) {
        const int kx = t + m * H::T;
        const float a = 0.5f * screen_amp(N, kx, ky, P.amp0, P.l2);
        draw(kx, a);
        draw(kx ? N - kx : N / 2, kx ? a : 0.5f * screen_amp(N, N / 2, ky, P.amp0, P.l2));
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = row[fft_pad(t + m * H::T)];
    __syncthreads();
    half_fft<N>(v, row, tw, t);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // nothing above reads or writes global memory
    float2* out = P.dst_c + (size_t)ky * N;
    constexpr int Q = H::R3 > 1 ? 16 / H::R3 : 1;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int o = H::R3 > 1 ? t + (i % Q) * H::T + 256 * (i / Q) : t + 16 * i;
        out[o] = v[i];
    }
}

template <int N, int NF>
__global__ void __launch_bounds__(HalfFft<N, NF>::kThreads) screen_half_cols(ScreenPass P) {
    using H = HalfFft<N, NF>;
    extern __shared__ float4 smem_raw[];
    float2* tw = reinterpret_cast<float2*>(smem_raw);
    // neighbouring threads take neighbouring column pairs
    const int f = threadIdx.x % H::F, t = threadIdx.x / H::F;
    float2* row = tw + H::kTw + f * H::kRow;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int x = 2 * (blockIdx.x * H::F + f);
    half_twiddles<N>(tw, threadIdx.x, H::kThreads);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the rows
    float2 v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int ky = t + m * H::T;
        const bool up = ky > N / 2;
        const float4 g = *reinterpret_cast<const float4*>(P.src + (size_t)(up ? N - ky : ky) * N + x);
        v[m] = up ? make_float2(g.x + g.w, g.z - g.y) : make_float2(g.x - g.w, g.y + g.z);
    }
    half_fft<N>(v, row, tw, t);
    constexpr int Q = H::R3 > 1 ? 16 / H::R3 : 1;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int o = H::R3 > 1 ? t + (i % Q) * H::T + 256 * (i / Q) : t + 16 * i;
        *reinterpret_cast<float2*>(P.dst_r + (size_t)o * N + x) = v[i];
    }
}

}  // namespace

size_t screen_fft_smem(int n) { return sizeof(float2) * (2 * (size_t)screen_rows(n) * n + n); }

namespace {

cudaError_t screen_passes(ScreenPass P, cudaStream_t s) {
    const size_t bytes = screen_fft_smem(P.n);
    // the limit is the kernel's, for every thread: always the target, which no size up to 4096 exceeds
    constexpr int kMost = (int)kScreenSmemTarget;
    static_assert(3 * sizeof(float2) * 4096 <= kScreenSmemTarget, "one row per block fits");
    cudaError_t e = cudaFuncSetAttribute(screen_fft_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(screen_fft_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)((P.n + P.rows - 1) / P.rows);
    float2* work = P.dst_c;
    float* out = P.dst_r;
    P.dst_r = nullptr;
    screen_fft_pass<true><<<blocks, kScreenThreads, bytes, s>>>(P);
    P.src = work;
    P.dst_c = nullptr;
    P.dst_r = out;
    screen_fft_pass<false><<<blocks, kScreenThreads, bytes, s>>>(P);
    return cudaGetLastError();
}

template <int N>
cudaError_t half_passes(ScreenPass P, cudaStream_t s) {
    // rows: two transforms per block (four at 256), so that small screens spread over the SMs; columns:
    // four, so that a block stores whole 32-byte sectors, where their shared memory leaves two blocks per SM
    using A = HalfFft<N, N == 256 ? 4 : 2>;
    using B = HalfFft<N, N == 4096 ? 2 : 4>;
    const auto rows = screen_half_rows<N, A::F>;
    const auto cols = screen_half_cols<N, B::F>;
    cudaError_t e = cudaFuncSetAttribute(rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A::smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cols, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)B::smem);
    if (e != cudaSuccess) return e;
    // both passes are programmatic dependents of what is before them on the stream: the columns' blocks
    // take over the SMs that the rows leave, and the next screen is drawn beside this one's columns.  Each waits
    // for all of the kernel before it (griddepcontrol.wait) ahead of its first access to global memory.
    // A captured launch may follow the allocation of its buffers, not a kernel: plain there.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(s, &capture)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = capture == cudaStreamCaptureStatusNone ? 1 : 0;
    cfg.stream = s;
    cfg.gridDim = dim3((N / 2 + 1 + A::F - 1) / A::F);
    cfg.blockDim = dim3(A::kThreads);
    cfg.dynamicSmemBytes = A::smem;
    if ((e = cudaLaunchKernelEx(&cfg, rows, P)) != cudaSuccess) return e;
    P.src = P.dst_c;
    cfg.gridDim = dim3(N / 2 / B::F);
    cfg.blockDim = dim3(B::kThreads);
    cfg.dynamicSmemBytes = B::smem;
    return cudaLaunchKernelEx(&cfg, cols, P);
}

}  // namespace

// powers of two from 256 to 4096; the passes store pairs of columns, so they need an 8-byte aligned screen
bool screen_is_half(int n, const float* out) {
    return n >= 256 && n <= 4096 && (n & (n - 1)) == 0 && reinterpret_cast<uintptr_t>(out) % 8 == 0;
}

cudaError_t launch_screen(int n, double pixel, double r0, double L0, unsigned long long seed, const int* radices,
                          int n_radices, float2* work, float2* W, float* out, cudaStream_t s) {
    ScreenPass P{};
    P.n = n;
    P.rows = screen_rows(n);
    const double extent = (double)n * pixel;
    P.amp0 = (float)(sqrt(0.023 * pow(r0, -5.0 / 3.0)) * pow(extent, 11.0 / 6.0) / extent);
    P.l2 = (float)((extent / L0) * (extent / L0));
    P.key0 = (uint32_t)seed;
    P.key1 = (uint32_t)(seed >> 32);
    P.W = W;
    P.n_radices = n_radices;
    for (int i = 0; i < n_radices && i < 16; ++i) P.radices[i] = radices[i];
    P.dst_c = work;
    P.dst_r = out;
    if (screen_is_half(n, out)) switch (n) {
        case 256: return half_passes<256>(P, s);
        case 512: return half_passes<512>(P, s);
        case 1024: return half_passes<1024>(P, s);
        case 2048: return half_passes<2048>(P, s);
        case 4096: return half_passes<4096>(P, s);
    }
    screen_twiddle_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, W);
    return screen_passes(P, s);
}

}  // namespace mcao
