// Noise-free centre of gravity of a Shack-Hartmann spot, and its derivative with respect to the
// residual phase, straight from the lags of the field ("The closed loop": X and Y slopes of the
// residual phase; "The calibration of the interaction matrices": their response to each command).
//
// The detector image is B[m] = sum_u ACF(u) OTF(u) h(ux) h(uy) exp(2 pi i u.m / n_det) (k_wfs.cu),
// ACF(u) = sum_x E(x) conj(E(x + u)), h the factor of the shift by N/2 and of the binning.  Summed
// over the rows m_y, exp(2 pi i uy m_y / n_det) leaves only the lags uy = 0 mod n_det, and h is
// zero at every such lag but 0.  So the x slope needs the lags (ux, 0) alone, the y slope (0, uy):
//   s_x = sum_u ACF(u, 0) K(u) / ACF(0, 0),   K(u) = OTF(u, 0) h(u) D(u) / (b n_det),
//   D(u) = sum_m (m - c) exp(2 pi i u m / n_det)   (K Hermitian, K(0) = 0),
// and with C(x) = sum_b K(b - x) conj(E(b, y)) along the sample's row, z = E C:
//   s_x = sum Re z / sum |E|^2,   d s_x / d phi = -2 scale Im z / sum |E|^2
// (sum |E|^2 does not depend on the phase).  No spectrum, image or adjoint image is formed: n_px
// complex multiply-adds per sample and slope instead of 3 to 7 two-dimensional FFTs of the padded
// field.  Photon or read noise and kept frames need the image: those steps stay on k_wfs.cu.
// (39 m interaction matrix: 6 x 1.10 ms of FFTs before, 0.09 ms for all six sensors now; the wide-field sensors'
// noise-free slopes, 3504 subapertures of 16 samples: 420 us before, 30 us now.)
//
// What is left is bound by the gathers of the grids (one layer or DM is four loads per sample).
// Groups of threads per subaperture: one warp at 8 samples per side (8 subapertures per block, only
// warp barriers), 128 threads at 16, 1024 at 32 (these sensors have a few subapertures, so their
// time is one block's latency).
#include "device_common.cuh"
#include "mcao_internal.h"

namespace mcao {

namespace {

constexpr float kPi = 3.14159265358979323846f;

template <int NPX>
struct LagShape {
    static constexpr int G = NPX == 8 ? 32 : NPX == 16 ? 128 : 1024;   // threads per subaperture
    static constexpr int NG = NPX == 8 ? 8 : 1;                        // subapertures per block
    static constexpr int PPT = NPX * NPX / G;                          // samples per thread
};

struct LagGrid {
    const float* data;
    int n;
    float sign;
};

template <int NPX>
__device__ __forceinline__ void group_sync() {
    if constexpr (NPX == 8) __syncwarp();
    else __syncthreads();
}

// sums of three values over the group, in every thread
template <int NPX>
__device__ __forceinline__ void group_sum3(float (&v)[3], float (*red)[3], int t) {
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = warp_sum(v[i]);
    if constexpr (NPX != 8) {
        constexpr int NW = LagShape<NPX>::G / 32;
        if ((t & 31) == 0)
#pragma unroll
            for (int i = 0; i < 3; ++i) red[t >> 5][i] = v[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            v[i] = 0.0f;
            for (int q = 0; q < NW; ++q) v[i] += red[q][i];
        }
    }
}

// SENS: d slope / d phase rows into sens; otherwise the slopes
template <int NPX, bool SENS>
__global__ void __launch_bounds__(LagShape<NPX>::G* LagShape<NPX>::NG) wfs_lag_kernel(WfsLaunch L, int real0, float* sens) {
    using S = LagShape<NPX>;
    __shared__ AxisEnt s_e[S::NG][2][kMaxEntries * NPX];
    __shared__ LagGrid s_g[S::NG][kMaxEntries];
    __shared__ float2 s_E[S::NG][NPX * NPX];
    __shared__ float2 s_K[S::NG][2][2 * NPX - 1];
    __shared__ float s_red[S::G / 32][3];
    const int grp = NPX == 8 ? threadIdx.x >> 5 : 0, t = NPX == 8 ? threadIdx.x & 31 : threadIdx.x;
    const int sub = blockIdx.x * S::NG + grp;
    if (sub >= L.n_subaps) return;   // a whole warp at 8 samples; never at 16 and 32
    const int real = real0 + blockIdx.y;
    const SubapDev sd = L.subaps[sub];
    const WfsDev& w = L.ctx.wfs[sd.wfs];
    const int i0 = sd.sx * NPX, j0 = sd.sy * NPX;
    const int n_grids = L.ctx.n_grids;
    const GridView* V = L.ctx.views + real * L.ctx.view_stride + (long long)sd.wfs * n_grids;
    tile_entries<NPX>(V, n_grids, L.ctx.st->k, i0, j0, s_e[grp][0], s_e[grp][1], t, S::G);
    if (t < n_grids) s_g[grp][t] = LagGrid{V[t].data, V[t].n, V[t].sign};
    for (int q = t; q < 2 * (2 * NPX - 1); q += S::G) {
        const int axis = q / (2 * NPX - 1), u = q - axis * (2 * NPX - 1);
        float2 k = w.kap[u];
        if (sd.elong_a > 0.0f) {
            const float d = (float)(u - (NPX - 1)) * (axis ? sd.dir_y : sd.dir_x);
            const float o = expf(-sd.elong_a * d * d);
            k.x *= o;
            k.y *= o;
        }
        s_K[grp][axis][u] = k;
    }
    group_sync<NPX>();

    // field E = A exp(i (scale phi - pi (x + y) / N)) of the thread's samples
    float phi[S::PPT];
    float2 E[S::PPT];
#pragma unroll
    for (int i = 0; i < S::PPT; ++i) phi[i] = 0.0f;
#pragma unroll 2
    for (int g = 0; g < n_grids; ++g) {
        const LagGrid gm = s_g[grp][g];
#pragma unroll
        for (int i = 0; i < S::PPT; ++i) {
            const int q = t + i * S::G;
            phi[i] = fmaf(gm.sign, bilinear(gm.data, gm.n, s_e[grp][0][g * NPX + q % NPX], s_e[grp][1][g * NPX + q / NPX]), phi[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < S::PPT; ++i) {
        const int q = t + i * S::G, x = q % NPX, y = q / NPX;
        const float a = __ldg(w.amp + (long long)(j0 + y) * w.N + i0 + x);
        float sn, cs;
        sincosf(w.scale * phi[i] - kPi * (float)(x + y) / (float)w.n_fft, &sn, &cs);
        E[i] = make_float2(a * cs, a * sn);
        s_E[grp][q] = E[i];
    }
    group_sync<NPX>();

    // C along the sample's row (x slope) and column (y slope)
    float2 cx[S::PPT], cy[S::PPT];
#pragma unroll
    for (int i = 0; i < S::PPT; ++i) cx[i] = cy[i] = make_float2(0.0f, 0.0f);
    auto add = [](float2& c, float2 k, float2 e) {   // c += k conj(e)
        c.x = fmaf(k.x, e.x, fmaf(k.y, e.y, c.x));
        c.y = fmaf(k.y, e.x, fmaf(-k.x, e.y, c.y));
    };
#pragma unroll 8
    for (int b = 0; b < NPX; ++b)
#pragma unroll
        for (int i = 0; i < S::PPT; ++i) {
            const int q = t + i * S::G, x = q % NPX, y = q / NPX;
            add(cx[i], s_K[grp][0][b - x + NPX - 1], s_E[grp][y * NPX + b]);
            add(cy[i], s_K[grp][1][b - y + NPX - 1], s_E[grp][b * NPX + x]);
        }
    float v[3] = {0.0f, 0.0f, 0.0f};   // sum |E|^2, sum Re z_x, sum Re z_y
#pragma unroll
    for (int i = 0; i < S::PPT; ++i) {
        v[0] = fmaf(E[i].x, E[i].x, fmaf(E[i].y, E[i].y, v[0]));
        v[1] = fmaf(E[i].x, cx[i].x, fmaf(-E[i].y, cx[i].y, v[1]));
        v[2] = fmaf(E[i].x, cy[i].x, fmaf(-E[i].y, cy[i].y, v[2]));
    }
    group_sum3<NPX>(v, s_red, t);
    // without light no derivatives; a NaN phase gives NaN
    const float inv = v[0] != 0.0f ? 1.0f / v[0] : 0.0f;
    if constexpr (SENS) {
        float* rx = sens + w.sens0 + (long long)sd.rank * (NPX * NPX);
        float* ry = rx + (long long)w.n_valid * (NPX * NPX);
        const float f = -2.0f * w.scale * inv;
#pragma unroll
        for (int i = 0; i < S::PPT; ++i) {
            const int q = t + i * S::G;
            rx[q] = v[0] != 0.0f ? f * fmaf(E[i].x, cx[i].y, E[i].y * cx[i].x) : 0.0f;
            ry[q] = v[0] != 0.0f ? f * fmaf(E[i].x, cy[i].y, E[i].y * cy[i].x) : 0.0f;
        }
    } else if (t == 0) {
        const int ix = w.slope0 + sd.rank, iy = ix + w.n_valid;
        const bool live = v[0] > 0.0f && w.n_photons * sd.frac > 0.0f;   // a dark frame has no slopes
        const float gx = live ? v[1] * inv : 0.0f, gy = live ? v[2] * inv : 0.0f;
        const float vx = gx - (L.s_ref ? L.s_ref[ix] : 0.0f), vy = gy - (L.s_ref ? L.s_ref[iy] : 0.0f);
        float* slopes = L.slopes + (long long)real * L.slope_stride;
        slopes[ix] = vx;
        slopes[iy] = vy;
        if (L.slopes_pad) {
            float* pad = L.slopes_pad + (long long)real * L.pad_stride;
            pad[w.rcol0 + sd.rank] = vx;
            pad[w.rcol0 + w.n_valid + sd.rank] = vy;
        }
    }
}

template <int NPX, bool SENS>
cudaError_t launch(const WfsLaunch& L, int real0, int n_real, float* sens, cudaStream_t s) {
    using S = LagShape<NPX>;
    const unsigned blocks = (unsigned)((L.n_subaps + S::NG - 1) / S::NG);
    if (blocks) wfs_lag_kernel<NPX, SENS><<<dim3(blocks, (unsigned)n_real), S::G * S::NG, 0, s>>>(L, real0, sens);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_wfs_lag(const WfsLaunch& L, int n_px, cudaStream_t s) {
    switch (n_px) {
        case 8: return launch<8, false>(L, 0, L.ctx.n_real, nullptr, s);
        case 16: return launch<16, false>(L, 0, L.ctx.n_real, nullptr, s);
        case 32: return launch<32, false>(L, 0, L.ctx.n_real, nullptr, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sens(const WfsLaunch& L, int n_px, int real, float* sens, cudaStream_t s) {
    switch (n_px) {
        case 8: return launch<8, true>(L, real, 1, sens, s);
        case 16: return launch<16, true>(L, real, 1, sens, s);
        case 32: return launch<32, true>(L, real, 1, sens, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mcao
