// Adjoint of the DM and layer projections: what the derivatives of the slopes with respect to the
// residual phase (k_lag.cu) say about the DM commands, the pupil phase and the screens ("The
// calibration of the interaction matrices": the interaction matrix is the slopes' response to each
// command; here it is the Jacobian at the current state rather than a finite poke).
//
// phi(p) = ... - bilinear(S_m, p) and S_m = Gy C Gx^T, so
//   d phi(p) / d C[b][a] = -((1 - t_x) Gx[i0][a] + t_x Gx[i1][a]) ((1 - t_y) Gy[j0][b] + t_y Gy[j1][b]),
// the same fixed-point sample positions and clamped bilinear weights as the forward; actuators
// outside the union of the forward's per-tile bands (weights below 1e-10) are left out.  A
// rotated DM has no separable tables: its weights are evaluated at each bilinear corner.
//
// The interaction matrix is written row by row, zeros included, by one pass (dm_rows_kernel); the
// product of its transpose with given vectors never forms a row: the pupil-phase gradient of each
// sensor goes through the two separable weight tables (dm_project_x / dm_project_y).
#include <algorithm>

#include "device_common.cuh"
#include "mcao_internal.h"
#include "row_parts.h"

namespace mcao {

namespace {

constexpr int kAdjThreads = 256;
constexpr int kAdjMaxBand = 128;   // actuators per axis acting on one subaperture footprint

// d slope / d phase on the slope's n_px^2 samples (axis 0: x slope, 1: y slope)
__device__ __forceinline__ const float* sens_row(const float* sens, const WfsDev& w, int axis, int rank) {
    return sens + w.sens0 + ((long long)axis * w.n_valid + rank) * (w.n_px * w.n_px);
}

// 1 - t and t of a pupil column / row's two table rows, combined for actuator a
__device__ __forceinline__ float axis_weight(const float* G, int na, AxisEnt e, int a) {
    return (1.0f - e.t) * G[(long long)(e.idx & 0xffff) * na + a] + e.t * G[(long long)(e.idx >> 16) * na + a];
}

// surface samples [x, y] that a run of adjacent pupil samples meets, from its first and last entries:
// they ascend, or descend under a DM above the star (a DM grid does not wrap)
__device__ __forceinline__ int2 footprint(AxisEnt a, AxisEnt b) {
    return make_int2(min(a.idx & 0xffff, b.idx & 0xffff), max(a.idx >> 16, b.idx >> 16));
}

// Actuators [a0, a1) x [b0, b1) of a DM that act on surface samples [cx.x, cx.y] x [cy.x, cy.y]: for a
// separable DM the union of the forward's per-tile bands over the tiles the footprint touches, for a
// rotated one the actuators within rc pitches of the footprint's corners.
__device__ void actuator_range(const DmDesc& dd, const int2* band, int2 cx, int2 cy, int (&rng)[4]) {
    int a0 = dd.nx, a1 = 0, b0 = dd.ny, b1 = 0;
    if (dd.general) {
        const float c0 = 0.5f * (float)(dd.surf_n - 1), ca = 0.5f * (float)(dd.nx - 1), cb = 0.5f * (float)(dd.ny - 1);
        float lo_a = 1e30f, hi_a = -1e30f, lo_b = 1e30f, hi_b = -1e30f;
        for (int c = 0; c < 4; ++c) {
            const float x = ((float)((c & 1) ? cx.y : cx.x) - c0) * dd.dx - dd.shx;
            const float y = ((float)((c & 2) ? cy.y : cy.x) - c0) * dd.dx - dd.shy;
            const float ua = (dd.cr * x + dd.sr * y) * dd.inv_mag / dd.pitch + ca;
            const float ub = (-dd.sr * x + dd.cr * y) * dd.inv_mag / dd.pitch + cb;
            lo_a = fminf(lo_a, ua); hi_a = fmaxf(hi_a, ua);
            lo_b = fminf(lo_b, ub); hi_b = fmaxf(hi_b, ub);
        }
        a0 = max(0, (int)ceilf(lo_a - dd.rc)); a1 = min(dd.nx - 1, (int)floorf(hi_a + dd.rc)) + 1;
        b0 = max(0, (int)ceilf(lo_b - dd.rc)); b1 = min(dd.ny - 1, (int)floorf(hi_b + dd.rc)) + 1;
    } else {
        for (int t = cx.x / kDmTile; t <= cx.y / kDmTile; ++t) {
            const int2 bt = band[dd.tband_x + t];
            if (bt.y > bt.x) { a0 = min(a0, bt.x); a1 = max(a1, bt.y); }
        }
        for (int t = cy.x / kDmTile; t <= cy.y / kDmTile; ++t) {
            const int2 bt = band[dd.tband_y + t];
            if (bt.y > bt.x) { b0 = min(b0, bt.x); b1 = max(b1, bt.y); }
        }
    }
    rng[0] = a0; rng[1] = max(a0, a1); rng[2] = b0; rng[3] = max(b0, b1);
}

// Gauss-Newton terms of a DM misregistration fit, one block per slope row of one sensor, for DM m
// only.  The row of the model matrix D(p) (the exact Jacobian with the DM moved by p = (shift_x,
// shift_y, rotation, magnification)) and its four derivatives dD/dp_i are formed by evaluating
// each actuator's influence function at the four bilinear corners of every pupil sample, in the
// DM's own frame (as the general adjoint does), and differentiating that evaluation:
//   u = R(-theta)(q - shift) / mag  (q a surface grid point, metres),  phi = exp(-|u - x_a|^2 / 2 s^2),
//   d phi / dp = -phi (u - x_a) . du/dp / s^2, with du/d shift_x = (-cos, sin) / mag,
//   du/d shift_y = (-sin, -cos) / mag, du/d theta = (B, -A) / mag, du/d mag = -(A, B) / mag^2
// (A, B the rotated offset before the division).  Against the measured row (columns of DM m) the
// block accumulates in double: cost = sum e^2 (e = D - D_meas), Jte_i = sum dD_i e, the upper
// triangle of JtJ_ij = sum dD_i dD_j, and sum D_meas^2; one record of 16 doubles per row.
__global__ void __launch_bounds__(256) misreg_gn_kernel(ProjLaunch L, int m, const float* __restrict__ D_meas,
                                                        long long ld_meas, int cmd0, double* __restrict__ rec) {
    __shared__ float s_L[kMaxNpx * kMaxNpx];
    __shared__ AxisEnt s_ex[kMaxNpx], s_ey[kMaxNpx];
    __shared__ int s_rng[4];
    __shared__ double s_red[8][16];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int axis = blockIdx.x / L.n_valid, rank = blockIdx.x - axis * L.n_valid;
    const SubapDev sd = L.subaps[rank];
    const WfsDev& w = L.ctx.wfs[sd.wfs];
    const int npx = w.n_px;
    const int row = w.slope0 + axis * w.n_valid + sd.rank;
    const int i0 = sd.sx * npx, j0 = sd.sy * npx;
    const GridView* V = L.ctx.views + L.real * L.ctx.view_stride + (long long)sd.wfs * L.ctx.n_grids;
    const long long k = L.ctx.st->k;
    const float* sens = sens_row(L.sens, w, axis, sd.rank);
    for (int q = tid; q < npx * npx; q += nthr) s_L[q] = sens[q];
    const GridView& v = V[L.n_layers + m];
    const DmDesc dd = L.desc[m];
    if (tid < npx)
        s_ex[tid] = axis_entry(v.ax + (long long)(i0 + tid) * v.bp + k * v.vx, v.n, v.periodic, v.inv_n);
    else if (tid < 2 * npx)
        s_ey[tid - npx] = axis_entry(v.ay + (long long)(j0 + tid - npx) * v.bp + k * v.vy, v.n, v.periodic, v.inv_n);
    __syncthreads();
    const float c0 = 0.5f * (float)(dd.surf_n - 1), ca = 0.5f * (float)(dd.nx - 1), cb = 0.5f * (float)(dd.ny - 1);
    // offset of grid point (i, j) from the shift, rotated: (A, B), metres
    auto rot = [&](int i, int j, float& A, float& B) {
        const float x = ((float)i - c0) * dd.dx - dd.shx, y = ((float)j - c0) * dd.dx - dd.shy;
        A = dd.cr * x + dd.sr * y;
        B = -dd.sr * x + dd.cr * y;
    };
    if (tid == 0) {
        int cx0 = v.n, cx1 = 0, cy0 = v.n, cy1 = 0;
        for (int q = 0; q < npx; ++q) {
            cx0 = min(cx0, s_ex[q].idx & 0xffff);
            cx1 = max(cx1, s_ex[q].idx >> 16);
            cy0 = min(cy0, s_ey[q].idx & 0xffff);
            cy1 = max(cy1, s_ey[q].idx >> 16);
        }
        float lo_a = 1e30f, hi_a = -1e30f, lo_b = 1e30f, hi_b = -1e30f;
        for (int c = 0; c < 4; ++c) {
            float A, B;
            rot((c & 1) ? cx1 : cx0, (c & 2) ? cy1 : cy0, A, B);
            const float ua = A * dd.inv_mag / dd.pitch + ca, ub = B * dd.inv_mag / dd.pitch + cb;
            lo_a = fminf(lo_a, ua); hi_a = fmaxf(hi_a, ua);
            lo_b = fminf(lo_b, ub); hi_b = fmaxf(hi_b, ub);
        }
        int a0 = max(0, (int)ceilf(lo_a - dd.rc)), a1 = min(dd.nx - 1, (int)floorf(hi_a + dd.rc)) + 1;
        int b0 = max(0, (int)ceilf(lo_b - dd.rc)), b1 = min(dd.ny - 1, (int)floorf(hi_b + dd.rc)) + 1;
        if (a1 < a0) a1 = a0;
        if (b1 < b0) b1 = b0;
        s_rng[0] = a0; s_rng[1] = a1; s_rng[2] = b0; s_rng[3] = b1;
    }
    __syncthreads();
    const int a0 = s_rng[0], na = s_rng[1] - s_rng[0], b0 = s_rng[2], nbd = s_rng[3] - s_rng[2];
    const float im = dd.inv_mag, tws = 2.0f * dd.inv2s2;
    double acc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q] = 0.0;
    for (int idx = tid; idx < na * nbd; idx += nthr) {
        const int b = idx / na, a = idx - b * na;
        const int cmd = L.act_map[dd.map_off + (long long)(b0 + b) * dd.nx + a0 + a];
        if (cmd < 0) continue;
        const float xa = ((float)(a0 + a) - ca) * dd.pitch, yb = ((float)(b0 + b) - cb) * dd.pitch;
        float val = 0.0f, g0 = 0.0f, g1 = 0.0f, g2 = 0.0f, g3 = 0.0f;
        for (int y = 0; y < npx; ++y) {
            const AxisEnt ey = s_ey[y];
            const int r0 = ey.idx & 0xffff, r1 = ey.idx >> 16;
            for (int x = 0; x < npx; ++x) {
                const float lv = s_L[y * npx + x];
                if (lv == 0.0f) continue;
                const AxisEnt ex = s_ex[x];
                const int q0 = ex.idx & 0xffff, q1 = ex.idx >> 16;
                for (int c = 0; c < 4; ++c) {
                    const int i = (c & 1) ? q1 : q0, j = (c & 2) ? r1 : r0;
                    const float wl = lv * ((c & 1) ? ex.t : 1.0f - ex.t) * ((c & 2) ? ey.t : 1.0f - ey.t);
                    float A, B;
                    rot(i, j, A, B);
                    const float da = A * im - xa, db = B * im - yb;
                    const float ph = wl * expf(-(da * da + db * db) * dd.inv2s2);
                    val += ph;
                    const float gg = -tws * ph;   // d/dp of exp(-r^2 / 2 s^2) = -(r . dr/dp) / s^2 exp(..)
                    g0 = fmaf(gg, (-da * dd.cr + db * dd.sr) * im, g0);
                    g1 = fmaf(gg, (-da * dd.sr - db * dd.cr) * im, g1);
                    g2 = fmaf(gg, (da * B - db * A) * im, g2);
                    g3 = fmaf(gg, -(da * A + db * B) * im * im, g3);
                }
            }
        }
        const double dv = (double)(v.sign * val);
        const double d[4] = {(double)(v.sign * g0), (double)(v.sign * g1), (double)(v.sign * g2),
                             (double)(v.sign * g3)};
        const double meas = (double)D_meas[(long long)row * ld_meas + (cmd - cmd0)];
        const double e = dv - meas;
        acc[0] += e * e;
        acc[15] += meas * meas;
        int t = 5;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            acc[1 + p] += d[p] * e;
#pragma unroll
            for (int q = p; q < 4; ++q) acc[t++] += d[p] * d[q];
        }
    }
    // block sum in a fixed order: warp shuffles, then warp 0 over the warps
#pragma unroll
    for (int q = 0; q < 16; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    const int lane = tid & 31, warp = tid >> 5;
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 16; ++q) s_red[warp][q] = acc[q];
    __syncthreads();
    if (tid < 16) {
        double sum = 0.0;
        for (int wv = 0; wv < (nthr >> 5); ++wv) sum += s_red[wv][tid];
        rec[(long long)row * 16 + tid] = sum;
    }
}

// rows' records summed in row order into out[16] (one block; fixed order)
__global__ void misreg_sum_kernel(const double* __restrict__ rec, int n_rows, double* __restrict__ out) {
    __shared__ double s[256];
    for (int q = 0; q < 16; ++q) {
        double sum = 0.0;
        for (int r = threadIdx.x; r < n_rows; r += blockDim.x) sum += rec[(long long)r * 16 + q];
        s[threadIdx.x] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int i = 0; i < (int)blockDim.x; ++i) t += s[i];
            out[q] = t;
        }
        __syncthreads();
    }
}

// n floats from p set to zero by the warp: whole 16-byte vectors between the unaligned ends
__device__ __forceinline__ void zero_run(float* p, int n, int lane) {
    const int head = min(n, (int)((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15) / 4), vecs = (n - head) / 4;
    float4* v = reinterpret_cast<float4*>(p + head);
#pragma unroll 4
    for (int q = lane; q < vecs; q += 32) __stcs(v + q, make_float4(0.0f, 0.0f, 0.0f, 0.0f));
    const int rest = n - 4 * vecs;   // at most 3 before and 3 after
    if (lane < rest) __stcs(p + (lane < head ? lane : lane + 4 * vecs), 0.0f);
}

// Interaction-matrix rows of both slopes of one subaperture (block x) over a part of the commands
// (block z).  Every command of the part is written once, zero outside the actuators that reach the
// subaperture, so the matrix needs no clearing and its lines are written whole: the pass is bound by
// the matrix's own bytes.  Commands run along DM rows, so on each DM they are a run of zeros, the
// rows of the band (each command checked against the band's columns) and a run of zeros.  One block
// does every DM, so that the three barriers of the setup are paid once per 2 n_cmd stored floats and
// hide behind the other blocks' stores; a sensor of a few subapertures is cut into enough parts to
// fill the GPU, and no part writes another's commands (row_parts.h).  39 m (55608 x 8051, 1.79 GB), six
// laser stars: 470 us, bound by the instructions that form the weights and by the writes; clearing the
// matrix and scattering one slope's band per block took 6 x 160 us and 3 x 131 us more (natural
// stars), clearing whole rows first 580, a block per DM that checks every command 789.
// With gvec set (rotated DMs only) the rows are not stored: sum over both slopes of g row is added
// to the command gradients of every vector.
struct RowsDm {                // one DM's view from the block's subaperture
    AxisEnt ex[kMaxNpx], ey[kMaxNpx];
    int rng[4];                // actuators [a0, a1) x [b0, b1)
    CmdRange cmds;             // commands of rows [b0, b1) in the block's part
};

// nbw: most actuators per axis on a footprint, at most kAdjMaxBand (shared-memory row length)
template <bool ROTATED>
__global__ void __launch_bounds__(kAdjThreads, ROTATED ? 2 : 6) dm_rows_kernel(ProjLaunch L, int nbw) {
    extern __shared__ float rows_sm[];
    __shared__ RowsDm s_dm[kMaxDms];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const SubapDev sd = L.subaps[blockIdx.x];
    const WfsDev& w = L.ctx.wfs[sd.wfs];
    const int npx = w.n_px, i0 = sd.sx * npx, j0 = sd.sy * npx;
    const GridView* V = L.ctx.views + L.real * L.ctx.view_stride + (long long)sd.wfs * L.ctx.n_grids + L.n_layers;
    const int lane = tid & 31, warp = tid >> 5, n_warps = nthr >> 5;
    const bool staged = npx <= 16;                         // column weights kept (they fit)
    float* s_L = rows_sm;                                  // [2][npx][npx]
    float* s_T = s_L + 2 * npx * npx;                      // [n_dms][2][npx][nbw]
    float* s_gy = s_T + L.n_dms * 2 * npx * nbw;           // [n_dms][nbw][npx]
    float* s_gx = s_gy + L.n_dms * npx * nbw;              // [n_dms][npx][nbw], staged only
    const float *lx = sens_row(L.sens, w, 0, sd.rank), *ly = sens_row(L.sens, w, 1, sd.rank);
    for (int q = tid; q < npx * npx; q += nthr) {
        s_L[q] = lx[q];
        s_L[npx * npx + q] = ly[q];
    }
    for (int m = warp; m < 2 * L.n_dms; m += n_warps) {    // one warp per DM and axis
        const GridView& v = V[m >> 1];
        if (lane < npx) {
            if (m & 1) s_dm[m >> 1].ey[lane] = axis_entry(v.ay + (long long)(j0 + lane) * v.bp, v.n, v.periodic, v.inv_n);
            else s_dm[m >> 1].ex[lane] = axis_entry(v.ax + (long long)(i0 + lane) * v.bp, v.n, v.periodic, v.inv_n);
        }
    }
    __syncthreads();
    const CmdRange part = command_part(L.n_cmd, (int)gridDim.z, (int)blockIdx.z);
    if (lane == 0 && warp < L.n_dms) {
        RowsDm& d = s_dm[warp];
        const DmDesc& dd = L.desc[warp];
        int rng[4];
        actuator_range(dd, L.band, footprint(d.ex[0], d.ex[npx - 1]), footprint(d.ey[0], d.ey[npx - 1]), rng);
        if (rng[1] - rng[0] > nbw || rng[3] - rng[2] > nbw) {
            atomicExch(L.err, 1);
            rng[1] = rng[0];
            rng[3] = rng[2];
        }
        if (L.gvec && !dd.general) rng[3] = rng[2];
        for (int q = 0; q < 4; ++q) d.rng[q] = rng[q];
        const int* row0 = L.cmd_act + dd.row_off;          // commands before each DM row, and the total
        d.cmds = band_in_part(part, dd.cmd0 + row0[min(rng[2], dd.ny)], dd.cmd0 + row0[min(rng[3], dd.ny)]);
    }
    __syncthreads();
    const int row_x = w.slope0 + sd.rank, row_y = row_x + w.n_valid;
    float* out_x = L.D ? L.D + (long long)row_x * L.ld : nullptr;
    float* out_y = L.D ? L.D + (long long)row_y * L.ld : nullptr;
    // the zeros between the DMs' bands, one warp per run and row
    if (L.D)
        for (int r = warp; r < 2 * (L.n_dms + 1); r += n_warps) {
            const int m = r >> 1;
            const CmdRange z = zeros_between(part, m ? &s_dm[m - 1].cmds : nullptr, m < L.n_dms ? &s_dm[m].cmds : nullptr);
            zero_run((r & 1 ? out_y : out_x) + z.lo, z.hi - z.lo, lane);
        }
    // weights of the footprint's columns and rows
    for (int m = 0; m < L.n_dms; ++m) {
        const DmDesc& dd = L.desc[m];
        const RowsDm& d = s_dm[m];
        const int a0 = d.rng[0], na = d.rng[1] - a0, b0 = d.rng[2], nbd = d.rng[3] - b0;
        if ((ROTATED && dd.general) || d.cmds.lo == d.cmds.hi) continue;
        const float *Gx = L.g + dd.gx_off + a0, *Gy = L.g + dd.gy_off + b0;
        for (int y = warp; y < npx; y += n_warps) {
            if (staged)
                for (int a = lane; a < na; a += 32) s_gx[(m * npx + y) * nbw + a] = axis_weight(Gx, dd.nx, d.ex[y], a);
            for (int b = lane; b < nbd; b += 32) s_gy[(m * nbw + b) * npx + y] = axis_weight(Gy, dd.ny, d.ey[y], b);
        }
    }
    __syncthreads();
    // T[axis][y][a] = sum_x L[axis][y][x] gx_a(x)
    for (int m = 0; m < L.n_dms; ++m) {
        const DmDesc& dd = L.desc[m];
        const RowsDm& d = s_dm[m];
        const int a0 = d.rng[0], na = d.rng[1] - a0;
        if ((ROTATED && dd.general) || d.cmds.lo == d.cmds.hi) continue;
        const float* Gx = L.g + dd.gx_off + a0;
        float* T = s_T + m * 2 * npx * nbw;
        if (staged) {
            for (int y = warp; y < npx; y += n_warps)
                for (int a = lane; a < na; a += 32) {
                    float tx = 0.0f, ty = 0.0f;
#pragma unroll 8
                    for (int x = 0; x < npx; ++x) {
                        const float g = s_gx[(m * npx + x) * nbw + a];
                        tx = fmaf(s_L[y * npx + x], g, tx);
                        ty = fmaf(s_L[(npx + y) * npx + x], g, ty);
                    }
                    T[y * nbw + a] = tx;
                    T[(npx + y) * nbw + a] = ty;
                }
        } else {
            for (int idx = tid; idx < na * npx; idx += nthr) {
                const int y = idx / na, a = idx - y * na;
                float tx = 0.0f, ty = 0.0f;
#pragma unroll 4
                for (int x = 0; x < npx; ++x) {
                    const float g = axis_weight(Gx, dd.nx, d.ex[x], a);
                    tx = fmaf(s_L[y * npx + x], g, tx);
                    ty = fmaf(s_L[(npx + y) * npx + x], g, ty);
                }
                T[y * nbw + a] = tx;
                T[(npx + y) * nbw + a] = ty;
            }
        }
    }
    __syncthreads();
    for (int m = 0; m < L.n_dms; ++m) {
        const DmDesc& dd = L.desc[m];
        const RowsDm& d = s_dm[m];
        const int a0 = d.rng[0], na = d.rng[1] - a0, b0 = d.rng[2], nbd = d.rng[3] - b0;
        const float sign = V[m].sign;
        const float* T = s_T + m * 2 * npx * nbw;
        const float* gy = s_gy + m * npx * nbw;
        for (int j = d.cmds.lo + tid; j < d.cmds.hi; j += nthr) {
            const int ab = __ldg(L.cmd_act + j), a = (ab & 0xffff) - a0, b = (int)((unsigned)ab >> 16) - b0;
            float vx = 0.0f, vy = 0.0f;
            if ((unsigned)a < (unsigned)na && (unsigned)b < (unsigned)nbd) {
                if (!ROTATED || !dd.general) {
#pragma unroll 8
                    for (int y = 0; y < npx; ++y) {
                        const float g = gy[b * npx + y];
                        vx = fmaf(g, T[y * nbw + a], vx);
                        vy = fmaf(g, T[(npx + y) * nbw + a], vy);
                    }
                } else {
                    // influence function of actuator (a, b) at q(i, j) = R(-rot)((x_i, y_j) - shift) / mag,
                    // at the four bilinear corners of every sample
                    const float g0 = 0.5f * (float)(dd.surf_n - 1);
                    const float fa = (float)(a0 + a) - 0.5f * (float)(dd.nx - 1), fb = (float)(b0 + b) - 0.5f * (float)(dd.ny - 1);
                    for (int q = 0; q < npx * npx; ++q) {
                        const float l0 = s_L[q], l1 = s_L[npx * npx + q];
                        if (l0 == 0.0f && l1 == 0.0f) continue;
                        const AxisEnt ex = d.ex[q % npx], ey = d.ey[q / npx];
                        float wt = 0.0f;
                        for (int c = 0; c < 4; ++c) {
                            const int i = (c & 1) ? ex.idx >> 16 : ex.idx & 0xffff, k = (c & 2) ? ey.idx >> 16 : ey.idx & 0xffff;
                            const float wc = ((c & 1) ? ex.t : 1.0f - ex.t) * ((c & 2) ? ey.t : 1.0f - ey.t);
                            const float x = ((float)i - g0) * dd.dx - dd.shx, y = ((float)k - g0) * dd.dx - dd.shy;
                            const float ua = (dd.cr * x + dd.sr * y) * dd.inv_mag / dd.pitch;
                            const float ub = (-dd.sr * x + dd.cr * y) * dd.inv_mag / dd.pitch;
                            const float da = (ua - fa) * dd.pitch, db = (ub - fb) * dd.pitch;
                            wt = fmaf(wc, expf(-(da * da + db * db) * dd.inv2s2), wt);
                        }
                        vx = fmaf(l0, wt, vx);
                        vy = fmaf(l1, wt, vy);
                    }
                }
                vx *= sign;
                vy *= sign;
                if (L.gvec)
                    for (int vv = 0; vv < L.n_vec; ++vv) {
                        const float gx = L.gvec[(long long)vv * L.n_slopes + row_x], gy = L.gvec[(long long)vv * L.n_slopes + row_y];
                        // a slope that the vector leaves out adds nothing, a NaN derivative neither
                        const float add = fmaf(gx, gx != 0.0f ? vx : 0.0f, gy * (gy != 0.0f ? vy : 0.0f));
                        if (add != 0.0f) atomicAdd(L.gc + (long long)vv * L.n_cmd + j, add);
                    }
            }
            if (L.D) {
                __stcs(out_x + j, vx);
                __stcs(out_y + j, vy);
            }
        }
    }
    // padding columns past the last command
    if (L.D && blockIdx.z == gridDim.z - 1)
        for (long long j = L.n_cmd + tid; j < L.ld; j += nthr) out_x[j] = out_y[j] = 0.0f;
}

// Flags a subaperture whose footprint on a DM meets more actuators than the rows kernel takes (one
// thread per subaperture and DM), so that the products refuse what the matrix refuses.
__global__ void dm_range_kernel(ProjLaunch L) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n_valid * L.n_dms) return;
    const int m = i / L.n_valid;
    const SubapDev sd = L.subaps[i - m * L.n_valid];
    const WfsDev& w = L.ctx.wfs[sd.wfs];
    const GridView& v = L.ctx.views[L.real * L.ctx.view_stride + (long long)sd.wfs * L.ctx.n_grids + L.n_layers + m];
    auto at = [&](long long a, int i) {
        return footprint(axis_entry(a + (long long)i * v.bp, v.n, v.periodic, v.inv_n),
                         axis_entry(a + (long long)(i + w.n_px - 1) * v.bp, v.n, v.periodic, v.inv_n));
    };
    int rng[4];
    actuator_range(L.desc[m], L.band, at(v.ax, sd.sx * w.n_px), at(v.ay, sd.sy * w.n_px), rng);
    if (rng[1] - rng[0] > kAdjMaxBand || rng[3] - rng[2] > kAdjMaxBand) atomicExch(L.err, 1);
}

// D^T g of the separable DMs from the sensors' pupil-phase gradients, in two passes over the
// separable weights: U[y][a] = sum_x g(y, x) gx_a(x), then C[b][a] -= sum_y gy_b(y) U[y][a] over
// every sensor, in a fixed order.  The products are N^2 n_x + N n_x n_y per sensor and DM, whatever
// the number of subapertures (before: each slope's row, added into the gradient by atomics).
// Block: 8 pupil rows (one per warp) x 32 actuators; x in tiles of 32, and only the tiles whose band
// of actuators with a weight meets the block's 32 (found for all tiles at once, one thread each: the
// dependent reads of the band table one tile after another took most of the 39 us this pass took at
// 320 x 320 samples and 3 sensors; 27 us now).
constexpr int kProjMaxTiles = 512;   // pupil grids of at most 16384 samples per side
__global__ void __launch_bounds__(256) dm_project_x(ProjLaunch L, const float* __restrict__ g_phase, long long phase_stride,
                                                    float* __restrict__ U, int u_rows, int u_cols) {
    __shared__ float s_w[32][33];
    __shared__ float s_g[8][32];
    __shared__ int2 s_band[kProjMaxTiles];
    const int wi = blockIdx.y / L.n_dms, m = blockIdx.y - wi * L.n_dms;
    const int a_tiles = (u_cols + 31) / 32, vec = blockIdx.z / a_tiles, a0 = (blockIdx.z - vec * a_tiles) * 32;
    const WfsDev& w = L.ctx.wfs[wi];
    const DmDesc dd = L.desc[m];
    const int N = w.N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int y = blockIdx.x * 8 + warp;
    if (dd.general || a0 >= dd.nx || (int)blockIdx.x * 8 >= N) return;
    long long off = vec * phase_stride;
    for (int q = 0; q < wi; ++q) off += (long long)L.ctx.wfs[q].N * L.ctx.wfs[q].N;
    const GridView& v = L.ctx.views[L.real * L.ctx.view_stride + (long long)wi * L.ctx.n_grids + L.n_layers + m];
    auto entry = [&](int x) { return axis_entry(v.ax + (long long)x * v.bp, v.n, v.periodic, v.inv_n); };
    const int tiles = (N + 31) / 32;
    for (int t = threadIdx.x; t < tiles; t += 256) {
        int lo = dd.nx, hi = 0;
        const int2 c = footprint(entry(32 * t), entry(min(32 * t + 32, N) - 1));
        for (int q = c.x / kDmTile; q <= c.y / kDmTile; ++q) {
            const int2 bt = L.band[dd.tband_x + q];
            if (bt.y > bt.x) { lo = min(lo, bt.x); hi = max(hi, bt.y); }
        }
        s_band[t] = make_int2(lo, hi);
    }
    float acc = 0.0f;
    __syncthreads();
    for (int t = 0; t < tiles; ++t) {
        const int2 bt = s_band[t];
        if (bt.y <= a0 || bt.x >= a0 + 32) continue;   // the same for the whole block
        const int x0 = 32 * t;
        __syncthreads();
        for (int q = threadIdx.x; q < 32 * 32; q += 256) {
            const int x = x0 + (q >> 5), a = a0 + (q & 31);
            const float wt = (x < N && a >= bt.x && a < bt.y) ? axis_weight(L.g + dd.gx_off, dd.nx, entry(x), a) : 0.0f;
            s_w[q >> 5][q & 31] = wt < 1e-10f ? 0.0f : wt;   // the band is wider than this sample's own reach
        }
        s_g[warp][lane] = (y < N && x0 + lane < N) ? g_phase[off + (long long)y * N + x0 + lane] : 0.0f;
        __syncthreads();
#pragma unroll 8
        for (int x = 0; x < 32; ++x) {
            const float wt = s_w[x][lane];
            if (wt != 0.0f) acc = fmaf(s_g[warp][x], wt, acc);   // a NaN reaches the actuators with a weight alone
        }
    }
    if (y < N && a0 + lane < dd.nx) U[(((long long)vec * gridDim.y + blockIdx.y) * u_rows + y) * u_cols + a0 + lane] = acc;
}

// One block per (DM row b, 32 actuator columns).  The 32 warps take chunks of 32 pupil rows of each
// sensor in turn: lane l forms the weight of row l, then the rows with one are added in order.
// (A row at a time, each waiting for its band and table reads: 44 us; 23 us now.)
__global__ void __launch_bounds__(1024) dm_project_y(ProjLaunch L, int n_wfs, const float* __restrict__ U, int u_rows,
                                                    int u_cols) {
    __shared__ float s_sum[32][32];
    const int m = blockIdx.z % L.n_dms, vec = blockIdx.z / L.n_dms;
    const DmDesc dd = L.desc[m];
    const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, a = blockIdx.x * 32 + lane;
    if (dd.general || b >= dd.ny || (int)blockIdx.x * 32 >= dd.nx) return;
    float acc = 0.0f;
    int turn = 0;
    for (int wi = 0; wi < n_wfs; ++wi) {
        const WfsDev& w = L.ctx.wfs[wi];
        const GridView& v = L.ctx.views[L.real * L.ctx.view_stride + (long long)wi * L.ctx.n_grids + L.n_layers + m];
        const float* u = U + ((long long)vec * n_wfs + wi) * L.n_dms * u_rows * u_cols + (long long)m * u_rows * u_cols;
        for (int y0 = 0; y0 < w.N; y0 += 32, ++turn) {
            if ((turn & 31) != warp) continue;
            float gy = 0.0f;
            if (y0 + lane < w.N) {
                const AxisEnt e = axis_entry(v.ay + (long long)(y0 + lane) * v.bp, v.n, v.periodic, v.inv_n);
                const int2 b0 = L.band[dd.tband_y + (e.idx & 0xffff) / kDmTile], b1 = L.band[dd.tband_y + (e.idx >> 16) / kDmTile];
                if ((b >= b0.x && b < b0.y) || (b >= b1.x && b < b1.y)) gy = v.sign * axis_weight(L.g + dd.gy_off, dd.ny, e, b);
            }
            if (!__ballot_sync(0xffffffffu, gy != 0.0f)) continue;
#pragma unroll 8
            for (int q = 0; q < 32; ++q) {
                const float g = __shfl_sync(0xffffffffu, gy, q);
                if (g != 0.0f && a < dd.nx) acc = fmaf(g, u[(long long)(y0 + q) * u_cols + a], acc);
            }
        }
    }
    s_sum[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && a < dd.nx) {
        float s = 0.0f;
        for (int q = 0; q < 32; ++q) s += s_sum[q][lane];
        const int cmd = L.act_map[dd.map_off + (long long)b * dd.nx + a];
        if (cmd >= 0) L.gc[(long long)vec * L.n_cmd + cmd] = s;
    }
}

// Per subaperture and vector: g_phi = g_v[x slope] L_x + g_v[y slope] L_y on its pupil samples,
// stored in g_phase[v][sensor's offset + (j0 + y) N + i0 + x] and/or scattered onto the layers (the
// adjoint of the periodic bilinear sampling at the frozen-flow position of the step) in
// g_layers[v][...].  The subapertures of every sensor in one launch, block y = vector.  proj, for the
// command gradients, is laid out as g_phase and leaves slopes with g = 0 out: their derivatives may be NaN.
__global__ void __launch_bounds__(128) phase_adjoint_kernel(ProjLaunch L, float* g_phase, float* proj, long long phase_stride,
                                                            float* g_layers, long long layer_stride,
                                                            const long long* layer_off) {
    const SubapDev sd = L.subaps[blockIdx.x];
    const WfsDev& w = L.ctx.wfs[sd.wfs];
    const int npx = w.n_px, vv = blockIdx.y;
    const int i0 = sd.sx * npx, j0 = sd.sy * npx;
    const GridView* V = L.ctx.views + L.real * L.ctx.view_stride + (long long)sd.wfs * L.ctx.n_grids;
    const long long k = L.ctx.st->k;
    const float *lx = sens_row(L.sens, w, 0, sd.rank), *ly = sens_row(L.sens, w, 1, sd.rank);
    const float* g = L.gvec + (long long)vv * L.n_slopes + w.slope0 + sd.rank;
    const float gx = g[0], gy = g[w.n_valid];
    long long off = vv * phase_stride;
    for (int q = 0; q < sd.wfs; ++q) off += (long long)L.ctx.wfs[q].N * L.ctx.wfs[q].N;
    for (int q = threadIdx.x; q < npx * npx; q += blockDim.x) {
        const int x = q % npx, y = q / npx;
        const float gp = gx * lx[q] + gy * ly[q];
        const long long at = off + (long long)(j0 + y) * w.N + i0 + x;
        if (g_phase) g_phase[at] = gp;
        if (proj) proj[at] = gx * (gx != 0.0f ? lx[q] : 0.0f) + gy * (gy != 0.0f ? ly[q] : 0.0f);
        if (!g_layers || gp == 0.0f) continue;
        for (int l = 0; l < L.n_layers; ++l) {
            const GridView& v = V[l];
            const AxisEnt ex = axis_entry(v.ax + (long long)(i0 + x) * v.bp + k * v.vx, v.n, v.periodic, v.inv_n);
            const AxisEnt ey = axis_entry(v.ay + (long long)(j0 + y) * v.bp + k * v.vy, v.n, v.periodic, v.inv_n);
            float* gl = g_layers + vv * layer_stride + layer_off[l];
            const int c0 = ex.idx & 0xffff, c1 = ex.idx >> 16, r0 = ey.idx & 0xffff, r1 = ey.idx >> 16;
            const float s = v.sign * gp;
            atomicAdd(gl + (long long)r0 * v.n + c0, s * (1.0f - ex.t) * (1.0f - ey.t));
            atomicAdd(gl + (long long)r0 * v.n + c1, s * ex.t * (1.0f - ey.t));
            atomicAdd(gl + (long long)r1 * v.n + c0, s * (1.0f - ex.t) * ey.t);
            atomicAdd(gl + (long long)r1 * v.n + c1, s * ex.t * ey.t);
        }
    }
}

}  // namespace

cudaError_t launch_dm_rows(const ProjLaunch& L, int n_px, int sm_count, cudaStream_t s) {
    if (!L.n_valid || !L.n_dms) return cudaSuccess;
    const int nbw = std::max(1, std::min(L.max_band, kAdjMaxBand));
    const size_t bytes = sizeof(float) * (2 * n_px * n_px + L.n_dms * (n_px <= 16 ? 4 : 3) * n_px * nbw);
    const auto kernel = L.rotated ? dm_rows_kernel<true> : dm_rows_kernel<false>;
    // the limit is the kernel's, for every thread: always the largest, 4 DMs with full bands at 32 samples
    constexpr int kMost = (int)sizeof(float) * (2 * kMaxNpx * kMaxNpx + kMaxDms * 3 * kMaxNpx * kAdjMaxBand);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (e != cudaSuccess) return e;
    // parts of the commands: two blocks per SM where the subapertures alone do not give them
    const int parts = std::max(1, std::min(16, 2 * sm_count / L.n_valid));
    kernel<<<dim3((unsigned)L.n_valid, 1u, (unsigned)parts), kAdjThreads, bytes, s>>>(L, nbw);
    return cudaGetLastError();
}

cudaError_t launch_dm_range(const ProjLaunch& L, cudaStream_t s) {
    const int n = L.n_valid * L.n_dms;
    if (n) dm_range_kernel<<<(n + 127) / 128, 128, 0, s>>>(L);
    return cudaGetLastError();
}

cudaError_t launch_dm_project(const ProjLaunch& L, int n_wfs, int max_n, int max_nx, int max_ny, const float* g_phase,
                              long long phase_stride, float* U, cudaStream_t s) {
    if (!L.n_dms || !n_wfs) return cudaSuccess;
    dm_project_x<<<dim3((unsigned)((max_n + 7) / 8), (unsigned)(n_wfs * L.n_dms), (unsigned)(L.n_vec * ((max_nx + 31) / 32))),
                   256, 0, s>>>(
        L, g_phase, phase_stride, U, max_n, max_nx);
    dm_project_y<<<dim3((unsigned)((max_nx + 31) / 32), (unsigned)max_ny, (unsigned)(L.n_dms * L.n_vec)), 1024, 0, s>>>(
        L, n_wfs, U, max_n, max_nx);
    return cudaGetLastError();
}

cudaError_t launch_misreg_gn(const ProjLaunch& L, int m, const float* D_meas, long long ld_meas, int cmd0, double* rec,
                             cudaStream_t s) {
    if (L.n_valid) misreg_gn_kernel<<<(unsigned)(2 * L.n_valid), 256, 0, s>>>(L, m, D_meas, ld_meas, cmd0, rec);
    return cudaGetLastError();
}

cudaError_t launch_misreg_sum(const double* rec, int n_rows, double* out, cudaStream_t s) {
    misreg_sum_kernel<<<1, 256, 0, s>>>(rec, n_rows, out);
    return cudaGetLastError();
}

cudaError_t launch_phase_adjoint(const ProjLaunch& L, float* g_phase, float* proj, long long phase_stride, float* g_layers,
                                 long long layer_stride, const long long* layer_off, cudaStream_t s) {
    if (L.n_valid)
        phase_adjoint_kernel<<<dim3((unsigned)L.n_valid, (unsigned)L.n_vec), 128, 0, s>>>(L, g_phase, proj, phase_stride, g_layers,
                                                                                         layer_stride, layer_off);
    return cudaGetLastError();
}

}  // namespace mcao
