// stencil.cu -- the grid CWT as the paper evaluates it (Sec. 2.1): every grid
// node adds its mass times the wavelet sampled on a stencil around it.  The
// stencil is the cube of offsets |d_x|, |d_y|, |d_z| <= R (R = gdw_resolution
// of Table 1, read as a radius), periodic:
//   C(g) = sum_{d in cube} m(g - d) Psi(w, Delta |d|).
//
// On a cube the Mexican hat stays exactly separable: with G(d) = exp(-w^2
// Delta^2 d^2 / 4) and H(d) = w^2 Delta^2 d^2 G(d) (both even, |d| <= R),
//   Psi = w^1.5 [6 G_x G_y G_z - H_x G_y G_z - G_x H_y G_z - G_x G_y H_z],
// so the sum is seven 1D convolutions in three passes over the grid:
//   x:  A = G_x * m,  B = H_x * m
//   y:  P = G_y * (6A - B) - H_y * A,  Q = G_y * A
//   z:  C = w^1.5 (G_z * P - H_z * Q).
// Each pass reads and writes the grid once (8 + 8, 8 + 8, 8 + 4 bytes per
// cell), in fp32, with the int64 CIC masses converted on the first read.
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.cuh"

namespace cwthf {
namespace {

constexpr int kMaxR = CWTHF_MAX_STENCIL_R;

struct StencilTaps {
    float g[kMaxR + 1];  // G(d), d = 0..R
    float h[kMaxR + 1];  // H(d)
    int R;
};

// Radii up to kRegMaxR (Table 1's are 5 .. 20 in cells of the paper's grids)
// run register-window kernels, compiled per radius class (the radius rounded
// up to a multiple of four, with zero taps beyond R): a thread takes several
// neighbouring outputs, loads the window they share once, and adds the taps
// from registers in the same order as the general kernels below, which load
// 2 R + 1 shared-memory values per output and array and were bound by those
// loads.  256^3, R = 7: x 74 -> 44 us, y 125 -> 65 us, z 115 -> 58 us
// (the same bits).
constexpr int kRegMaxR = 16;
constexpr int kXWarps = 8;  // rows per CTA in the x passes

__host__ __device__ constexpr int x_pitch_r(int ng, int RC) { return (ng + 2 * RC + 7) & ~3; }

// x pass: one warp per row, staged in shared memory with RC wrapped cells on
// each side; each lane forms A and B for four neighbouring columns.
template <int RC>
__global__ void __launch_bounds__(32 * kXWarps) k_sten_x_reg(const int64_t* grid, int ng, StencilTaps t,
                                                             float* __restrict__ A, float* __restrict__ B) {
    pdl_wait();
    extern __shared__ __align__(16) float rows[];  // [kXWarps][pitch]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* buf = rows + warp * x_pitch_r(ng, RC);
    const int64_t row = int64_t(blockIdx.x) * kXWarps + warp;
    if (row >= int64_t(ng) * ng) return;  // warp-uniform; no block barrier below
    constexpr float kUnit = 9.3132257461547852e-10f;  // 2^-30: one CIC mass unit
    const int64_t* src = grid + row * ng;
    if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {  // ng is even
        for (int x = 2 * lane; x < ng; x += 64) {
            const longlong2 v = *reinterpret_cast<const longlong2*>(src + x);
            buf[RC + x] = ll2float(v.x) * kUnit;
            buf[RC + x + 1] = ll2float(v.y) * kUnit;
        }
    } else {
        for (int x = lane; x < ng; x += 32) buf[RC + x] = ll2float(src[x]) * kUnit;
    }
    __syncwarp();
    if (lane < RC) {  // RC <= ng: the radius class is at most R + 3, and ng >= 2 R + 1, ng >= 8
        buf[lane] = buf[ng + lane];
        buf[RC + ng + lane] = buf[RC + lane];
    }
    __syncwarp();
    float* a = A + row * ng;
    float* b = B + row * ng;
    for (int x = 4 * lane; x < ng; x += 128) {
        float w[4 + 2 * RC];  // buf[x + i] = m(x - RC + i)
#pragma unroll
        for (int i = 0; i < 4 + 2 * RC; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(buf + x + i);
            w[i] = v.x;
            w[i + 1] = v.y;
            w[i + 2] = v.z;
            w[i + 3] = v.w;
        }
        float sa[4], sb[4];
#pragma unroll
        for (int o = 0; o < 4; o++) {
            sa[o] = t.g[0] * w[o + RC];
            sb[o] = 0.0f;  // H(0) = 0
#pragma unroll
            for (int d = 1; d <= RC; d++) {
                const float s = w[o + RC - d] + w[o + RC + d];
                sa[o] = fmaf(t.g[d], s, sa[o]);
                sb[o] = fmaf(t.h[d], s, sb[o]);
            }
        }
        // row starts are 8-byte aligned (ng is even)
        *reinterpret_cast<float2*>(a + x) = make_float2(sa[0], sa[1]);
        *reinterpret_cast<float2*>(b + x) = make_float2(sb[0], sb[1]);
        if (x + 2 < ng) {
            *reinterpret_cast<float2*>(a + x + 2) = make_float2(sa[2], sa[3]);
            *reinterpret_cast<float2*>(b + x + 2) = make_float2(sb[2], sb[3]);
        }
    }
}

// y and z passes: a CTA takes 32 adjacent x columns of one line family (a
// plane z for the y pass, a row y for the z pass) and kLine outputs along the
// pass's axis, staging kLine + 2 RC input lines of both arrays in shared
// memory; a warp takes kOut neighbouring lines.
constexpr int kLine = 64;
constexpr int kLineThreads = 256;
constexpr int kOut = kLine / (kLineThreads / 32);  // 8

template <bool kZ, int RC>
__global__ void __launch_bounds__(kLineThreads) k_sten_yz_reg(const float* in0,
                                                             const float* in1, int ng, StencilTaps t,
                                                             float scale, float* __restrict__ out0,
                                                             float* __restrict__ out1) {
    pdl_wait();
    constexpr int H = kLine + 2 * RC, W = kOut + 2 * RC;
    extern __shared__ float tile[];  // [2][H][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* s0 = tile;
    float* s1 = tile + H * 32;
    const int nxc = (ng + 31) / 32, nlc = (ng + kLine - 1) / kLine;
    const int xc = int(blockIdx.x % nxc), lc = int((blockIdx.x / nxc) % nlc), fam = int(blockIdx.x / (nxc * nlc));
    const int x = xc * 32 + lane;
    const bool own = x < ng;
    const int64_t stride = kZ ? int64_t(ng) * ng : int64_t(ng);  // step along the pass's axis
    const int64_t base = (kZ ? int64_t(fam) * ng : int64_t(fam) * ng * ng) + x;
    const int l0 = lc * kLine;
    constexpr int kWarps = kLineThreads / 32, kLd = H / kWarps;  // lines per warp (H is a multiple of 8)
    static_assert(H % kWarps == 0, "whole lines per warp");
    float v0[kLd], v1[kLd];  // all loads in flight at once
#pragma unroll
    for (int i = 0; i < kLd; i++) {
        int l = l0 - RC + warp + i * kWarps;
        if (l < 0) l += ng;
        while (l >= ng) l -= ng;  // at most once for ng >= kLine + 2 RC
        v0[i] = own ? in0[base + l * stride] : 0.f;
        v1[i] = own ? in1[base + l * stride] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < kLd; i++) {
        const int j = warp + i * kWarps;
        // z pass: inputs P, Q as they are; y pass: inputs A, B, staged as U = 6A - B and A
        s0[j * 32 + lane] = kZ ? v0[i] : 6.0f * v0[i] - v1[i];
        s1[j * 32 + lane] = kZ ? v1[i] : v0[i];
    }
    __syncthreads();
    const int j0 = warp * kOut;  // lines l0 + j0 ..; line l's window starts at staged line l - l0
    if (!own || l0 + j0 >= ng) return;
    float r0[kOut], r1[kOut];
    {
        float w[W];
#pragma unroll
        for (int i = 0; i < W; i++) w[i] = s0[(j0 + i) * 32 + lane];
#pragma unroll
        for (int o = 0; o < kOut; o++) {  // G * P (z pass), G * U (y pass)
            float s = t.g[0] * w[o + RC];
#pragma unroll
            for (int d = 1; d <= RC; d++) s = fmaf(t.g[d], w[o + RC - d] + w[o + RC + d], s);
            r0[o] = s;
        }
    }
    float w[W];
#pragma unroll
    for (int i = 0; i < W; i++) w[i] = s1[(j0 + i) * 32 + lane];
#pragma unroll
    for (int o = 0; o < kOut; o++) {  // H * Q (z pass); G * A and H * A (y pass)
        float sa = kZ ? 0.f : t.g[0] * w[o + RC], sh = 0.0f;
#pragma unroll
        for (int d = 1; d <= RC; d++) {
            const float v = w[o + RC - d] + w[o + RC + d];
            if (!kZ) sa = fmaf(t.g[d], v, sa);
            sh = fmaf(t.h[d], v, sh);
        }
        r0[o] -= sh;
        r1[o] = sa;
    }
#pragma unroll
    for (int o = 0; o < kOut; o++) {
        const int l = l0 + j0 + o;
        if (l >= ng) break;
        out0[base + l * stride] = kZ ? scale * r0[o] : r0[o];
        if (!kZ) out1[base + l * stride] = r1[o];
    }
}

// ---- any radius ----

// x pass: one warp per row of the grid.  The row (with R wrapped cells on each
// side) is staged in shared memory; each lane then forms A and B for the
// columns lane, lane + 32, ...
__global__ void __launch_bounds__(32 * kXWarps) k_sten_x(const int64_t* grid, int ng, StencilTaps t,
                                                         float* __restrict__ A, float* __restrict__ B) {
    pdl_wait();
    extern __shared__ float rows[];  // [kXWarps][ng + 2R]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int R = t.R, W = ng + 2 * R;
    float* buf = rows + warp * W;
    const int64_t nrows = int64_t(ng) * ng;
    const int64_t row = int64_t(blockIdx.x) * kXWarps + warp;
    if (row >= nrows) return;  // warp-uniform; no block barrier below
    constexpr float kUnit = 9.3132257461547852e-10f;  // 2^-30: one CIC mass unit
    const int64_t* src = grid + row * ng;
    for (int j = lane; j < W; j += 32) {
        int x = j - R;
        x = x < 0 ? x + ng : (x >= ng ? x - ng : x);
        buf[j] = ll2float(src[x]) * kUnit;
    }
    __syncwarp();
    float* a = A + row * ng;
    float* b = B + row * ng;
    for (int x = lane; x < ng; x += 32) {
        const float* c = buf + x + R;  // c[d] = m(x + d)
        float sa = t.g[0] * c[0], sb = 0.0f;  // H(0) = 0
        for (int d = 1; d <= R; d++) {
            const float s = c[-d] + c[d];
            sa = fmaf(t.g[d], s, sa);
            sb = fmaf(t.h[d], s, sb);
        }
        a[x] = sa;
        b[x] = sb;
    }
}

// y and z passes: as above, each output's taps read from shared memory.

template <bool kZ>
__global__ void __launch_bounds__(kLineThreads) k_sten_yz(const float* in0, const float* in1,
                                                         int ng, StencilTaps t, float scale,
                                                         float* __restrict__ out0, float* __restrict__ out1) {
    pdl_wait();
    extern __shared__ float tile[];  // [2][kLine + 2R][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int R = t.R, H = kLine + 2 * R;
    float* s0 = tile;
    float* s1 = tile + H * 32;
    const int nxc = (ng + 31) / 32, nlc = (ng + kLine - 1) / kLine;
    const int xc = int(blockIdx.x % nxc), lc = int((blockIdx.x / nxc) % nlc), fam = int(blockIdx.x / (nxc * nlc));
    const int x = xc * 32 + lane;
    const bool own = x < ng;
    const int64_t stride = kZ ? int64_t(ng) * ng : int64_t(ng);  // step along the pass's axis
    const int64_t base = (kZ ? int64_t(fam) * ng : int64_t(fam) * ng * ng) + x;
    const int l0 = lc * kLine;
    for (int j = warp; j < H; j += kLineThreads / 32) {
        int l = l0 - R + j;
        l = ((l % ng) + ng) % ng;
        float v0 = 0.f, v1 = 0.f;
        if (own) {
            v0 = in0[base + l * stride];
            v1 = in1[base + l * stride];
        }
        if (kZ) {  // z pass: inputs P, Q as they are
            s0[j * 32 + lane] = v0;
            s1[j * 32 + lane] = v1;
        } else {  // y pass: inputs A, B; stage U = 6A - B and A
            s0[j * 32 + lane] = 6.0f * v0 - v1;
            s1[j * 32 + lane] = v0;
        }
    }
    __syncthreads();
    if (!own) return;
    for (int j = warp; j < kLine; j += kLineThreads / 32) {
        const int l = l0 + j;
        if (l >= ng) break;
        const float* c0 = s0 + (j + R) * 32 + lane;
        const float* c1 = s1 + (j + R) * 32 + lane;
        if (kZ) {  // C = scale (G * P - H * Q)
            float sp = t.g[0] * c0[0], sq = 0.0f;
            for (int d = 1; d <= R; d++) {
                sp = fmaf(t.g[d], c0[-32 * d] + c0[32 * d], sp);
                sq = fmaf(t.h[d], c1[-32 * d] + c1[32 * d], sq);
            }
            out0[base + l * stride] = scale * (sp - sq);
        } else {  // P = G * U - H * A,  Q = G * A
            float su = t.g[0] * c0[0], sa = t.g[0] * c1[0], sh = 0.0f;
            for (int d = 1; d <= R; d++) {
                const float a = c1[-32 * d] + c1[32 * d];
                su = fmaf(t.g[d], c0[-32 * d] + c0[32 * d], su);
                sa = fmaf(t.g[d], a, sa);
                sh = fmaf(t.h[d], a, sh);
            }
            out0[base + l * stride] = su - sh;
            out1[base + l * stride] = sa;
        }
    }
}

// The register-window passes of one radius class.
template <int RC>
int launch_reg(cwthf_ctx* ctx, const int64_t* grid, int ng, const StencilTaps& t, float scale, float* A, float* B,
               float* P, float* Q, float* cwt, cudaStream_t s) {
    const size_t xs = size_t(kXWarps) * x_pitch_r(ng, RC) * sizeof(float);
    CWTHF_LAUNCH(ctx, s, "k_sten_x",
                 pdl(k_sten_x_reg<RC>, div_up(int64_t(ng) * ng, kXWarps), 32 * kXWarps, xs, s)(grid, ng, t, A, B));
    const size_t ls = size_t(2) * (kLine + 2 * RC) * 32 * sizeof(float);
    const unsigned lblocks = unsigned(div_up(ng, 32) * div_up(ng, kLine) * ng);
    CWTHF_LAUNCH(ctx, s, "k_sten_y",
                 pdl(k_sten_yz_reg<false, RC>, lblocks, kLineThreads, ls, s)(A, B, ng, t, 1.0f, P, Q));
    CWTHF_LAUNCH(ctx, s, "k_sten_z",
                 pdl(k_sten_yz_reg<true, RC>, lblocks, kLineThreads, ls, s)(P, Q, ng, t, scale, cwt, nullptr));
    return cuda_status(cudaGetLastError());
}

}  // namespace

int transform_stencil_impl(cwthf_ctx* ctx, const int64_t* grid, int ng, double L, double mass_unit, double w, int R,
                           float* cwt, cudaStream_t s) {
    StencilTaps t = {};  // taps beyond R are zero
    t.R = R;
    const double dx = L / ng;
    for (int d = 0; d <= R; d++) {
        const double u2 = (dx * d) * (dx * d);
        const double gd = std::exp(-0.25 * w * w * u2);
        t.g[d] = float(gd);
        t.h[d] = float(w * w * u2 * gd);
    }
    const float scale = float(std::pow(w, 1.5) * mass_unit);
    const int64_t cells = int64_t(ng) * ng * ng;
    // scratch: A, B in the context's CWT and label buffers, P, Q in its int64
    // grid buffer (two float grids)
    float* A = ctx->cwt;
    float* B = reinterpret_cast<float*>(ctx->label);
    float* P = reinterpret_cast<float*>(ctx->grid);
    float* Q = P + cells;
    if (R <= 4) return launch_reg<4>(ctx, grid, ng, t, scale, A, B, P, Q, cwt, s);
    if (R <= 8) return launch_reg<8>(ctx, grid, ng, t, scale, A, B, P, Q, cwt, s);
    if (R <= 12) return launch_reg<12>(ctx, grid, ng, t, scale, A, B, P, Q, cwt, s);
    if (R <= kRegMaxR) return launch_reg<16>(ctx, grid, ng, t, scale, A, B, P, Q, cwt, s);
    const size_t xs = size_t(kXWarps) * (ng + 2 * R) * sizeof(float);
    const int xblocks = div_up(int64_t(ng) * ng, kXWarps);
    CWTHF_LAUNCH(ctx, s, "k_sten_x", pdl(k_sten_x, xblocks, 32 * kXWarps, xs, s)(grid, ng, t, A, B));
    const size_t ls = size_t(2) * (kLine + 2 * R) * 32 * sizeof(float);
    const unsigned lblocks = unsigned(div_up(ng, 32) * div_up(ng, kLine) * ng);
    cudaFuncSetAttribute(k_sten_yz<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(ls));
    cudaFuncSetAttribute(k_sten_yz<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(ls));
    CWTHF_LAUNCH(ctx, s, "k_sten_y", pdl(k_sten_yz<false>, lblocks, kLineThreads, ls, s)(A, B, ng, t, 1.0f, P, Q));
    CWTHF_LAUNCH(ctx, s, "k_sten_z", pdl(k_sten_yz<true>, lblocks, kLineThreads, ls, s)(P, Q, ng, t, scale, cwt, nullptr));
    return cuda_status(cudaGetLastError());
}

}  // namespace cwthf
