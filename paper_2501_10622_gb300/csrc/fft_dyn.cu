// fft_dyn.cu -- the run-time FFT pass kernels, for the plans a caller sets
// (cwthf_set_fft_plan: any radix order and tile width).  One butterfly per
// thread and stage, each radix's stage a function of its own; the built-in
// plans, also when a caller sets one, run compile-time instances instead
// (fft_ct.cuh), which take a third to a tenth of the time.
#include "fft.cuh"

namespace cwthf {
namespace fft {
namespace {

// Load the R inputs of butterfly j, apply the inter-stage twiddles, DFT.
template <int R, class A>
__device__ __forceinline__ void bfly_load(const float2* tile, A addr, const float2* tw, int L, int Ns, int j, int c,
                                          float2 (&v)[R]) {
    const int stride = L / R;
#pragma unroll
    for (int r = 0; r < R; r++) v[r] = tile[addr(j + r * stride, c)];
    if (Ns > 1) {
        const int k = j % Ns;
        const int step = L / (Ns * R);
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = cmul(v[r], tw[r * k * step]);  // r*k*step < Ns*R*step = L
    }
    RegDif<R>::template run<0>(v);  // output r now sits at v[dig_rev(R, r)]
}

template <int R, class A>
__device__ __forceinline__ void bfly_store(float2* tile, A addr, int Ns, int j, int c, const float2 (&v)[R]) {
    const int k = j % Ns;
    const int base = (j / Ns) * Ns * R + k;
    static_for<0, R>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        tile[addr(base + r * Ns, c)] = v[dig_rev(R, r)];
    });
}

// One full stage: every active thread reads, the block syncs, every active thread writes.
// Not inlined: each radix gets its own register allocation.
template <int R, class A>
__device__ __noinline__ void stage_r(float2* tile, A addr, const float2* tw, int L, int Ns, int C) {
    const int c = threadIdx.x % C, j = threadIdx.x / C;
    const bool on = j < L / R;
    float2 v[R];
    if (on) bfly_load<R>(tile, addr, tw, L, Ns, j, c, v);
    __syncthreads();
    if (on) bfly_store<R>(tile, addr, Ns, j, c, v);
    __syncthreads();
}

template <class A>
__device__ __forceinline__ void stage(int R, float2* tile, A addr, const float2* tw, int L, int Ns, int C) {
    switch (R) {
        case 2: stage_r<2>(tile, addr, tw, L, Ns, C); break;
        case 3: stage_r<3>(tile, addr, tw, L, Ns, C); break;
        case 4: stage_r<4>(tile, addr, tw, L, Ns, C); break;
        case 5: stage_r<5>(tile, addr, tw, L, Ns, C); break;
        case 6: stage_r<6>(tile, addr, tw, L, Ns, C); break;
        case 7: stage_r<7>(tile, addr, tw, L, Ns, C); break;
        case 8: stage_r<8>(tile, addr, tw, L, Ns, C); break;
        case 9: stage_r<9>(tile, addr, tw, L, Ns, C); break;
        case 10: stage_r<10>(tile, addr, tw, L, Ns, C); break;
        case 12: stage_r<12>(tile, addr, tw, L, Ns, C); break;
        case 14: stage_r<14>(tile, addr, tw, L, Ns, C); break;
        case 15: stage_r<15>(tile, addr, tw, L, Ns, C); break;
        case 16: stage_r<16>(tile, addr, tw, L, Ns, C); break;
        case 18: stage_r<18>(tile, addr, tw, L, Ns, C); break;
        case 20: stage_r<20>(tile, addr, tw, L, Ns, C); break;
        case 21: stage_r<21>(tile, addr, tw, L, Ns, C); break;
        case 24: stage_r<24>(tile, addr, tw, L, Ns, C); break;
        case 25: stage_r<25>(tile, addr, tw, L, Ns, C); break;
        case 27: stage_r<27>(tile, addr, tw, L, Ns, C); break;
        case 28: stage_r<28>(tile, addr, tw, L, Ns, C); break;
        case 30: stage_r<30>(tile, addr, tw, L, Ns, C); break;
        case 32: stage_r<32>(tile, addr, tw, L, Ns, C); break;
        default: break;
    }
}

// Forward DFT of all C sequences of the tile (natural order in and out).
template <class A>
__device__ __forceinline__ void fft_tile(const Plan& p, float2* tile, A addr, const float2* tw) {
    const int r0 = p.rad[0], r1 = p.rad[1], r2 = p.rad[2];
    stage(r0, tile, addr, tw, p.L, 1, p.C);
    if (p.nst > 1) stage(r1, tile, addr, tw, p.L, r0, p.C);
    if (p.nst > 2) stage(r2, tile, addr, tw, p.L, r0 * r1, p.C);
}

template <int R, class A>
__device__ __noinline__ void stage_fused_r(float2* tile, A addr, const float2* tw, int L, int Ns, int C,
                                              const Wave& wv) {
    const int c = threadIdx.x % C, j = threadIdx.x / C;
    const bool on = j < L / R;
    float2 v[R];
    if (on) {
        bfly_load<R>(tile, addr, tw, L, Ns, j, c, v);  // last forward stage: Ns * R == L
        // forward output r (frequency kz = j + r*Ns) sits at v[dig_rev(R, r)]; the first
        // inverse butterfly needs its inputs in natural order r
        float2 u[R];
        static_for<0, R>([&](auto rc) {
            constexpr int r = decltype(rc)::value;
            int kz = j + r * Ns;
            float psi = wv.a * wv.gz[kz] + wv.b * wv.hz[kz];
            float2 x = v[dig_rev(R, r)];
            u[r] = make_float2(x.x * psi, -(x.y * psi));  // multiply, then conj for the inverse
        });
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = u[r];
        RegDif<R>::template run<0>(v);  // first inverse stage (Ns = 1, no twiddles)
    }
    __syncthreads();
    if (on) bfly_store<R>(tile, addr, 1, j, c, v);
    __syncthreads();
}

template <class A>
__device__ __forceinline__ void stage_fused(int R, float2* tile, A addr, const float2* tw, int L, int Ns, int C,
                                            const Wave& wv) {
    switch (R) {
        case 2: stage_fused_r<2>(tile, addr, tw, L, Ns, C, wv); break;
        case 3: stage_fused_r<3>(tile, addr, tw, L, Ns, C, wv); break;
        case 4: stage_fused_r<4>(tile, addr, tw, L, Ns, C, wv); break;
        case 5: stage_fused_r<5>(tile, addr, tw, L, Ns, C, wv); break;
        case 6: stage_fused_r<6>(tile, addr, tw, L, Ns, C, wv); break;
        case 7: stage_fused_r<7>(tile, addr, tw, L, Ns, C, wv); break;
        case 8: stage_fused_r<8>(tile, addr, tw, L, Ns, C, wv); break;
        case 9: stage_fused_r<9>(tile, addr, tw, L, Ns, C, wv); break;
        case 10: stage_fused_r<10>(tile, addr, tw, L, Ns, C, wv); break;
        case 12: stage_fused_r<12>(tile, addr, tw, L, Ns, C, wv); break;
        case 14: stage_fused_r<14>(tile, addr, tw, L, Ns, C, wv); break;
        case 15: stage_fused_r<15>(tile, addr, tw, L, Ns, C, wv); break;
        case 16: stage_fused_r<16>(tile, addr, tw, L, Ns, C, wv); break;
        case 18: stage_fused_r<18>(tile, addr, tw, L, Ns, C, wv); break;
        case 20: stage_fused_r<20>(tile, addr, tw, L, Ns, C, wv); break;
        case 21: stage_fused_r<21>(tile, addr, tw, L, Ns, C, wv); break;
        case 24: stage_fused_r<24>(tile, addr, tw, L, Ns, C, wv); break;
        case 25: stage_fused_r<25>(tile, addr, tw, L, Ns, C, wv); break;
        case 27: stage_fused_r<27>(tile, addr, tw, L, Ns, C, wv); break;
        case 28: stage_fused_r<28>(tile, addr, tw, L, Ns, C, wv); break;
        case 30: stage_fused_r<30>(tile, addr, tw, L, Ns, C, wv); break;
        case 32: stage_fused_r<32>(tile, addr, tw, L, Ns, C, wv); break;
        default: break;
    }
}

// The run-time policy.
struct DynFft {
    static constexpr int kThreads = 512, kMinBlocks = 1;
    static constexpr bool kBlue = false, kLiteral = false;
    static constexpr int kMaxLen = CWTHF_MAX_NG / 2;  // longest x pass (the x kernels keep a row in registers)
    static __device__ __forceinline__ int cols(const Plan& p) { return p.C; }
    static __device__ __forceinline__ int len(const Plan& p) { return p.L; }
    // DFT, or the unnormalised inverse: conj(DFT(conj(x))) with the conjugations as passes
    template <class A>
    static __device__ __forceinline__ void dft(const Plan& p, float2* t, A addr, const float2* tw, uint32_t sign) {
        const int n = p.L * p.C;
        if (sign) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = conjf2(t[i]);
            __syncthreads();
        }
        fft_tile(p, t, addr, tw);
        if (sign)
            for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = conjf2(t[i]);
    }
    template <class A>
    static __device__ __forceinline__ void wave(const Plan& p, float2* t, A addr, const float2* tw, const Wave& wv) {
        const int L = p.L, C = p.C, r0 = p.rad[0], r1 = p.rad[1], r2 = p.rad[2];
        if (p.nst == 1) {
            stage_fused(r0, t, addr, tw, L, 1, C, wv);
        } else if (p.nst == 2) {
            stage(r0, t, addr, tw, L, 1, C);
            stage_fused(r1, t, addr, tw, L, r0, C, wv);
            stage(r0, t, addr, tw, L, r1, C);
        } else {
            stage(r0, t, addr, tw, L, 1, C);
            stage(r1, t, addr, tw, L, r0, C);
            stage_fused(r2, t, addr, tw, L, r0 * r1, C, wv);
            stage(r1, t, addr, tw, L, r2, C);
            stage(r0, t, addr, tw, L, r2 * r1, C);
        }
        const int n = L * C;
        for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = conjf2(t[i]);
    }
};

}  // namespace

YzKernel dyn_yz() { return k_fft_yz<DynFft>; }
XFwdKernel dyn_x_fwd() { return k_fft_x_fwd<DynFft>; }
XInvKernel dyn_x_inv() { return k_fft_x_inv<DynFft>; }

}  // namespace fft
}  // namespace cwthf
