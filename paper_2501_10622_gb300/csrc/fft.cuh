// fft.cuh -- the device side of the grid CWT's FFT passes: butterflies, stages
// over shared-memory tiles, and the pass kernels.  The host side (plans,
// tables, launches) is in fft.cu; the compile-time instances are spread over
// fft_ct0.cu ... fft_ct7.cu and the run-time ones are in fft_dyn.cu, so that
// they compile in parallel.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "internal.cuh"

namespace cwthf {

struct Tables {
    int ng = 0;
    const float2* twN = nullptr;  // [ng]   exp(-2 pi i m / ng)
    const float2* twM = nullptr;  // [ng/2] exp(-2 pi i m / (ng/2))
    // Bluestein passes (null for passes with a radix plan): chirp b_n of the
    // pass length, the transformed chirp of the inner length (scaled by its
    // inverse), the inner length's twiddles
    const float2* chirp_yz = nullptr;
    const float2* bhat_yz = nullptr;
    const float2* tw_yz = nullptr;
    const float2* chirp_x = nullptr;
    const float2* bhat_x = nullptr;
    const float2* tw_x = nullptr;
};

namespace fft {

// ---------------------------------------------------------------------------
// Compile-time twiddle constants (series evaluated in fp64, rounded to fp32).
// ---------------------------------------------------------------------------
constexpr double kPi = 3.14159265358979323846264338327950288;

__host__ __device__ constexpr double cx_sin(double x) {
    double term = x, sum = x;
    for (int k = 1; k < 30; k++) {
        term *= -x * x / double((2 * k) * (2 * k + 1));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double cx_cos(double x) {
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 30; k++) {
        term *= -x * x / double((2 * k - 1) * (2 * k));
        sum += term;
    }
    return sum;
}
// angle 2 pi e / n reduced into [-pi, pi]
__host__ __device__ constexpr double cx_angle(int e, int n) {
    int r = ((e % n) + n) % n;
    if (2 * r > n) r -= n;
    return 2.0 * kPi * double(r) / double(n);
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }

// a * exp(-2 pi i E / N), exact for the quarter turns.
template <int N, int E>
__device__ __forceinline__ float2 mul_w(float2 a) {
    constexpr int e = ((E % N) + N) % N;
    if constexpr (e == 0) {
        return a;
    } else if constexpr (4 * e == N) {
        return make_float2(a.y, -a.x);
    } else if constexpr (2 * e == N) {
        return make_float2(-a.x, -a.y);
    } else if constexpr (4 * e == 3 * N) {
        return make_float2(-a.y, a.x);
    } else {
        constexpr float wr = float(cx_cos(cx_angle(e, N)));
        constexpr float wi = float(-cx_sin(cx_angle(e, N)));
        return make_float2(a.x * wr - a.y * wi, a.x * wi + a.y * wr);
    }
}

template <int I, int End, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < End) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, End>(f);
    }
}

// Smallest prime factor of n (2, 3, 5 or 7 for the supported radices).
__host__ __device__ constexpr int small_factor(int n) {
    return n % 2 == 0 ? 2 : (n % 3 == 0 ? 3 : (n % 5 == 0 ? 5 : 7));
}

// Position of output k of the in-place DIF below: for N = p*M, X[p*m + s]
// ends in block s at the position its length-M sub-transform gives m.
__host__ __device__ constexpr int dig_rev(int n, int k) {
    int pos = 0, base = 0;
    while (n > 1) {
        int p = small_factor(n), m = n / p;
        base += m * (k % p);
        k /= p;
        n = m;
    }
    return base + pos;
}

// In-register forward DFT of N values (N = 2^a 3^b 5^c 7^d), decimation in
// frequency, in place on v[OFF .. OFF+N): input in natural order, output
// X[k] at v[OFF + dig_rev(N, k)].  All indices are compile-time constants.
// Each step splits N = P M on the smallest prime P: for k < M the P inputs
// k + p M go through a P-point DFT, output q is multiplied by
// exp(-2 pi i q k / N) and kept in block q, whose length-M DFT follows.
template <int N>
struct RegDif {
    static constexpr int P = small_factor(N);
    static constexpr int M = N / P;
    template <int OFF>
    static __device__ __forceinline__ void run(float2* v) {
        if constexpr (N > 1) {
            if constexpr (P == 2) {
                static_for<0, M>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    float2 a = v[OFF + k], b = v[OFF + k + M];
                    v[OFF + k] = cadd(a, b);
                    v[OFF + k + M] = mul_w<N, k>(csub(a, b));
                });
            } else if constexpr (P == 3) {
                constexpr float h = 0.866025403784438646763723170752936f;  // sqrt(3)/2
                static_for<0, M>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    float2 a = v[OFF + k], b = v[OFF + k + M], c = v[OFF + k + 2 * M];
                    float2 t1 = cadd(b, c);
                    float2 t2 = make_float2(a.x - 0.5f * t1.x, a.y - 0.5f * t1.y);
                    float2 d = make_float2(h * (b.x - c.x), h * (b.y - c.y));
                    v[OFF + k] = cadd(a, t1);
                    v[OFF + k + M] = mul_w<N, k>(make_float2(t2.x + d.y, t2.y - d.x));          // t2 - i d
                    v[OFF + k + 2 * M] = mul_w<N, 2 * k>(make_float2(t2.x - d.y, t2.y + d.x));  // t2 + i d
                });
            } else {  // P = 5 or 7: the P-point DFT with constant roots
                static_for<0, M>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    float2 a[P];
                    static_for<0, P>([&](auto pc) { a[decltype(pc)::value] = v[OFF + k + decltype(pc)::value * M]; });
                    static_for<0, P>([&](auto qc) {
                        constexpr int q = decltype(qc)::value;
                        float2 y = a[0];
                        static_for<1, P>([&](auto pc) {
                            constexpr int pp = decltype(pc)::value;
                            y = cadd(y, mul_w<P, (pp * q) % P>(a[pp]));
                        });
                        v[OFF + k + q * M] = mul_w<N, q * k>(y);
                    });
                });
            }
            static_for<0, P>([&](auto sc) {
                constexpr int sblk = decltype(sc)::value;
                RegDif<M>::template run<OFF + sblk * M>(v);
            });
        }
    }
};

// ---------------------------------------------------------------------------
// Plans.  A shared-memory tile holds C sequences of length L; a pass runs at
// most three radix stages over it, in place.
// ---------------------------------------------------------------------------
constexpr int kRadices[] = {2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16, 18, 20, 21, 24, 25, 27, 28, 30, 32};

constexpr bool is_radix(int r) {
    for (int x : kRadices)
        if (x == r) return true;
    return false;
}

struct Radices {
    int n = 0;  // stages (0: no plan)
    int r[3] = {1, 1, 1};
};
// Up to three radices from kRadices whose product is L, maximising the
// smallest radix (fewest threads, least shared-memory traffic).
constexpr Radices make_radices(int L) {
    Radices p;
    int best = -1;
    if (is_radix(L)) {
        p.n = 1;
        p.r[0] = L;
        return p;
    }
    for (int a : kRadices) {
        if (L % a) continue;
        const int rem = L / a, m = a < rem ? a : rem;
        if (is_radix(rem) && m > best) {
            best = m;
            p.n = 2;
            p.r[0] = a;
            p.r[1] = rem;
        }
    }
    if (best > 0) return p;
    for (int a : kRadices) {
        if (L % a) continue;
        for (int b : kRadices) {
            if (L % (a * b)) continue;
            const int c = L / (a * b);
            if (!is_radix(c)) continue;
            const int m0 = a < b ? a : b, m = m0 < c ? m0 : c;
            if (m > best) {
                best = m;
                p.n = 3;
                p.r[0] = a;
                p.r[1] = b;
                p.r[2] = c;
            }
        }
    }
    return p;
}

struct Plan {
    int L;       // transform length (the inner length of a Bluestein pass)
    int nst;     // number of stages (1..3)
    int rad[3];  // radices, applied in this order (Ns = product of the earlier ones)
    int C;       // sequences per tile (a power of two)
    int T;       // threads per block (multiple of 32)
    int Lb = 0;  // Bluestein pass: the pass length (L >= 2 Lb - 1), else 0
    const float2* chirp = nullptr;  // [Lb] b_n = exp(i pi n^2 / Lb)
    const float2* bhat = nullptr;   // [L]  DFT_L of the wrapped chirp, divided by L
};

// Element l of sequence c of a tile.
struct AddrPlain {  // [L][C], row-major (TMA tiles)
    int C;
    __device__ __forceinline__ int operator()(int l, int c) const { return l * C + c; }
};
struct AddrSwz {  // [L][C] with the column XOR-swizzled by the row (C a power of 2)
    int C;
    __device__ __forceinline__ int operator()(int l, int c) const { return l * C + (c ^ (l & (C - 1))); }
};

// Wavelet multiply between the forward and inverse z transforms, done in the
// registers of the last forward stage: the thread that finishes forward
// butterfly j holds X[j + r L/R], exactly the inputs of inverse butterfly j of
// an inverse plan that starts with the same radix R.
struct Wave {
    float a, b;            // this column's coefficients: Psi^(kz) = a G^(kz) + b H^(kz)
    const float* gz;       // G^ table
    const float* hz;       // H^ table
};

__device__ __forceinline__ float flip(float x, uint32_t sign) { return __uint_as_float(__float_as_uint(x) ^ sign); }

// ---------------------------------------------------------------------------
// Compile-time plans: length, columns, radices and block size are constants,
// so index arithmetic folds to shifts and constants, everything inlines into
// the kernel (one register allocation, no calls), and the conjugations of the
// inverse transforms ride on the first load and the last store.  A thread
// takes as many butterflies per stage as the block size asks for; the stage is
// in place (every thread loads all of its butterflies, the block syncs, every
// thread stores them).
// ---------------------------------------------------------------------------
// What a stage does to its inputs and outputs beside the butterflies.
enum : int {
    kIoNone = 0,   // nothing
    kIoSign = 1,   // flips the imaginary parts by a run-time sign bit (conjugation or not)
    kIoChirp = 2   // Bluestein: inputs, after the sign flip, times conj(b_l), zero from row Lb on;
                   // outputs of the rows below Lb only, times b_l, conjugated, then sign-flipped
};
// The pointwise operation of a fused stage.
enum : int {
    kMidPsi = 0,   // times Psi^, conjugated (wavelet, then the inverse transform)
    kMidBhat = 1,  // times the transformed chirp, conjugated (between a Bluestein pass's transforms)
    kMidPad = 2    // times Psi^, zero from row Lb on: between the two Bluestein transforms of a wavelet
                   // pass, where the chirps of the first one's end and the second one's start cancel
};

struct Chirp {
    const float2* b;     // [Lb]
    const float2* bhat;  // [L]
    int Lb;
};

template <int L, int C, int T, int R, int Ns, int kIn, class A>
__device__ __forceinline__ void ct_load(const float2* tile, A addr, const float2* tw, int j, int c, uint32_t sign,
                                        const Chirp& ch, float2 (&v)[R]) {
    constexpr int NB = L / R;
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int l = j + r * NB;
        if constexpr (kIn == kIoChirp) {
            float2 x = make_float2(0.f, 0.f);
            if (l < ch.Lb) {
                x = tile[addr(l, c)];
                x.y = flip(x.y, sign);
                x = cmul(x, conjf2(__ldg(ch.b + l)));
            }
            v[r] = x;
        } else {
            v[r] = tile[addr(l, c)];
            if constexpr (kIn == kIoSign) v[r].y = flip(v[r].y, sign);
        }
    }
    if constexpr (Ns > 1) {
        const int k = j % Ns;
        constexpr int step = L / (Ns * R);
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = cmul(v[r], tw[r * k * step]);
    }
    RegDif<R>::template run<0>(v);
}

template <int R, int Ns, int kOut, class A>
__device__ __forceinline__ void ct_store(float2* tile, A addr, int j, int c, uint32_t sign, const Chirp& ch,
                                         const float2 (&v)[R]) {
    const int base = (j / Ns) * Ns * R + j % Ns;
    static_for<0, R>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        const int l = base + r * Ns;
        float2 x = v[dig_rev(R, r)];
        if constexpr (kOut == kIoChirp) {
            if (l < ch.Lb) {
                x = conjf2(cmul(x, __ldg(ch.b + l)));
                x.y = flip(x.y, sign);
                tile[addr(l, c)] = x;
            }
        } else {
            if constexpr (kOut == kIoSign) x.y = flip(x.y, sign);
            tile[addr(l, c)] = x;
        }
    });
}

// The butterflies of a thread: b = thread + k T < C L / R, sequence b % C
// (T is a multiple of C), butterfly b / C.
template <int L, int C, int T, int R, int Ns, int kIn, int kOut, class A>
__device__ __forceinline__ void stage_ct(float2* tile, A addr, const float2* tw, uint32_t sign, const Chirp& ch) {
    constexpr int NB = L / R, K = (NB * C + T - 1) / T;
    const int c = int(threadIdx.x) % C;
    float2 v[K][R];
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int b = int(threadIdx.x) + k * T;
        if (b < NB * C) ct_load<L, C, T, R, Ns, kIn>(tile, addr, tw, b / C, c, sign, ch, v[k]);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int b = int(threadIdx.x) + k * T;
        if (b < NB * C) ct_store<R, Ns, kOut>(tile, addr, b / C, c, sign, ch, v[k]);
    }
    __syncthreads();
}

// The fused stage: the last stage of one transform (Ns R = L), the pointwise
// operation, and the first stage of the next transform.
template <int L, int C, int T, int R, int kIn, int kMid, int kOut, class A>
__device__ __forceinline__ void fused_ct(float2* tile, A addr, const float2* tw, const Wave& wv, uint32_t sign,
                                         const Chirp& ch) {
    constexpr int NB = L / R, K = (NB * C + T - 1) / T;
    const int c = int(threadIdx.x) % C;
    float2 v[K][R];
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int b = int(threadIdx.x) + k * T, j = b / C;
        if (b < NB * C) {
            ct_load<L, C, T, R, NB, kIn>(tile, addr, tw, j, c, sign, ch, v[k]);
            float2 u[R];
            static_for<0, R>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                const int l = j + r * NB;
                const float2 x = v[k][dig_rev(R, r)];
                if constexpr (kMid == kMidBhat) {
                    u[r] = conjf2(cmul(x, __ldg(ch.bhat + l)));
                } else if constexpr (kMid == kMidPad) {
                    const float psi = l < ch.Lb ? wv.a * wv.gz[l] + wv.b * wv.hz[l] : 0.f;
                    u[r] = make_float2(x.x * psi, x.y * psi);
                } else {
                    const float psi = wv.a * wv.gz[l] + wv.b * wv.hz[l];
                    u[r] = make_float2(x.x * psi, -(x.y * psi));
                }
            });
#pragma unroll
            for (int r = 0; r < R; r++) v[k][r] = u[r];
            RegDif<R>::template run<0>(v[k]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int b = int(threadIdx.x) + k * T;
        if (b < NB * C) ct_store<R, 1, kOut>(tile, addr, b / C, c, sign, ch, v[k]);
    }
    __syncthreads();
}

constexpr int kSmemPerSm = 225 * 1024;

// Tile width and block size of a compile-time plan.
struct CtShape {
    int C, T, blocks;
};
constexpr int ct_threads(Radices p, int L, int C, int E) {  // with at most E values per thread and stage
    int t = 32;
    for (int s = 0; s < p.n; s++) {
        const int nb = C * (L / p.r[s]), k = E / p.r[s];
        const int need = (nb + k - 1) / k;
        t = need > t ? need : t;
    }
    return (t + 31) / 32 * 32;
}
// Eight sequences per tile (64-byte row segments in the y/z passes) while two
// tiles fit an SM, else four.  The fewest values per thread (at least the
// largest radix) with a block of at most 512 threads; as many blocks per SM as
// their tiles and about 2 E + 16 registers per thread allow.  (512 = 16 32 with
// 128 threads and two radix-16 butterflies each instead of 256 threads with
// one: the 512^3 transform 1.43 -> 1.27 ms.)
constexpr CtShape ct_shape(int L) {
    CtShape s{8, 0, 1};
    if (2 * L * 8 * s.C > kSmemPerSm) s.C = 4;
    const Radices p = make_radices(L);
    int rmax = 0;
    for (int i = 0; i < p.n; i++) rmax = p.r[i] > rmax ? p.r[i] : rmax;
    int E = rmax;
    while (E < 32 && ct_threads(p, L, s.C, E) > 512) E++;
    s.T = ct_threads(p, L, s.C, E);
    const int by_smem = kSmemPerSm / (L * 8 * s.C + 1200), by_regs = 65536 / (s.T * (2 * E + 16));
    s.blocks = by_smem < by_regs ? by_smem : by_regs;
    if (s.blocks < 1) s.blocks = 1;
    if (s.blocks > 2048 / s.T) s.blocks = 2048 / s.T;
    if (s.blocks > 16) s.blocks = 16;
    return s;
}

// What bounds these kernels and why they are compile-time: a pass moves each
// value once, but every stage also costs a shared-memory round trip, twiddle
// loads and index arithmetic.  With run-time lengths the divides, calls and
// generic (not shared-space) addresses cost more than the butterflies, and the
// thread-per-butterfly rule forced narrow tiles (two columns, 16-byte row
// segments, at 1000 = 10 10 10).  Whole transform, run-time kernels ->
// compile-time instances: 128^3 112 -> 52 us, 384^3 1.52 -> 0.56 ms, 640^3
// 6.1 -> 2.9 ms, 1000^3 33 -> 14 ms; the results are the same to the bit.
// Bluestein lengths: 190^3 0.88 -> 0.23 ms, 562^3 26.9 -> 6.2 ms, 1150^3
// 236 -> 67 ms (the chirps ride on the first loads and last stores, the
// pointwise products sit in fused stages, whole boxes of up to 256 rows).
//
// A transform policy: the tile FFTs a kernel runs, and its tile width.
// CtFft<L, blue> is the compile-time plan of length L; blue: a Bluestein pass
// of that inner length.  With nk = (n^2 + k^2 - (k - n)^2) / 2,
//   X_k = conj(b_k) sum_n (x_n conj(b_n)) b_(k-n),   b_n = exp(i pi n^2 / Lb),
// a circular convolution of length L >= 2 Lb - 1 done as DFT_L, a multiply by
// the DFT of the wrapped chirp, and a conjugated DFT_L (in reversed radix
// order, so that its first stage fuses with the last one before it).
template <int L_, bool kBlue_>
struct CtFft {
    static constexpr Radices kRad = make_radices(L_);
    static constexpr CtShape kShape = ct_shape(L_);
    static constexpr int C_ = kShape.C, T_ = kShape.T, N_ = kRad.n;
    static constexpr int R0 = kRad.r[0], R1 = kRad.r[1], R2 = kRad.r[2];
    static constexpr int kThreads = T_, kMinBlocks = kShape.blocks;
    static constexpr bool kBlue = kBlue_;
    static constexpr int kMaxLen = kBlue_ ? (L_ + 1) / 2 : L_;  // the longest pass
    // The x passes' row loops take the length as a literal for powers of two from 256 on, else at
    // run time.  The compiler contracts their products in another order with a literal, for some
    // lengths, so either choice is one of a length's last bits, on which near ties of the
    // segmentation hang; each length keeps the choice its results were made with.  In time: 1024^3
    // 10.52 ms with the literal, 11.07 without; 512^3 1.25 and 1.24; 640^3 (and others) the same.
    static constexpr bool kLiteral = !kBlue_ && L_ >= 256 && (L_ & (L_ - 1)) == 0;
    static_assert(N_ >= 1 && R0 * R1 * R2 == L_, "radices multiply to the length");
    static_assert(!kBlue_ || N_ >= 2, "a Bluestein plan has two or three stages");
    static __device__ __forceinline__ int cols(const Plan&) { return C_; }
    static __device__ __forceinline__ int len(const Plan& p) { return kBlue_ ? p.Lb : L_; }

    template <int R, int Ns, int kIn, int kOut, class A>
    static __device__ __forceinline__ void st(float2* t, A addr, const float2* tw, uint32_t sign, const Chirp& ch) {
        stage_ct<L_, C_, T_, R, Ns, kIn, kOut>(t, addr, tw, sign, ch);
    }
    template <int R, int kIn, int kMid, int kOut, class A>
    static __device__ __forceinline__ void fu(float2* t, A addr, const float2* tw, const Wave& wv, uint32_t sign,
                                              const Chirp& ch) {
        fused_ct<L_, C_, T_, R, kIn, kMid, kOut>(t, addr, tw, wv, sign, ch);
    }
    // the stages of a transform but the last (forward order; a first stage with kIn) ...
    template <int kIn, class A>
    static __device__ __forceinline__ void head(float2* t, A addr, const float2* tw, uint32_t sign, const Chirp& ch) {
        if constexpr (N_ >= 2) st<R0, 1, kIn, kIoNone>(t, addr, tw, sign, ch);
        if constexpr (N_ >= 3) st<R1, R0, kIoNone, kIoNone>(t, addr, tw, sign, ch);
    }
    // ... and the stages of the reversed transform but the first (a last stage with kOut)
    template <int kOut, class A>
    static __device__ __forceinline__ void tail(float2* t, A addr, const float2* tw, uint32_t sign, const Chirp& ch) {
        if constexpr (N_ >= 3) st<R1, R2, kIoNone, kIoNone>(t, addr, tw, sign, ch);
        if constexpr (N_ >= 2) st<R0, L_ / R0, kIoNone, kOut>(t, addr, tw, sign, ch);
    }
    static constexpr int RL = kRad.r[N_ - 1];  // last radix

    // DFT (sign = 0), or the unnormalised inverse (sign = the sign bit:
    // conjugated inputs and outputs)
    template <class A>
    static __device__ __forceinline__ void dft(const Plan& p, float2* t, A addr, const float2* tw, uint32_t sign) {
        const Chirp ch{p.chirp, p.bhat, p.Lb};
        if constexpr (kBlue_) {
            const Wave wv{0.f, 0.f, nullptr, nullptr};
            head<kIoChirp>(t, addr, tw, sign, ch);
            fu<RL, kIoNone, kMidBhat, kIoNone>(t, addr, tw, wv, 0u, ch);
            tail<kIoChirp>(t, addr, tw, sign, ch);
        } else if constexpr (N_ == 1) {
            st<R0, 1, kIoSign, kIoSign>(t, addr, tw, sign, ch);
        } else {
            head<kIoSign>(t, addr, tw, sign, ch);
            st<RL, L_ / RL, kIoNone, kIoSign>(t, addr, tw, sign, ch);
        }
    }
    // forward, multiply by Psi^, inverse
    template <class A>
    static __device__ __forceinline__ void wave(const Plan& p, float2* t, A addr, const float2* tw, const Wave& wv) {
        const Chirp ch{p.chirp, p.bhat, p.Lb};
        constexpr uint32_t kNeg = 0x80000000u;
        if constexpr (kBlue_) {
            // first transform up to its last stage, which is also the second one's first
            head<kIoChirp>(t, addr, tw, 0u, ch);
            fu<RL, kIoNone, kMidBhat, kIoNone>(t, addr, tw, wv, 0u, ch);
            if constexpr (N_ >= 3) st<R1, R2, kIoNone, kIoNone>(t, addr, tw, 0u, ch);
            fu<R0, kIoNone, kMidPad, kIoNone>(t, addr, tw, wv, 0u, ch);
            if constexpr (N_ >= 3) st<R1, R0, kIoNone, kIoNone>(t, addr, tw, 0u, ch);
            fu<RL, kIoNone, kMidBhat, kIoNone>(t, addr, tw, wv, 0u, ch);
            tail<kIoChirp>(t, addr, tw, kNeg, ch);
        } else if constexpr (N_ == 1) {
            fu<R0, kIoNone, kMidPsi, kIoSign>(t, addr, tw, wv, kNeg, ch);
        } else {
            head<kIoNone>(t, addr, tw, 0u, ch);
            fu<RL, kIoNone, kMidPsi, kIoNone>(t, addr, tw, wv, 0u, ch);
            tail<kIoSign>(t, addr, tw, kNeg, ch);
        }
    }
};

// ---------------------------------------------------------------------------
// TMA and mbarrier helpers (inline PTX).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// Bounded wait on phase `parity`; returns false if the limit was reached.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
    uint32_t a = smem_u32(bar);
    for (long long it = 0; it < limit; it++) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(src))
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit_and_drain() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------------------
// y / z pencil pass: one CTA transforms C adjacent columns of one plane.
// ---------------------------------------------------------------------------
enum YzMode : int { kYzForward = 0, kYzInverse = 1, kYzWavelet = 2 };

struct YzArgs {
    Plan p;
    int ncc;         // column chunks per plane
    int boxr;        // rows per TMA box
    int nbox;        // boxes per tile (boxr * nbox >= pass length: the last box may overhang the end of
                     // the axis, its loads read zeros there and its stores are clipped)
    int trows;       // tile rows: at least nbox * boxr and the plan's length
    int mode;
    int along_z;     // 1: transform along z (plane index o = y), 0: along y (o = z)
    int nplanes;     // planes (ng)
    int M;           // ng / 2 (highest valid kx)
    const float2* tw;   // [L]
    const float* ghat;  // [L]  G^(k)   (wavelet mode)
    const float* hhat;  // [L]  H^(k)
    float scale;        // w^1.5 * mass_unit / ng^3
    int* status;
    // fault injection (tests): CTA no_copy_block arms its barrier for the tile
    // but issues no copy, so its bounded wait (no_copy_spin polls) runs out
    // with nothing in flight; -1: off
    int no_copy_block;
    long long no_copy_spin;
};

// One CTA per tile: TMA brings the [L][C] pencil tile into shared memory
// (mbarrier completion), the block transforms it, TMA stores it back.
// Several CTAs per SM overlap their load, compute and store phases.
template <class F>
__global__ void __launch_bounds__(F::kThreads, F::kMinBlocks)
    k_fft_yz(const __grid_constant__ CUtensorMap in_map, const __grid_constant__ CUtensorMap out_map, YzArgs a) {
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Plan& p = a.p;
    const int C = F::cols(p);
    // TMA boxes land at 128-byte aligned offsets of the tile
    unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float2* tile = reinterpret_cast<float2*>(base);
    // twiddle and wavelet tables are read through the cache (three CTAs fit an SM)
    const float2* tw = a.tw;
    uint64_t* bar = reinterpret_cast<uint64_t*>(tile + a.trows * C);
    const int cc = blockIdx.x % a.ncc, o = blockIdx.x / a.ncc;

    const bool no_copy = int(blockIdx.x) == a.no_copy_block;
    if (threadIdx.x == 0) mbar_init(bar, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        // whole boxes (the last one may overhang the axis: the rows past it
        // arrive as zeros and count like the others)
        mbar_expect_tx(bar, uint32_t(a.nbox) * uint32_t(a.boxr) * C * 8u);
        for (int b = 0; b < a.nbox && !no_copy; b++) {
            const int r = b * a.boxr;
            if (a.along_z) tma_load_3d(tile + r * C, &in_map, bar, 2 * cc * C, o, r);
            else tma_load_3d(tile + r * C, &in_map, bar, 2 * cc * C, r, o);
        }
    }
    Wave wv{0.f, 0.f, a.ghat, a.hhat};
    if (a.mode == kYzWavelet) {
        // column c <-> kx = cc*C + c, this plane <-> ky = o
        const int kx = cc * C + int(threadIdx.x % C);
        if (kx <= a.M) {
            const float gx = a.ghat[kx], hx = a.hhat[kx], gy = a.ghat[o], hy = a.hhat[o];
            wv.a = a.scale * (6.f * gx * gy - hx * gy - gx * hy);
            wv.b = -a.scale * gx * gy;
        }
    }
    __syncthreads();
    // the whole block agrees on the outcome of its bounded wait before leaving
    // together.  After a timeout the call's results are unspecified (the status
    // word says so); a copy that is still outstanding gets a second bounded wait.
    const bool loaded = mbar_wait(bar, 0, no_copy ? a.no_copy_spin : kSpinLimit);
    if (__syncthreads_or(!loaded)) {
        if (threadIdx.x == 0) set_status(a.status, CWTHF_E_TIMEOUT);
        if (!no_copy) mbar_wait(bar, 0, kSpinLimit);
        return;
    }
    AddrPlain addr{C};
    if (a.mode == kYzWavelet) F::wave(p, tile, addr, tw, wv);  // forward, multiply, inverse
    else F::dft(p, tile, addr, tw, a.mode == kYzInverse ? 0x80000000u : 0u);
    fence_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int b = 0; b < a.nbox; b++) {
            const int r = b * a.boxr;
            if (a.along_z) tma_store_3d(&out_map, tile + r * C, 2 * cc * C, o, r);
            else tma_store_3d(&out_map, tile + r * C, 2 * cc * C, r, o);
        }
        tma_store_commit_and_drain();
    }
}

// ---------------------------------------------------------------------------
// x passes: C rows of one real transform each (plain coalesced loads).
// ---------------------------------------------------------------------------
struct XArgs {
    Plan p;          // complex FFT of length M = ng / 2 over C rows
    int ng, M, P;
    unsigned long long inv_ng;  // floor((2^64 - 1) / ng)
    int64_t rows;    // ng * ng
    const float2* twM;  // [M]   exp(-2 pi i m / M)  (Bluestein: the inner length's twiddles)
    const float2* twN;  // [ng]  exp(-2 pi i k / ng)
};

// floor(s / n) with inv = floor((2^64 - 1) / n): the high product is at most two
// short (s < 2^63).
__device__ __forceinline__ unsigned long long row_mean(unsigned long long s, unsigned n, unsigned long long inv) {
    unsigned long long q = __umul64hi(s, inv), r = s - q * n;
    if (r >= n) {
        q++;
        r -= n;
    }
    if (r >= n) q++;
    return q;
}

// Bound by DRAM and the latency of a tile's phases (1024^3: 12.9 GB in 3.0 ms);
// 64-bit conversions and a 64-bit divide per row took another 6 %.
template <class F>
__global__ void __launch_bounds__(F::kThreads, F::kMinBlocks) k_fft_x_fwd(XArgs a, const int64_t* grid,
                                                                          float2* __restrict__ spec) {
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Plan& p = a.p;
    const int M = F::kLiteral ? F::len(p) : a.M, C = F::cols(p);
    float2* tile = reinterpret_cast<float2*>(smem_raw);
    float2* tws = tile + a.p.L * C;
    double* rowdc = reinterpret_cast<double*>(tws + M);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const float2* tw = tws;
    if constexpr (F::kBlue) tw = a.twM;  // the inner length's twiddles, through the cache
    else
        for (int i = threadIdx.x; i < M; i += blockDim.x) tws[i] = a.twM[i];
    AddrSwz addr{C};
    // load, exact row sum, remove the row's integer mean exactly, round to fp32.
    // Dropping the mean's fractional part only shifts the row's DC bin, which is
    // replaced by the exact row sum below.  The spectrum is in units of 2^-30 of
    // the grid (mass_unit is applied with the wavelet).
    constexpr float kUnit = 9.3132257461547852e-10f;  // 2^-30, exact
    constexpr int kRowVec = (F::kMaxLen + 31) / 32;  // a row's int64 pairs per lane
    const bool vec = (reinterpret_cast<uintptr_t>(grid) & 15u) == 0;  // (rows are an even number of cells)
    for (int r = warp; r < C; r += nwarp) {
        int64_t row = int64_t(blockIdx.x) * C + r;
        longlong2 v[kRowVec];
        long long sum = 0;
        const int64_t* src = grid + row * a.ng;
        if (vec) {
#pragma unroll
            for (int i = 0; i < kRowVec; i++) {
                int k = lane + 32 * i;
                v[i] = (row < a.rows && k < M) ? reinterpret_cast<const longlong2*>(src)[k] : make_longlong2(0, 0);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kRowVec; i++) {
                int k = lane + 32 * i;
                v[i] = (row < a.rows && k < M) ? make_longlong2(src[2 * k], src[2 * k + 1]) : make_longlong2(0, 0);
            }
        }
#pragma unroll
        for (int i = 0; i < kRowVec; i++) sum += v[i].x + v[i].y;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const long long q0 = sum >= 0 ? (long long)row_mean((unsigned long long)sum, unsigned(a.ng), a.inv_ng) : sum / a.ng;
        if (lane == 0) rowdc[r] = double(__ll2float_rn(sum) * kUnit);
#pragma unroll
        for (int i = 0; i < kRowVec; i++) {
            int k = lane + 32 * i;
            if (k < M) {
                float re = ll2float(v[i].x - q0) * kUnit;
                float im = ll2float(v[i].y - q0) * kUnit;
                tile[addr(k, r)] = make_float2(re, im);
            }
        }
    }
    __syncthreads();
    F::dft(p, tile, addr, tw, 0u);
    // r2c post-processing: X[k] = (Z[k] + Z*[M-k])/2 - (i/2) W_N^k (Z[k] - Z*[M-k])
    for (int r = warp; r < C; r += nwarp) {
        int64_t row = int64_t(blockIdx.x) * C + r;
        if (row >= a.rows) continue;
        float2* out = spec + row * a.P;
        for (int k = lane; k <= M / 2; k += 32) {
            float2 zk = tile[addr(k, r)];
            float2 zm = tile[addr((M - k) % M, r)];
            if (k == 0) {
                out[0] = make_float2(float(rowdc[r]), 0.f);
                out[M] = make_float2(zk.x - zk.y, 0.f);
                continue;
            }
            float2 w = a.twN[k];
            // k side
            float2 e = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));   // (Z[k] + conj Z[M-k]) / 2
            float2 d = make_float2(0.5f * (zk.x - zm.x), 0.5f * (zk.y + zm.y));   // (Z[k] - conj Z[M-k]) / 2
            float2 wd = cmul(w, d);
            out[k] = make_float2(e.x + wd.y, e.y - wd.x);  // e - i w d
            if (2 * k != M) {
                // M-k side: the same with Z[k] and Z[M-k] swapped and W^(M-k) = -conj(W^k)
                float2 e2 = make_float2(e.x, -e.y);
                float2 d2 = make_float2(-d.x, d.y);
                float2 w2 = make_float2(-w.x, w.y);
                float2 wd2 = cmul(w2, d2);
                out[M - k] = make_float2(e2.x + wd2.y, e2.y - wd2.x);
            }
        }
        for (int k = M + 1 + lane; k < a.P; k += 32) out[k] = make_float2(0.f, 0.f);
    }
}

template <class F>
__global__ void __launch_bounds__(F::kThreads, F::kMinBlocks) k_fft_x_inv(XArgs a, const float2* spec,
                                                                          float* __restrict__ cwt) {
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Plan& p = a.p;
    const int M = F::kLiteral ? F::len(p) : a.M, C = F::cols(p);
    float2* tile = reinterpret_cast<float2*>(smem_raw);
    float2* tws = tile + a.p.L * C;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const float2* tw = tws;
    if constexpr (F::kBlue) tw = a.twM;
    else
        for (int i = threadIdx.x; i < M; i += blockDim.x) tws[i] = a.twM[i];
    AddrSwz addr{C};
    // c2r pre-processing: Z'[k] = (X[k] + X*[M-k]) + i W_N^-k (X[k] - X*[M-k]); stored conjugated.
    // All of a row's loads are issued before any is used (memory parallelism).
    for (int r = warp; r < C; r += nwarp) {
        int64_t row = int64_t(blockIdx.x) * C + r;
        const float2* in = spec + (row < a.rows ? row : 0) * a.P;
        constexpr int kPairs = F::kMaxLen / 64 + 1;  // k = lane + 32 i covers k <= M/2
        float2 xk[kPairs], xm[kPairs];
#pragma unroll
        for (int i = 0; i < kPairs; i++) {
            const int k = lane + 32 * i;
            if (k <= M / 2) {
                xk[i] = in[k];
                xm[i] = in[M - k];
            }
        }
#pragma unroll
        for (int i = 0; i < kPairs; i++) {
            const int k = lane + 32 * i;
            if (k > M / 2) continue;
            float2 a0 = xk[i], a1 = xm[i];
            if (k == 0) {
                a0.y = 0.f;
                a1.y = 0.f;
            }
            float2 e = make_float2(a0.x + a1.x, a0.y - a1.y);  // X[k] + conj X[M-k]
            float2 d = make_float2(a0.x - a1.x, a0.y + a1.y);  // X[k] - conj X[M-k]
            float2 winv = conjf2(a.twN[k]);                     // W_N^-k
            float2 wd = cmul(winv, d);
            float2 zk = make_float2(e.x - wd.y, e.y + wd.x);   // e + i W^-k d
            tile[addr(k, r)] = conjf2(zk);
            if (k != 0 && 2 * k != M) {
                float2 e2 = make_float2(e.x, -e.y);
                float2 d2 = make_float2(-d.x, d.y);
                float2 w2 = make_float2(-winv.x, winv.y);      // W_N^-(M-k) = -conj(W_N^-k)
                float2 wd2 = cmul(w2, d2);
                float2 zm = make_float2(e2.x - wd2.y, e2.y + wd2.x);
                tile[addr(M - k, r)] = conjf2(zm);
            }
        }
    }
    __syncthreads();
    F::dft(p, tile, addr, tw, 0u);
    const bool vec = (reinterpret_cast<uintptr_t>(cwt) & 7u) == 0;
    for (int r = warp; r < C; r += nwarp) {
        int64_t row = int64_t(blockIdx.x) * C + r;
        if (row >= a.rows) continue;
        float* out = cwt + row * a.ng;
        for (int n = lane; n < M; n += 32) {
            float2 z = tile[addr(n, r)];
            z.y = -z.y;  // conj back; z[n] = x[2n] + i x[2n+1]
            if (vec) {
                reinterpret_cast<float2*>(out)[n] = z;
            } else {
                out[2 * n] = z.x;
                out[2 * n + 1] = z.y;
            }
        }
    }
}


using YzKernel = void (*)(const CUtensorMap, const CUtensorMap, YzArgs);
using XFwdKernel = void (*)(XArgs, const int64_t*, float2*);
using XInvKernel = void (*)(XArgs, const float2*, float*);

// One compile-time length: its kernels (y/z only where a grid of that size
// exists), tile width and block size.
struct CtEntry {
    int L = 0;
    bool blue = false;
    int C = 0, T = 0;
    YzKernel yz = nullptr;
    XFwdKernel xf = nullptr;
    XInvKernel xi = nullptr;
};

// Compile-time lengths of radix passes: every 7-smooth length of a y/z pass
// (even, 8 .. 1152) or of an x pass (half of one).
constexpr bool smooth7(int n) {
    for (int p : {2, 3, 5, 7})
        while (n % p == 0) n /= p;
    return n == 1;
}
constexpr bool is_yz_len(int n) { return n >= CWTHF_MIN_NG && n <= CWTHF_MAX_NG && n % 2 == 0 && smooth7(n); }
constexpr bool is_x_len(int n) { return is_yz_len(2 * n); }

// Inner lengths of Bluestein passes (any other length): products of large
// radices, close enough together that every pass length Lb finds one between
// 2 Lb - 1 and 2.25 Lb + 64.
constexpr int kInner[] = {48,  64,  80,  96,  128, 144, 160, 192,  224,  256,  288,  320,  384,  448,  512,  576,
                          640, 720, 768, 864, 960, 1024, 1152, 1280, 1440, 1536, 1728, 1920, 2048, 2304};

// The entries of translation unit k (fft_ct<k>.cu) of kCtUnits.
constexpr int kCtUnits = 8;
template <int K>
void ct_entries(std::vector<CtEntry>& out);

// Run-time kernels, for the plans callers set (fft_dyn.cu).
YzKernel dyn_yz();
XFwdKernel dyn_x_fwd();
XInvKernel dyn_x_inv();

}  // namespace fft
}  // namespace cwthf
