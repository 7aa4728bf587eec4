// segment.cu -- local maxima and steepest-ascent segmentation of the CWT field
// (Sec. 2 steps 4-5, Sec. 2.3).
//
// Order on cells: a beats b iff C[a] > C[b], or C[a] == C[b] and a < b
// (a, b linear indices).  parent(c) = the best of c and its 26 periodic
// neighbours; c is a local maximum iff parent(c) == c.  A maximum with
// C > cwt_min is a seed; the label of a cell is the seed its parent chain
// reaches, or -1 when the chain ends at a maximum that is not a seed.
//
// k_seg_tile finds the parents of a tile's cells and keeps them as pointers in
// shared memory, resolves every chain that stays inside the tile, and writes
// the labels.  A chain that leaves the tile is written as a flagged pointer
// (-2 - g) to the first cell g outside; the global pass then replaces flagged
// pointers by the label of their target (bounded walks, then, only if a chain
// outlived them, pointer-doubling rounds in one cooperative launch; hitting the
// round bound is reported as CWTHF_E_NOT_CONVERGED).  The result does not
// depend on update order: every update moves a pointer further along the
// (unique) chain.
#include <cuda/atomic>

#include "internal.cuh"

namespace cwthf {
namespace {

// Chain tiles: 64 x 16 x 16 cells.  A warp owns kSegRows rows of 64 columns in
// every plane, each lane two adjacent columns.  A tile row's flagged cells go
// out as 32 masks: word 2 lz + p holds plane lz's columns of parity p (bit =
// lane).
constexpr int kChTX = 64, kChTY = 16, kChTZ = 16;
constexpr int kRowWords = 2 * kChTZ;  // flagged-cell masks per tile row (32)
constexpr int kSegRows = 2, kSegThreads = 32 * (kChTY / kSegRows);  // 256
static_assert(kRowWords == 32 && kChTX == 64, "mask layout");
// Shared-memory pointers: the 16-bit shared address of the target's own entry,
// in a box with one cell of halo on each side (rows padded to 68 entries, so
// that a lane's column pair is 4-byte aligned); a root points at itself.  One
// more entry stands for "no seed".  (The block's shared memory starts in the
// first few KB of the window, which the kernel checks.)
constexpr int kSRow = 2 * (kChTX + 4), kSPlane = kSRow * (kChTY + 2);  // bytes
constexpr int kSNone = kSPlane * (kChTZ + 2), kSBytes = kSNone + 8;
static_assert( kSRow == 136 && kSPlane == 2448, "quotient below");
// A flagged pointer (a chain still to be followed) to cell g is stored as
// -2 - g, apart from -1 (no seed) and the final labels (seed cells, >= 0).
__device__ __forceinline__ bool is_flagged(int32_t v) { return v <= -2; }
__device__ __forceinline__ int32_t flag_target(int32_t v) { return -2 - v; }
constexpr int kJumpRoundsInTile = 16;  // in-place jumping rounds (each triples the distance)
// Seeds of one tile: at most one local maximum per 2 x 2 x 2 block of cells
// (any two cells of such a block are neighbours).
constexpr int kTileSeedCap = (kChTX / 2) * (kChTY / 2) * (kChTZ / 2);
// pointers, the tile's seeds (addresses), cell counts of kCountSeeds of them at a time and of the rest, rows
constexpr int kCountSeeds = 1024;
constexpr int kSegLines = (kChTY + 2) * (kChTZ + 2);  // rows of the box, with their global indices
static_assert(kSBytes + 2 * kTileSeedCap + 4 * kCountSeeds < 60000, "16-bit addresses");
constexpr int kSegSmem =  // (a row for "no seed")
    kSBytes + 2 * kTileSeedCap + 4 * (kCountSeeds + 1) + 4 * (kSegLines + 1);

// o / kSRow for offsets o <= kSNone
constexpr uint32_t kYMul = 30841;
constexpr int kYShift = 22;

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Shared-memory accesses by 32-bit address: the pointers are addresses, so
// following one takes no arithmetic at all.  (Through C++ pointers every access
// recomputed the window's base; with that, branches and 64-bit addressing a
// cell took 186 instructions.)
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts16(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(uint16_t(v)));
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v)); }
__device__ __forceinline__ void reds32(uint32_t a, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v));
}

// The better of two candidates under the strict order, the first one coming
// earlier in position order: the second wins if it is greater, or, with `tie`
// (one of the two lies across the periodic boundary, which reverses their
// index order), if it is equal.
template <bool kInner>
__device__ __forceinline__ void best2(float m1, int q1, float m2, int q2, bool tie, float& m, int& q) {
    const bool w = kInner ? m2 > m1 : (m2 > m1 || (tie && m2 == m1));
    m = fmaxf(m1, m2);
    q = w ? q2 : q1;
}

// One tile.  The best of the 27 cells around c is the first cell, in wrapped
// (z, y, x) lexicographic order, holding the window's maximum, so it is found
// separably: the x windows of every row (shuffles), the y windows over the
// warp's rows, the z windows over the planes as they come.  Neighbouring
// windows of three share a pair (columns 2k, 2k+1; the warp's two rows), so two
// windows take three two-way choices instead of four.  Each choice carries the
// candidate's offset in the pointer array: the x choice is relative to the
// lane's first column, the row's offset rides in it as a constant, and the
// plane's is added once, so the z choice is the pointer itself.  kInner: the
// tile and its halo are clear of the periodic boundary.
//
// What bounds it and what it replaced: instruction issue, not DRAM.  Two
// kernels did this before (one-byte parent codes through memory, then a tile
// kernel that decoded them to 32-bit pointers): 250 instructions per cell,
// 3.34 + 4.52 ms per scale at 1024^3 and 0.26 + 0.26 ms at 384^3, against
// 4.47 and 0.27 ms here (of which the parents take half, the chains a fifth,
// the labels the rest).  16-bit pointers in a box with a halo need no decoding
// and no test for neighbours outside the tile, and leave room for four blocks
// per SM.  Two rows per warp rather than four: the halo rows' x windows cost 4
// instructions per cell more, but half the code and 64 registers per thread
// keep 32 warps on an SM (1024^3: 7.16 ms with four rows, 128 registers and 16
// warps).
template <bool kInner>
__device__ __forceinline__ void seg_tile(const float* __restrict__ C, int N, float cwt_min, int32_t* __restrict__ label,
                                         uint32_t* __restrict__ seed_bits, uint32_t* __restrict__ seed_cells,
                                         uint32_t* __restrict__ ballots, int* status, uint32_t sb, uint32_t* n_seeds) {
    const uint32_t seeds = sb + kSBytes, cnt = seeds + 2 * kTileSeedCap, line = cnt + 4 * (kCountSeeds + 1);
    const uint32_t none = sb + kSNone;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ntx = (N + kChTX - 1) / kChTX, nty = (N + kChTY - 1) / kChTY;
    const int t = int(blockIdx.x);
    const int tx = t % ntx, ty = (t / ntx) % nty, tz = t / (ntx * nty);
    const int x0 = tx * kChTX, y0 = ty * kChTY, z0 = tz * kChTZ;
    const int wx = min(kChTX, N - x0), wy = min(kChTY, N - y0), wz = min(kChTZ, N - z0);  // all even
    const int32_t plane = N * N;
    // every entry a root (the halo and what a ragged tile leaves out stay that way)
    for (uint32_t o = 4 * threadIdx.x; o < uint32_t(kSBytes); o += 4 * kSegThreads)
        sts32(sb + o, (sb + o) | ((sb + o + 2) << 16));
    // global index of each row's x = 0
    for (int i = threadIdx.x; i < kSegLines; i += kSegThreads) {
        const int z = z0 - 1 + i / (kChTY + 2), y = y0 - 1 + i % (kChTY + 2);
        sts32(line + 4 * i, uint32_t(kInner ? z * plane + y * N : ((z + N) % N) * plane + ((y + N) % N) * N));
    }
    // ("no seed" reads as a root whose label is -1)
    if (threadIdx.x == 0) sts32(line + 4 * kSegLines, uint32_t(-1 - (kInner ? x0 - 2 : wrap(x0 - 2, N))));
    __syncthreads();

    // ---- parents ----
    constexpr int R = kSegRows, NR = R + 2;
    const int lx = 2 * lane, r0 = warp * R;  // this lane's columns lx, lx + 1; the warp's rows r0 .. r0 + R - 1
    const int xa = kInner ? x0 + lx : (x0 + lx) % N;
    // lanes 0 and 31 fetch the columns beside the tile as well
    const int xe = kInner ? 0 : (lane == 0 ? (x0 - 1 + N) % N : (x0 + kChTX) % N);
    const bool first_lane = lane == 0, last_lane = lane == 31;
    uint32_t roff[NR];  // this lane's first column in the fetched rows of the plane fetched next
    const int zfirst = kInner ? z0 - 1 : (z0 - 1 + N) % N;
#pragma unroll
    for (int j = 0; j < NR; j++) {
        const int y = y0 + r0 - 1 + j;
        roff[j] = uint32_t(zfirst * plane + (kInner ? y : (y + N) % N) * N + xa);
    }
    int zf = zfirst;  // (boundary tiles) the plane fetched next
    const bool vec = (reinterpret_cast<uintptr_t>(C) & 7u) == 0;  // N and xa are even
    const bool tie_xl = !kInner && xa == 0, tie_xr = !kInner && xa + 1 == N - 1;
    bool bad = false;
    float2 va[NR];
    float ve[NR];
    auto fetch = [&]() {
#pragma unroll
        for (int j = 0; j < NR; j++) {
            const float* a = C + roff[j];
            if (vec) va[j] = *reinterpret_cast<const float2*>(a);
            else va[j] = make_float2(a[0], a[1]);
            if (kInner) {
                if (first_lane) ve[j] = a[-1];
                if (last_lane) ve[j] = a[2];
            } else if (first_lane || last_lane) {
                ve[j] = C[roff[j] - uint32_t(xa) + uint32_t(xe)];
            }
        }
        uint32_t step = uint32_t(plane);
        if (!kInner && ++zf == N) {
            zf = 0;
            step -= uint32_t(plane) * uint32_t(N);  // back to plane 0 (mod 2^32)
        }
#pragma unroll
        for (int j = 0; j < NR; j++) roff[j] += step;
    };
    // x and y windows of the plane fetched last; qz: the address of (that
    // plane, row r0 - 1, this lane's first column)
    auto xy = [&](float (&M)[2 * R], uint32_t (&Q)[2 * R], uint32_t qz) {
        float m[2 * NR];
        int q[2 * NR];
#pragma unroll
        for (int j = 0; j < NR; j++) {
            const float a = va[j].x, b = va[j].y;
            if (j >= 1 && j <= R) bad |= (a != a) | (b != b);  // (the halo rows are other warps')
            float l = __shfl_up_sync(full, b, 1), r = __shfl_down_sync(full, a, 1);
            if (first_lane) l = ve[j];
            if (last_lane) r = ve[j];
            const int o = j * kSRow;
            const float pm = fmaxf(a, b);
            const int pq = b > a ? o + 2 : o;
            best2<kInner>(l, o - 2, pm, pq, tie_xl, m[2 * j], q[2 * j]);
            best2<kInner>(pm, pq, r, o + 4, tie_xr, m[2 * j + 1], q[2 * j + 1]);
        }
#pragma unroll
        for (int k = 0; k < R; k += 2) {  // rows k, k + 1 of the warp (fetched rows k + 1, k + 2)
            const int y = y0 + r0 + k;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                float pm;
                int pq, qa, qb;
                best2<true>(m[2 * (k + 1) + c], q[2 * (k + 1) + c], m[2 * (k + 2) + c], q[2 * (k + 2) + c], false, pm, pq);
                best2<kInner>(m[2 * k + c], q[2 * k + c], pm, pq, !kInner && y == 0, M[2 * k + c], qa);
                best2<kInner>(pm, pq, m[2 * (k + 3) + c], q[2 * (k + 3) + c], !kInner && y + 1 == N - 1,
                              M[2 * (k + 1) + c], qb);
                Q[2 * k + c] = qz + uint32_t(qa);
                Q[2 * (k + 1) + c] = qz + uint32_t(qb);
            }
        }
    };
    const uint32_t lane0 = sb + uint32_t(r0 * kSRow + 2 * (lx + 2));  // (plane 0, row r0 - 1, column lx)
    const bool own_x = lx < wx;
    // the lane's seeds: bit 2 lz + c of its row's mask (listed after the planes: a seed in half of all rows of
    // 64 made the listing inside the loop a third of its instructions)
    uint32_t smask[R] = {};
    uint32_t bit = 1;
    // stores the pointers of tile plane p - 1 from the choices (m1, q1), (m2, q2) along z
    auto emit = [&](int p, const float (&m1)[2 * R], const uint32_t (&q1)[2 * R], const float (&m2)[2 * R],
                    const uint32_t (&q2)[2 * R], bool tie, bool first) {
        const uint32_t own0 = lane0 + uint32_t(p * kSPlane + kSRow), half = sb + uint32_t(kSPlane);
#pragma unroll
        for (int k = 0; k < R; k++) {
            const uint32_t own = own0 + uint32_t(k * kSRow);
            const bool in = own_x && r0 + k < wy;
            uint32_t q[2];
            // (first: the pair's choice may lie in the plane across the boundary, which loses ties)
#pragma unroll
            for (int c = 0; c < 2; c++) {
                const int i = 2 * k + c;
                const bool w = kInner ? m2[i] > m1[i]
                                      : (m2[i] > m1[i] || ((tie || (first && q1[i] < half)) && m2[i] == m1[i]));
                const float m = fmaxf(m1[i], m2[i]);
                q[c] = w ? q2[i] : q1[i];
                if (q[c] == own + 2 * c) {  // a local maximum
                    if (!(m > cwt_min)) q[c] = none;
                    else if (in) smask[k] |= bit << c;
                }
            }
            if (in) sts32(own, q[0] | (q[1] << 16));
        }
        bit <<= 2;
    };
    // along z: the better of the last two planes, and the last plane
    float mP[2 * R], mL[2 * R], mN[2 * R];
    uint32_t qP[2 * R], qL[2 * R], qN[2 * R];
    fetch();
    xy(mP, qP, lane0);
    fetch();
    xy(mL, qL, lane0 + kSPlane);
    fetch();
    // planes 0 and 1: the first one wins ties unless it lies across the boundary
#pragma unroll
    for (int i = 0; i < 2 * R; i++) {
        const bool w = mL[i] > mP[i] || (!kInner && z0 == 0 && mL[i] == mP[i]);
        mP[i] = fmaxf(mP[i], mL[i]);
        qP[i] = w ? qL[i] : qP[i];
    }
#pragma unroll 1
    for (int p = 1; p <= wz; p++) {
        xy(mN, qN, lane0 + uint32_t((p + 1) * kSPlane));
        if (p < wz) fetch();
        emit(p, mP, qP, mN, qN, !kInner && z0 + p == N, !kInner && z0 == 0 && p == 1);
#pragma unroll
        for (int i = 0; i < 2 * R; i++) {
            const bool w = mN[i] > mL[i];
            mP[i] = fmaxf(mL[i], mN[i]);
            qP[i] = w ? qN[i] : qL[i];
            mL[i] = mN[i];
            qL[i] = qN[i];
        }
    }
    if (bad) set_status(status, CWTHF_E_BAD_INPUT);
    const uint32_t mine = lane0 + kSPlane + kSRow;  // (plane lz 0, row r0)
    {  // list the warp's seeds
        uint32_t n = 0;
#pragma unroll
        for (int k = 0; k < R; k++) n += uint32_t(__popc(smask[k]));
        uint32_t incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t j = 0;
        if (last_lane && incl) j = atomicAdd(n_seeds, incl);
        j = __shfl_sync(full, j, 31) + incl - n;
#pragma unroll
        for (int k = 0; k < R; k++)
            for (uint32_t m = smask[k]; m; m &= m - 1, j++) {
                const int i = __ffs(m) - 1;
                if (j < uint32_t(kTileSeedCap))
                    sts16(seeds + 2 * j, mine + uint32_t(k * kSRow + (i >> 1) * kSPlane + 2 * (i & 1)));
            }
    }
    __syncthreads();

    // ---- chains inside the tile: pointer jumping in place, every cell in
    // lockstep; a pointer takes its target's target's target, until every
    // pointer names a root.  A value read while another thread rewrites it is
    // the old or the new pointer, both points of the same chain.  The loads of
    // kBatch pairs go together. ----
    constexpr int kBatch = 8;
    auto ok = [&](uint32_t u) { return index_ok(int64_t(u) - int64_t(sb), kSBytes, status); };
    for (int round = 0; round < kJumpRoundsInTile; round++) {
        bool more = false;
#pragma unroll 1
        for (int i0 = 0; i0 < R * kChTZ; i0 += kBatch) {  // plane pairs of row i0 / kChTZ
            const uint32_t a0 = mine + uint32_t((i0 / kChTZ) * kSRow + (i0 % kChTZ) * kSPlane);
            uint32_t u[kBatch], t0[kBatch], t1[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; i++) u[i] = lds32(a0 + i * kSPlane);
#pragma unroll
            for (int i = 0; i < kBatch; i++) {
                t0[i] = ok(u[i] & 0xffffu) ? lds16(u[i] & 0xffffu) : u[i] & 0xffffu;
                t1[i] = ok(u[i] >> 16) ? lds16(u[i] >> 16) : u[i] >> 16;
            }
#pragma unroll
            for (int i = 0; i < kBatch; i++) {
                const uint32_t tt = t0[i] | (t1[i] << 16);
                if (tt != u[i]) {
                    const uint32_t w = lds16(t0[i]) | (lds16(t1[i]) << 16);
                    sts32(a0 + i * kSPlane, w);
                    more |= w != tt;
                }
            }
        }
        if (!__syncthreads_or(more)) break;
    }
    // global index of the cell of the entry at address u (inside the tile or in its halo)
    const uint32_t bias = sb * kYMul;
    const int xb = 2 * (x0 - 2) - int(sb);
    auto cell_at = [&](uint32_t u) -> int32_t {
        const uint32_t r = (u * kYMul - bias) >> kYShift;
        const int x = (int(u - r * uint32_t(kSRow)) + xb) >> 1;
        return int32_t(lds32(line + 4 * r)) + (kInner ? x : wrap(x, N));
    };
    // each seed's entry now holds the address of its counter (odd: addresses of entries are even), seeds
    // beyond the counters share one that is not read
    const uint32_t ns = min(*n_seeds, uint32_t(kTileSeedCap));
    if (threadIdx.x == 0 && *n_seeds > uint32_t(kTileSeedCap)) set_status(status, CWTHF_E_BAD_INPUT);
    auto mark = [&](uint32_t j0) {  // counters of seeds j0 .. j0 + kCountSeeds - 1
        for (uint32_t j = threadIdx.x; j < ns; j += kSegThreads)
            sts16(lds16(seeds + 2 * j), cnt + 4 * min(j - j0, uint32_t(kCountSeeds)) + 1);
        for (uint32_t j = threadIdx.x; j <= uint32_t(kCountSeeds); j += kSegThreads) sts32(cnt + 4 * j, 0u);
        if (threadIdx.x == 0) sts16(none, cnt + 4 * kCountSeeds + 1);
    };
    for (uint32_t j = threadIdx.x; j < ns; j += kSegThreads) {
        const uint32_t g = uint32_t(cell_at(lds16(seeds + 2 * j)));
        atomicOr(&seed_bits[g >> 5], 1u << (g & 31));
    }
    mark(0);
    __syncthreads();

    // ---- labels, and one count per cell for the tile's seeds ----
    auto finish = [&](uint32_t u, uint32_t own, uint32_t& flags, uint32_t fbit) -> int32_t {
        u = (u & 1u) ? own : u;  // a seed's own entry
        const uint32_t e = ok(u) ? lds16(u) : u;
        const int32_t g = cell_at(u);
        if (e & 1u) {
            reds32(e - 1, 1u);
            return g;
        }
        flags |= fbit;  // outside the tile (or not finished within the round bound)
        return -2 - g;
    };
    const bool lvec = (reinterpret_cast<uintptr_t>(label) & 7u) == 0;  // even cells: 8-byte label pairs
#pragma unroll 1
    for (int k = 0; k < R; k++) {
        const bool own = own_x && r0 + k < wy;
        int32_t* out = label + (size_t(z0) * N + (y0 + r0 + k)) * N + x0 + lx;
        uint32_t flags = 0;  // bit 2 lz + p: this lane's cell of plane lz, column parity p is flagged
        if (own) {
            uint32_t o = mine + uint32_t(k * kSRow), fbit = 1;
#pragma unroll 4
            for (int lz = 0; lz < wz; lz++, out += plane, o += kSPlane, fbit <<= 2) {
                const uint32_t u = lds32(o);
                int2 res;
                res.x = finish(u & 0xffffu, o, flags, fbit);
                res.y = finish(u >> 16, o + 2, flags, fbit << 1);
                if (lvec) {
                    *reinterpret_cast<int2*>(out) = res;
                } else {
                    out[0] = res.x;
                    out[1] = res.y;
                }
            }
        }
        __syncwarp();
        // transposed over the warp: word w (lane w) gets bit w of every lane
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const uint32_t low = d == 16 ? 0x0000ffffu
                               : d == 8  ? 0x00ff00ffu
                               : d == 4  ? 0x0f0f0f0fu
                               : d == 2  ? 0x33333333u
                                         : 0x55555555u;
            const uint32_t other = __shfl_xor_sync(full, flags, d);
            flags = (lane & d) ? ((flags & ~low) | ((other & ~low) >> d)) : ((flags & low) | ((other & low) << d));
        }
        ballots[(size_t(t) * kChTY + r0 + k) * kRowWords + lane] = flags;
    }
    __syncthreads();
    // in-tile cell counts of this tile's seeds (cells reaching them from other
    // tiles are added by the global pass)
    for (uint32_t j0 = 0;;) {  // one turn but for tiles of more than kCountSeeds seeds
        for (uint32_t j = j0 + threadIdx.x; j < min(ns, j0 + uint32_t(kCountSeeds)); j += kSegThreads)
            seed_cells[size_t(cell_at(lds16(seeds + 2 * j)))] = lds32(cnt + 4 * (j - j0));
        j0 += uint32_t(kCountSeeds);
        if (j0 >= ns) break;  // block-uniform
        __syncthreads();
        mark(j0);
        __syncthreads();
        for (int k = 0; k < R; k++)
            if (own_x && r0 + k < wy)
                for (int lz = 0; lz < wz; lz++) {
                    const uint32_t o = mine + uint32_t(k * kSRow + lz * kSPlane), w = lds32(o);
                    for (int c = 0; c < 2; c++) {
                        const uint32_t u = c ? w >> 16 : w & 0xffffu;
                        const uint32_t e = (u & 1u) ? u : (ok(u) ? lds16(u) : u);
                        if (e & 1u) reds32(e - 1, 1u);
                    }
                }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kSegThreads, 4) k_seg_tile(const float* C, int ng, float cwt_min,
                                                             int32_t* __restrict__ label,
                                                             uint32_t* __restrict__ seed_bits,
                                                             uint32_t* __restrict__ seed_cells,
                                                             uint32_t* __restrict__ ballots, int* status) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char seg_smem[];
    __shared__ uint32_t n_seeds;
    if (threadIdx.x == 0) n_seeds = 0;  // (the tile's first barrier is before its first use)
    const uint32_t sb = uint32_t(__cvta_generic_to_shared(seg_smem));
    if (sb + uint32_t(kSegSmem) > 65535u) {  // pointers would not fit 16 bits: cannot happen (see above)
        set_status(status, CWTHF_E_CUDA);
        return;
    }
    const int ntx = (ng + kChTX - 1) / kChTX, nty = (ng + kChTY - 1) / kChTY;
    const int t = int(blockIdx.x), tx = t % ntx, ty = (t / ntx) % nty, tz = t / (ntx * nty);
    const bool inner = tx > 0 && (tx + 1) * kChTX < ng && ty > 0 && (ty + 1) * kChTY < ng && tz > 0 &&
                       (tz + 1) * kChTZ < ng;
    if (inner) seg_tile<true>(C, ng, cwt_min, label, seed_bits, seed_cells, ballots, status, sb, &n_seeds);
    else seg_tile<false>(C, ng, cwt_min, label, seed_bits, seed_cells, ballots, status, sb, &n_seeds);
}

constexpr int kResolveThreads = 256;
constexpr int kResTabBits = 10, kResTab = 1 << kResTabBits;  // per-tile count table (shared memory)

// The global pass over the cells whose chain left their tile.  A CTA takes
// `rows` rows of chain tiles at a time from a global counter, and its warps
// take them one at a time from a shared counter (the flagged cells crowd where
// the field is clumped, so a fixed split leaves some warps far more work than
// others).  A warp gathers the flagged cells of a row's non-empty plane masks
// into a shared batch; every full batch of 32 cells (and the warp's last,
// partial one) is resolved by the whole warp: each lane follows its cell's
// chain through the label grid (at most `limit` steps, kDefaultChaseLimit by
// default) and takes the label it reaches.  The cells are counted per seed in a
// shared table (one entry per distinct seed, one shared atomic per distinct
// seed of a batch) that is added to the counts kept at the seeds' cells once
// per turn (the tile pass wrote each seed's in-tile count there; seed slots are
// ranked only afterwards).  A cell still unfinished at the limit stays flagged
// and sets changed[0]; the doubling rounds then finish it and the cells are
// recounted.  Labels read while other threads update them are always a later
// point of the same chain, so the result does not depend on timing.
__device__ __forceinline__ void table_add(int32_t* tkey, uint32_t* tcnt, uint32_t* __restrict__ seed_cells,
                                          int32_t lab, uint32_t n) {
    uint32_t h = (uint32_t(lab) * 2654435761u) >> (32 - kResTabBits);
    for (int p = 0; p < 16; p++) {
        const int32_t k = tkey[h];
        if (k == lab) {
            atomicAdd(&tcnt[h], n);
            return;
        }
        if (k == -1) {
            const int32_t prev = atomicCAS(&tkey[h], -1, lab);
            if (prev == -1 || prev == lab) {
                atomicAdd(&tcnt[h], n);
                return;
            }
        }
        h = (h + 1) & (kResTab - 1);
    }
    atomicAdd(&seed_cells[lab], n);  // table crowded: straight to the seed's count
}

__device__ __forceinline__ void resolve_batch(int32_t* __restrict__ label, bool valid, uint32_t c, int32_t* tkey,
                                              uint32_t* tcnt, uint32_t* __restrict__ seed_cells, int limit,
                                              bool& left, int64_t cells, int* status) {
    int32_t lab = -1;
    if (valid) {
        int32_t w = label[c];
        int steps = 0;
        while (is_flagged(w) && steps < limit) {
            if (!index_ok(flag_target(w), cells, status)) {
                w = -1;
                break;
            }
            w = label[flag_target(w)];
            steps++;
        }
        label[c] = w;
        if (is_flagged(w)) left = true;
        else lab = w;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, lab);  // every lane
    if (lab >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1)
        table_add(tkey, tcnt, seed_cells, lab, uint32_t(__popc(peers)));
}

__global__ void __launch_bounds__(kResolveThreads) k_seg_resolve(int32_t* __restrict__ label, int ng,
                                                                 const uint32_t* ballots,
                                                                 uint32_t* __restrict__ seed_cells,
                                                                 int* __restrict__ changed,
                                                                 unsigned* __restrict__ next_rows, int limit,
                                                                 int rows, int* status) {
    pdl_wait();
    __shared__ uint32_t batch[kResolveThreads / 32][64];  // pending cells (fewer than 32 between batches)
    __shared__ int32_t tkey[kResTab];
    __shared__ uint32_t tcnt[kResTab];
    __shared__ unsigned s_end, s_row;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t* wl = batch[threadIdx.x >> 5];
    const int N = ng;
    const int ntx = (N + kChTX - 1) / kChTX, nty = (N + kChTY - 1) / kChTY, ntz = (N + kChTZ - 1) / kChTZ;
    const unsigned nrows = unsigned(ntx) * unsigned(nty) * unsigned(ntz) * unsigned(kChTY);  // rows of all tiles
    const uint32_t plane32 = uint32_t(N) * uint32_t(N);
    const int64_t cells = int64_t(plane32) * N;
    for (int i = threadIdx.x; i < kResTab; i += blockDim.x) {
        tkey[i] = -1;
        tcnt[i] = 0;
    }
    bool left = false;
    for (;;) {
        if (threadIdx.x == 0) {
            const unsigned r = atomicAdd(next_rows, 1u) * unsigned(rows);  // (far below 2^32: CTAs stop at nrows)
            s_row = r;
            s_end = r < nrows ? min(nrows, r + unsigned(rows)) : 0u;
        }
        __syncthreads();
        const unsigned row_end = s_end;
        if (row_end == 0u) break;  // block-uniform
        uint32_t k = 0;  // warp-uniform
        for (;;) {
            unsigned rw = 0;
            if (lane == 0) rw = atomicAdd(&s_row, 1u);
            rw = __shfl_sync(full, rw, 0);
            if (rw >= row_end) break;  // warp-uniform
            const unsigned t = rw / unsigned(kChTY), ly = rw % unsigned(kChTY);
            const int tx = int(t % unsigned(ntx)), ty = int((t / unsigned(ntx)) % unsigned(nty)),
                      tz = int(t / (unsigned(ntx) * unsigned(nty)));
            const int yc = ty * kChTY + int(ly);
            if (yc >= N) continue;  // warp-uniform
            const uint32_t mine = ballots[size_t(rw) * kRowWords + lane];  // plane lane / 2, columns of parity lane % 2
            uint32_t words = __ballot_sync(full, mine != 0u);
            const uint32_t cell0 =
                uint32_t((int64_t(tz) * kChTZ * N + yc) * N + int64_t(tx) * kChTX) + 2u * uint32_t(lane);
            while (words) {
                const int wd = __ffs(words) - 1;
                words &= words - 1u;
                const uint32_t b = __shfl_sync(full, mine, wd);
                if (b & (1u << lane)) wl[k + __popc(b & lt)] = cell0 + uint32_t(wd >> 1) * plane32 + uint32_t(wd & 1);
                k += __popc(b);
                if (k >= 32) {
                    __syncwarp();
                    resolve_batch(label, true, wl[lane], tkey, tcnt, seed_cells, limit, left, cells, status);
                    const uint32_t rest = wl[32 + lane];
                    __syncwarp();
                    if (uint32_t(lane) + 32 < k) wl[lane] = rest;
                    k -= 32;
                    __syncwarp();
                }
            }
        }
        __syncwarp();
        if (k)
            resolve_batch(label, uint32_t(lane) < k, uint32_t(lane) < k ? wl[lane] : 0u, tkey, tcnt, seed_cells,
                          limit, left, cells, status);
        __syncthreads();
        // the rows' counts go to the seeds' cells; the table is cleared for the next ones
        for (int i = threadIdx.x; i < kResTab; i += blockDim.x) {
            const int32_t key = tkey[i];
            if (key >= 0) {
                atomicAdd(&seed_cells[key], tcnt[i]);
                tkey[i] = -1;
                tcnt[i] = 0;
            }
        }
        __syncthreads();
    }
    if (__any_sync(full, left) && lane == 0) changed[0] = 1;
}

// Fallback for chains that outlived the bounded walks (changed[0] set by the
// resolve pass); returns at once otherwise.  Round r (1 <= r <= rounds)
// replaces every flagged pointer by its target's label, which moves it 2^(r-1)
// or more links further, so 31 rounds finish any chain of a grid of at most
// 2^30 cells; changed[r] records whether a pointer is still flagged after it.
// Rounds are separated by grid barriers.  Then the cell counts of every seed
// (kept at the seed's cell) are cleared and recounted from the finished
// labels.  A flag still set after
// the last round is reported as CWTHF_E_NOT_CONVERGED (the labels are then
// unspecified, and flagged values are skipped by the recount).
__global__ void __launch_bounds__(256) k_seg_fallback(int32_t* __restrict__ label, int64_t cells, int* changed,
                                                      int rounds, const uint32_t* bits,
                                                      uint32_t* __restrict__ seed_cells, unsigned* bar, int* status) {
    pdl_wait();
    if (*reinterpret_cast<volatile int*>(&changed[0]) == 0) return;  // the same answer in every CTA
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t gid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    bool done = false;
    for (int r = 1; r <= rounds; r++) {
        bool any = false;
        for (int64_t c = gid; c < cells; c += stride) {
            const int32_t v = label[c];
            if (is_flagged(v) && index_ok(flag_target(v), cells, status)) {
                const int32_t w = label[flag_target(v)];
                label[c] = w;
                any |= is_flagged(w);  // still a pointer: another round is needed
            }
        }
        if (__any_sync(0xffffffffu, any) && (threadIdx.x & 31) == 0) atomicOr(&changed[r], 1);
        if (!grid_sync(bar, status)) return;
        if (*reinterpret_cast<volatile int*>(&changed[r]) == 0) {
            done = true;
            break;
        }
    }
    if (!done && gid == 0) set_status(status, CWTHF_E_NOT_CONVERGED);
    auto is_seed = [&](int64_t c) { return (bits[c >> 5] >> (c & 31)) & 1u; };
    for (int64_t c = gid; c < cells; c += stride)
        if (is_seed(c)) seed_cells[c] = 0;
    if (!grid_sync(bar, status)) return;
    for (int64_t c = gid; c < cells; c += stride) {
        const int32_t l = label[c];
        if (l >= 0 && int64_t(l) < cells && is_seed(l)) atomicAdd(&seed_cells[l], 1u);
    }
}

// slot -> seed cell, in increasing cell order.  *n_slots = number of seeds,
// clamped to slot_cap (more seeds than that can only come from an inconsistent
// label grid, reported as bad input).
__global__ void k_seed_list(const uint32_t* bits, const uint32_t* prefix, int64_t nwords,
                            int64_t slot_cap, int32_t* __restrict__ seed_list, uint32_t* __restrict__ n_slots,
                            int* status) {
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        uint32_t total = prefix[nwords];
        if (int64_t(total) > slot_cap) set_status(status, CWTHF_E_BAD_INPUT);
        *n_slots = uint32_t(min(int64_t(total), slot_cap));
    }
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < nwords; i += stride) {
        uint32_t b = bits[i];
        if (!b) continue;
        uint32_t s = prefix[i];
        while (b && int64_t(s) < slot_cap) {
            seed_list[s++] = int32_t(i * 32 + __ffs(b) - 1);
            b &= b - 1;
        }
    }
}

// Clears the slots' accumulators; the cell count starts from the tile pass's
// count at the seed's cell when given.  With the clearing inside the list's
// loop over the bitmap, each seed's gather and 48 bytes of stores waited for the
// seed before it in the same word (0.68 ms per scale at 1024^3, 0.14 + 0.40 now).
__global__ void k_seed_acc(const int32_t* seed_list, const uint32_t* seed_cells,
                           HaloAcc* __restrict__ acc, const uint32_t* n_slots) {
    pdl_wait();
    // an accumulator is three 16-byte pieces, all zero but the count in the last one's upper half; one
    // thread per piece, so that a warp's stores are contiguous
    static_assert(sizeof(HaloAcc) == 48 && offsetof(HaloAcc, n_cells) == 40, "piece layout");
    const uint64_t n = uint64_t(*n_slots) * 3;
    ulonglong2* out = reinterpret_cast<ulonglong2*>(acc);
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t s = uint32_t(i / 3);
        out[i] = make_ulonglong2(0ull, seed_cells && i == 3ull * s + 2 ? seed_cells[seed_list[s]] : 0ull);
    }
}

// Seeds from a label grid: the cells labelled with their own index.
__global__ void k_seeds_from_labels(const int32_t* label, int64_t cells, uint32_t* __restrict__ bits,
                                    int* status) {
    pdl_wait();
    constexpr int kIlp = 4;  // labels in flight (one at a time: 256^3 37 us, 28 with four)
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t c0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; c0 < cells; c0 += kIlp * stride) {
        int32_t l[kIlp];
#pragma unroll
        for (int u = 0; u < kIlp; u++) l[u] = c0 + u * stride < cells ? label[c0 + u * stride] : -1;
#pragma unroll
        for (int u = 0; u < kIlp; u++) {
            const int64_t c = c0 + u * stride;
            if (l[u] < -1 || l[u] >= cells) set_status(status, CWTHF_E_BAD_INPUT);
            if (l[u] == c) atomicOr(&bits[c >> 5], 1u << (c & 31));
        }
    }
}

// Seeds of the last segmentation and their segments' cell counts.
__global__ void k_segment_sizes(const int32_t* seed_list, const HaloAcc* acc,
                                const uint32_t* n_slots, int64_t cap, int32_t* __restrict__ seeds,
                                int64_t* __restrict__ n_cells, int64_t* __restrict__ n_out) {
    pdl_wait();
    const int64_t ns = *n_slots;
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_out = ns;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < min(ns, cap); i += stride) {
        seeds[i] = seed_list[i];
        n_cells[i] = int64_t(acc[i].n_cells);
    }
}

}  // namespace

int segment_sizes_impl(cwthf_ctx* ctx, int32_t* seeds, int64_t* n_cells, int64_t cap, int64_t* n_seeds,
                       cudaStream_t s) {
    CWTHF_LAUNCH(ctx, s, "k_segment_sizes",
                 pdl(k_segment_sizes, ctx->sm_count, 256, 0, s)(ctx->seed_list, ctx->acc, ctx->n_seeds, cap, seeds,
                                                               n_cells, n_seeds));
    return cuda_status(cudaGetLastError());
}

int seeds_rank(cwthf_ctx* ctx, int ng, const uint32_t* seed_cells, cudaStream_t s) {
    int64_t cells = int64_t(ng) * ng * ng;
    int64_t nwords = (cells + 31) / 32;
    const int blocks = int(std::min<int64_t>(div_up(nwords, 256), int64_t(ctx->sm_count) * 8));
    // (at most a seed per 8 cells)
    const int sblocks = int(std::min<int64_t>(div_up(3 * cells / 8, 256), int64_t(ctx->sm_count) * 8));
    int rc = scan_popc(ctx, ctx->seed_bits, ctx->seed_prefix, nwords, s);
    if (rc) return rc;
    CWTHF_LAUNCH(ctx, s, "k_seed_list",
                 pdl(k_seed_list, blocks, 256, 0, s)(ctx->seed_bits, ctx->seed_prefix, nwords, cells / 8 + 8,
                                                    ctx->seed_list, ctx->n_seeds, ctx->d_status));
    CWTHF_LAUNCH(ctx, s, "k_seed_acc",
                 pdl(k_seed_acc, sblocks, 256, 0, s)(ctx->seed_list, seed_cells, ctx->acc, ctx->n_seeds));
    return cuda_status(cudaGetLastError());
}

int seeds_from_labels(cwthf_ctx* ctx, const int32_t* label, int ng, cudaStream_t s) {
    int64_t cells = int64_t(ng) * ng * ng;
    int64_t nwords = (cells + 31) / 32;
    cudaError_t e = cudaMemsetAsync(ctx->seed_bits, 0, size_t(nwords) * 4, s);
    if (e != cudaSuccess) return cuda_status(e);
    CWTHF_LAUNCH(ctx, s, "k_seeds_from_labels",
                 pdl(k_seeds_from_labels, ctx->sm_count * 8, 256, 0, s)(label, cells, ctx->seed_bits, ctx->d_status));
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e);
    return seeds_rank(ctx, ng, nullptr, s);
}

// CTAs of the cooperative fallback launch: all resident at once (its grid
// barriers need that), at most four per SM.
int fallback_blocks(int sm_count) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_seg_fallback, 256, 0) != cudaSuccess || per_sm < 1)
        return -1;
    return std::min(per_sm, 4) * sm_count;
}

int launch_fallback(cwthf_ctx* ctx, int32_t* label, int64_t cells, cudaStream_t s) {
    if (ctx->fallback_blocks <= 0) return CWTHF_E_CUDA;
    int* changed = ctx->jump_changed;
    unsigned* bar = reinterpret_cast<unsigned*>(changed + kJumpBarrier);
    int rounds = ctx->dbg_jump_rounds;
    // fewer CTAs for small grids: a cooperative launch waits until all of its CTAs fit beside what runs on
    // other streams, and nearly always has nothing to do (a batch of 24 finds on 8 streams 2.94 -> 2.52 ms,
    // together with the launches sized by their work)
    const unsigned blocks = unsigned(std::min<int64_t>(ctx->fallback_blocks, cells / 16384 + 1));
    void* args[] = {&label, &cells, &changed, &rounds, &ctx->seed_bits, &ctx->seed_cells, &bar, &ctx->d_status};
    cudaError_t e;
    CWTHF_LAUNCH(ctx, s, "k_seg_fallback",
                 e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_seg_fallback),
                                                 dim3(blocks), dim3(256), args, 0, s));
    return cuda_status(e);
}

int segment_impl(cwthf_ctx* ctx, const float* cwt, int ng, float cwt_min, int32_t* label, bool,
                 cudaStream_t s) {
    int64_t cells = int64_t(ng) * ng * ng;
    int64_t nwords = (cells + 31) / 32;
    cudaError_t e = cudaMemsetAsync(ctx->seed_bits, 0, size_t(nwords) * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->jump_changed, 0, sizeof(int) * kJumpWords, s);
    if (e != cudaSuccess) return cuda_status(e);
    // the flagged-cell masks of every chain tile (one bit per cell) in the context's int64 grid buffer
    // (8 bytes per cell, free once the forward transform has read it)
    uint32_t* ballots = reinterpret_cast<uint32_t*>(ctx->grid);
    const int64_t ntiles = int64_t(div_up(ng, kChTX)) * div_up(ng, kChTY) * div_up(ng, kChTZ);
    if (ntiles * (kChTY * kRowWords * 4) > cells * 8) return CWTHF_E_UNSUPPORTED_SIZE;
    cudaFuncSetAttribute(k_seg_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, kSegSmem);
    CWTHF_LAUNCH(ctx, s, "k_seg_tile",
                 pdl(k_seg_tile, unsigned(ntiles), kSegThreads, kSegSmem, s)(cwt, ng, cwt_min, label, ctx->seed_bits,
                                                                            ctx->seed_cells, ballots, ctx->d_status));
    // chains that left their tile, counted at their seed's cell
    int blocks = ctx->sm_count * 8;
    int* changed = ctx->jump_changed;  // see kJumpWords
    // rows per turn: four tiles' where there are many turns per CTA (the barriers around a turn's table flush
    // were the pass's largest stall with one tile: 2.14 ms per scale at 1024^3, 1.93 with four), two rows where
    // tiles are too few to fill the GPU (64^3: 38 us with 16 whole tiles, 27 us)
    const int rows = ntiles < 2 * ctx->sm_count ? 2 : (ntiles < 16 * blocks ? kChTY : 4 * kChTY);
    const int rblocks = int(std::min<int64_t>(blocks, ntiles * kChTY / rows));
    CWTHF_LAUNCH(ctx, s, "k_seg_resolve",
                 pdl(k_seg_resolve, rblocks, kResolveThreads, 0, s)(
                     label, ng, ballots, ctx->seed_cells, changed,
                     reinterpret_cast<unsigned*>(changed + kJumpTileCounter), ctx->dbg_chase_limit, rows,
                     ctx->d_status));
    // pointer doubling and a recount for whatever the bounded walks left
    // (normally nothing: the kernel then returns at once)
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e);
    int rc = launch_fallback(ctx, label, cells, s);
    if (rc) return rc;
    // seed slots in cell order, each with its segment's cell count
    return seeds_rank(ctx, ng, ctx->seed_cells, s);
}

}  // namespace cwthf
