// fft.cu -- the grid CWT of Sec. 2.1 (Eq. 2-4) as a 3D real FFT, a multiply
// by the exact DFT of the sampled Mexican-hat wavelet, and an inverse FFT.
//
// Data flow for an ng^3 grid (M = ng/2, P = complex row pitch, even):
//   x-fwd   int64 grid -> fp32 -> real FFT along x -> spec [z][y][0..M]   (k_fft_x_fwd)
//   y-fwd   complex FFT along y, in place                                (k_fft_yz, TMA)
//   z       complex FFT along z, multiply by Psi^, inverse FFT along z    (k_fft_yz, TMA)
//   y-inv   inverse complex FFT along y, in place                        (k_fft_yz, TMA)
//   x-inv   half spectrum -> real row, written to the CWT field          (k_fft_x_inv)
//
// Every 1D transform of length L runs in shared memory as a Stockham
// autosort FFT with at most three radix stages (radices 2^a 3^b 5^c 7^d
// <= 32); each thread performs one or more radix-R butterflies per
// stage entirely in registers, with compile-time constants inside the
// butterfly and fp32 twiddles (rounded once from fp64 on the host) between
// stages.  Lengths with a prime factor above 7 run as Bluestein passes.  The
// device side is in fft.cuh.  Inverse transforms use
// IDFT(x) = conj(DFT(conj(x))).  The forward transform is unnormalised; the
// 1/ng^3 of the inverse is folded into the wavelet spectrum.
//
// Wavelet spectrum (exact DFT of the sampled kernel): with G(u) =
// exp(-w^2 u^2/4) and H(u) = w^2 u^2 G(u) sampled at minimum-image offsets,
//   Psi = w^1.5 [6 G_x G_y G_z - H_x G_y G_z - G_x H_y G_z - G_x G_y H_z],
// so its DFT is the same combination of the 1D DFTs G^ and H^ (real, even),
// tabulated per grid size and scale in fp64 on the host.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "fft.cuh"

namespace cwthf {

using namespace fft;

namespace {

// ---------------------------------------------------------------------------
// Host side: plans, tables, tensor maps, launches.
// ---------------------------------------------------------------------------
// The compile-time instances, by length.
const std::vector<CtEntry>& ct_table() {
    static const std::vector<CtEntry> tab = [] {
        std::vector<CtEntry> t;
        ct_entries<0>(t);
        ct_entries<1>(t);
        ct_entries<2>(t);
        ct_entries<3>(t);
        ct_entries<4>(t);
        ct_entries<5>(t);
        ct_entries<6>(t);
        ct_entries<7>(t);
        return t;
    }();
    return tab;
}
const CtEntry* ct_find(int L, bool blue) {
    for (const CtEntry& e : ct_table())
        if (e.L == L && e.blue == blue) return &e;
    return nullptr;
}

// The built-in plan of a pass: its compile-time instance and, for a length
// that has none, the Bluestein instance of the smallest inner length
// Mb >= 2 L - 1 (at most 2.25 L + 64: the tables' slots are sized for that).
struct PassPlan {
    Plan p;
    const CtEntry* ct = nullptr;
};
bool pass_plan_for(int L, bool x, PassPlan& out) {
    auto use = [&](int len, bool blue) {
        const CtEntry* e = ct_find(len, blue);
        if (!e || !(x ? bool(e->xf) : bool(e->yz))) return false;
        const Radices r = make_radices(len);
        out.p = Plan();
        out.p.L = len;
        out.p.nst = r.n;
        for (int i = 0; i < 3; i++) out.p.rad[i] = r.r[i];
        out.p.C = e->C;
        out.p.T = e->T;
        out.p.Lb = blue ? L : 0;
        out.ct = e;
        return true;
    };
    if (use(L, false)) return true;
    for (int Mb : kInner)
        if (Mb >= 2 * L - 1 && Mb <= 2 * L + L / 4 + 64) return use(Mb, true);
    return false;
}

// Rows per TMA box for a y/z pass of length L with C columns: as few boxes of
// at most 256 rows as cover the pass, each spanning a multiple of 128 bytes;
// the last one may overhang the end of the axis (its loads read zeros there
// and its stores are clipped).
int pick_boxr(int L, int C) {
    const int align = std::max(1, 16 / C);
    const int n = div_up(L, 256);
    return div_up(div_up(L, n), align) * align;
}

// The built-in plans of a grid size (host arithmetic on the size alone),
// worked out once per size and process.
struct SizePlans {
    PassPlan yz, x;
    bool ok = false;
};
const SizePlans& size_plans(int ng) {
    static SizePlans tab[CWTHF_MAX_NG / 2 + 1];
    static std::once_flag once[CWTHF_MAX_NG / 2 + 1];
    const int i = ng / 2;
    std::call_once(once[i], [&] {
        SizePlans& s = tab[i];
        s.ok = pass_plan_for(ng, false, s.yz) && pass_plan_for(ng / 2, true, s.x);
    });
    return tab[i];
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}

// 3D view of a spectrum as floats: dim0 = 2P floats (contiguous), dim1 = y,
// dim2 = z.  A box is C complex columns by boxr rows of the transform axis
// (y: {2C, boxr, 1}; z: {2C, 1, boxr}); either lands in shared memory as a
// dense [boxr][C] complex tile.
int make_spec_map(CUtensorMap* map, float2* base, int ng, bool along_z, int C, int boxr) {
    auto fn = encode_fn();
    if (!fn) return CWTHF_E_CUDA;
    const int P = spec_pitch(ng);
    cuuint64_t dims[3] = {cuuint64_t(2 * P), cuuint64_t(ng), cuuint64_t(ng)};
    cuuint64_t row = cuuint64_t(P) * 8, plane = row * ng;
    cuuint64_t strides[2] = {row, plane};
    cuuint32_t box[3] = {cuuint32_t(2 * C), along_z ? 1u : cuuint32_t(boxr), along_z ? cuuint32_t(boxr) : 1u};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? CWTHF_OK : CWTHF_E_CUDA;
}

// Dynamic shared memory: alignment slack, the tile and the transfer barrier;
// the tile, the twiddles and the row sums.
size_t yz_smem(const Plan& p, int trows) { return 128 + size_t(trows) * p.C * 8 + 16; }
size_t x_smem(const Plan& p) { return size_t(p.L) * p.C * 8 + size_t(p.L) * 8 + size_t(p.C) * 8; }

void host_twiddles(int n, std::vector<float2>& out) {
    out.resize(n);
    for (int m = 0; m < n; m++) {
        double ang = 2.0 * kPi * double(m) / double(n);
        out[m] = make_float2(float(std::cos(ang)), float(-std::sin(ang)));
    }
}

// The twiddle table of a grid size: twN [ng] and twM [ng/2], then for each
// Bluestein pass its chirp, transformed chirp and inner twiddles (float
// offsets; 0 = absent).
struct TwLayout {
    size_t n = 0;
    size_t chirp_yz = 0, bhat_yz = 0, tw_yz = 0, chirp_x = 0, bhat_x = 0, tw_x = 0;
    int lb_yz = 0, mb_yz = 0, lb_x = 0, mb_x = 0;
};
TwLayout tw_layout(int ng) {
    TwLayout t;
    size_t o = 3 * size_t(ng);
    if (const Plan& p = size_plans(ng).yz.p; p.Lb) {
        t.lb_yz = p.Lb;
        t.mb_yz = p.L;
        t.chirp_yz = o;
        o += 2 * size_t(p.Lb);
        t.bhat_yz = o;
        o += 2 * size_t(p.L);
        t.tw_yz = o;
        o += 2 * size_t(p.L);
    }
    if (const Plan& p = size_plans(ng).x.p; p.Lb) {
        t.lb_x = p.Lb;
        t.mb_x = p.L;
        t.chirp_x = o;
        o += 2 * size_t(p.Lb);
        t.bhat_x = o;
        o += 2 * size_t(p.L);
        t.tw_x = o;
        o += 2 * size_t(p.L);
    }
    t.n = o;
    return t;
}

// Bluestein tables in fp64, stored as fp32: the chirp b_n = exp(i pi n^2 / Lb),
// n < Lb (n^2 reduced mod 2 Lb exactly); the DFT of length Mb of the wrapped
// chirp (b_n at n and at Mb - n, zero between), divided by Mb; the twiddles of Mb.
void host_bluestein(int Lb, int Mb, float* chirp, float* bhat, float* tw) {
    std::vector<double> br(Lb), bi(Lb);
    for (int n = 0; n < Lb; n++) {
        const long long q = (static_cast<long long>(n) * n) % (2LL * Lb);
        const double ang = kPi * double(q) / double(Lb);
        br[n] = std::cos(ang);
        bi[n] = std::sin(ang);
        chirp[2 * n] = float(br[n]);
        chirp[2 * n + 1] = float(bi[n]);
    }
    std::vector<double> cm(Mb), sm(Mb);
    for (int m = 0; m < Mb; m++) {
        cm[m] = std::cos(2.0 * kPi * double(m) / double(Mb));
        sm[m] = std::sin(2.0 * kPi * double(m) / double(Mb));
    }
    for (int k = 0; k < Mb; k++) {
        double sr = 0.0, si = 0.0;
        auto add = [&](int n, int j) {  // B_n = b_j, times exp(-2 pi i n k / Mb)
            const int e = int((static_cast<long long>(n) * k) % Mb);
            sr += br[j] * cm[e] + bi[j] * sm[e];
            si += bi[j] * cm[e] - br[j] * sm[e];
        };
        for (int n = 0; n < Lb; n++) add(n, n);
        for (int n = Mb - Lb + 1; n < Mb; n++) add(n, Mb - n);
        bhat[2 * k] = float(sr / Mb);
        bhat[2 * k + 1] = float(si / Mb);
    }
    std::vector<float2> w;
    host_twiddles(Mb, w);
    std::memcpy(tw, w.data(), w.size() * 8);
}

// G^(k) and H^(k), k < ng: 1D DFTs (real, even sequences) of the sampled
// Gaussian factor and of its w^2 u^2 multiple, in fp64, stored as fp32
// (out[k] = G^(k), out[ng + k] = H^(k)).
void host_wavelet_tables(int ng, double L, double w, float* out) {
    const double dx = L / ng;
    std::vector<double> gn(ng), hn(ng), cosn(ng);
    for (int n = 0; n < ng; n++) {
        int d = (2 * n <= ng) ? n : n - ng;
        double u2 = (dx * d) * (dx * d);
        gn[n] = std::exp(-0.25 * w * w * u2);
        hn[n] = w * w * u2 * gn[n];
        cosn[n] = std::cos(2.0 * kPi * double(n) / double(ng));
    }
    for (int k = 0; k < ng; k++) {
        double sg = 0.0, sh = 0.0;
        for (int n = 0; n < ng; n++) {
            double c = cosn[(int64_t(k) * n) % ng];
            sg += gn[n] * c;
            sh += hn[n] * c;
        }
        out[k] = float(sg);
        out[ng + k] = float(sh);
    }
}

// The context's table slots (allocated by cwthf_create, never grown).  A
// miss fills a slot on the host (the slot's pinned staging) and queues one
// copy to the device on the call's stream, so a call allocates nothing and
// never waits for the device, except when it must reuse a slot whose
// previous copy may still be pending.  Slots read by work captured into a
// CUDA graph are never reused.  A captured call records the copy of a table
// that no uncaptured call has put on the device yet, so such a graph brings
// its own tables on every replay; a table already copied by an uncaptured
// call (cwthf_prepare, or an earlier call) is only read, and that copy must
// be complete before the graph runs.  An uncaptured call that finds a slot
// filled only inside a capture queues the copy itself.  During a capture only
// free slots can be filled; with none left the call fails with
// CWTHF_E_TABLE_CACHE.
int table_lookup(cwthf_ctx* ctx, int kind, int ng, double L, double w, cudaStream_t s, const float** out) {
    std::lock_guard<std::mutex> g(ctx->table_mu);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) return CWTHF_E_CUDA;
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    const size_t stride = ctx->table_slot_floats;
    const TwLayout lay = kind == kTableTwiddles ? tw_layout(ng) : TwLayout();
    const size_t n = kind == kTableTwiddles ? lay.n : 2 * size_t(ng);
    if (n > stride) return CWTHF_E_UNSUPPORTED_SIZE;
    int pick = -1;
    for (int i = 0; i < kTableSlots && pick < 0; i++) {
        const TableSlot& t = ctx->table_slot[i];
        if (t.kind == kind && t.ng == ng && t.L == L && t.w == w) pick = i;
    }
    bool fill = pick < 0;
    if (fill) {
        for (int i = 0; i < kTableSlots && pick < 0; i++)
            if (ctx->table_slot[i].kind < 0) pick = i;
        if (pick < 0 && !capturing)  // least recently used slot that no graph reads
            for (int i = 0; i < kTableSlots; i++) {
                const TableSlot& t = ctx->table_slot[i];
                if (!t.graph_ref && (pick < 0 || t.last_use < ctx->table_slot[pick].last_use)) pick = i;
            }
        if (pick < 0) return CWTHF_E_TABLE_CACHE;
    }
    TableSlot& t = ctx->table_slot[pick];
    float* host = ctx->table_host + pick * stride;
    float* dev = ctx->table_dev + pick * stride;
    if (fill) {
        // an evicted slot (only ever filled outside a capture): its last copy
        // must have read the staging before the staging is rewritten
        if (t.kind >= 0 && cudaEventSynchronize(t.filled) != cudaSuccess) return CWTHF_E_CUDA;
        t = TableSlot{-1, 0, 0.0, 0.0, 0, false, false, t.filled};
        if (kind == kTableTwiddles) {  // exp(-2 pi i m / ng), m < ng, then exp(-2 pi i m / (ng/2)), m < ng/2
            std::vector<float2> a, b;
            host_twiddles(ng, a);
            host_twiddles(ng / 2, b);
            std::memcpy(host, a.data(), a.size() * 8);
            std::memcpy(host + 2 * ng, b.data(), b.size() * 8);
            if (lay.lb_yz)
                host_bluestein(lay.lb_yz, lay.mb_yz, host + lay.chirp_yz, host + lay.bhat_yz, host + lay.tw_yz);
            if (lay.lb_x) host_bluestein(lay.lb_x, lay.mb_x, host + lay.chirp_x, host + lay.bhat_x, host + lay.tw_x);
        } else {
            host_wavelet_tables(ng, L, w, host);
        }
        t.kind = kind;
        t.ng = ng;
        t.L = L;
        t.w = w;
        ctx->table_fills++;
    }
    // a captured call that finds the table already on the device (an earlier
    // uncaptured copy) records no copy: the graph reads the slot, which is
    // kept from now on; otherwise the graph carries the copy itself
    if (!t.on_device) {  // a fill always clears on_device
        if (cudaMemcpyAsync(dev, host, n * 4, cudaMemcpyHostToDevice, s) != cudaSuccess) return CWTHF_E_CUDA;
        if (!capturing) {
            if (cudaEventRecord(t.filled, s) != cudaSuccess) return CWTHF_E_CUDA;
            t.on_device = true;
        }
    }
    t.graph_ref |= capturing;
    t.last_use = ++ctx->table_clock;
    *out = dev;
    return CWTHF_OK;
}

int get_tables(cwthf_ctx* ctx, int ng, cudaStream_t s, Tables& t) {
    const float* p = nullptr;
    int rc = table_lookup(ctx, kTableTwiddles, ng, 0.0, 0.0, s, &p);
    if (rc) return rc;
    t.ng = ng;
    t.twN = reinterpret_cast<const float2*>(p);
    t.twM = reinterpret_cast<const float2*>(p + 2 * ng);
    const TwLayout lay = tw_layout(ng);
    auto at = [&](size_t o) { return o ? reinterpret_cast<const float2*>(p + o) : nullptr; };
    t.chirp_yz = at(lay.chirp_yz);
    t.bhat_yz = at(lay.bhat_yz);
    t.tw_yz = at(lay.tw_yz);
    t.chirp_x = at(lay.chirp_x);
    t.bhat_x = at(lay.bhat_x);
    t.tw_x = at(lay.tw_x);
    return CWTHF_OK;
}

// A caller's plan (which = 0: y/z passes of length ng, 1: x passes of length
// ng/2), checked against what the run-time kernels can run: radices from
// kRadices whose product is the length, C in {2, 4, 8, 16}, <= 64 KB of tile,
// <= 512 threads, and for the y/z passes whole 128-byte multiples of rows that
// divide the length.
bool plan_from(int L, int which, int C, const int* rad, int nst, Plan& p) {
    if (nst < 1 || nst > 3 || !(C == 2 || C == 4 || C == 8 || C == 16)) return false;
    int prod = 1, rmin = 64;
    for (int i = 0; i < nst; i++) {
        if (!is_radix(rad[i])) return false;
        prod *= rad[i];
        rmin = std::min(rmin, rad[i]);
    }
    if (prod != L) return false;
    p = Plan();
    p.L = L;
    p.nst = nst;
    for (int i = 0; i < 3; i++) p.rad[i] = i < nst ? rad[i] : 1;
    p.C = C;
    p.T = (C * (L / rmin) + 31) / 32 * 32;
    if (which != 0) p.T = std::max(p.T, 32 * std::min(C, 16));
    if (size_t(L) * C * 8 > 65536 || p.T > 512) return false;
    bool box = which != 0;
    for (int b = std::min(L, 256); b >= 1 && !box; b--) box = L % b == 0 && (size_t(b) * C * 8) % 128 == 0;
    return box;
}

// The plan a pass of this context uses: the caller's (on the run-time kernels,
// unless it is the built-in one), else the built-in one.
bool pass_plan(cwthf_ctx* ctx, int ng, int which, PassPlan& p) {
    {
        std::lock_guard<std::mutex> g(ctx->table_mu);
        for (const auto& o : ctx->fft_plans)
            if (o.ng == ng && o.which == which) {
                const int len = which == 0 ? ng : ng / 2;
                p.ct = nullptr;
                if (!plan_from(len, which, o.C, o.rad, o.nst, p.p)) return false;
                // the built-in plan's own radices and width: its compile-time instance
                const PassPlan& b = which == 0 ? size_plans(ng).yz : size_plans(ng).x;
                bool same = size_plans(ng).ok && !b.p.Lb && b.p.C == o.C && b.p.nst == o.nst;
                for (int i = 0; i < o.nst && same; i++) same = b.p.rad[i] == o.rad[i];
                if (same) p = b;
                return true;
            }
    }
    const SizePlans& s = size_plans(ng);
    p = which == 0 ? s.yz : s.x;
    return s.ok;
}

int launch_yz(cwthf_ctx* ctx, float2* src, float2* dst, int ng, bool along_z, int mode, const Tables* t,
              const float* wtab, double w, double mass_unit, cudaStream_t s) {
    PassPlan pp;
    if (!pass_plan(ctx, ng, 0, pp)) return CWTHF_E_UNSUPPORTED_SIZE;
    Plan& p = pp.p;
    const int boxr = pick_boxr(ng, p.C);
    if (p.Lb && !(t->chirp_yz && t->bhat_yz && t->tw_yz)) return CWTHF_E_UNSUPPORTED_SIZE;
    p.chirp = t->chirp_yz;
    p.bhat = t->bhat_yz;
    CUtensorMap in_map, out_map;
    int rc = make_spec_map(&in_map, src, ng, along_z, p.C, boxr);
    if (!rc) rc = make_spec_map(&out_map, dst, ng, along_z, p.C, boxr);
    if (rc) return rc;
    YzArgs a;
    a.p = p;
    a.M = ng / 2;
    a.ncc = div_up(a.M + 1, p.C);
    a.boxr = boxr;
    a.nbox = div_up(ng, boxr);
    a.trows = std::max(a.nbox * boxr, p.L);
    a.mode = mode;
    a.along_z = along_z ? 1 : 0;
    a.nplanes = ng;
    a.tw = p.Lb ? t->tw_yz : t->twN;
    a.ghat = wtab;
    a.hhat = wtab ? wtab + ng : nullptr;
    // w^1.5 (Eq. 4), the 1/ng^3 of the inverse DFT, and the mass of one spectrum
    // unit (the x pass already scaled the int64 grid by 2^-30: units of mass_unit)
    a.scale = float(std::pow(w, 1.5) * mass_unit / (double(ng) * ng * ng));
    a.status = ctx->d_status;
    a.no_copy_block = -1;
    a.no_copy_spin = 0;
    if (ctx->dbg_tma_no_copy) {  // one-shot fault injection (cwthf_debug_set)
        ctx->dbg_tma_no_copy = 0;
        a.no_copy_block = 0;
        a.no_copy_spin = 1 << 12;
    }
    const YzKernel k = pp.ct ? pp.ct->yz : dyn_yz();
    const size_t smem = yz_smem(p, a.trows);
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    CWTHF_LAUNCH(ctx, s, "k_fft_yz", pdl(k, unsigned(a.ncc) * ng, p.T, smem, s)(in_map, out_map, a));
    return cuda_status(cudaGetLastError());
}

int x_args(cwthf_ctx* ctx, int ng, const Tables* t, XArgs& a, const CtEntry*& ct) {
    PassPlan pp;
    if (!pass_plan(ctx, ng, 1, pp)) return CWTHF_E_UNSUPPORTED_SIZE;
    Plan& p = pp.p;
    ct = pp.ct;
    if (p.Lb && !(t->chirp_x && t->bhat_x && t->tw_x)) return CWTHF_E_UNSUPPORTED_SIZE;
    p.chirp = t->chirp_x;
    p.bhat = t->bhat_x;
    a.p = p;
    a.ng = ng;
    a.M = ng / 2;
    a.P = spec_pitch(ng);
    a.rows = int64_t(ng) * ng;
    a.inv_ng = ~0ull / unsigned(ng);
    a.twM = p.Lb ? t->tw_x : t->twM;
    a.twN = t->twN;
    return CWTHF_OK;
}

}  // namespace

int transform_forward_xy(cwthf_ctx* ctx, const int64_t* grid, int ng, float2* spec, cudaStream_t s) {
    if (ng > CWTHF_MAX_NG) return CWTHF_E_UNSUPPORTED_SIZE;
    Tables tb;
    int rc = get_tables(ctx, ng, s, tb);
    if (rc) return rc;
    const Tables* t = &tb;
    XArgs a;
    const CtEntry* ct = nullptr;
    rc = x_args(ctx, ng, t, a, ct);
    if (rc) return rc;
    const XFwdKernel k = ct ? ct->xf : dyn_x_fwd();
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(x_smem(a.p)));
    CWTHF_LAUNCH(ctx, s, "k_fft_x_fwd", pdl(k, div_up(a.rows, a.p.C), a.p.T, x_smem(a.p), s)(a, grid, spec));
    if ((rc = cuda_status(cudaGetLastError()))) return rc;
    return launch_yz(ctx, spec, spec, ng, false, kYzForward, t, nullptr, 0.0, 1.0, s);
}

int transform_tables(cwthf_ctx* ctx, int ng, double L, const double* w, int n, const float** wtab,
                     cudaStream_t s) {
    if (n + 1 > kTableSlots) return CWTHF_E_TABLE_CACHE;
    Tables tb;
    int rc = get_tables(ctx, ng, s, tb);
    for (int i = 0; i < n && !rc; i++) rc = table_lookup(ctx, kTableWavelet, ng, L, w[i], s, &wtab[i]);
    return rc;
}

int transform_wavelet_inverse(cwthf_ctx* ctx, float2* src, float2* dst, int ng, double L, double w,
                              double mass_unit, const float* wtab, float* cwt, cudaStream_t s) {
    Tables tb;
    int rc = get_tables(ctx, ng, s, tb);
    if (rc) return rc;
    const Tables* t = &tb;
    rc = launch_yz(ctx, src, dst, ng, true, kYzWavelet, t, wtab, w, mass_unit, s);
    if (!rc) rc = launch_yz(ctx, dst, dst, ng, false, kYzInverse, t, nullptr, 0.0, 1.0, s);
    if (rc) return rc;
    XArgs a;
    const CtEntry* ct = nullptr;
    if ((rc = x_args(ctx, ng, t, a, ct))) return rc;
    const XInvKernel k = ct ? ct->xi : dyn_x_inv();
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(x_smem(a.p)));
    CWTHF_LAUNCH(ctx, s, "k_fft_x_inv", pdl(k, div_up(a.rows, a.p.C), a.p.T, x_smem(a.p), s)(a, dst, cwt));
    return cuda_status(cudaGetLastError());
}

int set_fft_plan(cwthf_ctx* ctx, int ng, int which, int C, const int* rad, int nst) {
    if (which != 0 && which != 1) return CWTHF_E_INVALID_ARG;
    std::lock_guard<std::mutex> g(ctx->table_mu);
    auto& v = ctx->fft_plans;
    v.erase(std::remove_if(v.begin(), v.end(), [&](const cwthf_ctx::PlanOverride& o) {
                return o.ng == ng && o.which == which;
            }), v.end());
    if (nst == 0) return CWTHF_OK;  // back to the built-in rule
    Plan p;
    if (!rad || !plan_from(which == 0 ? ng : ng / 2, which, C, rad, nst, p)) return CWTHF_E_INVALID_ARG;
    cwthf_ctx::PlanOverride o{ng, which, C, nst, {1, 1, 1}};
    for (int i = 0; i < nst; i++) o.rad[i] = rad[i];
    v.push_back(o);
    return CWTHF_OK;
}

// The same plans the launches use.
bool fft_size_supported(int ng) { return ng >= 2 && ng % 2 == 0 && ng <= CWTHF_MAX_NG && size_plans(ng).ok; }

void free_tables(cwthf_ctx* ctx) {
    for (TableSlot& t : ctx->table_slot) {
        if (t.filled) cudaEventDestroy(t.filled);
        t = TableSlot();
    }
}

int init_tables(cwthf_ctx* ctx) {
    for (TableSlot& t : ctx->table_slot)
        if (cudaEventCreateWithFlags(&t.filled, cudaEventDisableTiming) != cudaSuccess) return CWTHF_E_CUDA;
    return CWTHF_OK;
}

}  // namespace cwthf
