// fft_ct.cuh -- instantiates the compile-time FFT lengths of one translation
// unit (every kCtUnits-th length, so that the units take about as long).
#pragma once

#include <utility>

#include "fft.cuh"

namespace cwthf {
namespace fft {

template <int L, bool kBlue>
CtEntry ct_entry() {
    using F = CtFft<L, kBlue>;
    CtEntry e;
    e.L = L;
    e.blue = kBlue;
    e.C = F::C_;
    e.T = F::T_;
    if constexpr (kBlue || is_yz_len(L)) e.yz = k_fft_yz<F>;
    if constexpr (kBlue ? L <= 1152 + 288 : is_x_len(L)) {
        e.xf = k_fft_x_fwd<F>;
        e.xi = k_fft_x_inv<F>;
    }
    return e;
}

// index of L among the compile-time radix lengths
constexpr int ct_index(int L) {
    int k = 0;
    for (int n = 4; n < L; n++) k += is_yz_len(n) || is_x_len(n);
    return k;
}

template <int K, int L>
void ct_add(std::vector<CtEntry>& out) {
    if constexpr (is_yz_len(L) || is_x_len(L)) {
        if constexpr (ct_index(L) % kCtUnits == K) out.push_back(ct_entry<L, false>());
    }
}
template <int K, int I>
void ct_add_blue(std::vector<CtEntry>& out) {
    if constexpr (I % kCtUnits == K) out.push_back(ct_entry<kInner[I], true>());
}
template <int K, int... L>
void ct_all(std::vector<CtEntry>& out, std::integer_sequence<int, L...>) {
    (ct_add<K, L>(out), ...);
}
template <int K, int... I>
void ct_all_blue(std::vector<CtEntry>& out, std::integer_sequence<int, I...>) {
    (ct_add_blue<K, I>(out), ...);
}

#define CWTHF_CT_UNIT(k)                                                                                  \
    template <>                                                                                           \
    void ct_entries<k>(std::vector<CtEntry> & out) {                                                      \
        ct_all<k>(out, std::make_integer_sequence<int, CWTHF_MAX_NG + 1>{});                              \
        ct_all_blue<k>(out, std::make_integer_sequence<int, int(sizeof(kInner) / sizeof(kInner[0]))>{});  \
    }

}  // namespace fft
}  // namespace cwthf
