// Helpers for the compile-time unrolled Clebsch-Gordan contractions (cg_terms.cuh) and the host-side match of a path's tensor
// with them.
#pragma once
#include <math.h>

#include <utility>
#include <vector>

#include "cg_terms.cuh"

namespace sobek {

constexpr int CG_LMAX = 4;

// Destination orders that (LS, LB) reaches with l_dst = LS + LB + PAR (mod 2): LD0, LD0 + 2, ... (at most three), their
// components side by side.
template <int LS, int LB, int PAR>
struct CGSpan {
    static constexpr int lo = LS > LB ? LS - LB : LB - LS;
    static constexpr int LD0 = lo + ((lo + LS + LB + PAR) & 1);
    static constexpr int hi = LS + LB < CG_LMAX ? LS + LB : CG_LMAX;
    static constexpr int n = hi >= LD0 ? (hi - LD0) / 2 + 1 : 0;
    static __host__ __device__ constexpr int ld(int j) { return LD0 + 2 * j; }
    static __host__ __device__ constexpr int off(int j) { return j * (2 * LD0 + 1) + 2 * j * (j - 1); }
    static constexpr int NO = off(n);
};

// the terms of component S: [first, last) of the tensor's list
template <int LS, int LB, int LD, int S>
struct CGRange {
    using T = CGTerms<LS, LB, LD>;
    static __host__ __device__ constexpr int below(int s) { int k = 0; while (k < T::n && (T::id[k] >> 8) < s) ++k; return k; }
    static constexpr int first = below(S), count = below(S + 1) - below(S);
};

// host view of one tensor
struct CGHost { int n; const uint16_t* id; const float* c; };
namespace cg_detail {
template <int A, int B, int C>
CGHost view() {
    if constexpr (CGTerms<A, B, C>::n > 0) return CGHost{CGTerms<A, B, C>::n, CGTerms<A, B, C>::id, CGTerms<A, B, C>::c};
    else return CGHost{0, nullptr, nullptr};
}
template <int... I>
CGHost pick(int k, std::integer_sequence<int, I...>) {
    CGHost r{0, nullptr, nullptr};
    (void)((k == I ? (r = view<I / 25, I / 5 % 5, I % 5>(), true) : false) || ...);
    return r;
}
}  // namespace cg_detail
inline CGHost cg_host(int ls, int lb, int ld) {
    if (ls > CG_LMAX || lb > CG_LMAX || ld > CG_LMAX) return CGHost{0, nullptr, nullptr};
    return cg_detail::pick(ls * 25 + lb * 5 + ld, std::make_integer_sequence<int, 125>());
}

}  // namespace sobek
