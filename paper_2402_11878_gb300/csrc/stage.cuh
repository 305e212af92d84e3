// Staging of one slot in floating point: the RY coefficients, gradient scales and
// diagonal table of its gated bits.  For the floating-point passes (k_layers.cu) and
// for the passes that the fixed-point kernels leave in FP64 (k_layers_fx.cu).
#pragma once

#include <cstdint>

#include "pass_core.cuh"
#include "vqe_internal.h"

namespace vqe {

// All threads of the block; `rows` is the slot's coefficient row (one entry per tile
// bit, gated ones written), `tab` its diagonal table.
template <typename T, class Row>
__device__ __forceinline__ void stage_slot(const StageSlot &S, int n, const double *pr, Row *rows,
                                           typename V2<T>::type *tab) {
    using C = typename V2<T>::type;
    __shared__ double ph_c[kMaxTileBits], ph_s[kMaxTileBits], scl[kMaxTileBits], ph_v[kMaxTileBits];
    __shared__ int ph_m[kMaxTileBits];
    __shared__ double2 half_tab[2][1 << (kMaxTileBits / 2)];
    __shared__ double sigma;
    if (threadIdx.x < (unsigned)S.n_gated) {
        const int j = threadIdx.x;
        const int q = S.qubit[j];
        const double th = pr[((size_t)S.layer * n + q) * 2];
        const double phi = pr[((size_t)S.layer * n + q) * 2 + 1];
        double s, c;
        sincos(0.5 * th, &s, &c);
        if (fabs(c) >= fabs(s)) { ph_v[j] = s / c; ph_m[j] = 0; scl[j] = c; }
        else                    { ph_v[j] = c / s; ph_m[j] = 1; scl[j] = s; }
        double sp, cp;
        sincos(0.5 * phi, &sp, &cp);
        ph_c[j] = cp;
        ph_s[j] = sp;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double p = 1.0;
        for (int u = 0; u < S.n_gated; ++u) p *= scl[u];
        sigma = p;
    }
    __syncthreads();
    if (threadIdx.x < (unsigned)S.n_gated) {
        const int j = threadIdx.x;
        double pb = 1.0;
        for (int u = 0; u < S.n_gated; ++u)
            if ((S.before[j] >> S.tile_bit[u]) & 1u) pb *= scl[u];
        const double f = sigma / pb;
        Row rc{};
        rc.v = (T)ph_v[j];
        rc.gs = (T)(1.0 / (f * f));
        rc.mode = ph_m[j];
        rows[S.tile_bit[j]] = rc;
    }
    // table[e] = sigma * prod_j (bit_j(e) ? e^{+i phi_j/2} : e^{-i phi_j/2}).  The
    // gated bits are the tile's top ones (all of them in the low group): e counts
    // them from the lowest, t0.  The product of one factor for their low and one
    // for their high half: 4 FP64 multiply-adds per entry.
    const int kt = S.n_gated, kl = kt >> 1, kh = kt - kl;
    const double sg = sigma;
    for (uint32_t i = threadIdx.x; i < (1u << kl) + (1u << kh); i += blockDim.x) {
        const bool high = i >= (1u << kl);
        const uint32_t e = high ? i - (1u << kl) : i;
        double re = high ? sg : 1.0, im = 0.0;
        for (int j = 0; j < (high ? kh : kl); ++j) {
            const int q = high ? kl + j : j;
            const double c = ph_c[q];
            const double s = ((e >> j) & 1u) ? ph_s[q] : -ph_s[q];
            const double nr = re * c - im * s;
            const double ni = re * s + im * c;
            re = nr;
            im = ni;
        }
        half_tab[high][e] = make_double2(re, im);
    }
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < (1u << kt); e += blockDim.x) {
        const double2 x = half_tab[0][e & ((1u << kl) - 1u)], y = half_tab[1][e >> kl];
        C d;
        d.x = (T)(x.x * y.x - x.y * y.y);
        d.y = (T)(x.x * y.y + x.y * y.x);
        tab[e] = d;
    }
}

}  // namespace vqe
