// FP64 ansatz passes in block fixed point: staging and the tile-pass kernel.
//
// Same pass programs, tiles and memory traffic as the floating-point kernels of
// k_layers.cu: a tile of 2^k amplitudes goes through registers (8 per thread)
// and shared memory, and a program of rounds, butterflies, diagonals and
// (backward) flushes runs on it.  The arithmetic is that of fx.cuh: doubles in
// global memory, 64-bit integers in registers and shared memory.  One compiled
// body serves every program: the 3 register bits of a round are the same code
// wherever the round's chunk lies, only the addresses depend on it.  A state whose
// angles spread a tile's amplitudes too far for one exponent (kFxMaxSpread) goes
// through the same launch in FP64 (WideEnv).
#include <cstddef>

#include "fx.cuh"
#include "pass_core.cuh"
#include "pdl.cuh"
#include "smem_limit.h"
#include "stage.cuh"
#include "vqe_internal.h"

namespace vqe {

static_assert(sizeof(RotFx) == sizeof(RotCoef<double>), "the coefficient buffer holds either");

namespace {

constexpr int kR = 3, kNR = 8;

// ---------------------------------------------------------------- staging

// Integers scaled by 2^62: every factor of a diagonal table and every scale is
// made unitary to 2^-60 (one Newton step on the rounded FP64 values) and the
// products are taken in integers, so a table entry's modulus is exact to about
// 2^-57; only the angles carry FP64 rounding.
__device__ __forceinline__ long long mul62(long long a, long long b) { return __mul64hi(a, b) << 2; }

__device__ __forceinline__ longlong2 cmul62(longlong2 a, longlong2 b) {
    return make_longlong2((__mul64hi(a.x, b.x) - __mul64hi(a.y, b.y)) << 2,
                          (__mul64hi(a.x, b.y) + __mul64hi(a.y, b.x)) << 2);
}

// x (1 + r) scaled by 2^62, |x| <= 1, r a small correction
__device__ __forceinline__ long long to62(double x, double r) {
    return __double2ll_rn(x * 0x1p62) + __double2ll_rn(x * r * 0x1p62);
}

// Bits by which the amplitudes of a tile of the slot's pass spread (fx.cuh): per
// qubit of the tile the layers' largest tangent, 16 threads each.  The same for every
// slot of a pass, bit for bit.  A qubit that no layer turns leaves exact zeros.
__device__ __forceinline__ float tile_spread(const StageSlot &S, int n, int depth, const double *pr) {
    __shared__ float bits[kMaxTileBits];
    static_assert(kMaxTileBits <= 16, "16 threads per tile bit");
    const int j = threadIdx.x >> 4, t0 = S.tile_bit[0];   // the tile's ungated bits are qubits 0 .. t0 - 1
    if (j < S.k) {
        const int q = j < t0 ? j : S.qubit[j - t0];
        double w = 0.0;
        for (int l = threadIdx.x & 15; l < depth; l += 16) {
            const double th = pr[((size_t)l * n + q) * 2];
            const double turns = rint(th * 0.31830988618379067);   // 1 / pi
            const double d = fma(-turns, 1.2246467991473532e-16, fma(-turns, 3.141592653589793, th));
            w = fmax(w, fabs(d));   // an angle that is not a number does not count
        }
        float bit = w == 0.0 ? 0.f : w < 1e-30 ? 100.f : -log2f(tanf(fminf((float)(0.5 * w), 0.78539816f)));
        const unsigned group = 0xffffu << (threadIdx.x & 16u);
        for (int o = 8; o > 0; o >>= 1) {
            const double ow = __shfl_xor_sync(group, w, o);
            const float ob = __shfl_xor_sync(group, bit, o);
            if (ow > w) {
                w = ow;
                bit = ob;
            }
        }
        if ((threadIdx.x & 15u) == 0) bits[j] = fmaxf(bit, 0.f);
    }
    __syncthreads();
    float sum = 0.f;
    for (int i = 0; i < S.k; ++i) sum += bits[i];
    return sum;
}

// One block per slot and state: coefficients, gradient scales and shift
// schedule of the slot's gated bits, and the slot's diagonal table
//   d[l] = 2^S sigma prod_j (phase and quarter-turn sign of bit j of l),
// sigma the product of the gates' scales, S the shifts made in the slot, so
// that 1/2 < 2^S sigma <= 1.  The table is the product of one factor for the
// low and one for the high half of the tile bits.
__global__ void k_stage_fx(const StageSlot *__restrict__ slots, int n, int depth,
                           const double *__restrict__ params, RotFx *__restrict__ coefs,
                           size_t coef_stride, longlong2 *__restrict__ dtab, size_t dtab_stride) {
    pdl_trigger();
    __shared__ longlong2 half_tab[2][1 << (kMaxTileBits / 2)];
    __shared__ longlong2 d0[kMaxTileBits], d1[kMaxTileBits];
    __shared__ long long scl[kMaxTileBits];
    __shared__ float lg[kMaxTileBits];
    __shared__ long long scale_at[kMaxTileBits];   // of the buffers when the bit's theta gradient is taken
    __shared__ int turns_of[kMaxTileBits], order[kMaxTileBits], shb[kMaxTileBits];
    __shared__ RotFx rot[kMaxTileBits];
    __shared__ long long sigma;   // 2^S sigma
    __shared__ int table_shift;
    const StageSlot S = slots[blockIdx.x];
    const int b = blockIdx.y;
    const double *pr = params + (size_t)b * (2 * (size_t)n * depth);
    if (tile_spread(S, n, depth, pr) > kFxMaxSpread) {   // the pass stays in FP64
        stage_slot<double>(S, n, pr, reinterpret_cast<RotWide *>(coefs + (size_t)b * coef_stride + S.coef_off),
                           reinterpret_cast<double2 *>(dtab + (size_t)b * dtab_stride + S.dtab_off));
        return;
    }
    // Latency is what staging costs (FP64 instructions issue once per 64 clocks): theta
    // and phi in a warp each, the serial schedule in FP32 and integers, divisions in
    // parallel (64 states of 8 qubits, one slot: 24.7 -> 16.3 us).
    const int j = threadIdx.x & 31;
    const bool mine = j < S.n_gated;
    if (threadIdx.x < 32 && mine) {
        const int q = S.qubit[j];
        const double th = pr[((size_t)S.layer * n + q) * 2], phi = pr[((size_t)S.layer * n + q) * 2 + 1];
        double s, c;
        sincos(0.5 * th, &s, &c);
        // quarter turns taken off until the angle lies in [-pi/8, 3 pi/8):
        // the turn nearest pi/8, cos(pi/8) = 0.9239, sin(pi/8) = 0.3827
        int turns = 0;
        double best = -2.0, cq = c, sq = s;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const double ct = t == 0 ? c : t == 1 ? s : t == 2 ? -c : -s;
            const double st = t == 0 ? s : t == 1 ? -c : t == 2 ? -s : c;
            const double v = 0.9238795325112867 * ct + 0.3826834323650898 * st;
            if (v > best) {
                best = v;
                turns = t;
                cq = ct;
                sq = st;
            }
        }
        const bool half_turn = sq > 0.4142135623730950 * cq;
        const double tt = half_turn ? (sq - cq) / (sq + cq) : sq / cq;
        // scale 1 / sqrt(1 + t^2), its residual 1 - s^2 (1 + t^2) without rounding
        const double s0 = 1.0 / sqrt(fma(tt, tt, 1.0));
        const double p = s0 * s0, pe = fma(s0, s0, -p), u = tt * tt, ue = fma(tt, tt, -u);
        const double pu = p * u, pue = fma(p, u, -pu);
        const double res = ((((1.0 - p) - pu) - pue) - pe * (1.0 + u)) - p * ue;
        long long sc = to62(s0, 0.5 * res);
        if (half_turn) sc = __mul64hi(sc, 0x5A827999FCEF3242ll) << 1;   // 2^63 / sqrt(2)
        scl[j] = sc;
        lg[j] = -log2f((float)sc * 0x1p-62f);
        turns_of[j] = turns;
        const bool bad = !(isfinite(th) && isfinite(phi));
        const long long T = bad ? 0ll : __double2ll_rn(tt * 0x1p64);
        rot[j].tl = fx_lo(T);
        rot[j].th = fx_hi(T);
        rot[j].meta = ((turns & 1) ? kFxFlip : 0u) | (half_turn ? kFx45 : 0u) | (bad ? kFxBad : 0u);
        rot[j].wide = 0;
    } else if (threadIdx.x >= 32 && threadIdx.x < 64 && mine) {
        const double phi = pr[((size_t)S.layer * n + S.qubit[j]) * 2 + 1];
        double sp, cp;
        sincos(0.5 * phi, &sp, &cp);
        const double c2 = cp * cp, c2e = fma(cp, cp, -c2), s2 = sp * sp, s2e = fma(sp, sp, -s2);
        const double half_res = 0.5 * ((((1.0 - fmax(c2, s2)) - fmin(c2, s2)) - c2e) - s2e);
        const long long ci = to62(cp, half_res), si = to62(sp, half_res);
        d0[j] = make_longlong2(ci, -si);
        d1[j] = make_longlong2(ci, si);
    }
    __syncthreads();
    if (threadIdx.x >= 32 && threadIdx.x < 64 && mine) {
        // J^q: logical bit 0 takes -1 for q = 1, 2 and bit 1 for q = 2, 3
        const int turns = turns_of[j];
        const longlong2 a = d0[j], b1 = d1[j];
        if (turns == 1 || turns == 2) d0[j] = make_longlong2(-a.x, -a.y);
        if (turns >= 2) d1[j] = make_longlong2(-b1.x, -b1.y);
    }
    if (threadIdx.x == 0) {
        // shift schedule: A = log2 of the norm's growth since the slot began
        const int ng = S.n_gated;
        float A = 0.f;
        int total = 0;
        long long sig = 1ll << 62;
        for (int j = 0; j < ng; ++j) order[__popc(S.fbefore[j])] = j;
        for (int i = 0; i < ng; ++i) {
            const int j = order[i];
            A += lg[j];
            const int sh = A >= 1.f ? 1 : 0;   // lg < 0.62: at most one
            A -= (float)sh;
            total += sh;
            sig = mul62(sig, scl[j]) << sh;
            rot[j].meta |= (uint32_t)sh << kFxShiftF;
        }
        const bool near_one = sig > (1ll << 62) - (1ll << 32);
        sigma = sig;
        table_shift = near_one ? 0 : 1;
        for (int j = 0; j < ng; ++j) order[__popc(S.before[j])] = j;
        A = (float)total;
        for (int j = 0; j < ng; ++j) A -= lg[j];
        int done = 0;
        for (int i = 0; i < ng; ++i) {
            // A < 0.75 where the next gate's theta gradient is taken (after its turn)
            A += lg[order[i]];
            const float limit = i + 1 < ng && (rot[order[i + 1]].meta & kFx45) ? 0.25f : 0.75f;
            int sh = A >= limit && done < total ? 1 : 0;
            A -= (float)sh;
            if (i == ng - 1) sh = min(3, total - done);
            done += sh;
            shb[i] = sh;
        }
        long long f = 1ll << 62;   // scale of the buffers, back from the slot's end
        for (int i = ng - 1; i >= 0; --i) {
            const int j = order[i];
            f = mul62(f, scl[j]) << shb[i];
            scale_at[j] = f;
            rot[j].meta |= ((uint32_t)shb[i] << kFxShiftB) | ((uint32_t)total << kFxSlotShift) |
                           (near_one ? kFxHalf : 0u);
        }
    }
    __syncthreads();
    // one row per tile bit; the gated bits are the tile's top ones (all of them in
    // the low group), and the table has no index bits below them
    const int t0 = S.tile_bit[0], kt = S.k - t0;
    if (threadIdx.x < (unsigned)S.k) {
        RotFx r{0, 0, 0u, 0, 0.0};
        if ((int)threadIdx.x >= t0) {
            r = rot[threadIdx.x - t0];
            const double fd = (double)scale_at[threadIdx.x - t0] * 0x1p-62;
            // the theta gradient is taken after the bit's 45-degree turn (x sqrt 2)
            r.gs = 0.125 / (fd * fd * ((r.meta & kFx45) ? 2.0 : 1.0));
        }
        coefs[(size_t)b * coef_stride + S.coef_off + threadIdx.x] = r;
    }
    const int kl = kt >> 1, kh = kt - kl;
    for (uint32_t i = threadIdx.x; i < (1u << kl) + (1u << kh); i += blockDim.x) {
        const bool high = i >= (1u << kl);
        const uint32_t e = high ? (i - (1u << kl)) << kl : i;
        longlong2 v = make_longlong2(high ? sigma : 1ll << 62, 0ll);
        for (int j = high ? kl : 0; j < (high ? kt : kl); ++j) v = cmul62(v, ((e >> j) & 1u) ? d1[j] : d0[j]);
        half_tab[high][high ? i - (1u << kl) : i] = v;
    }
    __syncthreads();
    longlong2 *tab = dtab + (size_t)b * dtab_stride + S.dtab_off;
    for (uint32_t l = threadIdx.x; l < (1u << kt); l += blockDim.x) {
        const longlong2 v = cmul62(half_tab[0][l & ((1u << kl) - 1u)], half_tab[1][l >> kl]);
        tab[l] = make_longlong2(v.x << table_shift, v.y << table_shift);
    }
}

// ---------------------------------------------------------------- tile pass

// The parts of a pass that the kernel needs before its shared copy of the
// descriptor has arrived, by value.
struct FxHead {
    int k, m, a, n_ops, n_slots, chunk0;
    uint32_t zmask, gated;   // every slot of a pass gates the same tile bits
    int coef0, grad0;        // first slot's offsets; the slots follow one another
};

struct FxShared {
    PassDesc d;
    uint32_t flip[kMaxSlots];      // tile bits with an odd number of quarter turns, per slot
    uint32_t half[kMaxSlots];      // the slot's table is scaled by 2^62 (kFxHalf)
    uint32_t wmax[2][16];
    float wsum[2][16];
    long long total[2 * kMaxTileBits];   // block totals of a flush
};

// Sum over the lanes of a warp (the low `lanes` of them, a power of two).
__device__ __forceinline__ long long warp_sum64(long long v, unsigned mask, int lanes) {
    if (lanes == 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    for (int o = lanes >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}

// Block sums of one value per thread (256 threads) with the sign of each of the
// 8 thread bits, by one warp in one butterfly: entry 2 q + 1 of `out` for thread
// bit tb, q = tb below the chunk and tb + 3 above.
__device__ __forceinline__ void total_row_sums(const long long *src, int lane, int chunk, long long *out) {
    long long v[8], d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = src[lane + 32 * i];
#pragma unroll
    for (int j = 0; j < 3; ++j) {   // thread bits 5, 6, 7
        d[5 + j] = 0;
#pragma unroll
        for (int c = 0; c < (8 >> (j + 1)); ++c) {
            const long long x0 = v[2 * c], x1 = v[2 * c + 1];
            d[5 + j] += x0 - x1;
            v[c] = x0 + x1;
        }
    }
    long long s = v[0];
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        const long long o = __shfl_xor_sync(0xffffffffu, s, 1 << b);
        d[b] = ((lane >> b) & 1) ? o - s : s - o;
        s += o;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < b || c >= 5) d[c] += __shfl_xor_sync(0xffffffffu, d[c], 1 << b);
    }
    if (lane < 8) {
        long long x = d[0];
#pragma unroll
        for (int c = 1; c < 8; ++c) x = lane == c ? d[c] : x;
        out[2 * (lane < chunk ? lane : lane + kR) + 1] = x;
    }
}

__device__ __forceinline__ uint32_t abs_hi(long long bits) {
    return (uint32_t)((unsigned long long)bits >> 32) & 0x7fffffffu;
}

// Doubles to integers in place: the tile's exponent from its largest component
// and its 2-norm (in FP32 relative to that component: no overflow, no FP64),
// both block-wide.  E: unit exponent, V = x 2^-E.  bad: the tile holds an
// infinity or a NaN.
template <int NB>
__device__ __forceinline__ void fx_load_tile(long long (&re)[NB][kNR], long long (&im)[NB][kNR],
                                             FxShared &sh, unsigned wmask, int nwarps, int (&E)[NB],
                                             bool (&bad)[NB]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        uint32_t mx = 0u;
#pragma unroll
        for (int r = 0; r < kNR; ++r) mx = max(mx, max(abs_hi(re[u][r]), abs_hi(im[u][r])));
        mx = __reduce_max_sync(wmask, mx);
        if (lane == 0) sh.wmax[u][warp] = mx;
    }
    __syncthreads();
    int ef[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        uint32_t mx = 0u;
        for (int w = 0; w < nwarps; ++w) mx = max(mx, sh.wmax[u][w]);
        ef[u] = (int)(mx >> 20);
        const int base = (ef[u] - 127) * (1 << 20);
        float sum = 0.f;
#pragma unroll
        for (int r = 0; r < kNR; ++r) {
            const float x = __int_as_float(max((int)abs_hi(re[u][r]) - base, 0) << 3);
            const float y = __int_as_float(max((int)abs_hi(im[u][r]) - base, 0) << 3);
            sum = fmaf(x, x, sum);
            sum = fmaf(y, y, sum);
        }
        for (int o = 16; o > 0; o >>= 1)
            if ((wmask >> o) & 1u) sum += __shfl_xor_sync(wmask, sum, o);
        if (lane == 0) sh.wsum[u][warp] = sum;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        float tot = 0.f;
        for (int w = 0; w < nwarps; ++w) tot += sh.wsum[u][w];
        // |tile| < 2^((es + 1) / 2) 2^(ef - 1023); 1.001 covers the truncated mantissas
        const int es = (int)(__float_as_uint(tot * 1.001f) >> 23) - 127;
        E[u] = ef[u] - 1023 + ((es + 2) >> 1) - kFxNormBits;
        bad[u] = ef[u] == 0x7ff;
        if (ef[u] == 0) E[u] = 0;   // all zero (or subnormal)
        if (fx_plain_exponent(E[u])) {
#pragma unroll
            for (int r = 0; r < kNR; ++r) {
                re[u][r] = fx_from_bits(re[u][r], E[u]);
                im[u][r] = fx_from_bits(im[u][r], E[u]);
            }
        } else {
#pragma unroll
            for (int r = 0; r < kNR; ++r) {
                re[u][r] = fx_from_bits_any(re[u][r], E[u]);
                im[u][r] = fx_from_bits_any(im[u][r], E[u]);
            }
        }
    }
}

// One tile bit's gate on the thread's 8 amplitudes of each buffer, register
// bit J.  Forward: RY; backward: its inverse, and the theta gradient
//   Re<l1|p0> - Re<l0|p1>
// of the thread's pairs (buffer 0 = psi, 1 = lambda), in units of 2^61.
template <int J, bool BWD>
__device__ __forceinline__ long long fx_gate(long long (&re)[BWD ? 2 : 1][kNR],
                                             long long (&im)[BWD ? 2 : 1][kNR], const RotFx &c,
                                             bool neg) {
    constexpr int NB = BWD ? 2 : 1;
    if (c.meta & kFx45) {
        // (x - y, x + y), or (x + y, y - x); the difference as 2x minus the sum,
        // so that no operand is copied
        auto turn = [](long long &x, long long &y) {
            y += x;
            x = (x + x) - y;
        };
#pragma unroll
        for (int u = 0; u < NB; ++u) {
#pragma unroll
            for (int r = 0; r < kNR; ++r) {
                if ((r & (1 << J)) || neg) continue;
                turn(re[u][r], re[u][r | (1 << J)]);
                turn(im[u][r], im[u][r | (1 << J)]);
            }
#pragma unroll
            for (int r = 0; r < kNR; ++r) {
                if ((r & (1 << J)) || !neg) continue;
                turn(re[u][r | (1 << J)], re[u][r]);
                turn(im[u][r | (1 << J)], im[u][r]);
            }
        }
    }
    const long long T = ((long long)c.th << 32) + c.tl;
    const long long Tp = neg ? -T : T, Tn = neg ? T : -T;
    const int ph = fx_hi(Tp), pl = fx_lo(Tp), nh = fx_hi(Tn), nl = fx_lo(Tn);
    long long hp = 0, ap = 0, bp = 0, hn = 0, an = 0, bn = 0;
    int cp = 0, cn = 0;
#pragma unroll
    for (int r = 0; r < kNR; ++r) {
        if (r & (1 << J)) continue;
        const int r1 = r | (1 << J);
#pragma unroll
        for (int c2 = 0; c2 < 2; ++c2) {
            long long(&v)[NB][kNR] = c2 ? im : re;
            int xh[NB], xl[NB], yh[NB], yl[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                xh[u] = fx_hi(v[u][r]);
                xl[u] = fx_lo(v[u][r]);
                yh[u] = fx_hi(v[u][r1]);
                yl[u] = fx_lo(v[u][r1]);
            }
            if constexpr (BWD) {
                fx_acc(hp, yh[1], xh[0]);   // l1 p0
                fx_acc(ap, yh[1], xl[0]);
                fx_acc(bp, yl[1], xh[0]);
                cp += __mulhi(xl[0], yl[1] >> 3);
                fx_acc(hn, xh[1], yh[0]);   // l0 p1
                fx_acc(an, xh[1], yl[0]);
                fx_acc(bn, xl[1], yh[0]);
                cn += __mulhi(yl[0], xl[1] >> 3);
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const long long x = v[u][r], y = v[u][r1];
                v[u][r] = fx_ma(x, nh, nl, yh[u], yl[u]);
                v[u][r1] = fx_ma(y, ph, pl, xh[u], xl[u]);
            }
        }
    }
    if constexpr (!BWD) return 0ll;
    // h 2^64 + (a + b) 2^32 + c 2^35 in units of 2^61, rounded (a bias would add
    // up over the threads).  The norms are at most 2^61.75 here and the 16
    // high halves of a thread sum to at most 4 times theirs, so ap - an and
    // bp - bn stay below 2^62.8.
    const long long lo = ((ap - an) >> 1) + ((bp - bn) >> 1) + 4ll * ((long long)cp - cn);
    return ((hp - hn) << 3) + ((lo + (1ll << 27)) >> 28);
}

// A pass in FP64, for run_tile: bound by the FP64 pipe.  24 qubits, depth 8, energy /
// gradient: normal angles of deviation 0.1 in FP64 13.4 / 54.5 ms (54.5 with a row of
// partials per bit, 61.9 with a warp sum per gate), uniform angles in fixed point 6.7
// / 22.5.  Asking which it is costs the fixed-point passes 0.7 % forward (20 qubits,
// 64 energies: 24.51 -> 24.71 ms) and nothing backward (28 qubits: 394.4 -> 394.2).
struct WideEnv {
    using C = double2;
    static constexpr int kLoad = 1;
    static constexpr bool kRows = true;
    const PassDesc *d;
    const RotWide *cf;
    const double2 *dt;
    double *gout;
    uint64_t gslot;
    double2 *P, *L;
    int init_zero;
    int t0;
    __device__ RotCoef<double> coef(int slot, int bit) const {
        const RotWide &r = cf[slot * d->k + bit];
        return RotCoef<double>{r.v, r.gs, r.mode};
    }
    __device__ C diag(int slot, uint32_t e) const { return chain_load(dt + d->slot_dtab_off[slot] + (e >> t0)); }
    __device__ void grad(int slot, int bit, int comp, double v) const { gout[slot * gslot + bit * 2 + comp] = v; }
};

// Forward inlined, backward called: neither then takes registers from the
// fixed-point path (a call reserves some, which the forward's 64 cannot spare).
__device__ __noinline__ void wide_backward(const PassDesc &d, int n_ops, uint64_t base, double2 *buf, double *gsh,
                                           uint32_t size, WideEnv &env) {
    run_tile<double, kR, true>(d, d.ops, n_ops, base, buf, buf + size, gsh, env);
}

// One CTA per (tile, state).  A tile's phases (load, conversion, diagonal,
// gates, exchanges, store) use different pipes, so what counts beside the
// instructions (backward 760, forward 330 per amplitude in a slot of 7 gates) is
// how well the CTAs of an SM overlap: 4 forward CTAs of 64 registers (28 qubits:
// 92.7 ms against 97.2 with 3 of 80), 2 backward ones of 128, few barriers, and
// loads issued before anything else.  4 or 16 amplitudes per thread instead of 8
// are slower backward (348 and 375 against 276 ms).
// Against the same passes in FP64 multiply-adds, whole calls: 28-qubit energy +
// gradient (depth 8) 961 -> 395 ms, 64 energies at 20 qubits (depth 10) 54.6 ->
// 24.7 ms, gradient at 13 qubits (depth 6) 713 -> 433 us.
template <bool BWD, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
k_pass_fx(const FxHead H, const PassDesc *__restrict__ desc, int init_zero, double2 *psi,
          double2 *lam, size_t stride, const RotFx *coefs,
          size_t coef_stride, const longlong2 *dtab, size_t dtab_stride,
          double *gpart, size_t grad_stride) {
    constexpr int NB = BWD ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ FxShared sh;
    const int b = blockIdx.y;
    const uint32_t t = threadIdx.x;
    const int k = H.k, m = H.m, a = H.a;
    // dynamic shared memory: tile(s) | gradient rows (backward) | coefficient rows
    const uint32_t size = tile_buf_elems(k, 16);
    longlong2 *sbuf = reinterpret_cast<longlong2 *>(smem_raw);
    long long *rows = reinterpret_cast<long long *>(sbuf + NB * size);
    RotFx *scf = reinterpret_cast<RotFx *>(rows + (BWD ? (size_t)blockDim.x * (k + 1 + kR) : 0));
    const int mid = a - m;
    const uint32_t lowmask = (1u << m) - 1u;
    const uint64_t tile = blockIdx.x;
    const uint64_t base = ((tile & ((1ull << mid) - 1ull)) << m) | ((tile >> mid) << (a + (k - m)));
    double2 *P = psi + (size_t)b * stride;
    double2 *L = BWD ? lam + (size_t)b * stride : nullptr;
    // gradient partials: slot s at s * gridDim.x * 2 k, then tile-major
    double *gout = BWD ? gpart + (size_t)b * grad_stride + H.grad0 + tile * (uint64_t)(2 * k) : nullptr;
    const uint64_t gslot = (uint64_t)gridDim.x * (2 * k);
    const longlong2 *dt = dtab + (size_t)b * dtab_stride;
    const int t0 = __ffs(H.gated) - 1;   // the tables have no index bits below t0
    auto g32 = [&](uint32_t e) -> uint32_t {
        return (uint32_t)(base | (uint64_t)(e & lowmask) | ((uint64_t)(e >> m) << a));
    };
    pdl_trigger();
    {   // the plan's tables do not depend on earlier kernels
        static_assert(sizeof(PassDesc) % 4 == 0, "descriptor copied in words");
        const uint32_t *src = reinterpret_cast<const uint32_t *>(desc);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&sh.d);
        for (int i = t; i < (int)(offsetof(PassDesc, ops) / 4) + H.n_ops; i += blockDim.x) dst[i] = src[i];
    }
    pdl_wait();
    if (base & H.zmask) {   // block-uniform: psi is zero on this tile (see PassDesc::zmask)
        if (BWD) {
            for (int s = 0; s < H.n_slots; ++s)
                for (int i = t; i < 2 * k; i += blockDim.x) gout[s * gslot + i] = 0.0;
        } else {
            for (uint32_t e = t; e < (1u << k); e += blockDim.x) P[g32(e)] = make_double2(0.0, 0.0);
        }
        return;
    }

    // Global position of the register bits of a round: tile bit b sits at
    // global bit b below m and a + b - m above.
    auto reg_strides = [&](int p, uint32_t (&gs)[kR]) {
#pragma unroll
        for (int j = 0; j < kR; ++j) gs[j] = p + j < m ? 1u << (p + j) : 1u << (a + p + j - m);
    };
    auto reg_xor = [](int r, const uint32_t (&gs)[kR]) -> uint32_t {
        uint32_t x = 0u;
#pragma unroll
        for (int j = 0; j < kR; ++j)
            if ((r >> j) & 1) x ^= gs[j];
        return x;
    };

    // the tile's loads first: the coefficients arrive under them.
    // The state streams past L1, which the tables then stay in.
    long long re[NB][kNR], im[NB][kNR];
    int chunk = H.chunk0;
    {
        const uint32_t g0 = g32(elem_of(t, 0, chunk, kR));
        uint32_t gs[kR];
        reg_strides(chunk, gs);
#pragma unroll
        for (int r = 0; r < kNR; ++r) {
            const uint32_t g = g0 ^ reg_xor(r, gs);
            if (!BWD && init_zero) {
                re[0][r] = g == 0u ? 1ll << (kFxNormBits - 1) : 0ll;
                im[0][r] = 0ll;
            } else {
                const longlong2 x = __ldcg(reinterpret_cast<const longlong2 *>(P + g));
                re[0][r] = x.x;
                im[0][r] = x.y;
            }
            if constexpr (BWD) {
                const longlong2 y = __ldcg(reinterpret_cast<const longlong2 *>(L + g));
                re[1][r] = y.x;
                im[1][r] = y.y;
            }
        }
    }
    const PassDesc &d = sh.d;
    int any_bad = 0, wide = 0;
    {
        const RotFx *src = coefs + (size_t)b * coef_stride + H.coef0;
        if constexpr (!BWD) wide = chain_load(&src[t0].wide);   // (backward has no register to spare)
        for (int i = t; i < H.n_slots * k; i += blockDim.x) {
            const RotFx c = src[i];
            scf[i] = c;
            any_bad |= (int)(c.meta & kFxBad);
        }
    }
    any_bad = __syncthreads_or(any_bad);
    if (BWD ? scf[t0].wide : wide) {   // block-uniform
        WideEnv env{&d, reinterpret_cast<const RotWide *>(scf), reinterpret_cast<const double2 *>(dt), gout, gslot,
                    P, L, init_zero, t0};
        double2 *buf = reinterpret_cast<double2 *>(sbuf);
        if (!BWD && init_zero && H.n_slots == 1) {   // the tile at base 0
            write_product_tile<double>(d, reinterpret_cast<const RotWide *>(scf), env.dt, P, base, lowmask, m, a, k);
            return;
        }
        if constexpr (BWD) wide_backward(d, H.n_ops, base, buf, reinterpret_cast<double *>(rows), size, env);
        else run_tile<double, kR, false>(d, d.ops, H.n_ops, base, buf, nullptr, nullptr, env);
        return;
    }
    for (int s = t; s < H.n_slots; s += blockDim.x) {
        uint32_t f = 0u;
        for (int j = t0; j < k; ++j)
            if (scf[s * k + j].meta & kFxFlip) f |= 1u << j;
        sh.flip[s] = f;
        sh.half[s] = scf[s * k + t0].meta & kFxHalf;
    }
    if (!BWD && init_zero) __syncthreads();   // other tiles: fx_load_tile's
    const uint32_t nthr = blockDim.x;   // 2^(k - 3)
    const int nwarps = (int)((nthr + 31) >> 5);
    const int warp = t >> 5, lane = t & 31;
    const unsigned wmask = nthr >= 32 ? 0xffffffffu : ((1u << nthr) - 1u);
    const int wlanes = nthr >= 32 ? 32 : (int)nthr;

    int E[NB];
    bool bad[NB];
    if (!BWD && init_zero) {
        E[0] = 1 - kFxNormBits;
        bad[0] = false;
    } else {
        fx_load_tile<NB>(re, im, sh, wmask, nwarps, E, bad);
    }
    const int gexp = 64 + E[0] + E[NB - 1];   // gradient partials: integers scaled by 2^gexp
    const bool gplain = gexp > -900 && gexp < 900;
    const double gscale = gplain ? __hiloint2double((gexp + 1023) * (1 << 20), 0) : 0.0;
    const bool gbad = any_bad || bad[0] || bad[NB - 1];
    uint32_t F = 0u;          // flips: stored element e holds logical index e ^ F
    uint32_t Fdiag = 0u;      // F at the last diagonal (phi gradients)
    int dchunk = 0;
    for (int oi = 1; oi < H.n_ops; ++oi) {
        const PassOp op = d.ops[oi];
        if (op.kind == OP_ROUND) {
            const int p = op.chunk;
            uint32_t o[kR];
            // no barrier before the write: a thread writes the places it read last
            {
                longlong2 *bp = sbuf + pad_of<double>(elem_of(t, 0, chunk, kR));
#pragma unroll
                for (int j = 0; j < kR; ++j) o[j] = pad_of<double>(1u << (chunk + j));
#pragma unroll
                for (int r = 0; r < kNR; ++r) {
                    const uint32_t x = ((r & 1) ? o[0] : 0u) + ((r & 2) ? o[1] : 0u) + ((r & 4) ? o[2] : 0u);
#pragma unroll
                    for (int u = 0; u < NB; ++u) bp[u * size + x] = make_longlong2(re[u][r], im[u][r]);
                }
            }
            // with both chunks at or below 5 the warp's number is tile bits 8 and up
            // on both sides: the exchange stays inside the warp
            if (chunk <= 5 && p <= 5) __syncwarp(wmask);
            else __syncthreads();
            {
                const longlong2 *bp = sbuf + pad_of<double>(elem_of(t, 0, p, kR));
#pragma unroll
                for (int j = 0; j < kR; ++j) o[j] = pad_of<double>(1u << (p + j));
#pragma unroll
                for (int r = 0; r < kNR; ++r) {
                    const uint32_t x = ((r & 1) ? o[0] : 0u) + ((r & 2) ? o[1] : 0u) + ((r & 4) ? o[2] : 0u);
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        const longlong2 y = bp[u * size + x];
                        re[u][r] = y.x;
                        im[u][r] = y.y;
                    }
                }
            }
            chunk = p;
        } else if (op.kind == OP_BF) {
            auto gate = [&](auto jc) {
                constexpr int j = decltype(jc)::value;
                if (!((op.mask >> j) & 1)) return;
                const RotFx c = scf[op.slot * k + chunk + j];
                const bool neg = (((F >> (chunk + j)) & 1u) != 0u) != BWD;
                const long long g = fx_gate<j, BWD>(re, im, c, neg);
                if constexpr (BWD) rows[(chunk + j) * nthr + t] = g;
                const int s = (int)((c.meta >> (BWD ? kFxShiftB : kFxShiftF)) & 3u);
                if (s) {
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
#pragma unroll
                        for (int r = 0; r < kNR; ++r) {
                            re[u][r] >>= s;
                            im[u][r] >>= s;
                        }
                    }
                }
            };
            gate(IdxC<0>{});
            gate(IdxC<1>{});
            gate(IdxC<2>{});
        } else if (op.kind == OP_DIAG) {
            const uint32_t cz = d.slot_czmask[op.slot];
            if constexpr (!BWD) F ^= sh.flip[op.slot];
            const uint32_t e0 = elem_of(t, 0, chunk, kR) ^ F;   // logical index of register 0
            const uint32_t g0 = g32(e0);
            // CZ signs of the 8 registers as one mask (see run_tile in pass_core.cuh)
            const uint32_t W = ((g0 & cz) << 1) ^ ((g0 >> 1) & cz);
            const int lo_cnt = min(max(m - chunk, 0), kR);
            uint32_t wv = (W >> chunk) & ((1u << lo_cnt) - 1u);
            if (lo_cnt < kR)
                wv |= ((W >> (a + max(chunk - m, 0))) & ((1u << (kR - lo_cnt)) - 1u)) << lo_cnt;
            uint32_t czt = 0u;
            if (m >= 1) {
                czt = cz & ((1u << (m - 1)) - 1u);
                if (a == m && k > m) czt |= cz & (1u << (m - 1));
            }
            if (k - m >= 2) czt |= ((cz >> a) & ((1u << (k - m - 1)) - 1u)) << m;
            const uint32_t adj = czt >> chunk;
            uint32_t sm = (__popc(g0 & (g0 >> 1) & cz) & 1u) ? 0xffu : 0u;
#pragma unroll
            for (int j = 0; j < kR; ++j) {
                if ((wv >> j) & 1u) sm ^= reg_bit_table(j);
                if (j + 1 < kR && ((adj >> j) & 1u)) sm ^= reg_bit_table(j) & reg_bit_table(j + 1);
            }
            const longlong2 *tab = dt + d.slot_dtab_off[op.slot];
            const uint32_t half = sh.half[op.slot];   // 2 entries per unit: one more doubling
            FxWide ua[BWD ? kNR : 1];
#pragma unroll
            for (int r = 0; r < kNR; ++r) {
                const longlong2 e = chain_load(tab + ((e0 ^ ((uint32_t)r << chunk)) >> t0));
                // signs by complement: one unit of 2^-63 off
                const long long sg = -(long long)((sm >> r) & 1u);
                const long long dre = e.x ^ sg, dim = e.y ^ sg, dng = e.y ^ ~sg;
                const int drh = fx_hi(dre), drl = fx_lo(dre), dih = fx_hi(dim), dil = fx_lo(dim);
                const int dnh = fx_hi(dng), dnl = fx_lo(dng);
                int xh[NB], xl[NB], yh[NB], yl[NB];
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    xh[u] = fx_hi(re[u][r]);
                    xl[u] = fx_lo(re[u][r]);
                    yh[u] = fx_hi(im[u][r]);
                    yl[u] = fx_lo(im[u][r]);
                }
                // dE/dphi_q = Im<l|Z_q|p> = sum_i u_i (-1)^{bit_q(i)}, u = Im(conj(l) p)
                if constexpr (BWD)
                    ua[r] = fx_cross(xh[1], xl[1], yh[0], yl[0], yh[1], yl[1], xh[0], xl[0]);
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    if constexpr (!BWD) {
                        re[u][r] = fx_dot(xh[u], xl[u], drh, drl, yh[u], yl[u], dnh, dnl);
                        im[u][r] = fx_dot(xh[u], xl[u], dih, dil, yh[u], yl[u], drh, drl);
                    } else {
                        re[u][r] = fx_dot(xh[u], xl[u], drh, drl, yh[u], yl[u], dih, dil);
                        im[u][r] = fx_dot(xh[u], xl[u], dnh, dnl, yh[u], yl[u], drh, drl);
                    }
                }
            }
            if (half) {
#pragma unroll
                for (int u = 0; u < NB; ++u) {
#pragma unroll
                    for (int r = 0; r < kNR; ++r) {
                        re[u][r] <<= 1;
                        im[u][r] <<= 1;
                    }
                }
            }
            if constexpr (BWD) {
                // the thread's total (row k) and its signed sums over the chunk's
                // bits (rows k + 1 + j), in units of 2^60; the flush takes the sign
                // of the other bits from the thread's element base
                Fdiag = F;
                dchunk = chunk;
#pragma unroll
                for (int j = 0; j < kR; ++j) {
                    long long dh = 0, dm = 0;
#pragma unroll
                    for (int c = 0; c < (kNR >> (j + 1)); ++c) {
                        const FxWide x0 = ua[2 * c], x1 = ua[2 * c + 1];
                        dh += x0.h - x1.h;
                        dm += x0.m - x1.m;
                        ua[c] = FxWide{x0.h + x1.h, x0.m + x1.m};
                    }
                    rows[(k + 1 + j) * nthr + t] = (dh << 4) + ((dm + (1ll << 24)) >> 25);
                }
                rows[k * nthr + t] = (ua[0].h << 4) + ((ua[0].m + (1ll << 24)) >> 25);
                F ^= sh.flip[op.slot];
            }
        } else if (BWD) {   // OP_FLUSH: block totals of the slot's gradient partials
            // Integer sums: exact and independent of their order.
            __syncthreads();
            const uint32_t gated = H.gated;
            if (nthr == 256) {
                if (warp == 0) {
                    total_row_sums(rows + k * nthr, lane, dchunk, sh.total);
                } else {
                    // the theta rows and the chunk's phi rows
                    for (int row = warp - 1; row < k + kR; row += 7) {
                        const int q = row < k ? row : dchunk + row - k;
                        if (!((gated >> q) & 1u)) continue;
                        const long long *src = rows + (row < k ? row : row + 1) * 256;
                        long long sum = src[lane];
#pragma unroll
                        for (int i = 1; i < 8; ++i) sum += src[lane + 32 * i];
                        sum = warp_sum64(sum, wmask, 32);
                        if (lane == 0) sh.total[2 * q + (row < k ? 0 : 1)] = sum;
                    }
                }
            } else {
                for (int idx = warp; idx < 2 * k; idx += nwarps) {
                    const int q = idx >> 1;
                    if (!((gated >> q) & 1u)) continue;
                    const bool theta = (idx & 1) == 0;
                    const bool in_chunk = q >= dchunk && q < dchunk + kR;
                    const long long *src = rows + (theta ? q : (in_chunk ? k + 1 + q - dchunk : k)) * nthr;
                    // phi of a bit outside the chunk: the total row with the sign of
                    // thread bit tb; bits below 5 are the lane's
                    const int tb = theta || in_chunk ? -1 : (q < dchunk ? q : q - kR);
                    const uint32_t imask = tb >= 5 ? 1u << (tb - 5) : 0u;
                    long long sum = 0;
                    for (uint32_t i = 0; i < (uint32_t)nwarps; ++i) {
                        const long long v = src[lane + 32 * i];
                        sum += (i & imask) ? -v : v;
                    }
                    if (tb >= 0 && tb < 5 && ((lane >> tb) & 1)) sum = -sum;
                    sum = warp_sum64(sum, wmask, wlanes);
                    if (lane == 0) sh.total[idx] = sum;
                }
            }
            __syncthreads();
            // one thread per row: to doubles, scaled
            if (t < 2u * k || nthr < 2u * k) {
                for (int idx = t; idx < 2 * k; idx += nthr) {
                    const int q = idx >> 1;
                    if (!((gated >> q) & 1u)) continue;
                    const bool theta = (idx & 1) == 0;
                    double v = (double)sh.total[idx] * (theta ? scf[op.slot * k + q].gs : 0.0625);
                    v = gplain ? v * gscale : ldexp(v, gexp);
                    if (((theta ? F : Fdiag) >> q) & 1u) v = -v;
                    if (gbad) v = __longlong_as_double(0x7ff8000000000000ll);
                    gout[op.slot * gslot + idx] = v;
                }
            }
        }
    }
    {   // store: logical index e ^ F
        const uint32_t g0 = g32(elem_of(t, 0, chunk, kR) ^ F);
        uint32_t gs[kR];
        reg_strides(chunk, gs);
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            double2 *out = u ? L : P;
            if (any_bad || bad[u]) {
                const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
                for (int r = 0; r < kNR; ++r) out[g0 ^ reg_xor(r, gs)] = make_double2(nan, nan);
            } else if (fx_plain_exponent(E[u])) {
#pragma unroll
                for (int r = 0; r < kNR; ++r)
                    *reinterpret_cast<longlong2 *>(out + (g0 ^ reg_xor(r, gs))) =
                        make_longlong2(fx_to_bits(re[u][r], E[u]), fx_to_bits(im[u][r], E[u]));
            } else {
#pragma unroll
                for (int r = 0; r < kNR; ++r)
                    *reinterpret_cast<longlong2 *>(out + (g0 ^ reg_xor(r, gs))) =
                        make_longlong2(fx_to_bits_any(re[u][r], E[u]), fx_to_bits_any(im[u][r], E[u]));
            }
        }
    }
}

// What vqe_set_plan_options accepts by the tile buffers alone fits with the rows, the
// coefficients and the static part: the largest plan is 2^12 amplitudes, 512 threads.
constexpr int kFxMaxTileBits = kR + 9;
static_assert(2 * tile_buf_elems(kFxMaxTileBits, 16) * 16 +
                      (1u << (kFxMaxTileBits - kR)) * (kFxMaxTileBits + 1 + kR) * sizeof(long long) +
                      kMaxSlots * kFxMaxTileBits * sizeof(RotFx) + sizeof(FxShared) <=
                  227 * 1024,
              "the largest fixed-point plan fits the shared memory of a block");

template <bool BWD, int MAXT, int MINB>
cudaError_t launch_k(const PassDesc *desc_dev, const PassDesc &dh, int n_qubits, int batch, void *psi,
                     void *lam, size_t stride, const RotFx *coefs, size_t coef_stride,
                     const void *dtab, size_t dtab_stride, double *gpart, size_t grad_stride,
                     int init_zero, cudaStream_t s) {
    const int threads = 1 << (dh.k - kR);
    size_t smem = size_t(tile_buf_elems(dh.k, 16)) * 16 * (BWD ? 2 : 1) +
                  size_t(dh.n_slots) * dh.k * sizeof(RotFx);
    if (BWD) smem += size_t(threads) * (dh.k + 1 + kR) * sizeof(long long);
    auto kern = k_pass_fx<BWD, MAXT, MINB>;
    if (const cudaError_t e = allow_smem((const void *)kern, smem); e != cudaSuccess) return e;
    dim3 grid((unsigned)(1ull << (n_qubits - dh.k)), batch);
    const FxHead head{dh.k, dh.m, dh.a, dh.n_ops, dh.n_slots, dh.ops[0].chunk, dh.zmask,
                      dh.slot_gated[0], dh.slot_coef_off[0], dh.slot_grad_off[0]};
    return pdl_launch(kern, grid, threads, smem, s, pdl_pays(grid), head, desc_dev, init_zero, static_cast<double2 *>(psi),
                                     static_cast<double2 *>(lam), stride, coefs, coef_stride,
                                     static_cast<const longlong2 *>(dtab), dtab_stride, gpart,
                                     grad_stride);
}

}  // namespace

cudaError_t launch_stage_fx(const StageSlot *slots_dev, int n_slots, int n_qubits, int depth,
                            const double *params, int batch, RotFx *coefs, size_t coef_stride,
                            void *dtab, size_t dtab_stride, cudaStream_t s) {
    if (n_slots == 0 || batch == 0) return cudaSuccess;
    dim3 grid(n_slots, batch);
    k_stage_fx<<<grid, 256, 0, s>>>(slots_dev, n_qubits, depth, params, coefs, coef_stride,
                                    static_cast<longlong2 *>(dtab), dtab_stride);
    return cudaGetLastError();
}

cudaError_t launch_pass_fx(const PassDesc *desc_dev, const PassDesc &dh, int n_qubits, int batch,
                           void *psi, void *lam, size_t stride, const RotFx *coefs,
                           size_t coef_stride, const void *dtab, size_t dtab_stride, double *gpart,
                           size_t grad_stride, bool backward, int init_zero, cudaStream_t s) {
    const int threads = 1 << (dh.k - kR);
    if (dh.R != kR || threads > 512) return cudaErrorInvalidConfiguration;
    if (threads <= 256)
        return backward ? launch_k<true, 256, 2>(desc_dev, dh, n_qubits, batch, psi, lam, stride, coefs,
                                                 coef_stride, dtab, dtab_stride, gpart, grad_stride, 0, s)
                        : launch_k<false, 256, 4>(desc_dev, dh, n_qubits, batch, psi, nullptr, stride,
                                                  coefs, coef_stride, dtab, dtab_stride, gpart,
                                                  grad_stride, init_zero, s);
    return backward ? launch_k<true, 512, 1>(desc_dev, dh, n_qubits, batch, psi, lam, stride, coefs,
                                             coef_stride, dtab, dtab_stride, gpart, grad_stride, 0, s)
                    : launch_k<false, 512, 1>(desc_dev, dh, n_qubits, batch, psi, nullptr, stride, coefs,
                                              coef_stride, dtab, dtab_stride, gpart, grad_stride,
                                              init_zero, s);
}

}  // namespace vqe
