// Kernels of the particle-conserving ansatz (Sec. II-B, Eqs. 5-6):
// psi(theta) = U(theta) psi_HF with U a product of fermionic excitation gates
// exp(theta (T - T^dag)), T = a_p^dag a_r (single) or a_p^dag a_q^dag a_r a_s
// (double), under the Jordan-Wigner mapping.
//
// A gate pairs each basis state j whose annihilated modes are occupied and
// created modes empty with j' = j ^ (amask | cmask); on the pair it is the
// rotation
//     psi_j  <- cos t psi_j  - sgn sin t psi_j'
//     psi_j' <- cos t psi_j' + sgn sin t psi_j,   sgn = (-1)^(sign0 + popc(j & smask)),
// and leaves every other amplitude alone.  A pass stages tiles of 2^k amplitudes
// in shared memory (the low m tile bits are a contiguous run of the state, the
// other k - m the modes of its gates) and applies a run of consecutive gates
// whose modes lie in the tile, one barrier per gate.  The sign factors into a
// per-tile part (the sign mask's bits outside the tile, fixed by the tile's
// base) and a per-element parity over the tile bits.
//
// Excitations keep the number of electrons, so every amplitude whose index does
// not have n_elec ones is zero for good.  Inside a tile the live amplitudes are
// the tile words with n_elec - popc(base) ones: at most binomial(11, 5) = 462 of
// 2048 (FP64) or 924 of 4096.  Shared memory holds just this class, in the order
// of a constant table of the words sorted by popcount; a gate's live pairs are a
// class of the words of its free bits; elements that no gate of the pass pairs
// are not read or written.  Where every gate also keeps the electrons of one
// spin's modes, elements with another number of those are left out too.
// lambda = H psi is needed, and kept up, in the sector alone, because psi is zero
// elsewhere and the gates do not leave it.
//
// At 28 qubits and half filling 15 % of the amplitudes have the right number of
// ones, 4.4 % the right spins.  118 excitations in FP64, forward / backward:
// whole tiles 59.1 / 176.6 ms, the number sector 16.0 / 33.5, with the spins
// 12.7 / 22.2; complex64 at 27 qubits 13.0 / 27.5, 4.7 / 8.0, 4.5 / 5.9 ms.
//
// Before the wait for the kernel before, a warp per gate lists the gate's live
// pairs (their places in shared memory, from the table), so that a gate is one
// list entry, the rotation and a barrier (FP64, 14 qubits, 60 excitations: forward
// 66 -> 48 us, backward 93 -> 73, against looking the places up at the gate).
// FP64 gives a pair two lanes, one per component: half the FP64 instructions per
// warp where the 35 pairs of a double (11 tile bits, 5 electrons) are all there is.
//
// What bounds it now: at small sizes the chain of launch, staging and one
// barrier per gate; at large ones the latency of a tile (nine or more blocks per
// SM hide it) and the memory's 32-byte sectors, of which the scattered elements
// fill a half.
//
// The backward (adjoint) pass un-applies the gates in reverse on psi and
// lambda = H psi and, before un-applying gate g, takes
//     dE/dtheta_g = 2 Re <lambda| G_g |psi>,  G_g = T_g - T_g^dag,
// per pair sgn * (Re conj(lambda_j') psi_j - Re conj(lambda_j) psi_j').
#include "csum.cuh"
#include "pdl.cuh"
#include "sector.cuh"
#include "smem_limit.h"
#include "vqe_internal.h"

namespace vqe {

template <typename T> struct XV2;
template <> struct XV2<float> { using type = float2; };
template <> struct XV2<double> { using type = double2; };

constexpr int kExcMaxHigh = 7;   // k - m <= 7: 128 high-part offsets per pass
constexpr int kExcWide = 256;             // threads of a block of a grid that leaves the chip room
constexpr uint64_t kExcWideBlocks = 608;   // four per SM

template <typename T>
__global__ void k_exc_stage(const double *__restrict__ params, int total, T *__restrict__ cs) {
    pdl_trigger();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    double s, c;
    sincos(params[i], &s, &c);
    cs[2 * i] = (T)c;
    cs[2 * i + 1] = (T)s;
}

template <typename T>
cudaError_t launch_exc_stage(const double *params, int n_exc, int batch, T *cs, cudaStream_t s) {
    const int total = n_exc * batch;
    if (total == 0) return cudaSuccess;
    k_exc_stage<T><<<(total + 255) / 256, 256, 0, s>>>(params, total, cs);
    return cudaGetLastError();
}

// A gate of the pass as the tile's threads use it.
struct TileGate {
    uint32_t amask, flip;    // flip = amask | cmask
    uint32_t smask_t, sign;  // sign of the tile's base included
    uint32_t fixed, n_fixed; // four tile bits, a byte each
    uint32_t word, pairs;    // its live pairs' free bits: kClass.word[word ...]
};

// Places of both elements of pair f of a gate, whether it is dead for its spins
// (bit 30) and its sign (bit 31).
__device__ __forceinline__ uint32_t locate(const TileGate &G, uint32_t f, uint32_t at, uint32_t up, int up_left) {
    uint32_t e = kClass.word[G.word + f];
    uint32_t fx = G.fixed;
    for (uint32_t i = 0; i < G.n_fixed; ++i, fx >>= 8) {   // zero bits at the gate's modes
        const uint32_t low = (1u << (fx & 31u)) - 1u;
        e += e & ~low;
    }
    e |= G.amask;
    return kClass.place[at + e] | (uint32_t)kClass.place[at + (e ^ G.flip)] << 15 |
           (uint32_t)(__popc(e & up) != up_left) << 30 |
           (G.sign ^ (__popc(e & G.smask_t) & 1u)) << 31;
}

__device__ __forceinline__ double xflip(double v, uint32_t s) {
    return __longlong_as_double(__double_as_longlong(v) ^ ((unsigned long long)s << 63));
}
__device__ __forceinline__ float xflip(float v, uint32_t s) {
    return __int_as_float(__float_as_int(v) ^ (int)(s << 31));
}

template <typename T, bool BWD, int TH>
__global__ void __launch_bounds__(TH)
k_exc_pass(ExcPass P, const ExcGate *__restrict__ gates, const uint32_t *__restrict__ hoff,
           typename XV2<T>::type *psi, typename XV2<T>::type *lam,
           size_t stride, const T *cs, int n_exc, double *gpart,
           size_t grad_stride, int init_hf, uint64_t hf, uint32_t spin, int room, int span) {
    using C = typename XV2<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ TileGate sg[kExcMaxGates];
    __shared__ T scs[2 * kExcMaxGates];
    __shared__ uint32_t shoff[1 << kExcMaxHigh];
    const int k = P.k, m = P.m, ng = P.n_gates;
    const uint32_t size = 1u << k, at = size - 1u;
    const uint32_t tid = threadIdx.x;
    C *sp = reinterpret_cast<C *>(smem_raw);   // the live elements of the tile
    C *sl = BWD ? sp + room : nullptr;
    // backward: per-thread gradient partials, one row of TH per gate
    // (FP64 values, or compensated FP32 pairs in the FP32 kernel)
    unsigned char *rows = reinterpret_cast<unsigned char *>(sp + (BWD ? 2 * room : room));
    // the gates' live pairs (locate), `span` words each
    uint32_t *list = reinterpret_cast<uint32_t *>(rows + (BWD ? (size_t)ng * TH * 8 : 0));
    const int b = blockIdx.y;
    C *Pp = psi + (size_t)b * stride;
    C *Lp = BWD ? lam + (size_t)b * stride : nullptr;
    uint64_t base = 0;   // the tile number's bits at the bits of bmask, run by run
    {
        uint32_t bm = P.bmask;
        uint64_t t = blockIdx.x;
        while (bm) {
            const int lo = __ffs(bm) - 1;
            const uint32_t up = bm >> lo;
            const int len = up == 0xffffffffu ? 32 : __ffs(~up) - 1;
            const uint64_t run = (1ull << len) - 1ull;
            base |= (t & run) << lo;
            t >>= len;
            bm &= ~(uint32_t)(run << lo);
        }
    }
    // the plan's tables do not depend on earlier kernels; they are on their way
    // while the block waits
    pdl_trigger();
    static_assert(2 * kExcMaxGates <= TH, "one entry per thread");
    const uint32_t lowmask = (1u << m) - 1u;
    const int left = __popcll(hf) - __popcll(base);   // electrons in the tile's modes
    // and those of them in the modes of `spin`, of which the tile has n_up
    const int up_left = __popc((uint32_t)hf & spin) - __popc((uint32_t)base & spin);
    const int n_up = __popc(spin & ~P.bmask);
    const bool live = left >= 0 && left <= k && up_left >= 0 && up_left <= n_up &&
                      left - up_left >= 0 && left - up_left <= k - n_up &&
                      (BWD ? (base & P.bzmask) == P.bzval : (base & P.zmask) == P.zval);   // block-uniform
    constexpr int kPer = (sizeof(T) == 8 ? 512 : 1024) / TH;   // C(11,5) = 462, C(12,6) = 924 live ones
    constexpr uint32_t kSplit = sizeof(T) == 8 ? 2 : 1;   // lanes per pair; FP64: one per component
    constexpr uint32_t kNone = ~0u;
    uint32_t at_g[kPer];     // where this thread's elements of the class lie in the state
    uint32_t mine = 0u;      // which of them the pass moves
    uint32_t up = 0u;        // the modes of `spin` among the tile bits
    if (live) {
        if ((int)tid < ng) {
            const ExcGate my = gates[P.g_begin + tid];
            TileGate &G = sg[tid];
            G.amask = my.amask;
            G.flip = my.amask | my.cmask;
            G.smask_t = my.smask_t;
            G.sign = (uint32_t)((__popcll(base & (uint64_t)my.smask_g) + my.sign0) & 1);
            G.fixed = my.fixed[0] | my.fixed[1] << 8 | my.fixed[2] << 16 | (uint32_t)my.fixed[3] << 24;
            G.n_fixed = my.n_fixed;
            const int nb = k - my.n_fixed, p = left - my.n_fixed / 2;
            const bool some = p >= 0 && p <= nb;
            G.word = some ? (1u << nb) - 1u + kClass.begin[nb][p] : 0u;
            G.pairs = some ? kClass.begin[nb][p + 1] - kClass.begin[nb][p] : 0u;
        }
        for (uint32_t i = tid; i < (1u << (k - m)); i += TH) shoff[i] = hoff[P.hoff + i];
        const uint32_t first = kClass.begin[k][left], n_live = kClass.begin[k][left + 1] - first;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const uint32_t j = tid + u * TH;
            at_g[u] = j < n_live ? kClass.word[at + first + j] : kNone;
        }
        __syncthreads();
        {
            const uint32_t lane = tid & 31u;
            const bool in = (int)lane < k - m && (shoff[1u << lane] & spin) != 0u;
            up = (spin & lowmask) | __ballot_sync(0xffffffffu, in) << m;
        }
        // only elements that a gate pairs are read and written
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const uint32_t e = at_g[u];
            if (e == kNone) continue;
            bool used = !BWD && init_hf;
            for (int i = 0; i < ng; ++i) {
                const uint32_t v = e & sg[i].flip;
                used |= v == sg[i].amask || (v ^ sg[i].flip) == sg[i].amask;
            }
            used = used && ((!BWD && init_hf) || __popc(e & up) == up_left);
            mine |= (uint32_t)used << u;
            at_g[u] = (uint32_t)base | (e & lowmask) | shoff[e >> m];
        }
        // the gates' lists of live pairs, a gate per warp
        for (int i = tid >> 5; i < ng; i += TH / 32) {
            const uint32_t pairs = sg[i].pairs, lane = tid & 31u;
            uint32_t n = 0;
            for (uint32_t f = lane; f - lane < pairs; f += 32) {
                const uint32_t loc = f < pairs ? locate(sg[i], f, at, up, up_left) : 1u << 30;
                const bool ok = ((loc >> 30) & 1u) == 0u;
                const uint32_t votes = __ballot_sync(0xffffffffu, ok);
                if (ok) list[i * span + n + __popc(votes & ((1u << lane) - 1u))] = loc;
                n += __popc(votes);
            }
            if (lane == 0) sg[i].pairs = n;
        }
    }
    pdl_wait();
    if (!live) {
        if (BWD) {
            double *out = gpart + (size_t)b * grad_stride + P.grad_off + (size_t)blockIdx.x * ng;
            for (int i = tid; i < ng; i += TH) out[i] = 0.0;
        } else if (init_hf) {   // the first pass writes the whole state
            for (uint32_t e = tid; e < size; e += TH)
                Pp[base | (e & lowmask) | hoff[P.hoff + (e >> m)]] = C{};
        }
        return;
    }
    const T *my_cs = cs + (size_t)b * n_exc * 2;
    if ((int)tid < 2 * ng)   // gate g of the table has parameter g
        scs[tid] = my_cs[2 * P.g_begin + tid];
    T one = T(1);
    if (!BWD && init_hf && base == (hf & P.bmask)) {
        // an angle that is not a number shows in the energy, also where its
        // gate has no pair in the sector
        int bad = 0;
        for (int i = tid; i < n_exc; i += TH) bad |= !isfinite(my_cs[2 * i]);
        if (__syncthreads_or(bad)) one = T(NAN);
    }
    {
        C x[kPer], l[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (!((mine >> u) & 1u)) continue;
            if (!BWD && init_hf) {
                x[u].x = (at_g[u] == (uint32_t)hf) ? one : T(0);
                x[u].y = T(0);
            } else {
                x[u] = Pp[at_g[u]];
                if (BWD) l[u] = Lp[at_g[u]];
            }
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (!((mine >> u) & 1u)) continue;
            sp[tid + u * TH] = x[u];
            if (BWD) sl[tid + u * TH] = l[u];
        }
    }
    __syncthreads();
    for (int ii = 0; ii < ng; ++ii) {
        const int i = BWD ? ng - 1 - ii : ii;
        const TileGate &G = sg[i];
        const T c = scs[2 * i], s = scs[2 * i + 1];
        const uint32_t count = G.pairs * kSplit;
        double gd = 0.0;
        F32c gf = f32c_zero();
        for (uint32_t f = tid; f < count; f += TH) {
            const uint32_t loc = list[i * span + f / kSplit];
            const uint32_t i1 = loc & 0x7fffu, i2 = (loc >> 15) & 0x7fffu, par = loc >> 31;
            const T ss = xflip(s, par);
            if constexpr (sizeof(T) == 8) {
                double *p1 = reinterpret_cast<double *>(sp + i1) + (tid & 1u);
                double *p2 = reinterpret_cast<double *>(sp + i2) + (tid & 1u);
                const double x = *p1, y = *p2;
                if (!BWD) {
                    *p1 = fma(c, x, -ss * y);
                    *p2 = fma(c, y, ss * x);
                } else {
                    double *q1 = reinterpret_cast<double *>(sl + i1) + (tid & 1u);
                    double *q2 = reinterpret_cast<double *>(sl + i2) + (tid & 1u);
                    const double lx = *q1, ly = *q2;
                    gd += xflip(fma(ly, x, -(lx * y)), par);
                    *p1 = fma(c, x, ss * y);
                    *p2 = fma(c, y, -ss * x);
                    *q1 = fma(c, lx, ss * ly);
                    *q2 = fma(c, ly, -ss * lx);
                }
            } else {
                const C x = sp[i1], y = sp[i2];
                C nx, ny;
                if (!BWD) {
                    nx.x = fma(c, x.x, -ss * y.x);
                    nx.y = fma(c, x.y, -ss * y.y);
                    ny.x = fma(c, y.x, ss * x.x);
                    ny.y = fma(c, y.y, ss * x.y);
                } else {
                    const C lx = sl[i1], ly = sl[i2];
                    f32c_add(gf, xflip(fma(ly.x, x.x, fma(ly.y, x.y, -fma(lx.x, y.x, lx.y * y.y))), par));
                    nx.x = fma(c, x.x, ss * y.x);
                    nx.y = fma(c, x.y, ss * y.y);
                    ny.x = fma(c, y.x, -ss * x.x);
                    ny.y = fma(c, y.y, -ss * x.y);
                    C mx, my;
                    mx.x = fma(c, lx.x, ss * ly.x);
                    mx.y = fma(c, lx.y, ss * ly.y);
                    my.x = fma(c, ly.x, -ss * lx.x);
                    my.y = fma(c, ly.y, -ss * lx.y);
                    sl[i1] = mx;
                    sl[i2] = my;
                }
                sp[i1] = nx;
                sp[i2] = ny;
            }
        }
        if constexpr (BWD) {
            if constexpr (sizeof(T) == 8) reinterpret_cast<double *>(rows)[i * TH + tid] = gd;
            else reinterpret_cast<F32c *>(rows)[i * TH + tid] = gf;
        }
        __syncthreads();   // the next gate's pairs touch other threads' elements
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        if (!((mine >> u) & 1u)) continue;
        const uint32_t j = tid + u * TH;
        Pp[at_g[u]] = sp[j];
        if (BWD) Lp[at_g[u]] = sl[j];
    }
    if (!BWD && init_hf)   // the first pass writes the whole state
        for (uint32_t e = tid; e < size; e += TH)
            if (__popc(e) != left) Pp[base | (e & lowmask) | shoff[e >> m]] = C{};
    if constexpr (BWD) {
        // each warp sums whole rows in a fixed order (bitwise reproducible)
        double *out = gpart + (size_t)b * grad_stride + P.grad_off + (size_t)blockIdx.x * ng;
        const int warp = tid >> 5, lane = tid & 31;
        const int nw = TH / 32;
        for (int i = warp; i < ng; i += nw) {
            // threads beyond the gate's pairs hold zeros
            const int used = (int)min(sg[i].pairs * kSplit, (uint32_t)TH);
            if constexpr (sizeof(T) == 8) {
                const double *r = reinterpret_cast<const double *>(rows) + i * TH;
                double sum = 0.0;
                for (int t = lane; t < used; t += 32) sum += r[t];
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == 0) out[i] = 2.0 * sum;
            } else {
                const F32c *r = reinterpret_cast<const F32c *>(rows) + i * TH;
                F32c sum = f32c_zero();
                for (int t = lane; t < used; t += 32) sum = f32c_add(sum, r[t]);
                sum = f32c_warp_sum(sum, 0xffffffffu, 32);
                if (lane == 0) out[i] = 2.0 * f32c_value(sum);
            }
        }
    }
}

template <typename T>
cudaError_t launch_exc_pass(const ExcPass &P, const ExcGate *gates_dev, const uint32_t *hoff_dev,
                            int n_qubits, int batch, void *psi, void *lam, size_t state_stride,
                            const T *cs, int n_exc, double *gpart, size_t grad_stride,
                            bool backward, int init_hf, uint64_t hf_index, uint32_t spin, cudaStream_t s) {
    using C = typename XV2<T>::type;
    const dim3 grid(1u << (n_qubits - P.k), batch);
    int room = 1;   // the largest class: binomial(k, k / 2)
    for (int i = 1; i <= P.k / 2; ++i) room = room * (P.k + 1 - i) / i;
    if (P.k > (sizeof(T) == 8 ? 11 : 12)) return cudaErrorInvalidValue;
    const size_t row = sizeof(T) == 8 ? sizeof(double) : sizeof(F32c);
    // 256 threads where a grid leaves the chip room, for a shorter chain per gate;
    // 128 beyond, for more tiles per SM.  FP64, forward + backward of 100
    // excitations, 128 / 256 threads: 14 qubits (8 blocks) 200 / 184 us, 18 (128)
    // 304 / 242, 20 (512) 390 / 327, 21 (1024) 471 / 578; complex64: 18 (64) 183 /
    // 160 us, 21 (512) 293 / 304, 22 (1024) 409 / 547.
    // FP64 forward has half the rows to move and no partials: 64 threads from 2048
    // blocks on (22 qubits 276 -> 232 us, 24 789 -> 709, 28 14.7 -> 12.7 ms; at 1024
    // blocks 163 -> 192 us, and backward and complex64 are slower with 64).
    const uint64_t blocks = uint64_t(grid.x) * grid.y;
    const bool small = sizeof(T) == 8 && !backward && blocks >= 2048;
    const int th = small ? 64 : blocks <= kExcWideBlocks ? kExcWide : kExcThreads;
    int span = 1;   // the most pairs: a single's, binomial(k - 2, (k - 2) / 2)
    for (int i = 1; i <= (P.k - 2) / 2; ++i) span = span * (P.k - 1 - i) / i;
    const size_t smem = room * sizeof(C) * (backward ? 2 : 1) +
                        P.n_gates * ((backward ? th * row : 0) + span * sizeof(uint32_t));
    auto launch = [&](auto kern) {
        if (const cudaError_t e = allow_smem((const void *)kern, smem); e != cudaSuccess) return e;
        return pdl_launch(kern, grid, th, smem, s, true, P, gates_dev, hoff_dev, static_cast<C *>(psi),
                          static_cast<C *>(lam), state_stride, cs, n_exc, gpart, grad_stride, init_hf, hf_index,
                          spin, room, span);
    };
    if (th == kExcWide) return backward ? launch(k_exc_pass<T, true, kExcWide>) : launch(k_exc_pass<T, false, kExcWide>);
    if constexpr (sizeof(T) == 8)
        if (small) return launch(k_exc_pass<T, false, 64>);
    return backward ? launch(k_exc_pass<T, true, kExcThreads>) : launch(k_exc_pass<T, false, kExcThreads>);
}

template cudaError_t launch_exc_stage<float>(const double *, int, int, float *, cudaStream_t);
template cudaError_t launch_exc_stage<double>(const double *, int, int, double *, cudaStream_t);
template cudaError_t launch_exc_pass<float>(const ExcPass &, const ExcGate *, const uint32_t *, int,
                                            int, void *, void *, size_t, const float *, int,
                                            double *, size_t, bool, int, uint64_t, uint32_t, cudaStream_t);
template cudaError_t launch_exc_pass<double>(const ExcPass &, const ExcGate *, const uint32_t *, int,
                                             int, void *, void *, size_t, const double *, int,
                                             double *, size_t, bool, int, uint64_t, uint32_t, cudaStream_t);

}  // namespace vqe
