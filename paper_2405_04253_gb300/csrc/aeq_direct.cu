// aeq_direct.cu -- the AEQ (4x4 real-valued MIMO, RDE update of eq. (6)) with its
// convolutions and gradient as exact integer dot products.
//
// The transform kernels (aeq.cu, aeq_serial.cu) form each convolution through
// Fermat number transforms because a multiplication is what the paper's datapath
// cannot afford.  Constraint (5) makes every such convolution exact, so it equals
// the plain integer sum, and an SM multiplies as fast as it shifts: dp2a (two
// 16-bit by 8-bit products and an add) issues at the half rate of every shift,
// prmt and 32-bit multiply-add here (64 lanes a clock and SM, 4.4 cycles latency
// measured).  Per symbol and output the direct form takes 4 x 16 products, 32
// dp2a; the transforms took about 25 times as many instructions for a block.
// Results are the same integers for every input inside the documented ranges
// (5-bit symbols, 14-bit taps).
//
// Per block of SA = N - 16 symbols and output:
//   convolution  y_o[i] = sum_s1,k W_o,s1[k] x_s1[t0 + i - k]
//   error        z = sat16(y >> 7), one shuffle for the other output, e in 32 bits
//   gradient     G = sum_i e z_o[i] x_s1[t0 + i - k] with e z = c1 2^16 + c0
//                (c0 16 bits, c1 signed 16 bits) and, only when some |e z| of the
//                block reaches 2^31, c2 2^32: two (three) dp2a for two products;
//                limb sums are exact in 32 bits, then combined in 64
//   update       eq. (6) on the master taps, published as 16-bit taps
//
// Staged symbols.  xq[q] holds, for the four inputs, the four bytes of symbols
// q .. q + 3 (a 4 x 4 byte transpose at every q, 16 bytes a symbol), so both the
// convolution (four taps of an input against one word) and the gradient (four
// symbols of an input) read aligned 16-byte words at any offset.  A batch of
// blocks is transposed at once while the next batch's words arrive by cp.async.
//
// Two layouts; aeq_direct_split picks one (rule and figures there).
//   aeq_duo_kernel    a warp per (chain, polarisation): many chains, bound by dp2a issue
//                     and shared-memory loads
//   aeq_split_kernel  six or eight warps per (chain, polarisation), by role: few
//                     chains, bound by the latency of one block
#include <algorithm>

#include <cuda_runtime.h>

#include "host.h"
#include "internal.h"

namespace fnt {

namespace {

template <int NA, int PB_>
struct DirCfg {
    static constexpr int K = kAeqK;
    static constexpr int SA = NA - K;                     // symbols per block
    static constexpr int NG = SA / 4;                     // groups of four symbols
    static constexpr int PB = PB_;                        // blocks per staged batch
    static constexpr int B = PB * SA;                     // symbols per staged batch
    static constexpr int XW = K + B;                      // staged words: K of history
    static_assert(K == 16 && SA % 16 == 0, "shapes");
};

template <bool AS, bool HI>
__device__ __forceinline__ int32_t dp2a(uint32_t a, uint32_t b, int32_t c) {
    // a: two 16-bit values (signed when AS), b: bytes 0, 1 (2, 3 when HI), signed
    int32_t d;
    if constexpr (AS && HI)
        asm("dp2a.hi.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    else if constexpr (AS)
        asm("dp2a.lo.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    else if constexpr (HI)
        asm("dp2a.hi.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    else
        asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

__device__ __forceinline__ uint32_t word_of(const uint4 &v, int s) {
    return s == 0 ? v.x : s == 1 ? v.y : s == 2 ? v.z : v.w;
}

// 4-byte asynchronous global -> shared copy; invalid ones write zeros.
__device__ __forceinline__ void cp_async4(uint32_t *smem, const uint32_t *gmem, bool valid) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 4 : 0)
                 : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <int ID, int N>
__device__ __forceinline__ void bar_sync() {
    asm volatile("bar.sync %0, %1;\n" ::"n"(ID), "n"(N) : "memory");
}

// clamp(T + d, 30-bit master tap range): the sum saturated to 32 bits, then clamped
__device__ __forceinline__ int32_t add_tap(int32_t T, int64_t d) {
    const int64_t v = T + d;
    const int32_t lo = (int32_t)v, hi = (int32_t)(v >> 32);
    const int32_t w = hi == (lo >> 31) ? lo : (hi >> 31) ^ INT32_MAX;
    return min(max(w, -(1 << 29)), (1 << 29) - 1);
}

// add_tap(T, g >> mu) for g = l1 2^16 + l0 with |l1| < 2^26 and T inside the 30-bit
// range, in 32 bits: g = h 2^16 + r, 0 <= r < 2^16.  Below mu = 16 the step is h 2^(16-mu)
// plus r's top bits, h first cut to where the sum is past the range anyway.
__device__ __forceinline__ int32_t add_tap32(int32_t T, int32_t l1, int32_t l0, int mu) {
    const int32_t h = l1 + (l0 >> 16);
    int32_t d;
    if (mu >= 16)
        d = h >> min(mu - 16, 31);
    else
        d = (min(max(h, -(3 << (13 + mu))), 1 << (14 + mu)) << (16 - mu)) + ((l0 & 0xFFFF) >> mu);
    return min(max(T + d, -(1 << 29)), (1 << 29) - 1);
}

__device__ __forceinline__ bool tap_in_range(int32_t T) { return T >= -(1 << 29) && T < (1 << 29); }

// Copies of symbols tb - K + q, q < XW (zero outside [lo, end)), to xn, by NTHR threads.
template <class C, int NTHR = 32>
__device__ __forceinline__ void stage(uint32_t *xn, const uint32_t *xin, int64_t tb, int64_t lo, int64_t end,
                                      int lane) {
    const int64_t t0 = tb - C::K;
    const uint32_t *src = xin + t0;
    // positions with t inside [lo, end)
    const int q0 = (int)min(max(lo - t0, (int64_t)0), (int64_t)C::XW);
    const int q1 = (int)min(max(end - t0, (int64_t)0), (int64_t)C::XW);
#pragma unroll
    for (int q = lane; q < (C::XW + NTHR - 1) / NTHR * NTHR; q += NTHR) {
        if (q >= C::XW) break;
        const bool ok = q >= q0 && q < q1;
        cp_async4(xn + q, ok ? src + q : xin, ok);
    }
}

// xq[q] <- the byte transpose of the staged words q .. q + 3, by NTHR threads, four
// words of q a thread at a time (loads before stores).
template <class C, int NTHR = 32, bool PLANES = false>
__device__ __forceinline__ void transpose(const uint32_t *xn, uint4 *xq, int lane, uint32_t *xp = nullptr) {
    constexpr int NQ = C::XW - 3;
#pragma unroll
    for (int q0 = 0; q0 < NQ; q0 += 4 * NTHR) {
        uint32_t w[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) w[j][c] = q0 + NTHR * j < NQ ? xn[min(q0 + NTHR * j + lane, NQ - 1) + c] : 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = q0 + NTHR * j + lane;
            const uint32_t ab0 = __byte_perm(w[j][0], w[j][1], 0x5140), ab1 = __byte_perm(w[j][0], w[j][1], 0x7362);
            const uint32_t cd0 = __byte_perm(w[j][2], w[j][3], 0x5140), cd1 = __byte_perm(w[j][2], w[j][3], 0x7362);
            if (q0 + NTHR * j < NQ && q < NQ) {
                const uint4 v = make_uint4(__byte_perm(ab0, cd0, 0x5410), __byte_perm(ab0, cd0, 0x7632),
                                           __byte_perm(ab1, cd1, 0x5410), __byte_perm(ab1, cd1, 0x7632));
                xq[q] = v;
                if constexpr (PLANES) {
#pragma unroll
                    for (int s = 0; s < 4; ++s) xp[s * C::XW + q] = word_of(v, s);
                }
            }
        }
    }
}

// e z of one output of a symbol: limbs c0 (16 bits), c1 (signed 16) and c2 with
// e z = c2 2^32 + c1 2^16 + c0; c2 = 0 where e z fits 32 bits.  r2 <= 2^31 and
// 18 A2 < 2^29 are exact in 32 bits unsigned, R - r2 in 32 bits signed.
struct RdeLimbs {
    uint32_t lo;
    int32_t c2;
};

__device__ __forceinline__ RdeLimbs rde_limbs(int32_t z, int32_t zp, uint32_t A2, bool valid) {
    const uint32_t r2 = (uint32_t)(z * z) + (uint32_t)(zp * zp);
    const uint32_t R = 2 * A2 + (r2 < 6 * A2 ? 0 : 8 * A2) + (r2 < 14 * A2 ? 0 : 8 * A2);
    const int32_t e = valid ? (int32_t)(R - r2) : 0;
    const int64_t v = (int64_t)e * z;
    return {(uint32_t)v, (int32_t)(v >> 32) + (int32_t)((uint32_t)v >> 31)};
}

// Limbs in shared memory, per output a row of NG groups of four symbols: ez holds
// (c0 of symbols 0, 1; c0 of 2, 3; c1 of 0, 1; c1 of 2, 3), ez2 (c2 of 0, 1; of 2, 3).
__device__ __forceinline__ void store_limbs(uint4 *ezrow, int si, RdeLimbs v) {
    uint16_t *e16 = (uint16_t *)(ezrow + (si >> 2)) + (si & 3);
    e16[0] = (uint16_t)v.lo;
    e16[4] = (uint16_t)(v.lo >> 16);
}

__device__ __forceinline__ void store_limb2(uint2 *ez2row, int si, RdeLimbs v) {
    ((uint16_t *)(ez2row + (si >> 2)))[si & 3] = (uint16_t)v.c2;
}

// Taps in shared memory, per output a row of eight 16-byte words: word
// 4 (s1 / 2) + kg holds taps 4 kg + 3 .. 4 kg of inputs s1 and s1 + 1 in that order,
// as they meet the bytes of xq.  Halfword of (s1, tap k) in the row:
__device__ __forceinline__ int tap_slot(int s1, int k) {
    return (s1 >> 1) * 32 + (k >> 2) * 8 + (s1 & 1) * 4 + 3 - (k & 3);
}

// Adds taps 4 kg .. 4 kg + 3 of the four inputs against x to two partial sums.
__device__ __forceinline__ void conv4(const uint4 &wa, const uint4 &wb, const uint4 &x, int32_t &y0, int32_t &y1) {
    y0 = dp2a<true, false>(wa.x, x.x, y0);
    y1 = dp2a<true, true>(wa.y, x.x, y1);
    y0 = dp2a<true, false>(wa.z, x.y, y0);
    y1 = dp2a<true, true>(wa.w, x.y, y1);
    y0 = dp2a<true, false>(wb.x, x.z, y0);
    y1 = dp2a<true, true>(wb.y, x.z, y1);
    y0 = dp2a<true, false>(wb.z, x.w, y0);
    y1 = dp2a<true, true>(wb.w, x.w, y1);
}

// Four symbols of one input against the limbs c0, c1.
__device__ __forceinline__ void grad4(const uint4 &e, uint32_t x, int32_t &l0, int32_t &l1) {
    l0 = dp2a<false, false>(e.x, x, l0);
    l1 = dp2a<true, false>(e.z, x, l1);
    l0 = dp2a<false, true>(e.y, x, l0);
    l1 = dp2a<true, true>(e.w, x, l1);
}

__device__ __forceinline__ int32_t out_of(int32_t y) { return min(max(y >> 7, -32768), 32767); }

// ------------------------------------------------------------ few chains ----
//
// One CTA per (chain, polarisation), its warps by role, so that only what the next
// step waits for lies between two of them:
//   NC = SA / 16 output warps: lane = 2 i + o, output o, symbol i of the warp's 16
//     (no reduction), the error and the limbs of e z; between blocks they store the
//     outputs and load the next block's symbols
//   4 gradient warps, one per input s1: lane = 2 k + o, the gradient of one tap over
//     the block and its update; between blocks they load the next block's symbols
//   1 staging warp: the next batch into the other half of xq, once a batch
// Limbs go from output to gradient warps at barrier 1, which also tells whether any
// e z needs its third limb, taps back at barrier 3 (the writers arrive, the readers
// wait); barrier 2 joins all warps once a batch.
// What a block takes is the latency of that round trip: 0.21 us at N = 32 and 0.29 us
// at N = 64 for a lone chain (0.60 and 0.83 us with the transforms on a CTA); with a
// whole block in one warp it was 0.34 and 0.61 us, about 200 and 500 dependent
// instructions at 3 to 4 cycles each.  The launch bound of four CTAs an SM (64
// registers at N = 64) lets four items share an SM and takes 9 % (N = 32) and 7 % off a
// block of a lone chain against no bound (0.2078, 0.2885 us against 0.2278, 0.3092); a
// bound of two gives less (0.2117, 0.3029), five and six cost time.
template <int NA>
struct SplitCfg {
    // batches of 16 (N = 32) and 8 blocks: with half that a block of a lone chain takes
    // 0.2139 and 0.3061 us, not 0.2078 and 0.2885; twice that takes 0.2057 us at N = 32
    // and passes the static shared memory at N = 64
    using C = DirCfg<NA, NA == 64 ? 8 : 16>;
    static constexpr int NC = (NA - kAeqK) / 16;          // output warps
    static constexpr int NGW = 4;                         // gradient warps
    static constexpr int NCG = 32 * (NC + NGW);
    static constexpr int NT = NCG + 32;
};

template <int ID, int N>
__device__ __forceinline__ void bar_arrive() {
    asm volatile("bar.arrive %0, %1;\n" ::"n"(ID), "n"(N) : "memory");
}

// Barrier that returns whether v was true in any of its threads.
template <int ID, int N>
__device__ __forceinline__ bool bar_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(ID), "n"(N)
        : "memory");
    return r != 0;
}

template <int NA, bool PER>
__global__ void __launch_bounds__(SplitCfg<NA>::NT, 4) aeq_split_kernel(const DevFrame *__restrict__ frames,
                                                                     const AeqChain *__restrict__ chains,
                                                                     AeqParams prm,
                                                                     const __grid_constant__ SingleFrame one) {
    using R = SplitCfg<NA>;
    using C = typename R::C;
    constexpr int K = C::K, SA = C::SA, NG = C::NG, NC = R::NC, NCG = R::NCG;
    constexpr int WO = 12;                        // 16-byte words per tap row: the outputs 16 banks apart
    __shared__ uint4 s_xq[2][C::XW];
    __shared__ uint32_t s_xp[2][4 * C::XW];       // the same words, an input after the other
    __shared__ uint32_t s_xn[C::XW];
    __shared__ uint4 s_w[2 * WO];
    __shared__ uint4 s_ez[2 * NG];
    __shared__ uint2 s_ez2[2 * NG];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const AeqChain ch = chains ? chains[blockIdx.x >> 1] : single_chain(one, blockIdx.x >> 1);
    const int p = blockIdx.x & 1;
    const DevFrame &fr = chains ? frames[ch.frame] : one.fr;
    // (read once: nothing may be kept over the barriers' memory clobbers)
    const uint32_t *const xin = (const uint32_t *)fr.aeq_in;
    int16_t *const out = (int16_t *)fr.out;
    int32_t *const state = fr.state;
    const int64_t nblk = (ch.end - ch.begin + SA - 1) / SA;
    const int64_t nbatch = (nblk + C::PB - 1) / C::PB;
    const int mu = prm.mu_shift;
    const int o = lane & 1, i = lane >> 1;

    if (warp == NC + R::NGW) {
        // ---- staging
        stage<C>(s_xn, xin, ch.begin, ch.lo, ch.end, lane);
        for (int64_t j = 0; j < nbatch; ++j) {
            cp_async_wait_all();
            __syncwarp();
            transpose<C, 32, true>(s_xn, s_xq[j & 1], lane, s_xp[j & 1]);
            __syncwarp();
            if (j + 1 < nbatch) stage<C>(s_xn, xin, ch.begin + (j + 1) * C::B, ch.lo, ch.end, lane);
            bar_sync<2, R::NT>();                 // batch j staged; batch j - 1 consumed
        }
    } else if (warp < NC) {
        // ---- outputs: symbol si of output o
        const uint32_t A2 = (uint32_t)prm.rde_a * (uint32_t)prm.rde_a;
        const int si = 16 * warp + i;
        const uint4 *wr = s_w + o * WO;
        for (int64_t j = 0; j < nbatch; ++j) {
            bar_sync<2, R::NT>();                 // (j = 0: also the initial taps)
            const int64_t tb = ch.begin + j * C::B;
            const int nb = (int)min((int64_t)C::PB, nblk - j * C::PB);
            // valid and kept symbols relative to the batch, less the lane's
            const int left = (int)min(ch.end - tb, (int64_t)C::B) - si;
            const int skip = (int)min(max(ch.keep - tb, (int64_t)0), (int64_t)C::B) - si;
            int16_t *dst = out + (tb + si) * 4 + 2 * p;
            const uint4 *xb = s_xq[j & 1] + K + si - 3;
            uint4 x[4];                           // a block ahead
#pragma unroll
            for (int kg = 0; kg < 4; ++kg) x[kg] = xb[-4 * kg];
            for (int bb = 0; bb < nb; ++bb) {
                const bool valid = bb * SA < left;
                int32_t y[4][2];
#pragma unroll
                for (int kg = 0; kg < 4; ++kg) {
                    y[kg][0] = y[kg][1] = 0;
                    conv4(wr[kg], wr[4 + kg], x[kg], y[kg][0], y[kg][1]);
                }
                const int32_t z =
                    out_of(((y[0][0] + y[0][1]) + (y[1][0] + y[1][1])) + ((y[2][0] + y[2][1]) + (y[3][0] + y[3][1])));
                const int32_t zp = __shfl_xor_sync(0xffffffffu, z, 1);
                if (mu < 63) {
                    const RdeLimbs v = rde_limbs(z, zp, A2, valid);
                    store_limbs(s_ez + o * NG, si, v);
                    store_limb2(s_ez2 + o * NG, si, v);
                    bar_or<1, NCG>(v.c2 != 0);     // limbs stored
                }
                xb += SA;
                if (bb + 1 < nb) {
#pragma unroll
                    for (int kg = 0; kg < 4; ++kg) x[kg] = xb[-4 * kg];
                }
                if (o == 0 && valid && bb * SA >= skip)
                    *(uint32_t *)(dst + bb * SA * 4) = ((uint32_t)z & 0xFFFFu) | ((uint32_t)zp << 16);
                if (mu < 63) bar_sync<3, NCG>();   // taps published, limbs free
            }
        }
    } else {
        // ---- gradient of eq. (6) and update: tap k = i of (o, input s1)
        const int s1 = warp - NC;
        int16_t *wtap = (int16_t *)(s_w + o * WO) + tap_slot(s1, i);
        int32_t T = ch.init[((2 * p + o) * 4 + s1) * K + i];
        *wtap = (int16_t)(T >> 16);
        // a caller's state may hold taps beyond the 30-bit range until the first update
        bool wide = __any_sync(0xffffffffu, !tap_in_range(T));
        int64_t acc = 0;
        int in_period = 0;
        const uint4 *er = s_ez + o * NG;
        for (int64_t j = 0; j < nbatch; ++j) {
            bar_sync<2, R::NT>();
            if (mu >= 63) continue;                // the taps never move
            const int nb = (int)min((int64_t)C::PB, nblk - j * C::PB);
            const uint32_t *xs = s_xp[j & 1] + s1 * C::XW + K - i;
            for (int bb = 0; bb < nb; ++bb, xs += SA) {
                uint32_t x[NG];
#pragma unroll
                for (int n = 0; n < NG; ++n) x[n] = xs[4 * n];
                const bool any = bar_or<1, NCG>(false);   // limbs stored; some c2 is not 0
                int32_t l0[4] = {0, 0, 0, 0}, l1[4] = {0, 0, 0, 0};
#pragma unroll
                for (int n = 0; n < NG; ++n) grad4(er[n], x[n], l0[n & 3], l1[n & 3]);
                const int32_t g0 = (l0[0] + l0[1]) + (l0[2] + l0[3]), g1 = (l1[0] + l1[1]) + (l1[2] + l1[3]);
                if (!PER && !any && !wide) {
                    T = add_tap32(T, g1, g0, mu);
                    *wtap = (int16_t)(T >> 16);
                } else {
                    int64_t g = (int64_t)g1 * 65536 + g0;
                    if (any) {
                        int32_t l2 = 0;
#pragma unroll
                        for (int n = 0; n < NG; ++n) {
                            const uint2 e = s_ez2[o * NG + n];
                            l2 = dp2a<true, false>(e.x, x[n], l2);
                            l2 = dp2a<true, true>(e.y, x[n], l2);
                        }
                        g += (int64_t)l2 << 32;
                    }
                    bool apply = true;
                    if constexpr (PER) {
                        g += acc;
                        apply = ++in_period == prm.period || (j + 1 == nbatch && bb + 1 == nb);
                        if (apply) in_period = 0;
                        acc = apply ? 0 : g;
                    }
                    if (apply) {
                        T = add_tap(T, g >> mu);
                        *wtap = (int16_t)(T >> 16);
                        wide = false;
                    }
                }
                bar_arrive<3, NCG>();              // taps published, limbs read
            }
        }
        if (ch.write_state) state[((2 * p + o) * 4 + s1) * K + i] = T;
    }
}

// ----------------------------------------------------------- many chains ----
//
// A CTA of two warps per chain, a warp per polarisation that holds a whole block:
// lane = 2 i + o forms symbols i, i + 16, ... of output o, then the gradient of tap i
// of o and all four inputs over the block, and updates those four taps, so nothing is
// reduced over lanes and two __syncwarp order a block.  The warps share the staged
// batch and meet twice a batch.  Lanes 2 i and 2 i + 1 read the same staged word, so a
// 16-byte load of the warp is two passes over shared memory, not four.  Bound by issue
// once four warps share a scheduler: 0.69 us a block for 1,216 chains at N = 32, 1.62
// us at N = 64.  (One warp for both polarisations shares more loads, but took 0.73 and
// 1.65 us there, and 0.49 and 0.73 us for 608 and 760 chains at N = 32 where this one
// takes 0.43 and 0.55.)
template <int NA, bool PER>
__global__ void __launch_bounds__(64) aeq_duo_kernel(const DevFrame *__restrict__ frames,
                                                     const AeqChain *__restrict__ chains, AeqParams prm,
                                                     const __grid_constant__ SingleFrame one) {
    // batches of 32 (N = 32) and 8 blocks: with 8 and 4, 1 to 10 % slower
    using C = DirCfg<NA, NA == 64 ? 8 : 32>;
    constexpr int K = C::K, SA = C::SA, NG = C::NG, M = SA / 16;
    constexpr int WO = 12;
    __shared__ uint4 s_xq[C::XW];
    __shared__ uint32_t s_xn[C::XW];
    __shared__ uint4 s_w[2][2 * WO];
    __shared__ uint4 s_ez[2][2 * NG];
    __shared__ uint2 s_ez2[2][2 * NG];

    const int tid = threadIdx.x, lane = tid & 31, p = tid >> 5;
    const int o = lane & 1, i = lane >> 1;
    const uint32_t A2 = (uint32_t)prm.rde_a * (uint32_t)prm.rde_a;
    const int mu = prm.mu_shift;
    const AeqChain ch = chains ? chains[blockIdx.x] : single_chain(one, blockIdx.x);
    const DevFrame &fr = chains ? frames[ch.frame] : one.fr;
    const uint32_t *const xin = (const uint32_t *)fr.aeq_in;
    int16_t *const out = (int16_t *)fr.out;
    int32_t *const state = fr.state;

    int16_t *wrow = (int16_t *)(s_w[p] + o * WO);
    uint4 *ez = s_ez[p] + o * NG;
    uint2 *ez2 = s_ez2[p] + o * NG;
    int32_t T[4];
    int64_t acc[4];
    bool wide = false;   // a caller's state may hold taps beyond the 30-bit range until the first update
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        T[s] = ch.init[((2 * p + o) * 4 + s) * K + i];
        wide |= !tap_in_range(T[s]);
        wrow[tap_slot(s, i)] = (int16_t)(T[s] >> 16);
        acc[s] = 0;
    }
    wide = __any_sync(0xffffffffu, wide);
    const int64_t nblk = (ch.end - ch.begin + SA - 1) / SA;
    stage<C, 64>(s_xn, xin, ch.begin, ch.lo, ch.end, tid);
    int in_period = 0;
    for (int64_t b0 = 0; b0 < nblk; b0 += C::PB) {
        const int64_t tb = ch.begin + b0 * SA;
        cp_async_wait_all();
        __syncthreads();
        transpose<C, 64>(s_xn, s_xq, tid);
        __syncthreads();
        if (b0 + C::PB < nblk) stage<C, 64>(s_xn, xin, tb + C::B, ch.lo, ch.end, tid);
        const int nb = (int)min((int64_t)C::PB, nblk - b0);
        const bool last_batch = b0 + C::PB >= nblk;
        const int rel_end = (int)min(ch.end - tb, (int64_t)C::B);
        const int rel_keep = (int)min(max(ch.keep - tb, (int64_t)0), (int64_t)C::B);
        int16_t *outb = out + tb * 4 + 2 * p;
        for (int bb = 0; bb < nb; ++bb) {
            const uint4 *xb = s_xq + K + bb * SA;
            // ---- convolution, outputs, RDE error, limbs of e z
            int32_t y0[M], y1[M];
            const uint4 *wr = s_w[p] + o * WO;
#pragma unroll
            for (int m = 0; m < M; ++m) y0[m] = y1[m] = 0;
#pragma unroll
            for (int kg = 0; kg < 4; ++kg) {
                const uint4 wa = wr[kg], wb = wr[4 + kg];
#pragma unroll
                for (int m = 0; m < M; ++m) conv4(wa, wb, xb[16 * m + i - 4 * kg - 3], y0[m], y1[m]);
            }
            bool big = false;
            RdeLimbs v[M];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const int si = i + 16 * m, rel = bb * SA + si;
                const int32_t z = out_of(y0[m] + y1[m]);
                const int32_t zp = __shfl_xor_sync(0xffffffffu, z, 1);
                const bool valid = rel < rel_end;
                v[m] = rde_limbs(z, zp, A2, valid);
                store_limbs(ez, si, v[m]);
                big |= v[m].c2 != 0;
                if (valid && rel >= rel_keep && o == 0)
                    *(uint32_t *)(outb + rel * 4) = ((uint32_t)z & 0xFFFFu) | ((uint32_t)zp << 16);
            }
            const bool any = __any_sync(0xffffffffu, big);
            if (any) {
#pragma unroll
                for (int m = 0; m < M; ++m) store_limb2(ez2, i + 16 * m, v[m]);
            }
            __syncwarp();
            if (mu >= 63) continue;                // the taps never move: no gradient

            // ---- gradient of eq. (6) and update
            int32_t l0[4], l1[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) l0[s] = l1[s] = 0;
#pragma unroll
            for (int n = 0; n < NG; ++n) {
                const uint4 e = ez[n], x = xb[4 * n - i];
#pragma unroll
                for (int s = 0; s < 4; ++s) grad4(e, word_of(x, s), l0[s], l1[s]);
            }
            if (!PER && !any && !wide) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    T[s] = add_tap32(T[s], l1[s], l0[s], mu);
                    wrow[tap_slot(s, i)] = (int16_t)(T[s] >> 16);
                }
            } else {
                int64_t g[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) g[s] = (PER ? acc[s] : 0) + (int64_t)l1[s] * 65536 + l0[s];
                if (any) {
                    int32_t l2[4] = {0, 0, 0, 0};
                    for (int n = 0; n < NG; ++n) {
                        const uint2 e = ez2[n];
                        const uint4 x = xb[4 * n - i];
#pragma unroll
                        for (int s = 0; s < 4; ++s) {
                            l2[s] = dp2a<true, false>(e.x, word_of(x, s), l2[s]);
                            l2[s] = dp2a<true, true>(e.y, word_of(x, s), l2[s]);
                        }
                    }
#pragma unroll
                    for (int s = 0; s < 4; ++s) g[s] += (int64_t)l2[s] << 32;
                }
                bool apply = true;
                if constexpr (PER) {
                    apply = ++in_period == prm.period || (last_batch && bb + 1 == nb);
                    if (apply) in_period = 0;
                }
                if (apply) {
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        T[s] = add_tap(T[s], g[s] >> mu);
                        wrow[tap_slot(s, i)] = (int16_t)(T[s] >> 16);
                    }
                    wide = false;
                }
                if constexpr (PER) {
#pragma unroll
                    for (int s = 0; s < 4; ++s) acc[s] = apply ? 0 : g[s];
                }
            }
            __syncwarp();                          // taps published, limbs free
        }
    }
    if (ch.write_state) {
#pragma unroll
        for (int s = 0; s < 4; ++s) state[((2 * p + o) * 4 + s) * K + i] = T[s];
    }
}

template <int NA>
void launch_na(bool split, const DevFrame *frames, const AeqChain *chains, int n_chains, AeqParams prm,
               cudaStream_t stream, const SingleFrame &one) {
    const unsigned n = (unsigned)n_chains;
    if (split && prm.period > 1)
        aeq_split_kernel<NA, true><<<2 * n, SplitCfg<NA>::NT, 0, stream>>>(frames, chains, prm, one);
    else if (split)
        aeq_split_kernel<NA, false><<<2 * n, SplitCfg<NA>::NT, 0, stream>>>(frames, chains, prm, one);
    else if (prm.period > 1)
        aeq_duo_kernel<NA, true><<<n, 64, 0, stream>>>(frames, chains, prm, one);
    else
        aeq_duo_kernel<NA, false><<<n, 64, 0, stream>>>(frames, chains, prm, one);
}

const SingleFrame kNoSingle{};

}  // namespace

// The split layout takes fewer cycles a block while the GPU is not full, the duo layout
// fewer cycles of an SM a block.  total / longest is how many chains of the longest
// one's length the launch amounts to.  Measured with equal chains, us a block (split,
// duo), by (chain, polarisation) items per SM (152 SMs):
//                  1            2            3            4            5            6
//   N = 64         .293  .590   .397  .590   .518  .597   .649  .601   .861  .892   .984  .894
//   N = 32         .209  .322   .227  .322   .288  .326   .322  .327   .489  .419   .518  .419
//   N = 64, P = 4  .309  .559   .414  .562   .545  .569   .685  .568   .886  .877   1.02  .876
//   N = 32, P = 4  .212  .292   .238  .291   .307  .295   .350  .297   .505  .393   .544  .392
// so the lines lie between 3 and 4 items, at 4, and (update period P > 1, N = 32)
// between 2 and 3.
bool aeq_direct_split(int na, int period, int64_t total_symbols, int64_t longest_symbols, int n_sm) {
    const double items = 2.0 * (double)total_symbols / (double)std::max<int64_t>(longest_symbols, 1);
    return items < (na == 64 ? 3.5 : period > 1 ? 2.8 : 4.0) * n_sm;
}

cudaError_t aeq_direct_launch(int na, bool split, const DevFrame *frames, const AeqChain *chains, int n_chains,
                              AeqParams prm, cudaStream_t stream, const SingleFrame *one) {
    if (n_chains <= 0) return cudaSuccess;
    const SingleFrame &single = one ? *one : kNoSingle;
    if (one) frames = nullptr, chains = nullptr;
    if (na == 64)
        launch_na<64>(split, frames, chains, n_chains, prm, stream, single);
    else
        launch_na<32>(split, frames, chains, n_chains, prm, stream, single);
    return cudaGetLastError();
}

}  // namespace fnt
