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
// One item is a (chain, polarisation): the outputs 2p and 2p + 1 of one run, whose
// blocks of SA = N - 16 symbols follow each other through the tap update.  A warp
// holds lane = 16 o + i: first output o, symbol i of 16 (convolution, RDE error),
// then output o, tap k = i of all four inputs (gradient, update), so a block of 16
// symbols needs no reduction over lanes and two __syncwarp.
//   convolution  y_o[i] = sum_s1,k W_o,s1[k] x_s1[t0 + i - k]: four 16-byte loads of
//                symbol bytes, eight of taps, 32 dp2a
//   error        z = sat16(y >> 7), one shuffle for the other output, e in 32 bits
//   gradient     G = sum_i e z_o[i] x_s1[t0 + i - k] with e z = c1 2^16 + c0
//                (c0 16 bits, c1 signed 16 bits) and, only when some |e z| of the
//                warp's symbols reaches 2^31, c2 2^32: two (three) dp2a for two
//                products; limb sums are exact in 32 bits, then combined in 64
//   update       eq. (6) on the lane's own four master taps
//
// Staged symbols.  xq[q] holds, for the four inputs, the four bytes of symbols
// q .. q + 3 (a 4 x 4 byte transpose at every q, 16 bytes a symbol), so both the
// convolution (four taps of an input against one word) and the gradient (four
// symbols of an input) read aligned 16-byte words at any offset.  A batch of
// blocks is transposed at once while the next batch's words arrive by cp.async.
//
// Layouts <SYM, GRP, Q>: SA = 16 SYM GRP symbols, GRP Q warps per item.
//   SYM  symbol groups of 16 a warp works through (3 x 16 at N = 64)
//   GRP  warps that share a block by symbols.  Each keeps a copy of the taps, forms
//        the gradient of its own 16 symbols, and the partial sums cross once per
//        update through shared memory: one barrier a block.
//   Q    warps that share the gradient and the update by input s1; each repeats the
//        convolution (its pipes would idle).  One barrier a block, taps double
//        buffered.
// aeq_direct_launch picks the layout (rule and figures there).
#include <algorithm>

#include <cuda_runtime.h>

#include "host.h"
#include "internal.h"

namespace fnt {

namespace {

template <int SYM_, int GRP_, int Q_>
struct DirCfg {
    static constexpr int K = kAeqK;
    static constexpr int SYM = SYM_, GRP = GRP_, Q = Q_;
    static constexpr int SA = 16 * SYM * GRP;             // symbols per block
    static constexpr int W = GRP * Q;                     // warps per item
    static constexpr int NT = 32 * W;
    static constexpr int NS = 4 / Q;                      // inputs s1 whose gradient a lane holds
    static constexpr int PB = SA == 48 ? 4 : 8;           // blocks per staged batch
    static constexpr int B = PB * SA;                     // symbols per staged batch
    static constexpr int XW = K + B;                      // staged words: K of history
    static constexpr int WO = 36;                         // words per output in a tap set (bank shift 4)
    static constexpr int WS = 2 * WO;                     // words per tap set
    static constexpr int NG = 4 * SYM * GRP;              // groups of four symbols
    static_assert(K == 16 && (GRP == 1 || Q == 1) && 4 % Q == 0, "layouts");
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

template <int W>
__device__ __forceinline__ void item_sync() {
    if constexpr (W == 1)
        __syncwarp();
    else
        __syncthreads();
}

// clamp(T + d, 30-bit master tap range): the sum saturated to 32 bits, then clamped
__device__ __forceinline__ int32_t add_tap(int32_t T, int64_t d) {
    const int64_t v = T + d;
    const int32_t lo = (int32_t)v, hi = (int32_t)(v >> 32);
    const int32_t w = hi == (lo >> 31) ? lo : (hi >> 31) ^ INT32_MAX;
    return min(max(w, -(1 << 29)), (1 << 29) - 1);
}

// xn: staged words of symbols tb - K + q, q < XW; xq: their byte transposes.
template <class C>
__device__ __forceinline__ void stage(uint32_t *xn, const uint32_t *xin, int64_t tb, int64_t lo, int64_t end,
                                      int tid) {
    for (int q = tid; q < C::XW; q += C::NT) {
        const int64_t t = tb - C::K + q;
        const bool ok = t >= lo && t < end;
        cp_async4(xn + q, ok ? xin + t : xin, ok);
    }
}

template <class C>
__device__ __forceinline__ void transpose(const uint32_t *xn, uint4 *xq, int tid) {
    for (int q = tid; q < C::XW - 3; q += C::NT) {
        const uint32_t a = xn[q], b = xn[q + 1], c = xn[q + 2], d = xn[q + 3];
        const uint32_t ab0 = __byte_perm(a, b, 0x5140), ab1 = __byte_perm(a, b, 0x7362);   // (a0 b0 a1 b1), (a2 b2 a3 b3)
        const uint32_t cd0 = __byte_perm(c, d, 0x5140), cd1 = __byte_perm(c, d, 0x7362);
        xq[q] = make_uint4(__byte_perm(ab0, cd0, 0x5410), __byte_perm(ab0, cd0, 0x7632),
                           __byte_perm(ab1, cd1, 0x5410), __byte_perm(ab1, cd1, 0x7632));
    }
}

template <int SYM, int GRP, int Q, bool PER>
__global__ void __launch_bounds__(32 * GRP * Q) aeq_direct_kernel(const DevFrame *__restrict__ frames,
                                                                   const AeqChain *__restrict__ chains,
                                                                   AeqParams prm) {
    using C = DirCfg<SYM, GRP, Q>;
    constexpr int K = C::K, SA = C::SA, NS = C::NS;
    __shared__ uint4 s_xq[C::XW];
    __shared__ uint32_t s_xn[C::XW];
    // tap sets: GRP > 1 one per warp; Q > 1 two for the item, used in turn
    __shared__ uint4 s_w[(GRP > 1 ? GRP : Q > 1 ? 2 : 1) * C::WS / 4];
    // limbs of e z: [o][group of 4 symbols] (c0 01, c0 23, c1 01, c1 23); Q > 1: per warp
    __shared__ uint4 s_ez[Q * 2 * C::NG];
    __shared__ uint2 s_ez2[Q * 2 * C::NG];
    __shared__ longlong2 s_part[GRP > 1 ? 2 * GRP * 64 : 1];   // partial gradients [parity][warp][pair][lane]

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int grp = GRP > 1 ? warp : 0;
    const int q4 = Q > 1 ? warp : 0;
    const int o = lane >> 4, i = lane & 15;       // i: symbol of 16, then tap k
    const uint32_t A2 = (uint32_t)prm.rde_a * (uint32_t)prm.rde_a;
    const int mu = prm.mu_shift;
    const int period = PER ? prm.period : 1;

    const AeqChain ch = chains[blockIdx.x >> 1];
    const int p = blockIdx.x & 1;
    const DevFrame &fr = frames[ch.frame];
    const uint32_t *xin = (const uint32_t *)fr.aeq_in;
    int16_t *out = (int16_t *)fr.out;

    uint32_t *wset = (uint32_t *)s_w + (GRP > 1 ? grp * C::WS : 0);
    uint4 *ez = s_ez + q4 * 2 * C::NG;
    uint2 *ez2 = s_ez2 + q4 * 2 * C::NG;
    // tap k of (o, s1): halfword 3 - (k & 3) of the group of four taps k / 4
    const int tapw = (o * C::WO + (i >> 2) * 8) * 2 + (3 - (i & 3));
    int32_t T[NS];
    int64_t acc[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        T[s] = ch.init[((2 * p + o) * 4 + q4 * NS + s) * K + i];
        acc[s] = 0;
        ((int16_t *)wset)[tapw + 4 * (q4 * NS + s)] = (int16_t)(T[s] >> 16);
    }

    const int64_t nblk = (ch.end - ch.begin + SA - 1) / SA;
    stage<C>(s_xn, xin, ch.begin, ch.lo, ch.end, tid);
    int in_period = 0;
    int par = 0;                                   // parity of the tap set (Q > 1) or the partial sums (GRP > 1)
    for (int64_t b0 = 0; b0 < nblk; b0 += C::PB) {
        const int64_t tb = ch.begin + b0 * SA;
        cp_async_wait_all();
        item_sync<C::W>();                         // words staged; the last batch's reads of xq done
        transpose<C>(s_xn, s_xq, tid);
        item_sync<C::W>();
        if (b0 + C::PB < nblk) stage<C>(s_xn, xin, tb + C::B, ch.lo, ch.end, tid);
        const int nb = (int)min((int64_t)C::PB, nblk - b0);
        const bool last_batch = b0 + C::PB >= nblk;
        // valid and kept symbols relative to the batch
        const int rel_end = (int)min(ch.end - tb, (int64_t)C::B);
        const int rel_keep = (int)min(max(ch.keep - tb, (int64_t)0), (int64_t)C::B);
        int16_t *outb = out + tb * 4 + 2 * p;
        for (int bb = 0; bb < nb; ++bb) {
            const uint4 *xb = s_xq + K + bb * SA;

            // ---- convolution: y of (o, symbol 16 (grp SYM + m) + i)
            const uint4 *wr = (const uint4 *)(wset + (Q > 1 ? par * C::WS : 0) + o * C::WO);
            int32_t y[SYM][2];
#pragma unroll
            for (int m = 0; m < SYM; ++m) y[m][0] = y[m][1] = 0;
#pragma unroll
            for (int kg = 0; kg < 4; ++kg) {
                const uint4 wa = wr[2 * kg], wb = wr[2 * kg + 1];
#pragma unroll
                for (int m = 0; m < SYM; ++m) {
                    const uint4 x = xb[16 * (grp * SYM + m) + i - 4 * kg - 3];
                    y[m][0] = dp2a<true, false>(wa.x, x.x, y[m][0]);
                    y[m][1] = dp2a<true, true>(wa.y, x.x, y[m][1]);
                    y[m][0] = dp2a<true, false>(wa.z, x.y, y[m][0]);
                    y[m][1] = dp2a<true, true>(wa.w, x.y, y[m][1]);
                    y[m][0] = dp2a<true, false>(wb.x, x.z, y[m][0]);
                    y[m][1] = dp2a<true, true>(wb.y, x.z, y[m][1]);
                    y[m][0] = dp2a<true, false>(wb.z, x.w, y[m][0]);
                    y[m][1] = dp2a<true, true>(wb.w, x.w, y[m][1]);
                }
            }

            // ---- outputs, RDE error, limbs of e z
            bool big = false;
#pragma unroll
            for (int m = 0; m < SYM; ++m) {
                const int si = 16 * (grp * SYM + m) + i;
                const int32_t z = min(max((y[m][0] + y[m][1]) >> 7, -32768), 32767);
                const int32_t zp = __shfl_xor_sync(0xffffffffu, z, 16);
                // r2 <= 2^31 and 18 A2 < 2^29: exact in 32 bits unsigned
                const uint32_t r2 = (uint32_t)(z * z) + (uint32_t)(zp * zp);
                const uint32_t Rr = r2 < 6 * A2 ? 2 * A2 : (r2 < 14 * A2 ? 10 * A2 : 18 * A2);
                const int rel = bb * SA + si;
                const bool valid = rel < rel_end;
                if (valid && rel >= rel_keep && o == 0 && q4 == 0)
                    *(uint32_t *)(outb + rel * 4) = ((uint32_t)z & 0xFFFFu) | ((uint32_t)zp << 16);
                const int64_t v = valid ? (int64_t)(int32_t)(Rr - r2) * z : 0;
                // e z = c2 2^32 + c1 2^16 + c0 with c1 signed: c2 is 0 where e z fits 32 bits
                const uint32_t vl = (uint32_t)v;
                const int32_t c2 = (int32_t)(v >> 32) + (int32_t)(vl >> 31);
                big |= c2 != 0;
                uint16_t *e16 = (uint16_t *)(ez + o * C::NG + (si >> 2)) + (si & 3);
                e16[0] = (uint16_t)vl;
                e16[4] = (uint16_t)(vl >> 16);
                ((uint16_t *)(ez2 + o * C::NG + (si >> 2)))[si & 3] = (uint16_t)c2;
            }
            // (also orders the limbs before the gradient's reads, within the warp)
            const bool any = __any_sync(0xffffffffu, big);
            __syncwarp();

            // ---- gradient of eq. (6) for (o, s1, tap k = i) over the warp's symbols
            if (mu < 63) {
                int32_t l0[NS], l1[NS];
                int64_t g[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) l0[s] = l1[s] = 0;
#pragma unroll
                for (int n = 0; n < 4 * SYM; ++n) {
                    const int ig = 4 * SYM * grp + n;
                    const uint4 e = ez[o * C::NG + ig];
                    const uint4 x = xb[4 * ig - i];
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const uint32_t xs = Q == 1 ? word_of(x, s) : ((const uint32_t *)(xb + 4 * ig - i))[q4 * NS + s];
                        l0[s] = dp2a<false, false>(e.x, xs, l0[s]);
                        l1[s] = dp2a<true, false>(e.z, xs, l1[s]);
                        l0[s] = dp2a<false, true>(e.y, xs, l0[s]);
                        l1[s] = dp2a<true, true>(e.w, xs, l1[s]);
                    }
                }
#pragma unroll
                for (int s = 0; s < NS; ++s) g[s] = (int64_t)l1[s] * 65536 + l0[s];
                if (any) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        int32_t l2 = 0;
                        for (int n = 0; n < 4 * SYM; ++n) {
                            const int ig = 4 * SYM * grp + n;
                            const uint2 e = ez2[o * C::NG + ig];
                            const uint32_t xs = ((const uint32_t *)(xb + 4 * ig - i))[q4 * NS + s];
                            l2 = dp2a<true, false>(e.x, xs, l2);
                            l2 = dp2a<true, true>(e.y, xs, l2);
                        }
                        g[s] += (int64_t)l2 << 32;
                    }
                }
                bool apply = true;
                if constexpr (PER) {
                    apply = ++in_period == period || (last_batch && bb + 1 == nb);
                    if (apply) in_period = 0;
#pragma unroll
                    for (int s = 0; s < NS; ++s) g[s] = acc[s] += g[s];
                }
                if (apply) {
                    if constexpr (GRP > 1) {
                        // the other warps' partial sums over the period; two buffers in
                        // turn, so one barrier an update
                        longlong2 *part = s_part + par * GRP * 64;
                        part[grp * 64 + lane] = make_longlong2(g[0], g[1]);
                        part[grp * 64 + 32 + lane] = make_longlong2(g[2], g[3]);
                        __syncthreads();
#pragma unroll
                        for (int w = 1; w < GRP; ++w) {
                            const int og = grp + w < GRP ? grp + w : grp + w - GRP;
                            const longlong2 u = part[og * 64 + lane], v = part[og * 64 + 32 + lane];
                            g[0] += u.x;
                            g[1] += u.y;
                            g[2] += v.x;
                            g[3] += v.y;
                        }
                    }
                    if constexpr (GRP > 1 || Q > 1) par ^= 1;
                    int16_t *wn = (int16_t *)(wset + (Q > 1 ? par * C::WS : 0));
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        T[s] = add_tap(T[s], g[s] >> mu);
                        wn[tapw + 4 * (q4 * NS + s)] = (int16_t)(T[s] >> 16);
                        acc[s] = 0;
                    }
                    item_sync<Q>();                // the item's new taps, before the next block reads them
                } else {
                    __syncwarp();                  // the limbs are rewritten by the next block
                }
            }
        }
    }
    if (ch.write_state && grp == 0) {
#pragma unroll
        for (int s = 0; s < NS; ++s) fr.state[((2 * p + o) * 4 + q4 * NS + s) * K + i] = T[s];
    }
}

template <int SYM, int GRP, int Q>
cudaError_t launch_layout(const DevFrame *frames, const AeqChain *chains, int n_chains, AeqParams prm,
                          cudaStream_t stream) {
    const unsigned grid = 2u * (unsigned)n_chains;
    if (prm.period > 1)
        aeq_direct_kernel<SYM, GRP, Q, true><<<grid, 32 * GRP * Q, 0, stream>>>(frames, chains, prm);
    else
        aeq_direct_kernel<SYM, GRP, Q, false><<<grid, 32 * GRP * Q, 0, stream>>>(frames, chains, prm);
    return cudaGetLastError();
}

}  // namespace

cudaError_t aeq_direct_launch(int na, const DevFrame *frames, const AeqChain *chains, int n_chains,
                              int64_t total_symbols, int64_t longest_symbols, AeqParams prm, int n_sm,
                              cudaStream_t stream) {
    if (n_chains <= 0) return cudaSuccess;
    const bool spread = 2.0 * total_symbols < 8.0 * n_sm * (double)longest_symbols;
    if (na == 64)
        return spread ? launch_layout<1, 3, 1>(frames, chains, n_chains, prm, stream)
                      : launch_layout<3, 1, 1>(frames, chains, n_chains, prm, stream);
    return spread ? launch_layout<1, 1, 4>(frames, chains, n_chains, prm, stream)
                  : launch_layout<1, 1, 1>(frames, chains, n_chains, prm, stream);
}

}  // namespace fnt
