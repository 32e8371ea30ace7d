// cdc_direct.cu -- the CDC's complex convolution as exact integer dot products.
//
// z[t] = sum_k h[k] x[t-k] over at most 31 complex taps of 6 bits and 5-bit samples
// lies inside constraint (5), so it is the plain integer sum.  dp4a adds four 8-bit
// products per instruction at the rate of one shift (64 lanes a clock and SM
// measured), so two complex taps cost one dp4a for the real and one for the
// imaginary part: L + 1 instructions an output, where the 64-point transforms of
// eqs. (7)/(8) (cdc.cu) take about 90 a sample whatever L is.  The chain keeps every
// second sample (the AEQ runs at one sample a symbol), and only those are computed.
//
// A warp computes 256 outputs of a frame, all polarisations: consecutive samples
// (CDC) or symbols (chain).  It first stages pair words
//   pw[u] = (x[t-1], x[t]) as bytes re, im, re, im,   t = 2 u + parity
// per polarisation (and, CDC, per parity) in shared memory: tap pair m of output u
// then reads pw[u - m], so a lane's four outputs at consecutive u slide over aligned
// 16-byte words and every tap word serves all of a lane's 8 outputs x polarisations.
// Stores are 16 bytes (chain) or, where the buffer is 32-byte aligned, 32 bytes a
// lane (CDC).
//
// The polarisations run one after the other (56 registers, 36 warps an SM; both at
// once took 80 registers and 65.5 us) with the tap loop unrolled, so no register moves
// between tap groups.
//
// Bound: dp4a issue (40 a PDM sample at L = 19 against 12 bytes moved, about equal to
// the HBM time) for the CDC: 2^24 PDM samples, 19 taps in 51 us, 3.9 TB/s (245 us with
// the transforms).  Latency for small frames.
#include <algorithm>

#include <cuda_runtime.h>

#include "host.h"
#include "internal.h"

namespace fnt {

namespace {

constexpr int kHistPairs = 16;                   // pair words before a tile: 32 taps of history
constexpr int kTile = kCdcDirectTile;            // outputs per warp
constexpr int kHalf = kTile / 2;

// Shared words of a warp: pair words [group][pol][row] (CDC: a group per parity) or
// [pol][row] (chain: both halves of the tile in one row), then the tap words.  The
// row pitch puts the parities on different banks of the staging stores.
template <bool CHAIN, int NPOL>
struct CdcDirect {
    static constexpr int ROW = CHAIN ? kHistPairs + kTile : kHistPairs + kHalf + (NPOL == 2 ? 8 : 0);
    static constexpr int WORDS = CHAIN ? NPOL * ROW : 2 * NPOL * ROW;
    static_assert(ROW % 4 == 0 && WORDS % 4 == 0, "16-byte rows");
    // row start of group g (CDC: parity, chain: half) and polarisation p
    static __device__ __forceinline__ int base(int g, int p) {
        return CHAIN ? p * ROW + g * kHalf : (g * NPOL + p) * ROW;
    }
};

__device__ __forceinline__ int32_t sat5(int32_t v) { return min(max(v, -16), 15); }

__device__ __forceinline__ void store32(uint32_t *dst, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(dst), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// item: (frame, first tile, tiles); the CTA has a warp per tile of the longest item.
template <bool CHAIN, int NPOL>
__device__ __forceinline__ void cdc_tile(const DevFrame &fr, int64_t tile, uint32_t *pw, int2 *tw, int lane) {
    using C = CdcDirect<CHAIN, NPOL>;
    const int64_t n = fr.n;
    const int np = (fr.L + 1) >> 1;              // tap pairs

    // tap words of pair m: (h[2m+1], h[2m]) against (x[t-2m-1], x[t-2m]); the taps
    // are zero beyond L, and -im fits 8 bits (|im| <= 32)
    if (lane < kHistPairs) {
        const char4 h = *(const char4 *)(fr.taps + 4 * lane);         // re, im of taps 2m and 2m + 1
        const uint32_t r0 = (uint8_t)h.x, i0 = (uint8_t)h.y, r1 = (uint8_t)h.z, i1 = (uint8_t)h.w;
        const uint32_t n0 = (uint8_t)(-h.y), n1 = (uint8_t)(-h.w);
        tw[lane] = make_int2((int)(r1 | n1 << 8 | r0 << 16 | n0 << 24), (int)(i1 | r1 << 8 | i0 << 16 | r0 << 24));
    }
    // pair words; samples outside the frame are zero
    const int64_t t0 = CHAIN ? 2 * tile * kTile + fr.phase : tile * kTile;
    constexpr int NP = CHAIN ? kHistPairs + kTile : 2 * kHistPairs + kTile;
    const int64_t tfirst = t0 - 2 * kHistPairs;
    const bool inside = tfirst >= 1 && tfirst + (CHAIN ? 2 * (int64_t)NP : (int64_t)NP) <= n;
    auto put = [&](int q, uint32_t a, uint32_t b) {      // samples t - 1 and t
        const int idx = CHAIN ? q : (q & 1) * NPOL * C::ROW + (q >> 1);
        if constexpr (NPOL == 2) {
            pw[idx] = __byte_perm(a, b, 0x5410);
            pw[idx + C::ROW] = __byte_perm(a, b, 0x7632);
        } else {
            pw[idx] = a | b << 16;
        }
    };
    auto load = [&](int64_t t) -> uint32_t {
        if constexpr (NPOL == 2)
            return __ldg((const uint32_t *)fr.in + t);
        else
            return __ldg((const uint16_t *)fr.in + t);
    };
    constexpr int IT = (NP + 31) / 32;
    uint32_t a[IT], b[IT];
    if (inside) {
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const int q = min(lane + 32 * it, NP - 1);
            const int64_t t = tfirst + (CHAIN ? 2 * q : q);
            a[it] = load(t - 1);
            b[it] = load(t);
        }
    } else {
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const int64_t t = tfirst + (int64_t)(lane + 32 * it) * (CHAIN ? 2 : 1);
            a[it] = t >= 1 && t - 1 < n ? load(t - 1) : 0;
            b[it] = t >= 0 && t < n ? load(t) : 0;
        }
    }
#pragma unroll
    for (int it = 0; it < IT; ++it)
        if (lane + 32 * it < NP) put(lane + 32 * it, a[it], b[it]);
    __syncwarp();

    // one polarisation after the other: res packs its 8 outputs (CDC: re, im as 16
    // bits; chain: the two requantised bytes)
    uint32_t res[NPOL][2][4];
    [[maybe_unused]] const int sft = CHAIN ? fr.shift : 0;
    [[maybe_unused]] const int32_t rnd = sft > 0 ? (1 << (sft - 1)) : 0;
#pragma unroll
    for (int p = 0; p < NPOL; ++p) {
        int32_t re[2][4] = {}, im[2][4] = {};
        uint4 cur[2];                            // pw[u0 .. u0 + 3] of the chunk's first pair
#pragma unroll
        for (int g = 0; g < 2; ++g) cur[g] = *(const uint4 *)(pw + C::base(g, p) + kHistPairs + 4 * lane);
#pragma unroll
        for (int c = 0; c < kHistPairs / 4; ++c) {
            if (4 * c >= np) break;
            const int4 h01 = *(const int4 *)(tw + 4 * c), h23 = *(const int4 *)(tw + 4 * c + 2);
            uint32_t w[2][7];
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const uint4 A = cur[g];
                const uint4 B = *(const uint4 *)(pw + C::base(g, p) + kHistPairs - 4 + 4 * lane - 4 * c);
                w[g][0] = B.y, w[g][1] = B.z, w[g][2] = B.w;
                w[g][3] = A.x, w[g][4] = A.y, w[g][5] = A.z, w[g][6] = A.w;
                cur[g] = B;
            }
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                if (m > 0 && 4 * c + m >= np) break;
                const int hr = m == 0 ? h01.x : m == 1 ? h01.z : m == 2 ? h23.x : h23.z;
                const int hi = m == 0 ? h01.y : m == 1 ? h01.w : m == 2 ? h23.y : h23.w;
#pragma unroll
                for (int g = 0; g < 2; ++g)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        re[g][j] = __dp4a((int)w[g][3 + j - m], hr, re[g][j]);
                        im[g][j] = __dp4a((int)w[g][3 + j - m], hi, im[g][j]);
                    }
            }
        }
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                res[p][g][j] = CHAIN ? __byte_perm((uint32_t)sat5((re[g][j] + rnd) >> sft),
                                                   (uint32_t)sat5((im[g][j] + rnd) >> sft), 0x0040)
                                     : __byte_perm((uint32_t)re[g][j], (uint32_t)im[g][j], 0x5410);
    }

    if constexpr (CHAIN) {
        // symbols s0 + 128 g + 4 lane + j, a word (XI, XQ, YI, YQ) each
        uint32_t *dst = (uint32_t *)fr.aeq_in;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            uint32_t v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = __byte_perm(res[0][g][j], res[NPOL - 1][g][j], 0x5410);
            const int64_t s = tile * kTile + g * kHalf + 4 * lane;
            if (s + 4 <= fr.n_sym) {
                *(uint4 *)(dst + s) = make_uint4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (s + j < fr.n_sym) dst[s + j] = v[j];
            }
        }
    } else {
        // |z| <= 31 * 1024 fits 16 bits; samples t0 + 8 lane + 2 j + g
        uint32_t *dst = (uint32_t *)fr.out;
        const int64_t t = t0 + 8 * lane;
        if (t + 8 <= n && ((uintptr_t)dst & 31) == 0) {
            if constexpr (NPOL == 2) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t v[8] = {res[0][0][2 * h], res[1][0][2 * h], res[0][1][2 * h], res[1][1][2 * h],
                                           res[0][0][2 * h + 1], res[1][0][2 * h + 1], res[0][1][2 * h + 1],
                                           res[1][1][2 * h + 1]};
                    store32(dst + 2 * t + 8 * h, v);
                }
            } else {
                const uint32_t v[8] = {res[0][0][0], res[0][1][0], res[0][0][1], res[0][1][1],
                                       res[0][0][2], res[0][1][2], res[0][0][3], res[0][1][3]};
                store32(dst + t, v);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    if (t + 2 * j + g >= n) continue;
                    if constexpr (NPOL == 2)
                        *(uint2 *)(dst + 2 * (t + 2 * j + g)) = make_uint2(res[0][g][j], res[1][g][j]);
                    else
                        dst[t + 2 * j + g] = res[0][g][j];
                }
        }
    }
}

template <bool CHAIN>
__global__ void __launch_bounds__(32 * kCdcDirectWarps) cdc_direct_kernel(const DevFrame *__restrict__ frames,
                                                                          const int4 *__restrict__ items,
                                                                          const __grid_constant__ SingleFrame one) {
    __shared__ __align__(16) uint32_t s_pw[kCdcDirectWarps][CdcDirect<CHAIN, 2>::WORDS];
    __shared__ __align__(16) int2 s_tw[kCdcDirectWarps][kHistPairs];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // (no tables for a single frame: they would cost two dependent loads, and a call
    // their upload)
    int64_t tile = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const DevFrame *pf = &one.fr;
    if (items) {
        const int4 item = items[blockIdx.x];
        if (warp >= item.z) return;
        pf = frames + item.x;
        tile = (int64_t)item.y + warp;
    } else if (tile * kTile >= (CHAIN ? one.fr.n_sym : one.fr.n)) {
        return;
    }
    const DevFrame &fr = *pf;
    if (CHAIN || fr.n_pol == 2)
        cdc_tile<CHAIN, 2>(fr, tile, s_pw[warp], s_tw[warp], lane);
    else if constexpr (!CHAIN)
        cdc_tile<false, 1>(fr, tile, s_pw[warp], s_tw[warp], lane);
}

const SingleFrame kNoSingle{};

}  // namespace

cudaError_t cdc_direct_launch(const DevFrame *frames, const int4 *items, int n_items, bool chain, int warps,
                              cudaStream_t stream, const SingleFrame *one) {
    if (n_items <= 0) return cudaSuccess;
    const SingleFrame &single = one ? *one : kNoSingle;
    if (one) frames = nullptr, items = nullptr;
    if (chain)
        cdc_direct_kernel<true><<<n_items, 32 * warps, 0, stream>>>(frames, items, single);
    else
        cdc_direct_kernel<false><<<n_items, 32 * warps, 0, stream>>>(frames, items, single);
    return cudaGetLastError();
}

}  // namespace fnt
