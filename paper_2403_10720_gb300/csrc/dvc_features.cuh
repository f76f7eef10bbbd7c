// dvc_features.cuh -- the value network's input bits of a state.
#pragma once
#include "dvc_device.cuh"

namespace dvc {

constexpr int kFeatures = 640;
constexpr int kFeatWords = kFeatures / 32;  // 20
constexpr int kFeatPitch = kFeatWords + 1;  // 21: 32 rows start in 32 different banks

__device__ __forceinline__ uint32_t unknown_mask(const G& g) { return g.tmask & ~g.hand(g.cur) & ~g.rev; }

// OR a field of `width` bits into the bit vector f at position pos (both
// known at compile time once the caller's loops are unrolled).
__device__ __forceinline__ void or_bits(uint32_t* f, int pos, uint32_t field, int width) {
    const int w = pos >> 5, sh = pos & 31;
    f[w] |= field << sh;
    if (sh + width > 32) f[w + 1] |= field >> (32 - sh);
}

// The bits of part `part` of one row (0: the tiles; k: the slots of opponent
// k), ORed into its kFeatWords words in shared memory (zeroed before).  Positions
// are fixed, every loop is unrolled, so bits gather in registers.
__device__ __forceinline__ void feature_bits(const G& g, int part, uint32_t* mine) {
    uint32_t q1 = g.cur + 1u, q2 = g.cur + 2u, q3 = g.cur + 3u;
    q1 = q1 >= g.np ? q1 - g.np : q1;
    q2 = q2 >= g.np ? q2 - g.np : q2;
    q3 = q3 >= g.np ? q3 - g.np : q3;
    const uint32_t M1 = g.hand(q1), M2 = g.np > 2u ? g.hand(q2) : 0u, M3 = g.np > 3u ? g.hand(q3) : 0u;
    if (part == 0) {
        uint32_t f[6] = {0u, 0u, 0u, 0u, 0u, 0u};  // bits 0..181
        const uint32_t held = g.h0 | g.h1 | g.h2 | g.h3;
        // tiles: bit 7t + (owner seat relative to the mover), 7t + 4 + face-up,
        // 7t + 6 if drawn this turn; tiles in the pool have none
#pragma unroll
        for (int t = 0; t < 26; ++t) {
            const uint32_t r = ((M1 >> t) & 1u) | (((M2 >> t) & 1u) << 1) | (((M3 >> t) & 1u) * 3u);
            const uint32_t grp = (1u << r) | (16u << ((g.rev >> t) & 1u)) | ((uint32_t)t == g.drawn ? 64u : 0u);
            or_bits(f, 7 * t, ((held >> t) & 1u) ? grp : 0u, 7);
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) atomicOr(&mine[k], f[k]);
    } else if ((uint32_t)part < g.np) {
        const int k = part;
        const uint32_t U = unknown_mask(g);
        const uint32_t jok = (U & kJokerMask) ? 1u << 12 : 0u;
        // opponent k (seat cur + k), slot s: 13 bits at 182 + ((k - 1) * 11 + s) * 13;
        // a face-up tile sets its value (a joker 12); a face-down slot sets every
        // value the mover cannot see strictly between its face-up numbered
        // neighbours, plus bit 12 if a joker is unseen.  Slots are walked left
        // to right: numbered tiles ascend by id, each joker stands where its
        // gap puts it, and a joker's right-hand threshold is the next numbered
        // tile of the row (or 24).
        uint32_t f[5] = {0u, 0u, 0u, 0u, 0u};  // the opponent's 143 bits
        const uint32_t hq = k == 1 ? M1 : (k == 2 ? M2 : M3);
        const uint32_t len = (uint32_t)k < g.np ? (uint32_t)__popc(hq) : 0u;
        const uint32_t num = hq & kNumMask, R = num & g.rev;
        const uint32_t jp0 = (hq >> 24) & 1u ? joker_pos(g, hq, 0u) : 0xFFu;
        const uint32_t jp1 = (hq >> 25) & 1u ? joker_pos(g, hq, 1u) : 0xFFu;
        uint32_t rem = num;
#pragma unroll
        for (int sl = 0; sl < 11; ++sl) {
            if ((uint32_t)sl < len) {
                const bool j0 = (uint32_t)sl == jp0, j1 = (uint32_t)sl == jp1;
                const uint32_t low = rem ? (uint32_t)__ffs(rem) - 1u : 24u;
                const uint32_t t = j0 ? 24u : (j1 ? 25u : low);
                const uint32_t thr = low;  // a numbered slot's own tile, or the tile right of a joker
                if (!j0 && !j1) rem &= rem - 1u;
                uint32_t field;
                if ((g.rev >> t) & 1u) {
                    field = 1u << (t < 24u ? t >> 1 : 12u);
                } else {
                    const uint32_t below_thr = thr >= 32u ? 0xFFFFFFFFu : (1u << thr) - 1u;
                    const uint32_t left = R & below_thr, right = R & ~below_thr;
                    const int lo = left ? 31 - __clz(left) : -1;
                    const int hi = right ? __ffs(right) - 1 : 24;
                    const uint32_t above = lo < 0 ? 0x00FFFFFFu : (0x00FFFFFFu & ~((2u << lo) - 1u));
                    const uint32_t below = (1u << hi) - 1u;
                    const uint32_t m = U & above & below;
                    uint32_t x = (m | (m >> 1)) & 0x00555555u;
                    x = (x | (x >> 1)) & 0x00333333u;
                    x = (x | (x >> 2)) & 0x000F0F0Fu;
                    x = ((x | (x >> 4)) & 0x000000FFu) | ((x >> 8) & 0x00000F00u);
                    field = x | jok;
                }
                or_bits(f, sl * 13, field, 13);
            }
        }
        const uint32_t at = 182u + 143u * (uint32_t)(k - 1), w0 = at >> 5, sh = at & 31u;
        uint32_t carry = 0u;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            atomicOr(&mine[w0 + i], (f[i] << sh) | carry);
            carry = sh ? f[i] >> (32u - sh) : 0u;
        }
        if (carry) atomicOr(&mine[w0 + 5], carry);
    }
}

// A byte of feature bits as 8 BF16 values (0 or 1).
__device__ __forceinline__ uint4 feature_bf16(uint32_t b) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t two = (b >> (2 * j)) & 3u;  // low bit to the low half, high bit to the high half
        w[j] = (two * 0x8001u & 0x00010001u) * 0x3F80u;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace dvc
