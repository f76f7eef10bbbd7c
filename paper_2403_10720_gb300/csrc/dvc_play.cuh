// dvc_play.cuh -- uniform random playouts (Sec. II-B), one game per lane.
//
// A warp plays 32 games side by side, every lane its own, from start to end
// with no divergent control flow: a lane that is done plays on harmlessly
// until its warp's longest game ends.  Refilling such lanes with further games
// was measured and loses (two-player games, 1.68e7 playouts: 1.88 ms against
// 1.37): the games of a warp then leave the common rhythm in which one
// evaluation of the Philox rounds serves all 32 lanes, and starting a game
// costs the whole warp about half a game step.
//
// What bounds it is integer issue (ALU and integer-multiply pipes about 65 %
// busy each, 73 % of issue slots), so the game state is chosen for few
// operations per step:
//   - two players without jokers: the mover's and the opponent's face-down
//     tiles, the pool and the drawn tile, all as bit sets.  Face-up tiles take
//     no further part (the mover's unknown identities are the pool and the
//     opponent's face-down tiles), so neither hands nor face-up tiles are kept;
//   - otherwise: hands by distance from the mover, the face-up set, and for
//     each joker the threshold tile it stands in front of, which, unlike a count of
//     tiles to its left, no insertion changes;
//   - a uniform pair (slot, identity) from one word w: k = floor(w ns ni / 2^32)
//     splits into slot floor(w ns / 2^32) and identity floor(f ni / 2^32), f the
//     low word of w ns: two multiplies and no division;
//   - the n-th set bit from byte tables (one lookup after two population
//     counts); words from a ring in shared memory, refilled warp-wide.
// 4.29e9 two-player playouts from mid-game roots, 256 per leaf: 70.8 warp
// instructions per playout against 120 with hands by seat, division by magic
// numbers, 64-bit table entries and a branch per outcome; 1.26e10 against
// 7.4e9 playouts/s.
#pragma once
#include "dvc_device.cuh"

namespace dvc {

// Byte tables of select_bit: for the byte of the mask that holds the bit, at
// [rank in byte][byte value], the bit's position in the whole mask.  One copy per
// byte position, at the offset that the address arithmetic of select_bit adds.
constexpr uint32_t kSelOff1 = 2048u + 8u, kSelOff2 = 4128u + 16u;
constexpr uint32_t kSelBytes = 6208u;  // kSelOff2 + 2048, to a multiple of 64
struct SelectTable {
    uint8_t b[kSelBytes];
    constexpr SelectTable() : b() {
        for (uint32_t c = 0; c < 256u; ++c) {
            uint32_t r = 0;
            for (uint32_t i = 0; i < 8u; ++i)
                if ((c >> i) & 1u) {
                    b[r * 256u + c] = (uint8_t)i;
                    b[kSelOff1 + r * 256u + c] = (uint8_t)(i + 8u);
                    b[kSelOff2 + r * 256u + c] = (uint8_t)(i + 16u);
                    ++r;
                }
        }
    }
};
__device__ __align__(16) const SelectTable kSelect = SelectTable();

__device__ __forceinline__ void fill_select(unsigned char* dst, uint32_t tid, uint32_t nthr) {
    for (uint32_t e = tid; e < kSelBytes / 16u; e += nthr)
        reinterpret_cast<uint4*>(dst)[e] = reinterpret_cast<const uint4*>(kSelect.b)[e];
}

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t shared_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Index of the n-th set bit of m (m < 2^24, n < popc(m), or m = n = 0: some
// index); tab: shared address of the byte tables.  q carries the shift of the
// byte that holds the bit in its low five bits and, above them, minus 256 times
// the ranks before that byte plus the place of that byte's table.
__device__ __forceinline__ uint32_t select_bit(uint32_t tab, uint32_t m, uint32_t n) {
    const uint32_t c0 = __popc(m & 0xFFu), c1 = __popc(m & 0xFFFFu);
    const uint32_t q1 = c0 * (uint32_t)-256 + kSelOff1, q2 = c1 * (uint32_t)-256 + kSelOff2;
    uint32_t q = 0u;
    if (n >= c0) q = q1;
    if (n >= c1) q = q2;
    const uint32_t byte = __funnelshift_r(m, 0u, q) & 0xFFu;  // shifts by q mod 32
    const uint32_t a = tab + (n * 256u + q) + byte;
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
static_assert(kSelOff1 % 32u == 8u && kSelOff2 % 32u == 16u, "the low five bits are the byte's shift");

// The words of one playout stream (seed, tree, j, i, tag 4) in a ring of 16
// words in shared memory, lane-interleaved (word w of lane l of a warp's ring
// at (w mod 16) * 128 + 4 l), the first rows repeated after the last so that
// a step's words are read at fixed offsets.  Positions are kept times 128.
// The first Philox round's words that do not depend on the block are computed
// once per stream.
constexpr uint32_t kRingRows = 16u + 3u;
constexpr uint32_t kRingBytes = kRingRows * 128u;  // per warp
struct PlayWords {
    uint32_t ring;         // shared address of this lane's word 0
    uint32_t head, tail;   // words handed out / appended, times 128
    uint32_t n0, lo1, k1;  // round-1 state of the stream, key word 1 (tree)
    __device__ __forceinline__ void open(uint64_t seed, uint32_t tree, uint32_t j, uint32_t i) {
        n0 = __umulhi(0xCD9E8D57u, i) ^ j ^ (uint32_t)seed;
        lo1 = 0xCD9E8D57u * i;
        k1 = tree;
        head = tail = 0u;
    }
    // At least `need` (<= 4) words for every lane with want set; all lanes of the warp call.
    __device__ __forceinline__ void ensure(uint32_t need, bool want, uint64_t seed) {
        const uint32_t left = tail - head;
        if (!__any_sync(0xFFFFFFFFu, want && left < need * 128u)) return;
        const uint32_t blk = tail >> 9;
        const uint32_t tw = kTagRoll + 16u * (uint32_t)(seed >> 32);
        uint32_t x0 = n0, x1 = lo1, x2 = __umulhi(0xD2511F53u, blk) ^ tw ^ k1, x3 = 0xD2511F53u * blk;
        uint32_t ka = (uint32_t)seed, kb = k1;
#pragma unroll
        for (int r = 1; r < 10; ++r) {
            ka += 0x9E3779B9u;
            kb += 0xBB67AE85u;
            const uint32_t l0 = 0xD2511F53u * x0, h0 = __umulhi(0xD2511F53u, x0);
            const uint32_t l1 = 0xCD9E8D57u * x2, h1 = __umulhi(0xCD9E8D57u, x2);
            x0 = h1 ^ x1 ^ ka;
            x1 = l1;
            x2 = h0 ^ x3 ^ kb;
            x3 = l0;
        }
        const bool room = left <= 12u * 128u;
        const uint32_t at = tail & (16u * 128u - 1u), a = ring + at;
        if (room) {
            sts32(a, x0);
            sts32(a + 128u, x1);
            sts32(a + 256u, x2);
            sts32(a + 384u, x3);
            if (at == 0u) {
                sts32(a + 16u * 128u, x0);
                sts32(a + 17u * 128u, x1);
                sts32(a + 18u * 128u, x2);
            }
            tail += 512u;
        }
    }
    __device__ __forceinline__ uint32_t at() const { return ring + (head & (16u * 128u - 1u)); }
    __device__ __forceinline__ uint32_t used() const { return head >> 7; }
};

// A two-player game without jokers.
struct Play2 {
    uint32_t own, opp, pool;  // the mover's and the opponent's face-down tiles, the pool
    uint32_t out;             // the tile a wrong guess reveals: the drawn one, or the lowest if none was drawn
    uint32_t cur;
    static constexpr uint32_t kWords = 3u;

    __device__ __forceinline__ void begin(const G& g, uint32_t) {
        const uint32_t mine = g.cur ? g.h1 : g.h0, his = g.cur ? g.h0 : g.h1;
        own = mine & ~g.rev;
        opp = his & ~g.rev;
        pool = kNumMask & ~(g.h0 | g.h1);
        out = g.drawn < 24u ? 1u << g.drawn : own & (0u - own);
        cur = g.cur;
    }
    __device__ __forceinline__ void idle() { own = opp = pool = out = cur = 0u; }

    // One guess with its resolution and the next draw (PEND: with pend set,
    // the continue coin of a mover that may stop instead of the guess).
    // Returns true when the game ends, with the winner in `winner`.
    template <bool PEND>
    __device__ __forceinline__ bool step(PlayWords& r, uint32_t thr, uint32_t tab, bool pend, uint32_t& winner) {
        const uint32_t a = r.at(), b = PEND && pend ? a : a + 128u;
        const uint32_t w0 = lds32(a), w1 = lds32(b), w2 = lds32(b + 128u);
        const uint32_t ns = __popc(opp), np = __popc(pool);
        const uint64_t y = (uint64_t)w0 * ns;
        const uint32_t s = (uint32_t)(y >> 32), i = __umulhi((uint32_t)y, ns + np);
        uint32_t tb = 1u << select_bit(tab, opp, s);
        bool hit = (uint32_t)__popc((pool | opp) & (tb - 1u)) == i;
        if (PEND && pend) {
            hit = true;
            tb = 0u;
        }
        const uint32_t x = hit ? tb : out;
        own &= ~x;
        opp &= ~x;
        winner = cur ^ (hit ? 0u : 1u);
        const bool over = own == 0u || opp == 0u;
        const bool coin = hit && thr != 0u, again = coin && w1 < thr;
        // the next mover draws; with an empty pool the lowest face-down tile
        // takes the drawn tile's place
        const uint32_t from = pool ? pool : opp;
        const uint32_t d = 1u << select_bit(tab, from, __umulhi(coin ? w2 : w1, np));
        r.head += (PEND && pend ? 0u : 128u) + (coin ? 128u : 0u);
        if (!again) {
            r.head += pool ? 128u : 0u;
            pool &= ~d;
            out = d;
            const uint32_t n = opp | d;
            opp = own;
            own = n;
            cur ^= 1u;
        }
        return over;
    }
};

// Any player count, jokers.
struct PlayN {
    uint32_t a0, a1, a2, a3;  // hands of seats cur, cur + 1, ... (modulo np; 0 from np on)
    uint32_t rev, out;        // face-up tiles; the drawn tile, 0 if none
    uint32_t th;              // joker j stands before numbered tile (th >> 8 j) & 31; bit 16: equal thresholds, white first
    uint32_t cur, np, tmask;
    static constexpr uint32_t kWords = 4u;

    // The threshold of a joker after `gap` numbered tiles of the row hn.
    __device__ __forceinline__ static uint32_t threshold(uint32_t tab, uint32_t hn, uint32_t gap) {
        const uint32_t g = min(gap, (uint32_t)__popc(hn));
        return g ? select_bit(tab, hn, g - 1u) + 1u : 0u;
    }
    __device__ __forceinline__ void begin(const G& g, uint32_t tab) {
        uint32_t q1 = g.cur + 1u, q2 = g.cur + 2u, q3 = g.cur + 3u;
        q1 = q1 >= g.np ? q1 - g.np : q1;
        q2 = q2 >= g.np ? q2 - g.np : q2;
        q3 = q3 >= g.np ? q3 - g.np : q3;
        a0 = g.hand(g.cur);
        a1 = g.hand(q1);
        a2 = g.np > 2u ? g.hand(q2) : 0u;
        a3 = g.np > 3u ? g.hand(q3) : 0u;
        rev = g.rev;
        out = g.drawn < 26u ? 1u << g.drawn : 0u;
        cur = g.cur;
        np = g.np;
        tmask = g.tmask;
        th = 0u;
        if (tmask & kJokerMask) {
            const uint32_t o0 = holder(24u), o1 = holder(25u);
            th = threshold(tab, o0 & kNumMask, g.jg0) | threshold(tab, o1 & kNumMask, g.jg1) << 8 | g.jflag << 16;
        }
    }
    __device__ __forceinline__ void idle() { a0 = a1 = a2 = a3 = rev = out = th = cur = tmask = 0u, np = 2u; }
    // The hand that holds tile t (0 if it is in the pool).
    __device__ __forceinline__ uint32_t holder(uint32_t t) const {
        return ((a0 >> t) & 1u) ? a0 : ((a1 >> t) & 1u) ? a1 : ((a2 >> t) & 1u) ? a2 : ((a3 >> t) & 1u) ? a3 : 0u;
    }
    // Places of the jokers in jk (bit 0 black, 1 white) among the numbered
    // tiles n of one row, left to right; 0xFF for one not in jk.
    __device__ __forceinline__ void joker_places(uint32_t n, uint32_t jk, uint32_t& i0, uint32_t& i1) const {
        const uint32_t t0 = th & 31u, t1 = (th >> 8) & 31u;
        const bool white = t1 < t0 || (t1 == t0 && (th >> 16));  // the white joker stands first
        i0 = (jk & 1u) ? __popc(n & ((1u << t0) - 1u)) + (jk == 3u && white ? 1u : 0u) : 0xFFu;
        i1 = (jk & 2u) ? __popc(n & ((1u << t1) - 1u)) + (jk == 3u && !white ? 1u : 0u) : 0xFFu;
    }

    template <bool PEND>
    __device__ __forceinline__ bool step(PlayWords& r, uint32_t thr, uint32_t tab, bool pend, uint32_t& winner) {
        const uint32_t a = r.at(), b = PEND && pend ? a : a + 128u;
        const uint32_t w0 = lds32(a), w1 = lds32(b), w2 = lds32(b + 128u);
        const uint32_t U = tmask & ~a0 & ~rev, ni = __popc(U);
        const uint32_t c1 = __popc(a1 & ~rev), c2 = __popc(a2 & ~rev), c3 = __popc(a3 & ~rev);
        const uint64_t y = (uint64_t)w0 * (c1 + c2 + c3);
        uint32_t s = (uint32_t)(y >> 32);
        const uint32_t i = __umulhi((uint32_t)y, ni);
        uint32_t hid = a1 & ~rev;
        if (s >= c1) {
            s -= c1;
            hid = a2 & ~rev;
            if (s >= c2) {
                s -= c2;
                hid = a3 & ~rev;
            }
        }
        // the tile in that face-down slot
        const uint32_t n = hid & kNumMask, jk = hid >> 24;
        uint32_t sn = s, jb = 0u;
        if (__any_sync(0xFFFFFFFFu, jk != 0u)) {
            uint32_t i0, i1;
            joker_places(n, jk, i0, i1);
            sn -= (i0 < s ? 1u : 0u) + (i1 < s ? 1u : 0u);
            jb = s == i0 ? 1u << 24 : s == i1 ? 2u << 24 : 0u;
            if (jb) sn = 0u;  // any valid rank
        }
        uint32_t tb = 1u << select_bit(tab, n, n ? sn : 0u);
        tb = jb ? jb : tb;
        bool hit = (uint32_t)__popc(U & (tb - 1u)) == i;
        if (PEND && pend) {
            hit = true;
            tb = 0u;
        }
        uint32_t own = out;
        if (__any_sync(0xFFFFFFFFu, !hit && out == 0u)) {  // nothing drawn: the leftmost face-down tile
            const uint32_t m = a0 & ~rev, mn = m & kNumMask;
            uint32_t i0, i1;
            joker_places(mn, m >> 24, i0, i1);
            const uint32_t first = i0 == 0u ? 1u << 24 : i1 == 0u ? 2u << 24 : mn & (0u - mn);
            own = out ? out : first;
        }
        rev |= hit ? tb : own;
        // seats still in: those with a face-down tile
        const uint32_t e1 = (a1 & ~rev) ? 1u : 0u, e2 = (a2 & ~rev) ? 1u : 0u, e3 = (a3 & ~rev) ? 1u : 0u;
        const uint32_t live = e1 + e2 + e3;
        const bool over = live == 0u || (live == 1u && !(a0 & ~rev));
        uint32_t d = e1 ? 1u : e2 ? 2u : 3u;  // distance to the next seat still in
        uint32_t nc = cur + d;
        nc = nc >= np ? nc - np : nc;
        winner = live ? nc : cur;
        const bool coin = hit && thr != 0u, again = coin && w1 < thr;
        r.head += (PEND && pend ? 0u : 128u) + (coin ? 128u : 0u);
        // the next seat moves: hands rotate by d; with np seats position k + np is position k
        const bool pass = !again;
        d = pass ? d : 0u;
        cur = pass ? nc : cur;
        if (d & 1u) {
            const uint32_t t = a0;
            a0 = a1;
            a1 = np == 2u ? t : a2;
            a2 = np == 3u ? t : a3;
            a3 = np == 4u ? t : 0u;
        }
        if (d & 2u) {
            const uint32_t t0 = a0, t1 = a1;
            a0 = a2;
            a1 = np == 3u ? t0 : a3;
            a2 = np == 3u ? t1 : t0;
            a3 = np == 3u ? 0u : t1;
        }
        // ... and draws
        const uint32_t pool = tmask & ~(a0 | a1 | a2 | a3), pn = pool & kNumMask;
        const uint32_t k = __umulhi(coin ? w2 : w1, __popc(pool)), nn = __popc(pn);
        uint32_t t = select_bit(tab, pn, k < nn ? k : 0u);
        const bool joker = k >= nn && pool != 0u;
        if (joker) t = (pool >> 24) == 2u || k > nn ? 25u : 24u;
        const uint32_t dbit = pool ? 1u << t : 0u;
        if (pass) {
            r.head += pool ? 128u : 0u;
            out = dbit;
        }
        if (__any_sync(0xFFFFFFFFu, pass && joker)) {  // a joker's place: uniform over the row's insertion points
            if (pass && joker) {
                const uint32_t w = lds32(r.at());
                r.head += 128u;
                const uint32_t j = t - 24u, hn = a0 & kNumMask, to = (th >> (8u * (j ^ 1u))) & 31u;
                const uint32_t pos = __umulhi(w, __popc(a0) + 1u);
                uint32_t gap = pos, white = 0u;
                if ((a0 >> (24u + (j ^ 1u))) & 1u) {
                    const uint32_t po = __popc(hn & ((1u << to) - 1u));  // the other joker's place
                    const bool first = pos <= po;
                    gap = first ? pos : pos - 1u;
                    if (gap == po) white = first ? j : j ^ 1u;
                }
                const uint32_t nt = threshold(tab, hn, gap);
                th = ((th & (j ? 0x001Fu : 0x1F00u)) | nt << (8u * j)) | white << 16;
            }
        }
        a0 |= pass ? dbit : 0u;
        return over;
    }
};

// The 32 games of a warp to their ends.  busy: this lane has a game (its
// state and stream begun); pend: it starts with the continue coin.  Returns
// the lane's winner, kNone if it has no game or, after 128 steps, no result (a
// game has at most |T| guesses, each turning one tile face up).  CNT: adds the
// words of this lane's game to `words` and the warp's steps to `steps` (the
// same on every lane).
template <class Game, bool PEND, bool CNT>
__device__ __forceinline__ uint32_t play_games(Game& g, PlayWords& r, bool busy, bool pend, uint64_t seed,
                                               uint32_t thr, uint32_t tab, uint32_t& words, uint32_t& steps) {
    uint32_t res = kNone;
    for (int it = 0; it < 128; ++it) {
        if constexpr (CNT) steps += __popc(__ballot_sync(0xFFFFFFFFu, busy));
        r.ensure(Game::kWords, busy, seed);
        uint32_t winner;
        const uint32_t before = r.used();
        const bool over = g.template step<PEND>(r, thr, tab, PEND && it == 0 && pend, winner);
        if (busy && over) {
            res = winner;
            if constexpr (CNT) words += before + 1u;  // the last guess; what step() read past it is not used
        }
        busy = busy && !over;
        if (!__any_sync(0xFFFFFFFFu, busy)) break;
    }
    return res;
}

// Credit the winners of a warp's games to wins[4 * leaf + seat] (global or
// shared); `leaf` is this lane's.  One add per seat when the warp's games
// share their leaf.
__device__ __forceinline__ void credit_wins(int32_t* wins, uint32_t leaf, uint32_t winner) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t l0 = __shfl_sync(0xFFFFFFFFu, leaf, 0);
    if (__all_sync(0xFFFFFFFFu, winner >= 4u || leaf == l0)) {
#pragma unroll
        for (uint32_t s = 0; s < 4u; ++s) {
            const uint32_t n = __popc(__ballot_sync(0xFFFFFFFFu, winner == s));
            if (lane == s && n) atomicAdd(&wins[4u * l0 + s], (int32_t)n);
        }
    } else if (winner < 4u) {
        atomicAdd(&wins[4u * leaf + winner], 1);
    }
}

}  // namespace dvc
