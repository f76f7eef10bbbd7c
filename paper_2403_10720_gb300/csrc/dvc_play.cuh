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
//   - otherwise: hands by distance from the mover and the face-up set, in an
//     order of the tiles in which a joker's bit stands between the tiles its
//     row has left and right of it (at the end while it is in the pool), so
//     that bit order is row order and only placing a joker moves bits;
//   - a uniform pair (slot, identity) from one word w: k = floor(w ns ni / 2^32)
//     splits into slot floor(w ns / 2^32) and identity floor(f ni / 2^32), f the
//     low word of w ns: two multiplies and no division;
//   - the n-th set bit from byte tables (one lookup after two population
//     counts); words from a ring in shared memory, refilled warp-wide.
// 32 four-player joker games on a warp alone take 18,400 cycles, against 29,200
// with hands in identity order and jokers placed by gap counts.
// 1.68e7 two-player playouts from mid-game roots, 256 per leaf: 70.8 warp
// instructions per playout against 120 with hands by seat, division by magic
// numbers, 64-bit table entries and a branch per outcome; 1.26e10 against
// 7.4e9 playouts/s.
#pragma once
#include "dvc_device.cuh"

namespace dvc {

// Byte tables of select_bit for masks of three CH-bit chunks: for the chunk that
// holds the bit, at [rank in chunk][chunk value], the bit's position in the whole
// mask.  One copy per chunk, at the offset that select_bit's address arithmetic
// adds (its low five bits are the chunk's shift).
template <uint32_t CH>
struct SelectTable {
    static constexpr uint32_t kRow = 1u << CH;
    static constexpr uint32_t kOff1 = (CH * kRow + 31u) / 32u * 32u + CH;
    static constexpr uint32_t kOff2 = (kOff1 + CH * kRow + 31u) / 32u * 32u + 2u * CH;
    static constexpr uint32_t kBytes = (kOff2 + CH * kRow + 15u) / 16u * 16u;
    uint8_t b[kBytes];
    constexpr SelectTable() : b() {
        for (uint32_t c = 0; c < kRow; ++c) {
            uint32_t r = 0;
            for (uint32_t i = 0; i < CH; ++i)
                if ((c >> i) & 1u) {
                    b[r * kRow + c] = (uint8_t)i;
                    b[kOff1 + r * kRow + c] = (uint8_t)(i + CH);
                    b[kOff2 + r * kRow + c] = (uint8_t)(i + 2u * CH);
                    ++r;
                }
        }
    }
};
// 24 numbered tiles in bytes (6.2 KB); 26 tiles in chunks of nine (13.9 KB)
__device__ __align__(16) const SelectTable<8> kSelect24 = SelectTable<8>();
__device__ __align__(16) const SelectTable<9> kSelect27 = SelectTable<9>();

template <uint32_t CH>
__device__ __forceinline__ void fill_select(unsigned char* dst, uint32_t tid, uint32_t nthr) {
    const uint4* src = reinterpret_cast<const uint4*>(CH == 8u ? kSelect24.b : kSelect27.b);
    for (uint32_t e = tid; e < SelectTable<CH>::kBytes / 16u; e += nthr) reinterpret_cast<uint4*>(dst)[e] = src[e];
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

// Index of the n-th set bit of m (m < 2^(3 CH), n < popc(m), or m = n = 0:
// some index); tab: shared address of the tables.  q carries the shift of the
// chunk that holds the bit in its low five bits and, above them, minus the row
// length times the ranks before that chunk plus the place of that chunk's table.
// ORDERED: the read stays behind the barrier that follows the fill whatever m and n
// come from, for callers that may have them from before it.
template <uint32_t CH, bool ORDERED = false>
__device__ __forceinline__ uint32_t select_bit(uint32_t tab, uint32_t m, uint32_t n) {
    using T = SelectTable<CH>;
    static_assert(T::kOff1 % 32u == CH && T::kOff2 % 32u == 2u * CH, "the low five bits are the chunk's shift");
    const uint32_t c0 = __popc(m & (T::kRow - 1u)), c1 = __popc(m & (T::kRow * T::kRow - 1u));
    const uint32_t q1 = c0 * (0u - T::kRow) + T::kOff1, q2 = c1 * (0u - T::kRow) + T::kOff2;
    uint32_t q = 0u;
    if (n >= c0) q = q1;
    if (n >= c1) q = q2;
    const uint32_t chunk = __funnelshift_r(m, 0u, q) & (T::kRow - 1u);  // shifts by q mod 32
    const uint32_t a = tab + (n * T::kRow + q) + chunk;
    uint32_t v;
    // otherwise not volatile: the tables do not change after they are filled, and a
    // step's n comes from its random words, which lds32 reads behind the barrier
    if constexpr (ORDERED) asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    else asm("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}

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
    // The block of words that the next append() adds.
    __device__ __forceinline__ uint4 block(uint64_t seed) const {
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
        return make_uint4(x0, x1, x2, x3);
    }
    // Append it if the ring has room.
    __device__ __forceinline__ void append(uint4 x) {
        if (tail - head > 12u * 128u) return;
        const uint32_t at = tail & (16u * 128u - 1u), a = ring + at;
        sts32(a, x.x);
        sts32(a + 128u, x.y);
        sts32(a + 256u, x.z);
        sts32(a + 384u, x.w);
        if (at == 0u) {
            sts32(a + 16u * 128u, x.x);
            sts32(a + 17u * 128u, x.y);
            sts32(a + 18u * 128u, x.z);
        }
        tail += 512u;
    }
    // At least NEED (<= 8) words for every lane with want set; all lanes of the warp call.
    template <uint32_t NEED>
    __device__ __forceinline__ void ensure(bool want, uint64_t seed) {
#pragma unroll
        for (uint32_t have = 0u; have < NEED; have += 4u) {
            if (!__any_sync(0xFFFFFFFFu, want && tail - head < NEED * 128u)) return;
            append(block(seed));
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
    static constexpr uint32_t kWords = 3u, kChunk = 8u;

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
    // EARLY: the draw is selected for either of the two words it may fall to
    // (a coin comes before it or not) beside the guess: more operations, a
    // shorter chain.
    template <bool PEND, bool EARLY>
    __device__ __forceinline__ bool step(PlayWords& r, uint32_t thr, uint32_t tab, bool pend, uint32_t& winner) {
        const uint32_t a = r.at(), b = PEND && pend ? a : a + 128u;
        const uint32_t w0 = lds32(a), w1 = lds32(b), w2 = lds32(b + 128u);
        const uint32_t ns = __popc(opp), np = __popc(pool);
        uint32_t t1 = 0u, t2 = 0u;
        if constexpr (EARLY) {
            t1 = select_bit<8>(tab, pool, __umulhi(w1, np));
            t2 = select_bit<8>(tab, pool, __umulhi(w2, np));
        }
        const uint64_t y = (uint64_t)w0 * ns;
        const uint32_t s = (uint32_t)(y >> 32), i = __umulhi((uint32_t)y, ns + np);
        uint32_t tb = 1u << select_bit<8>(tab, opp, s);
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
        uint32_t d;
        if constexpr (EARLY) {
            d = pool ? 1u << (coin ? t2 : t1) : opp & (0u - opp);
        } else {
            const uint32_t from = pool ? pool : opp;
            d = 1u << select_bit<8>(tab, from, __umulhi(coin ? w2 : w1, np));
        }
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

// Any player count, jokers.  Tiles stand in an order in which bit order is row
// order: numbered tiles ascending, each joker that has been dealt or drawn
// right after the tile of its row on its left (a numbered tile inserted later
// between the two would have gone to the joker's right, so the place stays
// right), jokers in the pool at the end, black first.  Identities compare in
// another order, numbered tiles before jokers, which only their rank needs.
struct PlayN {
    uint32_t a0, a1, a2, a3;  // hands of seats cur, cur + 1, ... (modulo np; 0 from np on)
    uint32_t rev, out;        // face-up tiles; the tile a wrong guess reveals: the drawn one, or the leftmost
    uint32_t j0, j1;          // the black and the white joker's bits (0 without jokers)
    uint32_t cur, np, all;
    static constexpr uint32_t kWords = 4u, kChunk = 9u;

    // Move a joker from bit `jb`, held by nobody, to bit p <= its own: the tiles
    // from p on go up one place.  Its bit is left out of every hand.
    __device__ __forceinline__ uint32_t place(uint32_t jb, uint32_t p) {
        const uint32_t to = 1u << p, mid = (jb - 1u) & ~(to - 1u);
        a0 += a0 & mid;
        a1 += a1 & mid;
        a2 += a2 & mid;
        a3 += a3 & mid;
        rev += rev & mid;
        j0 = j0 == jb ? to : j0 + (j0 & mid);
        j1 = j1 == jb ? to : j1 + (j1 & mid);
        return to;
    }
    // Joker j (bit jb) of a record: from the end to the place its gap gives it
    // among the numbered tiles of the hand that holds it; nothing if in the
    // pool.  `other`: bit of the other joker if that one, in a hand, comes first
    // in a gap they share.
    __device__ __forceinline__ void settle(uint32_t tab, uint32_t jb, uint32_t gap, uint32_t other) {
        const uint32_t held = a0 | a1 | a2 | a3;
        if (!(held & jb)) return;
        const uint32_t h = (a0 & jb) ? a0 : (a1 & jb) ? a1 : (a2 & jb) ? a2 : a3;
        const uint32_t hn = h & ~(j0 | j1), k = min(gap, (uint32_t)__popc(hn));
        // ordered: the record may have been loaded before the tables were filled
        uint32_t p = k ? select_bit<9, true>(tab, hn, k - 1u) + 1u : 0u;
        if (other == 1u << p) ++p;
        const uint32_t in0 = a0 & jb, in1 = a1 & jb, in2 = a2 & jb, up = rev & jb;
        a0 &= ~jb;
        a1 &= ~jb;
        a2 &= ~jb;
        a3 &= ~jb;
        rev &= ~jb;
        const uint32_t drawn = out == jb ? 1u : 0u;
        if (!drawn) out += out & (jb - 1u) & ~((1u << p) - 1u);
        const uint32_t to = place(jb, p);
        if (in0) a0 |= to;
        else if (in1) a1 |= to;
        else if (in2) a2 |= to;
        else a3 |= to;
        if (up) rev |= to;
        if (drawn) out = to;
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
        // a tile is in one hand at most (a valid record's are; place() relies on it)
        a1 &= ~a0;
        a2 &= ~(a0 | a1);
        a3 &= ~(a0 | a1 | a2);
        rev = g.rev;
        out = g.drawn < 26u ? 1u << g.drawn : 0u;
        cur = g.cur;
        np = g.np;
        all = g.tmask;
        j0 = g.tmask & (1u << 24);
        j1 = g.tmask & (1u << 25);
        if (j0) {
            settle(tab, j0, g.jg0, 0u);
            // of two jokers in one gap the white one comes after the black one unless flagged
            const uint32_t held = a0 | a1 | a2 | a3;
            settle(tab, j1, g.jg1, g.jflag ? 0u : held & j0);
        }
        const uint32_t m = a0 & ~rev;
        if (!out) out = m & (0u - m);
    }
    __device__ __forceinline__ void idle() { a0 = a1 = a2 = a3 = rev = out = j0 = j1 = cur = all = 0u, np = 2u; }

    template <bool PEND, bool EARLY>
    __device__ __forceinline__ bool step(PlayWords& r, uint32_t thr, uint32_t tab, bool pend, uint32_t& winner) {
        const uint32_t a = r.at(), b = PEND && pend ? a : a + 128u;
        const uint32_t w0 = lds32(a), w1 = lds32(b), w2 = lds32(b + 128u);
        const uint32_t pool = all & ~(a0 | a1 | a2 | a3), npool = __popc(pool);
        uint32_t t1 = 0u, t2 = 0u;
        if constexpr (EARLY) {
            t1 = select_bit<9>(tab, pool, __umulhi(w1, npool));
            t2 = select_bit<9>(tab, pool, __umulhi(w2, npool));
        }
        const uint32_t U = all & ~a0 & ~rev;
        const uint32_t c1 = __popc(a1 & ~rev), c2 = __popc(a2 & ~rev), c3 = __popc(a3 & ~rev);
        const uint64_t y = (uint64_t)w0 * (c1 + c2 + c3);
        uint32_t s = (uint32_t)(y >> 32);
        const uint32_t i = __umulhi((uint32_t)y, __popc(U));
        uint32_t hid = a1 & ~rev;
        if (s >= c1) {
            s -= c1;
            hid = a2 & ~rev;
            if (s >= c2) {
                s -= c2;
                hid = a3 & ~rev;
            }
        }
        uint32_t tb = 1u << select_bit<9>(tab, hid, s);
        // rank of its identity among the unknown ones: jokers come last, black before white
        const uint32_t Un = U & ~(j0 | j1);
        const uint32_t below = tb & (j0 | j1) ? 0xFFFFFFFFu : tb - 1u;
        bool hit = (uint32_t)__popc(Un & below) + (tb == j1 && (U & j0) ? 1u : 0u) == i;
        if (PEND && pend) {
            hit = true;
            tb = 0u;
        }
        rev |= hit ? tb : out;
        // seats still in: those with a face-down tile
        const bool e1 = (a1 & ~rev) != 0u, e2 = (a2 & ~rev) != 0u, e3 = (a3 & ~rev) != 0u;
        const uint32_t live = (e1 ? 1u : 0u) + (e2 ? 1u : 0u) + (e3 ? 1u : 0u);
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
            const uint32_t t0 = a0, t1_ = a1;
            a0 = a2;
            a1 = np == 3u ? t0 : a3;
            a2 = np == 3u ? t1_ : t0;
            a3 = np == 3u ? 0u : t1_;
        }
        // ... and draws; with an empty pool its leftmost face-down tile takes the drawn tile's place
        const uint32_t t = EARLY ? (coin ? t2 : t1) : select_bit<9>(tab, pool, __umulhi(coin ? w2 : w1, npool));
        uint32_t db = pool ? 1u << t : 0u;
        if (pass) r.head += pool ? 128u : 0u;
        const bool joker = pass && (db & (j0 | j1));
        if (__any_sync(0xFFFFFFFFu, joker)) {  // a joker's place: uniform over the row's insertion points
            if (joker) {
                const uint32_t pos = __umulhi(lds32(r.at()), __popc(a0) + 1u);
                r.head += 128u;
                db = place(db, pos ? select_bit<9>(tab, a0, pos - 1u) + 1u : 0u);
            }
        }
        if (pass) {
            a0 |= db;
            const uint32_t m = a0 & ~rev;
            out = pool ? db : m & (0u - m);
        }
        return over;
    }
};

// The 32 games of a warp to their ends.  busy: this lane has a game (its
// state and stream begun); pend: it starts with the continue coin.  Returns
// the lane's winner, kNone if it has no game or, after 128 steps, no result (a
// game has at most |T| guesses, each turning one tile face up).  CNT: adds the
// words and steps of this lane's game to `words` and `steps`.
// ALONE: for a warp that has its scheduler nearly to itself (two-player games in
// the fused engine, by the rule play_alone in dvc_shape.cuh), where a step costs the
// length of its dependent chain and not its operations: two steps and the next
// block of words, which neither needs, form one stretch of code without a branch,
// and draws are selected early.  One game alone 10,400 -> 9,450 cycles, 32 games
// 11,900 -> 10,700.  The other games' step is twice as long and loses to instruction fetch that way (12 one-warp
// CTAs per SM: 40,400 -> 53,300 cycles).
template <class Game, bool PEND, bool CNT, bool ALONE>
__device__ __forceinline__ uint32_t play_games(Game& g, PlayWords& r, bool busy, bool pend, uint64_t seed,
                                               uint32_t thr, uint32_t tab, uint32_t& words, uint32_t& steps) {
    uint32_t res = kNone;
    constexpr int kSteps = ALONE ? 2 : 1;
    if constexpr (ALONE) {  // three blocks ahead: the loop adds what two plain steps use
#pragma unroll
        for (int k = 0; k < 3; ++k) r.append(r.block(seed));
    }
    for (int it = 0; it < 128; it += kSteps) {
        r.ensure<kSteps * Game::kWords>(busy, seed);
        uint4 next;
        if constexpr (ALONE) next = r.block(seed);
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
            if constexpr (CNT) steps += busy ? 1u : 0u;
            uint32_t winner;
            const uint32_t before = r.used();
            const bool over =
                g.template step<PEND, ALONE>(r, thr, tab, PEND && it + k == 0 && pend, winner);
            if (busy && over) {
                res = winner;
                if constexpr (CNT) words += before + 1u;  // the last guess; what step() read past it is not used
            }
            busy = busy && !over;
        }
        if constexpr (ALONE) r.append(next);
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
