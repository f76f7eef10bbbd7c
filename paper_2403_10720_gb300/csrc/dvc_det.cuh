// dvc_det.cuh -- uniform determinization of a root view (Sec. III-A: the
// plausible values of the tiles a player cannot see are re-drawn for every
// simulation), on the device.
//
// The unknown tiles (not in the observer's hand, not face up) are spread
// over the opponents' face-down slots and the pool.  A consistent deal keeps
// each opponent's face-up tiles where they are and its numbered tiles in
// ascending order; jokers may stand in any slot.  For opponent k the face-down
// slots between consecutive face-up numbered tiles ("anchors") form gaps; a
// gap takes numbered tiles from its id interval in order, and slots a gap
// still has open when the ascending walk over unknown numbered tiles passes
// its right anchor must hold jokers.  F(i, r, J) counts completions when the
// unknown numbered tile u_i is next, gap slots r[k] are still open and J
// unknown jokers are unplaced; closing a gap of c slots with o open ones
// multiplies by C(c, o) * J!/(J-o)!.  The table depends only on the root
// view, so it is filled once per search and sampled every iteration.  Few
// tiles have an anchor right after them: for the others (DetPlan::cross) no
// gap closes, and the destinations' counts stand at fixed distances in the next
// layer, four independent loads.  To sample, walk
// the tiles in id order, pick the destination (pool first, then opponents from
// observer+1) with weight = completions it leaves, as floor(r64 * W / 2^64)
// from two stream words, and pick each close's joker slots the same way.
#pragma once
#include "dvc_device.cuh"

namespace dvc {

constexpr uint32_t kDetMaxCells = 32768;  // table capacity for 3-4 players
constexpr uint32_t kDetMaxCells2p = 2048;  // two players: (m+1)(gap+1)(J+1) <= 25*25*3

struct DetPlan {
    uint8_t nq, m, J0, obs;
    uint8_t q[3];
    uint8_t nanch[3];
    uint8_t u[24];
    uint8_t jok[2];
    uint8_t gapsz[3][25];
    uint8_t G[3][25];
    uint8_t seqlen[3];
    uint8_t tpl[3][26];  // face-up slot: tile id; face-down slot: 0x80 | gap
    uint8_t cross[26];   // seats (bit k) with an anchor between unknown tiles i and i + 1 (i < m)
    uint32_t rads[26];   // gap slots that can be open at layer i, plus one, of the three seats (8 bits each)
    uint32_t off[26];    // first cell of layer i (i = 0..m), off[m+1] = cells
    uint32_t cells;
    uint32_t ok;         // 1 if the table fits
    unsigned long long total;
};

// The rows of a state laid out one tile per lane (lanes 0..25): the seat that
// holds tile `lane` (4: nobody) and the tile's place in that seat's row.
struct Rows {
    uint32_t owner, pos;
    __device__ __forceinline__ Rows(const G& g) {
        const uint32_t lane = threadIdx.x & 31u, bit = lane < 26u ? 1u << lane : 0u;
        uint32_t hp = 0u;
        owner = 4u;
        if (g.h0 & bit) { owner = 0u; hp = g.h0; }
        if (g.h1 & bit) { owner = 1u; hp = g.h1; }
        if (g.h2 & bit) { owner = 2u; hp = g.h2; }
        if (g.h3 & bit) { owner = 3u; hp = g.h3; }
        pos = __popc(hp & kNumMask & (bit - 1u));
        if (g.tmask & kJokerMask) {
            if (lane >= 24u) {
                if (owner < 4u) pos = joker_pos(g, hp, lane - 24u);
            } else {
                const uint32_t k = pos;
                if ((hp >> 24) & 1u) pos += g.jg0 <= k;
                if ((hp >> 25) & 1u) pos += g.jg1 <= k;
            }
        }
    }
    // Face-down places of seat q's row.
    __device__ __forceinline__ uint32_t hidden(const G& g, uint32_t q) const {
        const bool in = owner == q && !((g.rev >> (threadIdx.x & 31u)) & 1u) && ((g.alive >> q) & 1u);
        return __reduce_or_sync(0xFFFFFFFFu, in ? 1u << pos : 0u);
    }
};

// Index of (J, r) in layer i.
__device__ __forceinline__ uint32_t det_cell(const DetPlan& pl, uint32_t i, const uint32_t* r, uint32_t J) {
    const uint32_t rd = pl.rads[i];
    return pl.off[i] + ((J * (rd & 255u) + r[0]) * ((rd >> 8) & 255u) + r[1]) * (rd >> 16) + r[2];
}

// Ways to put o jokers into a gap of c slots, choosing from J distinct jokers.
__device__ __forceinline__ unsigned long long joker_ways(uint32_t c, uint32_t o, uint32_t J) {
    if (o == 0) return 1ull;
    if (o > J || o > c) return 0ull;
    if (o == 1) return (unsigned long long)c * J;
    return (unsigned long long)(c * (c - 1u) / 2u) * 2ull;  // o == 2, J == 2
}

// Pass from layer i to i+1 (i = -1: from the start to layer 0).  Returns the
// product of the close factors (0: no completion) and updates r, J.
__device__ __forceinline__ unsigned long long det_pass(const DetPlan& pl, int i, uint32_t* r, uint32_t& J) {
    unsigned long long mult = 1ull;
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) {
        if (k >= pl.nq) continue;
        const int from = i < 0 ? -1 : (int)pl.G[k][i];
        const int to = pl.G[k][i + 1];
        if (to == from) continue;
        for (int gg = from < 0 ? 0 : from; gg < to; ++gg) {
            const uint32_t c = pl.gapsz[k][gg];
            const uint32_t open = gg == from ? r[k] : c;
            const unsigned long long f = joker_ways(c, open, J);
            if (!f) return 0ull;
            J -= open;
            mult *= f;
        }
        r[k] = pl.gapsz[k][to];
    }
    return mult;
}

__device__ __forceinline__ unsigned long long det_finish(const DetPlan& pl, const uint32_t* r, uint32_t J) {
    unsigned long long mult = 1ull;
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) {
        if (k >= pl.nq) continue;
        const unsigned long long f = joker_ways(pl.gapsz[k][pl.nanch[k]], r[k], J);
        if (!f) return 0ull;
        J -= r[k];
        mult *= f;
    }
    return mult;
}

// Build the plan of the view of `obs` (a seat) in state g: one warp, every lane
// with the same arguments; pl in shared or global memory.  Lane t works on
// tile t, then lane i on layer i: a few hundred instructions where one thread
// walking rows and tiles took several thousand.
__device__ __forceinline__ void det_plan(const G& g, uint32_t obs, DetPlan& pl) {
    const uint32_t lane = threadIdx.x & 31u, bit = lane < 26u ? 1u << lane : 0u;
    if (obs >= g.np) obs = g.cur;
    const uint32_t nq = g.np - 1u;
    uint32_t R[3] = {0u, 0u, 0u};  // face-up numbered tiles (anchors) of the opponents
    for (uint32_t e = lane; e < sizeof(DetPlan) / 4u; e += 32u) reinterpret_cast<uint32_t*>(&pl)[e] = 0u;
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) {
        if (k >= nq) continue;
        uint32_t q = obs + 1u + k;
        q = q >= g.np ? q - g.np : q;
        R[k] = g.hand(q) & g.rev & kNumMask;
        if (lane == 0u) {
            pl.q[k] = (uint8_t)q;
            pl.seqlen[k] = (uint8_t)__popc(g.hand(q));
            pl.nanch[k] = (uint8_t)__popc(R[k]);
        }
    }
    const Rows v(g);
    const bool opp = v.owner < 4u && v.owner != obs, up = (g.rev & bit) != 0u;
    const uint32_t k = v.owner > obs ? v.owner - obs - 1u : v.owner + g.np - obs - 1u;
    const uint32_t mine = k == 0u ? R[0] : k == 1u ? R[1] : R[2];
    uint32_t gap = __popc(mine & (bit - 1u));  // anchors left of this tile
#pragma unroll
    for (uint32_t j = 24u; j < 26u; ++j) {  // a joker's: those of its row that stand before it
        const uint32_t po = __shfl_sync(0xFFFFFFFFu, v.pos, j), ow = __shfl_sync(0xFFFFFFFFu, v.owner, j);
        const uint32_t before = __ballot_sync(0xFFFFFFFFu, lane < 24u && up && v.owner == ow && v.pos < po);
        if (lane == j) gap = __popc(before);
    }
    if (opp) pl.tpl[k][v.pos] = (uint8_t)(up ? lane : 0x80u | gap);
    const uint32_t key = opp && !up ? k * 32u + gap : 0xFFu;
    const uint32_t same = __match_any_sync(0xFFFFFFFFu, key);
    if (opp && !up && lane == (uint32_t)__ffs(same) - 1u) pl.gapsz[k][gap] = (uint8_t)__popc(same);
    const uint32_t unk = g.tmask & ~g.hand(obs) & ~g.rev, un = unk & kNumMask, m = __popc(un);
    if (un & bit) {
        const uint32_t i = __popc(un & (bit - 1u));
        pl.u[i] = (uint8_t)lane;
        for (uint32_t a = 0; a < nq; ++a) pl.G[a][i] = (uint8_t)__popc(R[a] & (bit - 1u));
    }
    const uint32_t J0 = __popc(unk >> 24);
    if (lane == 0u) {
        pl.nq = (uint8_t)nq;
        pl.obs = (uint8_t)obs;
        pl.m = (uint8_t)m;
        pl.J0 = (uint8_t)J0;
        uint32_t n = 0u;
        if ((unk >> 24) & 1u) pl.jok[n++] = 24;
        if ((unk >> 25) & 1u) pl.jok[n++] = 25;
        for (uint32_t a = 0; a < nq; ++a) pl.G[a][m] = pl.nanch[a];
    }
    __syncwarp();
    uint32_t rd = 0u, cells = 0u, cross = 0u;
    if (lane <= m) {
        uint32_t r[3] = {1u, 1u, 1u};
        for (uint32_t a = 0; a < nq; ++a) {
            r[a] = pl.gapsz[a][pl.G[a][lane]] + 1u;
            if (lane < m && pl.G[a][lane + 1u] != pl.G[a][lane]) cross |= 1u << a;
        }
        rd = r[0] | r[1] << 8 | r[2] << 16;
        cells = (J0 + 1u) * r[0] * r[1] * r[2];
    }
    uint32_t sum = cells;  // inclusive prefix sum over the layers
#pragma unroll
    for (uint32_t o = 1u; o < 32u; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, sum, o);
        if (lane >= o) sum += x;
    }
    if (lane <= m) {
        pl.rads[lane] = rd;
        pl.off[lane] = sum - cells;
        if (lane < m) pl.cross[lane] = (uint8_t)cross;
    }
    if (lane == m) {
        if (m + 1u < 26u) pl.off[m + 1u] = sum;
        pl.cells = sum;
        pl.ok = sum <= kDetMaxCells ? 1u : 0u;
        pl.total = 0ull;
    }
    __syncwarp();
}

// Weight of each destination of unknown tile i (the pool, then the opponents)
// from gap slots r and J unplaced jokers: completions it leaves.
__device__ __forceinline__ void det_weights(const DetPlan& pl, const unsigned long long* F, uint32_t i,
                                            const uint32_t* r, uint32_t J, unsigned long long* w) {
    if (!pl.cross[i]) {
        // no anchor before the next tile: no gap closes, and a destination
        // only takes one slot of its gap
        const uint32_t rd = pl.rads[i + 1], s1 = rd >> 16, s0 = ((rd >> 8) & 255u) * s1;
        const uint32_t c = det_cell(pl, i + 1, r, J);
        w[0] = F[c];
        w[1] = r[0] ? F[c - s0] : 0ull;
        w[2] = r[1] ? F[c - s1] : 0ull;
        w[3] = r[2] ? F[c - 1u] : 0ull;
        return;
    }
#pragma unroll
    for (int d = -1; d < 3; ++d) {
        w[d + 1] = 0ull;
        if (d >= (int)pl.nq) continue;
        uint32_t rr[3] = {r[0], r[1], r[2]};
        uint32_t JJ = J;
        if (d >= 0) {
            if (rr[d] == 0) continue;
            rr[d]--;
        }
        const unsigned long long f = det_pass(pl, (int)i, rr, JJ);
        if (f) w[d + 1] = f * F[det_cell(pl, i + 1, rr, JJ)];
    }
}

// Fill the counting table F (pl.cells entries) for layers m down to 0, cells
// of one layer split over `nthr` cooperating threads (thread `tid`); `sync`
// must be a barrier over those threads.  Sets pl.total (by thread 0).
template <typename Sync>
__device__ void det_fill(DetPlan& pl, unsigned long long* F, uint32_t tid, uint32_t nthr, Sync sync) {
    for (int i = pl.m; i >= 0; --i) {
        const uint32_t rd = pl.rads[i], r0 = rd & 255u, r1 = (rd >> 8) & 255u, r2 = rd >> 16;
        const uint32_t ncell = (pl.J0 + 1u) * r0 * r1 * r2;
        for (uint32_t c = tid; c < ncell; c += nthr) {
            uint32_t rem = c;
            uint32_t r[3];
            r[2] = rem % r2;
            rem /= r2;
            r[1] = rem % r1;
            rem /= r1;
            r[0] = rem % r0;
            const uint32_t J = rem / r0;
            unsigned long long v = 0ull;
            if (i == pl.m) {
                v = det_finish(pl, r, J);
            } else {
                unsigned long long w[4];
                det_weights(pl, F, (uint32_t)i, r, J, w);
                v = w[0] + w[1] + w[2] + w[3];
            }
            F[pl.off[i] + c] = v;
        }
        sync();
    }
    if (tid == 0) {
        uint32_t r[3] = {0, 0, 0};
        uint32_t J = pl.J0;
        const unsigned long long f = det_pass(pl, -1, r, J);
        pl.total = f ? f * F[det_cell(pl, 0, r, J)] : 0ull;
    }
    sync();
}

// Joker slots chosen while sampling: per opponent, per gap-local slot.
struct JokerPick {
    uint8_t n;
    uint8_t k[2], gap[2], local[2], id[2];
};

// Choose which open slots of a closing gap hold jokers, and which jokers.
__device__ __forceinline__ void det_place(uint32_t k, uint32_t gap, uint32_t c, uint32_t open, uint32_t& J,
                                          uint32_t* jleft, Rng& rng, JokerPick& jp) {
    const unsigned long long opts = joker_ways(c, open, J);
    if (opts == 0ull || open > 2u || jp.n + open > 2u) return;  // only for a view with no completion
    const unsigned long long z = pick64(rng.next64(), opts);
    const unsigned long long perms = open == 1 ? J : 2ull;
    const unsigned long long posidx = z / perms, perm = z % perms;
    uint32_t pos0 = 0, pos1 = 0;
    if (open == 1) {
        pos0 = (uint32_t)posidx;
    } else {
        unsigned long long left = posidx;
        for (uint32_t a = 0; a < c; ++a) {
            const unsigned long long cnt = c - 1u - a;
            if (left < cnt) {
                pos0 = a;
                pos1 = a + 1u + (uint32_t)left;
                break;
            }
            left -= cnt;
        }
    }
    uint32_t id0, id1 = 0;
    if (open == 1) {
        id0 = jleft[perm];
    } else {
        id0 = jleft[perm == 0 ? 0 : 1];
        id1 = jleft[perm == 0 ? 1 : 0];
    }
    jp.k[jp.n] = (uint8_t)k;
    jp.gap[jp.n] = (uint8_t)gap;
    jp.local[jp.n] = (uint8_t)pos0;
    jp.id[jp.n] = (uint8_t)id0;
    jp.n++;
    if (open == 2) {
        jp.k[jp.n] = (uint8_t)k;
        jp.gap[jp.n] = (uint8_t)gap;
        jp.local[jp.n] = (uint8_t)pos1;
        jp.id[jp.n] = (uint8_t)id1;
        jp.n++;
    }
    // drop the chosen jokers from the ascending list of unplaced ones
    uint32_t keep[2], nk = 0;
    for (uint32_t a = 0; a < J; ++a) {
        const bool used = jleft[a] == id0 || (open == 2 && jleft[a] == id1);
        if (!used) keep[nk++] = jleft[a];
    }
    for (uint32_t a = 0; a < nk; ++a) jleft[a] = keep[a];
    J = nk;
}

// det_pass with joker placement on each close.
__device__ __forceinline__ void det_pass_sample(const DetPlan& pl, int i, uint32_t* r, uint32_t& J, uint32_t* jleft,
                                                Rng& rng, JokerPick& jp) {
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) {
        if (k >= pl.nq) continue;
        const int from = i < 0 ? -1 : (int)pl.G[k][i];
        const int to = pl.G[k][i + 1];
        if (to == from) continue;
        for (int gg = from < 0 ? 0 : from; gg < to; ++gg) {
            const uint32_t c = pl.gapsz[k][gg];
            const uint32_t open = gg == from ? r[k] : c;
            if (open) det_place(k, gg, c, open, J, jleft, rng, jp);
        }
        r[k] = pl.gapsz[k][to];
    }
}

// Sample one determinization of root g (whose view pl describes) into out.
__device__ __forceinline__ void det_sample(const DetPlan& pl, const unsigned long long* F, const G& g, Rng& rng,
                                           G& out) {
    if (!pl.ok || pl.total == 0ull) {  // no consistent deal: leave the state as it is
        out = g;
        return;
    }
    uint32_t r[3] = {0, 0, 0};
    uint32_t J = pl.J0;
    uint32_t jleft[2] = {pl.jok[0], pl.jok[1]};
    JokerPick jp;
    jp.n = 0;
    uint32_t got[3] = {0, 0, 0};  // numbered tiles dealt to each opponent (bitmask)
    det_pass_sample(pl, -1, r, J, jleft, rng, jp);
    for (uint32_t i = 0; i < pl.m; ++i) {
        unsigned long long w[4];
        det_weights(pl, F, i, r, J, w);
        unsigned long long x = pick64(rng.next64(), w[0] + w[1] + w[2] + w[3]);
        const uint32_t bit = 1u << pl.u[i];
        bool open = x >= w[0];  // not the pool
        x -= w[0];
#pragma unroll
        for (uint32_t k = 0; k < 3u; ++k) {
            const bool here = open && x < w[k + 1];
            if (here) {
                got[k] |= bit;
                r[k]--;
            }
            open = open && !here;
            x -= w[k + 1];
        }
        if (pl.cross[i]) det_pass_sample(pl, (int)i, r, J, jleft, rng, jp);
    }
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) {
        if (k >= pl.nq || !r[k]) continue;
        const uint32_t gg = pl.nanch[k];
        det_place(k, gg, pl.gapsz[k][gg], r[k], J, jleft, rng, jp);
    }
    // Rebuild the opponents' hands: face-up tiles, the numbered tiles dealt to
    // them, and the jokers placed; then the jokers' places.
    out = g;
    uint32_t jown[2] = {0xFFu, 0xFFu}, jseq[2] = {0u, 0u};  // owner and place in its row
#pragma unroll
    for (uint32_t j = 0; j < 2u; ++j) {
        const uint32_t bit = 1u << (24u + j);
        if (!(g.tmask & bit)) continue;
#pragma unroll
        for (uint32_t p = 0; p < 4u; ++p)  // the observer's jokers and face-up ones stay where they are
            if (p < g.np && (g.hand(p) & bit) && (p == pl.obs || (g.rev & bit))) {
                jown[j] = p;
                jseq[j] = joker_pos(g, g.hand(p), j);
            }
    }
    uint32_t joker_bits[3] = {0u, 0u, 0u};
    for (uint32_t e = 0; e < jp.n; ++e) {  // a joker placed in the local-th face-down slot of a gap
        uint32_t left = jp.local[e], s = 0u;
        const uint32_t k = jp.k[e], want = 0x80u | jp.gap[e];
        for (; s < pl.seqlen[k]; ++s)
            if (pl.tpl[k][s] == want && left-- == 0u) break;
        const uint32_t j = jp.id[e] - 24u;
        if (j == 0u) { jown[0] = pl.q[k]; jseq[0] = s; }
        else { jown[1] = pl.q[k]; jseq[1] = s; }
#pragma unroll
        for (uint32_t a = 0; a < 3u; ++a)
            if (a == k) joker_bits[a] |= 1u << jp.id[e];
    }
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) {
        if (k >= pl.nq) continue;
        const uint32_t q = pl.q[k];
        const uint32_t hand = (g.hand(q) & g.rev) | got[k] | joker_bits[k];
        if (q == 0) out.h0 = hand;
        if (q == 1) out.h1 = hand;
        if (q == 2) out.h2 = hand;
        if (q == 3) out.h3 = hand;
    }
    // a joker's gap: the numbered tiles before it, its place less the other joker if that comes first
    const bool together = jown[0] != 0xFFu && jown[0] == jown[1];
    const uint32_t g0 = jseq[0] - (together && jseq[1] < jseq[0] ? 1u : 0u);
    const uint32_t g1 = jseq[1] - (together && jseq[0] < jseq[1] ? 1u : 0u);
    out.jg0 = jown[0] == 0xFFu ? 0u : g0;
    out.jg1 = jown[1] == 0xFFu ? 0u : g1;
    out.jflag = together && g0 == g1 && jseq[1] < jseq[0] ? 1u : 0u;
}

}  // namespace dvc
