// dvc_tree.cuh -- device-resident UCT trees and one search iteration
// (Sec. II-B: select, expand, simulate, backpropagate; Sec. III-A: node =
// guess (slot, identity), determinized root per simulation, no extra guess in
// the tree, expansion depth limit).
//
// Arena layout, per tree: a slice of 16-byte node slots.  Slot 0 is the root.
// The children of a node live in blocks of consecutive slots -- the root's
// first block is sized to its legal-guess count (fixed for the whole search),
// other nodes' blocks grow 4, 8, 16, 32, 32, ... -- so a warp reads a block
// with one coalesced load.  Block k >= 1 of a node is recorded in `link` at
// the slot of the node's child k - 1: the first four links stand side by side
// at the first block, so a warp knows the places of up to 92 children after
// one load instead of following a chain of one link per block.  With blocks no
// larger than four times the children they hold, root block + 4 * budget slots
// always suffice.
//
// The walk is a chain of dependent steps of one warp, so what bounds it is
// latency: loads one after another, the instructions between them, and their
// fetch.  A level costs one load of the children (with their UCB1 terms, and
// all that the next level needs of them: child block, child count, exploration
// term) and, with more than four children, one of the links before it, both
// issued ahead of the work that does not need them.  The determinized rows are
// laid out one tile per lane, so slots, targets and draws are ballots and
// warp-wide reductions instead of bit selects through tables.
//
// Vanilla MCTS-dvc (Sec. III-A): the root's children are plausible-number
// sets, one per distinct assignment of the tiles the observer cannot see, and
// the guess tree of each hangs below it.  The root's single child block then
// holds `budget` slots (at most one set per iteration), and a per-tree open-
// addressing table maps an assignment to its set node.
#pragma once
#include "dvc_det.cuh"

namespace dvc {

struct __align__(16) Node {
    int32_t visits;
    int32_t wins;
    int32_t child;  // slot of the first child block, -1 if none
    uint32_t meta;  // action code (bits 0-11) | number of children (bits 12-23)
};

struct TreeMeta {
    long long node_off;   // first slot of this tree in the arena
    long long table_off;  // first cell of its determinization table
    int32_t cap;          // slots
    int32_t budget;       // iterations allowed in total
    int32_t done;         // iterations done
    int32_t next_free;    // next unused slot
    int32_t root_legal;   // legal guesses at the root
    uint32_t tree_id;     // stream key
    int32_t failed;       // arena exhausted, or view too large to determinize
    int32_t used;         // nodes in the tree
    long long set_off;    // vanilla: first cell of its plausible-set table
    int32_t set_cells;    // vanilla: cells of that table (2 * budget); 0 otherwise
    int32_t pad_;
};

// A tree's plausible-set table: open addressing with linear probing, cell i
// holds an assignment's key and the slot of its set node (-1: empty).  At
// most `budget` keys in 2 * budget cells, so an empty cell always ends a probe.
struct SetTable {
    uint4* key;
    int32_t* slot;
    uint32_t cells;  // 0: not a vanilla tree
};

// Key of a determinization's plausible-number set as seen by seat obs: the
// other seats' hands in seat order (three words, unused seats zero), then the
// joker gaps and the white-first flag, which place the jokers in the rows.
__device__ __forceinline__ uint4 set_key(const G& g, uint32_t obs) {
    uint32_t h[3] = {0u, 0u, 0u};
    uint32_t k = 0;
#pragma unroll
    for (uint32_t p = 0; p < 4; ++p)
        if (p < g.np && p != obs) h[k++] = g.hand(p);
    return make_uint4(h[0], h[1], h[2], g.jg0 | (g.jg1 << 8) | ((g.jflag & 1u) << 16));
}

// First probe cell of a key: a 64-bit mix (xor-shift-multiply rounds) of its
// words, scaled to the cell count by a multiply-high.
__device__ __forceinline__ uint32_t set_home(const uint4& k, uint32_t cells) {
    unsigned long long a = ((unsigned long long)k.y << 32 | k.x) ^ (((unsigned long long)k.w << 32 | k.z) * 0x9E3779B97F4A7C15ull);
    a ^= a >> 31;
    a *= 0xD6E8FEB86659FD93ull;
    a ^= a >> 32;
    return (uint32_t)(((unsigned long long)(uint32_t)a * cells) >> 32);
}

// Warp-parallel probe: lane j looks at the j-th cell of each round of 32; the
// first cell in probe order that is empty or holds the key ends the probe.
// Returns the set node's slot (-1 if absent) and the cell it sits in, or
// would be inserted into.  Lane-uniform.
__device__ __forceinline__ int32_t set_find(const SetTable& st, const uint4& k, uint32_t& cell) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t home = set_home(k, st.cells);
    for (uint32_t r = 0; r < st.cells; r += 32u) {
        uint32_t c = home + r + lane;
        c = c % st.cells;
        const int32_t s = st.slot[c];
        bool stop = s < 0;
        if (!stop) {
            const uint4 q = st.key[c];
            stop = q.x == k.x && q.y == k.y && q.z == k.z && q.w == k.w;
        }
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, stop);
        if (bal) {
            const uint32_t L = __ffs(bal) - 1u;
            cell = __shfl_sync(0xFFFFFFFFu, c, L);
            return __shfl_sync(0xFFFFFFFFu, s, L);
        }
    }
    cell = 0xFFFFFFFFu;  // unreachable while keys <= cells / 2
    return -1;
}

// Slots reserved for the root's child block: its legal-guess count is
// (face-down slots of opponents) x (unknown identities) <= 25 * 25.
constexpr int32_t kRootReserve = 640;

struct SearchParams {
    uint64_t seed;
    float c_uct;  // UCB1 exploration constant, rounded to float
    int32_t d_max;
    int32_t playouts;
    uint32_t cont_thr;
    int32_t policy;         // playout guesses: 0 uniform, 1 ordering-aware
    int32_t tree_continue;  // 1: a correct in-tree guess keeps the turn (Fig. 2a)
    const float2* terms;    // visit_terms of k * playouts visits, k = 1 .. n_terms
    int32_t n_terms;
    float inv_playouts;
};

// Child c of a node other than the root stands in block block_of(c) at
// block_off(c); block k holds block_size(k) slots.
__device__ __forceinline__ uint32_t block_of(uint32_t c) {
    return c < 4u ? 0u : c < 12u ? 1u : c < 28u ? 2u : 3u + ((c - 28u) >> 5);
}
__device__ __forceinline__ uint32_t block_off(uint32_t c) {
    return c < 4u ? c : c < 12u ? c - 4u : c < 28u ? c - 12u : (c - 28u) & 31u;
}
__device__ __forceinline__ uint32_t block_size(uint32_t k) { return k >= 3u ? 32u : 4u << k; }

// Slot of child c: block k >= 1 is linked from child k - 1, so block_of(k - 1)
// < k and the chain of blocks that leads to c is short (at most four for 4,095
// children).  single: the root, whose children are one block.
__device__ __forceinline__ int32_t child_slot(const int32_t* link, int32_t blk0, uint32_t c, bool single) {
    if (single) return blk0 + (int32_t)c;
    uint32_t at[4];
    int n = 0;
    uint32_t k = block_of(c);
    while (k > 0u && n < 4) {
        at[n++] = k - 1u;
        k = block_of(k - 1u);
    }
    int32_t blk = blk0;
    for (int i = n - 1; i >= 0; --i) blk = link[blk + (int32_t)block_off(at[i])];
    return blk + (int32_t)block_off(c);
}

// A node's blocks by lane: lane k holds block k's first slot, for as many of
// the first 32 blocks as nchild children need (they hold 956 children).  All
// lanes call.
constexpr uint32_t kDirChildren = 28u + 29u * 32u;
__device__ __forceinline__ int32_t block_dir(const int32_t* link, int32_t blk0, uint32_t nchild) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t last = block_of(nchild - 1u);  // callers have nchild > 0
    int32_t dir = blk0;
    if (lane >= 1u && lane <= min(last, 4u)) dir = link[blk0 + (int32_t)lane - 1];
    if (last > 4u) {  // blocks 5-12 are linked from block 1, 13-28 from block 2, the rest from block 3
        const int32_t b1 = __shfl_sync(0xFFFFFFFFu, dir, 1), b2 = __shfl_sync(0xFFFFFFFFu, dir, 2);
        const int32_t b3 = __shfl_sync(0xFFFFFFFFu, dir, 3);
        const int32_t from = lane < 13u ? b1 - 5 : lane < 29u ? b2 - 13 : b3 - 29;
        if (lane > 4u && lane <= last) dir = link[from + (int32_t)lane];
    }
    return dir;
}

// The words of an iteration's tree stream (tag 3), the same on every lane.
// b holds the block the next word is in; block 0 is given, as sampled ahead or by
// block(0).
struct TreeWords {
    uint32_t k0, k1, i, tw;
    uint4 b;
    uint32_t used;

    __device__ __forceinline__ uint4 block(uint32_t blk) const {
        uint32_t x0 = blk, x1 = 0u, x2 = i, x3 = tw;
        philox10(x0, x1, x2, x3, k0, k1);
        return make_uint4(x0, x1, x2, x3);
    }
    __device__ __forceinline__ void open(uint64_t seed, uint32_t tree, uint32_t it) {
        k0 = (uint32_t)seed;
        k1 = tree;
        i = it;
        tw = kTagTree + 16u * (uint32_t)(seed >> 32);
        used = 0u;
    }
    __device__ __forceinline__ uint32_t next() {
        const uint32_t n = used++, k = n & 3u;
        if (k == 0u && n) b = block(n >> 2);
        return k == 0u ? b.x : k == 1u ? b.y : k == 2u ? b.z : b.w;
    }
};

// tree_apply (dvc_device.cuh) by a whole warp: the same transition and words,
// the state the same on every lane before and after.
__device__ __forceinline__ void warp_apply(G& g, const Rows& v, uint32_t code, TreeWords& tw, bool cont) {
    const uint32_t lane = threadIdx.x & 31u, cur = g.cur;
    const bool was_stop = code == kStop;
    if (!was_stop) {
        const uint32_t q = code >> 10, sl = (code >> 5) & 31u, x = code & 31u;
        const unsigned at = __ballot_sync(0xFFFFFFFFu, v.owner == q && v.pos == sl);
        const uint32_t target = at ? (uint32_t)__ffs(at) - 1u : 0u;
        const bool hit = x == target;
        uint32_t tb = 1u << target;
        if (!hit) {
            uint32_t t = g.drawn;
            if (t == kNone) {  // the leftmost face-down tile
                const bool mine = v.owner == cur && !((g.rev >> lane) & 1u);
                t = __reduce_min_sync(0xFFFFFFFFu, mine ? v.pos << 5 | lane : 0xFFFFu) & 31u;
            }
            tb = 1u << t;
        }
        g.rev |= tb;
        const uint32_t seat = hit ? q : cur;
        if (!(g.hand(seat) & ~g.rev)) g.alive &= ~(1u << seat);
        g.mstop = 0u;
        if (__popc(g.alive) == 1) {
            g.winner = hit ? cur : (uint32_t)__ffs(g.alive) - 1u;
            return;
        }
        if (cont && hit) {
            g.mstop = 1u;
            return;
        }
    }
    g.mstop = 0u;
    g.cur = next_alive(g.alive, cur, g.np);
    const uint32_t pool = g.pool();
    if (!pool) {
        g.drawn = kNone;
        return;
    }
    const uint32_t n = __umulhi(tw.next(), __popc(pool));
    const bool here = ((pool >> lane) & 1u) && (uint32_t)__popc(pool & ((1u << lane) - 1u)) == n;
    const uint32_t t = (uint32_t)__ffs(__ballot_sync(0xFFFFFFFFu, here)) - 1u;
    insert_gaps(g, g.hand(g.cur), t, tw);
    g.add(g.cur, 1u << t);
    g.drawn = t;
}

// What a descent produced: a node to expand (found = 1, action act) or none
// (found = 0), and the state to score: after the new action, or at the node.
struct Descent {
    G s;
    int32_t node;     // slot reached
    int32_t found;    // 1: expand `act` below `node`
    uint32_t act;
    uint32_t who;     // the seat that makes it
    uint32_t meta;    // `node`'s action and number of children (Node::meta)
    int32_t blk;      // first child block of `node`, -1 if none
    int32_t dir;      // its blocks, by lane (block_dir); differs between lanes
    int32_t np;       // path length
    uint32_t set_cell;  // vanilla, act == kSet: the table cell for the new set
    uint4 set_key;      // vanilla, act == kSet: its key
};

// A node of the walk: slot, first child block, Node::meta, c * sqrt(ln visits).
struct WalkNode {
    int32_t slot, blk;
    uint32_t meta;
    float csl;
};

// Warp-cooperative descent from the root for one iteration.  All 32 lanes
// of the calling warp enter with the same arguments and leave with the same
// Descent; lane 0 records the path in path[] / mover[] (shared or global).
// at: the root's node.  E is a 4 x 26 word scratch (shared memory) for
// expanded-identity masks.  tw: the iteration's tree stream, opened.
// ucb[slot] = (wins/n, 1/sqrt(n)) and csl[slot] = c * sqrt(ln n) are the
// node's UCB1 terms, refreshed whenever its counts change (backprop), so a
// selection scan costs one multiply-add per child.  They are the same IEEE
// values a scan would compute from the counts.
// VANILLA: st is the tree's plausible-set table.  The determinization's set
// node is the first step below the root; a set not seen before is this
// iteration's expansion (act = kSet) and its leaf is the determinized root.
template <bool VANILLA>
__device__ __forceinline__ void descend(const G& det, uint32_t obs, WalkNode at, const Node* nodes,
                                        const int32_t* link, const float2* ucb, const float* csl_of,
                                        const SearchParams& sp, TreeWords& tw, int32_t* path, uint8_t* mover,
                                        uint32_t* E, Descent& d,
                                        const SetTable& st = SetTable{nullptr, nullptr, 0u}) {
    const uint32_t lane = threadIdx.x & 31u;
    d.s = det;
    d.found = 0;
    d.np = 1;
    if (lane == 0) {
        path[0] = 0;
        mover[0] = (uint8_t)obs;
    }
    uint32_t depth = 0;
    if (VANILLA && st.cells) {
        const uint4 key = set_key(d.s, obs);
        uint32_t cell;
        const int32_t slot = set_find(st, key, cell);
        if (slot < 0) {
            // a new set: appended to the root's single child block
            d.found = 1;
            d.act = kSet;
            d.who = d.s.cur;
            d.set_cell = cell;
            d.set_key = key;
            d.node = 0;
            d.meta = at.meta;
            d.blk = d.dir = at.blk;
            return;
        }
        if (lane == 0) {
            path[1] = slot;
            mover[1] = (uint8_t)obs;
        }
        d.np = 2;
        const Node sn = nodes[slot];
        at.slot = slot;
        at.blk = sn.child;
        at.meta = sn.meta;
        at.csl = csl_of[slot];
    }
    while (d.s.winner == kNone && depth < (uint32_t)sp.d_max) {
        const uint32_t cur = d.s.cur, np = d.s.np;
        const uint32_t nchild = at.meta >> 12;
        const bool wide = at.slot != 0 && nchild > 0u;
        const int32_t dir = wide ? block_dir(link, at.blk, nchild) : at.blk;
        // the legal actions of this determinization: STOP when allowed, and
        // face-down places of the opponents x identities the mover cannot see
        const uint32_t U = d.s.tmask & ~d.s.hand(cur) & ~d.s.rev;
        uint32_t q1 = cur + 1u, q2 = cur + 2u, q3 = cur + 3u;
        q1 = q1 >= np ? q1 - np : q1;
        q2 = q2 >= np ? q2 - np : q2;
        q3 = q3 >= np ? q3 - np : q3;
        const Rows rows(d.s);
        const uint32_t m1 = rows.hidden(d.s, q1);
        uint32_t m2 = 0u, m3 = 0u;
        if (np > 2u) m2 = rows.hidden(d.s, q2);
        if (np > 3u) m3 = rows.hidden(d.s, q3);
        const uint32_t legal =
            (uint32_t)(__popc(m1) + __popc(m2) + __popc(m3)) * (uint32_t)__popc(U) + (d.s.mstop ? 1u : 0u);
        if (legal == 0u) break;  // not in a running game
        // slot of child c (a lane's own; every lane of the warp calls)
        auto place = [&](uint32_t c) -> int32_t {
            if (!wide) return at.blk + (int32_t)c;
            const int32_t b = __shfl_sync(0xFFFFFFFFu, dir, block_of(c) & 31u);
            if (c >= kDirChildren && c < nchild) return child_slot(link, at.blk, c, false);
            return b + (int32_t)block_off(c);
        };
        uint32_t left = legal;  // legal actions without a child
        uint32_t act = kStop;
        float best_sc = 0.0f;
        uint32_t best_rank = 0xFFFFFFFFu, best_meta = 0u;
        int32_t best_slot = -1, best_blk = -1;
        float best_csl = 0.0f;
        if (nchild >= legal) {
            // perhaps every legal action has its child: score the legal ones,
            // two chunks of 32 children in flight
            uint32_t seen = 0u;
            for (uint32_t c0 = 0; c0 < nchild; c0 += 64u) {
                int2 ch[2];  // first child block, meta
                float2 u[2];
                float cs[2];
                int32_t sl[2];
#pragma unroll
                for (uint32_t h = 0; h < 2u; ++h) {
                    const uint32_t c = c0 + 32u * h + lane;
                    sl[h] = -1;
                    if (c0 + 32u * h < nchild) {
                        const int32_t s = place(c);
                        if (c < nchild) {
                            sl[h] = s;
                            ch[h] = reinterpret_cast<const int2*>(nodes + s)[1];
                            u[h] = ucb[s];  // set by the child's first backprop
                            cs[h] = csl_of[s];
                        }
                    }
                }
#pragma unroll
                for (uint32_t h = 0; h < 2u; ++h) {
                    if (sl[h] < 0) continue;
                    const uint32_t code = (uint32_t)ch[h].y & 0xFFFu;
                    const uint32_t q = code >> 10, x = code & 31u;
                    const uint32_t off = q > cur ? q - cur - 1u : q + np - cur - 1u;
                    const uint32_t m = off == 0u ? m1 : off == 1u ? m2 : m3;
                    bool ok = ((m >> ((code >> 5) & 31u)) & 1u) && ((U >> x) & 1u) && q != cur;
                    uint32_t rank = 1u + (off << 10 | (code & 1023u));  // canonical order, STOP first
                    if (code == kStop) {
                        ok = d.s.mstop != 0u;
                        rank = 0u;
                    }
                    if (!ok) continue;
                    ++seen;
                    const float sc = __fadd_rn(u[h].x, __fmul_rn(at.csl, u[h].y));
                    if (best_slot < 0 || sc > best_sc || (sc == best_sc && rank < best_rank)) {
                        best_sc = sc;
                        best_rank = rank;
                        best_slot = sl[h];
                        best_meta = (uint32_t)ch[h].y;
                        best_blk = ch[h].x;
                        best_csl = cs[h];
                    }
                }
            }
            left = legal - __reduce_add_sync(0xFFFFFFFFu, seen);
        }
        if (left) {
            // the first legal action without a child, in canonical order
            bool stop_child = false;
            if (nchild) {
                for (uint32_t e = lane; e < 104u; e += 32u) E[e] = 0u;
                __syncwarp();
                for (uint32_t c0 = 0; c0 < nchild; c0 += 32u) {
                    const uint32_t c = c0 + lane;
                    const int32_t s = place(c);
                    if (c >= nchild) continue;
                    const uint32_t code = nodes[s].meta & 0xFFFu;
                    const uint32_t sl = (code >> 5) & 31u;
                    if (code == kStop) stop_child = true;
                    else if (sl < 26u) atomicOr(&E[(code >> 10) * 26u + sl], 1u << (code & 31u));
                }
                __syncwarp();
            }
            if (!d.s.mstop || __any_sync(0xFFFFFFFFu, stop_child)) {
                for (uint32_t off = 0; off < 3u; ++off) {
                    const uint32_t m = off == 0u ? m1 : off == 1u ? m2 : m3;
                    const uint32_t q = off == 0u ? q1 : off == 1u ? q2 : q3;
                    uint32_t avail = (m >> lane) & 1u ? U : 0u;
                    if (avail && nchild) avail &= ~E[q * 26u + lane];
                    const unsigned bal = __ballot_sync(0xFFFFFFFFu, avail != 0u);
                    if (bal) {
                        const uint32_t sl = (uint32_t)__ffs(bal) - 1u;
                        const uint32_t av = __shfl_sync(0xFFFFFFFFu, avail, sl);
                        act = (q << 10) | (sl << 5) | ((uint32_t)__ffs(av) - 1u);
                        break;
                    }
                }
            }
            __syncwarp();  // E is read before a later walk of this warp clears it
            d.found = 1;
            d.who = cur;
            d.act = act;
            d.node = at.slot;
            d.meta = at.meta;
            d.blk = at.blk;
            d.dir = dir;
        } else {
            // UCB1 argmax over lanes: highest score (scores are not negative,
            // so their bits order like them), then lowest canonical rank
            const uint32_t key = best_slot < 0 ? 0u : __float_as_uint(best_sc) + 1u;
            const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, key);
            const uint32_t win =
                __reduce_min_sync(0xFFFFFFFFu, key == top ? best_rank << 5 | lane : 0xFFFFFFFFu) & 31u;
            const uint32_t meta = __shfl_sync(0xFFFFFFFFu, best_meta, win);
            at.slot = __shfl_sync(0xFFFFFFFFu, best_slot, win);
            at.blk = __shfl_sync(0xFFFFFFFFu, best_blk, win);
            at.csl = __shfl_sync(0xFFFFFFFFu, best_csl, win);
            at.meta = meta;
            act = meta & 0xFFFu;
            if (lane == 0) {
                path[d.np] = at.slot;
                mover[d.np] = (uint8_t)cur;
            }
            d.np++;
            ++depth;
        }
        warp_apply(d.s, rows, act, tw, sp.tree_continue != 0);
        if (d.found) break;
    }
}

// Create the child found by descend() (a new plausible set is entered in the
// tree's set table).  Lane-uniform; lane 0 writes memory.  next_free is the
// tree's allocator (uniform register copy).  Returns false if the arena is
// exhausted.
template <bool VANILLA>
__device__ __forceinline__ bool expand_child(Descent& d, Node* nodes, int32_t* link, int32_t* created,
                                             const TreeMeta& tm, int32_t& next_free, int32_t& used, uint32_t it,
                                             int32_t* path, uint8_t* mover,
                                             const SetTable& st = SetTable{nullptr, nullptr, 0u}) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t c = d.meta >> 12;
    const bool single = d.node == 0;  // the root's one block holds every child it can have
    // slot of a child i >= 1 of a node other than the root, from the walk's directory
    auto place = [&](uint32_t i) -> int32_t {
        if (c >= kDirChildren) return child_slot(link, d.blk, i, false);
        return __shfl_sync(0xFFFFFFFFu, d.dir, block_of(i)) + (int32_t)block_off(i);
    };
    int32_t slot;
    if (c == 0u || (!single && block_off(c) == 0u)) {
        // a new child block: first block of this node, or the last one is full
        const int32_t size = single ? (tm.root_legal > 0 ? tm.root_legal : 1) : (int32_t)block_size(block_of(c));
        if (next_free + size > tm.cap) return false;
        slot = next_free;
        next_free += size;
        const int32_t from = c ? place(block_of(c) - 1u) : 0;  // where the block is linked
        for (int32_t e = (int32_t)lane; e < size; e += 32) created[slot + e] = -1;  // slots not yet nodes
        if (lane == 0) {
            if (c == 0u) nodes[d.node].child = slot;
            else link[from] = slot;
        }
        __syncwarp();
    } else {
        if (single && (int32_t)c >= tm.root_legal) return false;  // unreachable: the block holds every child
        slot = single ? d.blk + (int32_t)c : place(c);
    }
    if (lane == 0) {
        Node n;
        n.visits = 0;
        n.wins = 0;
        n.child = -1;
        n.meta = d.act;
        nodes[slot] = n;
        created[slot] = (int32_t)it;
        nodes[d.node].meta = d.meta + (1u << 12);
        path[d.np] = slot;
        mover[d.np] = (uint8_t)d.who;
        if (VANILLA && d.act == kSet) {
            st.key[d.set_cell] = d.set_key;
            st.slot[d.set_cell] = slot;
        }
    }
    d.np++;
    ++used;
    return true;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// UCB1's terms of a node with v visits, 1 / sqrt(v) and c * sqrt(ln v).
__device__ __forceinline__ float2 visit_terms(float dv, float c_uct) {
    return make_float2(__fdiv_rn(1.0f, __fsqrt_rn(dv)), __fmul_rn(c_uct, __fsqrt_rn(ln_series(dv))));
}

// Backpropagation (Sec. II-B): every node on the path gains `playouts` visits
// and the playouts won by the seat that moved into it.  Visits are multiples of
// `playouts`, so their terms come from the forest's table (sp.terms, entry k
// for k * playouts visits).  One warp issues this step, an instruction every four
// cycles, so what bounds it is their number: with the two square roots, the division
// and the logarithm it took 1,600 cycles of a lone tree's iteration, now 980 (the
// search of 10,000 iterations 94.1 -> 92.4 ms with the list of leaves by ballots and
// the new child's block taken from the walk).
__device__ __forceinline__ void backprop(Node* nodes, float2* ucb, float* csl, const int32_t* path,
                                         const uint8_t* mover, int32_t np, const int32_t* wins,
                                         const SearchParams& sp) {
    const uint32_t lane = threadIdx.x & 31u;
    for (int32_t e = (int32_t)lane; e < np; e += 32) {
        const int32_t slot = path[e];
        Node* n = &nodes[slot];
        const int2 vw = *reinterpret_cast<const int2*>(n);
        const int32_t v = vw.x + sp.playouts;
        const int32_t w = vw.y + wins[mover[e]];
        *reinterpret_cast<int2*>(n) = make_int2(v, w);
        const float dv = __int2float_rn(v);
        // k is within 0.03 of the quotient for every k of the table
        const int32_t k = __float2int_rn(__fmul_rn(dv, sp.inv_playouts));
        float2 t;
        if ((uint32_t)(k - 1) < (uint32_t)sp.n_terms && k * sp.playouts == v) t = sp.terms[k];
        else t = visit_terms(dv, sp.c_uct);
        ucb[slot] = make_float2(__fdiv_rn(__int2float_rn(w), dv), t.x);
        csl[slot] = t.y;
    }
}

}  // namespace dvc
