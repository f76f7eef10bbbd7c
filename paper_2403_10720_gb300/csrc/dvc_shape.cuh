// dvc_shape.cuh -- which engine and launch shape a forest takes by default (host code).
#pragma once
#include <algorithm>
#include <cmath>

namespace dvc {

// Default engine for n trees on `sms` SMs with P playouts per leaf: 1 (fused) or 2
// (pipeline).  What counts is the CTA of the fused engine that holds most, with T =
// ceil(n / sms) trees: while its T P playouts are at most one per thread (512) and it
// has at most two trees per warp (32), its iteration is one walk and one pass of games;
// past that it takes a second pass over playouts, or a second wave of CTAs, and the
// pipeline, which spreads games over all SMs, is ahead.  Time per iteration (us, fused
// / pipeline, two players then four with jokers), the last size on the line and the
// first past it:
//   1 tree       512 playouts 10.5 / 10.8 and 19.2 / 16.8, 768: 15.4 / 10.8 and 29.9 /
//                16.8 (65,536: 920 / 13.9 and 1,971 / 24.2)
//   153 trees    256: 12.1 / 13.7 and 20.0 / 20.2, 300: 16.8 / 14.5 and 29.3 / 21.6
//   457 trees    128: 12.0 / 15.2 and 19.0 / 22.1, 170: 17.7 / 16.2 and 29.6 / 23.8
//   1,217 trees  56: 12.9 / 16.1 and 20.3 / 24.5, 57: 17.0 / 16.2 and 28.3 / 24.5
//   2,281 trees  32: 13.3 / 17.3 and 21.2 / 27.2, 33: 17.3 / 17.4 and 29.9 / 27.7
//   4,700 trees  16: 16.4 / 21.5 and 25.2 / 32.3
// (On the fused side the pipeline is ahead with four players and a few trees, up to 40,
// of 400 to 512 playouts.)
// Ordering-aware games differ most in length, and their pipeline pools a group's in one
// CTA, so that it gains nothing from idle SMs: up to two trees per SM the fused engine
// is ahead whatever the playouts (152 trees x 1,024: 80.9 / 177 and 620 / 1,304; 304 x
// 512: 80.5 / 95.6 and 571 / 632), with three but for a second pass of games (400 trees x
// 170: 41.4 / 57.5 and 288 / 347, x 200: 58.4 / 61.6 and 457 / 381, x 256: 68.1 / 64.7
// and 497 / 406, x 400: 94.6 / 105 and 758 / 745), with four up to one pass (608 trees x
// 128: 40.8 / 51.5 and 286 / 307, x 170: 63.2 / 58.5 and 473 / 377).  Beyond, the step
// waits for a CTA's longest game: the pipeline (one playout, four players: 1,200 trees
// 134 / 134, 2,432 trees 174 / 146).
inline int default_engine(int n, int sms, int P, bool ordered) {
    const int S = std::max(sms, 1);
    const long long T = ((long long)n + S - 1) / S, games = T * P;
    bool fused;
    if (!ordered) fused = T * std::max(P, 16) <= 512;
    else if (T <= 2) fused = true;
    else if (T == 3) fused = games <= 512 || games > 1024;
    else fused = T * std::max(P, 128) <= 512;
    return fused ? 1 : 2;
}

// Default launch shape of an engine for n trees on `sms` SMs with P playouts
// per leaf.  Pipeline: small rollout CTAs of at least two trees, warps enough
// for one playout per thread (4 to 16; the ordering-aware and compacting kernels
// only), and as many chains (up to 24) as give each chain about 1.1 trees per SM,
// so that the tree walks of some chains run beside the playouts of the others.  Fused: every SM holds a CTA, one
// warp per tree up to 16.
inline void default_shape(int n, int sms, int engine, int P, int& T, int& W, int& chains) {
    const int S = std::max(sms, 1);
    if (engine == 2) {
        chains = std::max(1, std::min(24, (int)std::lround(n / (1.12 * S))));
        T = std::max(2, std::min(64, (int)std::ceil(n / (chains * 0.85 * S))));
        W = std::max(4, std::min(16, (T * std::max(P, 1) + 31) / 32));
    } else {
        // a warp per tree, and enough warps for one playout per thread (16 at most)
        T = std::max(1, std::min(32, (n + S - 1) / S));
        W = std::min(16, std::max(T, (T * std::max(P, 1) + 31) / 32));
        chains = 1;
    }
}

// Iterations of one launch of the fused engine: as many as its lanes' 32-bit counts of
// random words hold, each lane playing T P games an iteration shared among 32 W lanes, of
// at most 128 steps of four words.  8.4 million for up to one game a lane (a minute and
// more); a longer step takes several launches.
inline int fused_launch_iterations(int T, int W, int P) {
    const long long lanes = 32LL * W, games = ((long long)T * P + lanes - 1) / lanes;
    return (int)std::max<long long>(1, ((1LL << 32) - 1) / (games * 128 * 4));
}

// Whether the fused engine's two-player playouts take the longer form that suits a warp
// with its scheduler nearly to itself (play_games, ALONE): up to three warps that play
// per scheduler, for `grid` CTAs of T trees and W warps (the builds of up to four warps
// stand on an SM by four, the others alone; warps 0, 4, 8, .. of every CTA share a
// scheduler).  Time per iteration (us, that form / the plain one): a lone tree, 32
// playouts 6.4 / 7.2, 512 (four warps per scheduler) 10.4 / 9.9; 152 trees x 256 (two)
// 8.9 / 9.4; 1,000 trees x 32 (two) 9.3 / 9.8, 2,000 x 32 (four) 13.2 / 12.8; CTAs of four trees and
// four warps, two per SM 9.2 / 9.9, three 11.4 / 11.4, four 13.8 / 12.9.
inline bool play_alone(int grid, int sms, int T, int W, int P) {
    const int S = std::max(sms, 1), ctas = std::min((grid + S - 1) / S, W <= 4 ? 4 : 1);
    const int warps = (int)std::min<long long>(W, ((long long)T * P + 31) / 32);
    return ctas * ((warps + 3) / 4) <= 3;
}

// Chains of value mode.  One chain's launches overlap one another (dvc_chain.cuh), so
// up to 16 trees per SM a second gains nothing (2,432 trees: 33.9 us per iteration
// against 34.7 with two and 35.1 with eight).  Beyond, the walks of one chain fill the
// SMs that the network of another leaves, as long as the tiles of 128 leaves of all
// eight, four SMs each, about fill the chip once (two players / four with jokers, one
// chain against eight): 4,096 trees 38.9 / 40.5 against 37.4 / 39.1, 4,864 53.1 / 55.2
// against 41.5 / 43.7, 5,000 46.9 / 49.1 against 41.7 / 44.1.  Past that (from 5,121
// trees on, six tiles a chain) the network runs layer by layer on the whole chip, and
// fewer, larger batches are better: 5,200 47.2 / 49.1 against 47.8 / 50.0, 6,000 48.4 /
// 50.9 against 49.6 / 52.2, 8,192 54.3 / 57.2 against 65.9 / 69.6.
inline int default_value_chains(int n, int sms) {
    const int S = std::max(sms, 1), tiles = (S + 16) / 32;  // of each of eight chains, to the nearest
    return n <= 16 * S || n > 8 * 128 * tiles ? 1 : 8;
}

}  // namespace dvc
