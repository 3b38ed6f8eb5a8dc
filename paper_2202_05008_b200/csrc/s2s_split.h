// Host arithmetic of the seq2seq kernels' launch (rollout_s2s.cu), without CUDA so that it can be tested anywhere.
#pragma once
#include <cstdint>

namespace evo {

// How the queries of all members come to blocks.  128 units (s2s_items): items of `chunk` queries of a member, `chunks` of them per member, which `places`
// blocks take in turn.  Narrower cells (s2s_split), in n-tiles of 8 queries: chunks of `chunk` n-tiles of a member, `chunks` of them per member, or
// (chunk = 0) a run of the tiles of all members for each of `places` blocks, worked off in pieces of one member.
struct S2sSplit { uint32_t chunk, chunks, places; };

constexpr uint32_t kS2sRunTiles64 = 14, kS2sRunTiles96 = 8;       // most n-tiles of a piece of a run

// 128 units: items of `chunk` queries of a member, `chunks` of them, for a block per SM that takes them in turn.  An item of q queries takes about
// 22 + T (1.36 + 0.0205 q) us for T steps (148 members, 3 digits: 32 queries 46 us, 64 51, 96 60, 128 66), so a population that leaves SMs idle
// with items of 128 takes smaller ones, as far as the rounds of the blocks do not eat up what that saves; where it is less than 3 %
// the items stay large.  `members`: of the whole population, so that shards sum up a member's loss alike.  Roll-outs, items of
// at most 128 and as few as possible / as here, us: 22 x 314, 3 digits 61 / 48; 36 x 128, 3 62 / 45; 48 x 47, 1 32 / 29; 76 x 240, 4 129 / 125; 160 x 250, 3 191 / 192.
inline S2sSplit s2s_items(uint32_t members, uint32_t queries, uint32_t digits, uint32_t sms)
{
    const uint64_t steps = 3u * digits + 2u;
    const uint32_t least = (queries + 127u) / 128u, most = (queries + 15u) / 16u;
    S2sSplit best = { 0u, 0u, sms };
    uint64_t best_time = 0;
    for (uint32_t n = least; n <= most && n <= least + sms; ++n) {
        uint32_t chunk = ((queries + n - 1u) / n + 7u) / 8u * 8u;
        if (chunk > 112u) chunk = 128u;                              // (the instance for these takes no longer for 128)
        const uint32_t chunks = (queries + chunk - 1u) / chunk;
        const uint64_t time = (static_cast<uint64_t>(members) * chunks + sms - 1u) / sms * (1100u + steps * (68u + chunk));       // units of 0.02 us
        if (best.chunks == 0u || time * 100u < best_time * 97u) { best.chunk = chunk; best.chunks = chunks; best_time = time; }
    }
    return best;
}

// Pieces of the run of n-tiles [first, end), `tiles` of them to a member
inline uint32_t s2s_pieces(uint32_t first, uint32_t end, uint32_t tiles, uint32_t most)
{
    const uint32_t a = first / tiles, b = (end - 1u) / tiles;      // first and last member
    if (tiles <= most) return b - a + 1u;
    auto pieces = [&](uint32_t n) { return (n + most - 1u) / most; };
    if (a == b) return pieces(end - first);
    return pieces((a + 1u) * tiles - first) + (b - a - 1u) * pieces(tiles) + pieces(end - b * tiles);
}

// Chunks of up to 64 queries, spread evenly over the fewest chunks; a small population takes smaller ones (down to one tile) until
// there are two blocks for every SM.  More chunks than the SMs hold at once (two blocks of 64 units, one of 96) end in a wave that may be nearly
// empty; runs are even, but every piece costs its weights and the latency of its steps.  In units of a sixth of a
// microsecond a piece of n tiles takes about 50 + 2 T + 2 T n for T steps, a wave of chunks as long as one of them, or, where
// the last one of 64 units leaves an SM no more than one block, two thirds.  Runs are taken where the longest of them is below the chunks by that
// (64 units: 4 % below).  Measured in 220 sizes each (30 to 2,500 members, 6 to 450 queries, 1 to 4 digits), against what the faster
// form takes, in the mean and at worst: 64 units 1.002 and 1.09, 96 units 1.003 and 1.10; runs whenever the chunks do not fit
// at once: 1.054 and 1.36, 1.021 and 1.19.  2 digits, chunks / runs: 64 units 300 x 100 77 / 67 us, 400 x 40 46 / 56, 100 x 56 28 / 34, 1,000 x 64 134 / 151;
// 96 units 300 x 100 165 / 139, 400 x 24 76 / 89.  Cells of 32 units hold six blocks to an SM and lose: 300 x 100 40 / 51.
inline S2sSplit s2s_split(uint32_t units, uint32_t members, uint32_t tiles, uint32_t digits, uint32_t sms)
{
    S2sSplit s;
    s.chunks = (tiles + 7u) / 8u;
    while (s.chunks < tiles && static_cast<uint64_t>(members) * s.chunks < 2u * sms) ++s.chunks;
    s.chunk = (tiles + s.chunks - 1u) / s.chunks;
    s.chunks = (tiles + s.chunk - 1u) / s.chunk;
    s.places = sms * (units == 64u ? 2u : 1u);
    const uint64_t blocks = static_cast<uint64_t>(members) * s.chunks, all = static_cast<uint64_t>(members) * tiles;
    if ((units != 64u && units != 96u) || blocks <= s.places || all > 0xFFFFFFFFull) return s;       // (a run counts its tiles in 32 bits)
    const uint64_t steps = 3u * digits + 2u, piece = 50u + 2u * steps;
    const uint64_t waves3 = 3u * (blocks / s.places) + (blocks % s.places == 0u ? 0u : units == 64u && blocks % s.places <= sms ? 2u : 3u);
    const uint64_t chunked = waves3 * (piece * s.chunks + 2u * steps * tiles);     // x 3 chunks
    uint64_t longest = 0;
    for (uint32_t b = 0; b < s.places; ++b) {
        const uint32_t first = static_cast<uint32_t>(all * b / s.places), end = static_cast<uint32_t>(all * (b + 1u) / s.places);
        const uint64_t run = piece * s2s_pieces(first, end, tiles, units == 64u ? kS2sRunTiles64 : kS2sRunTiles96) + 2u * steps * (end - first);
        if (run > longest) longest = run;
    }
    if (longest * 3u * s.chunks * 100u < chunked * (units == 64u ? 96u : 100u)) s.chunk = 0u;
    return s;
}

}  // namespace evo
