// How a reduce of many windows is cut over the GPU: host code only, no CUDA, so that
// it can be checked where there is no GPU.
#pragma once

#include <cstdint>

namespace hlf {

constexpr uint64_t kSmShared = 228 * 1024;  // shared memory of an SM
constexpr uint64_t kCtaShared = 1024;       // of it kept per CTA by the system

// CTAs of `threads`, `parts` of them per window, `per` indices per thread.
struct ReduceShape {
    unsigned threads, blocks;
    uint32_t parts;
    uint64_t per, runs;
    uint64_t align;  // runs start at multiples of align + 1
};

// The threads a window can use are one per Gray block of 2^U indices; a seed
// costs a few tens of solutions (kSeedCost), so short runs are worth it
// whenever they fill idle SMs. One window: one CTA if that holds them all (the
// result then needs no clearing), else all of them, up to one wave, in CTAs no
// larger than spreading them over every SM takes. Several windows: the CTA size and
// the cut whose waves cost least.
// With runs of at least 2048 indices and one CTA per window instead, 2^20
// four-word solutions took 694 us on one SM (now 10.8, two launches and the
// host's call among it), and 64 windows of 2^24 at W = 1 took 2.16 ms on 64
// CTAs of 256 threads (now 0.79).
//
// U: log2 of the Gray block; T: the most threads of a CTA; room: threads an SM's
// registers hold; smem: a CTA's shared memory.
inline ReduceShape reduce_shape(uint64_t chunk, uint64_t n_chunks, int U, uint64_t T, uint64_t sms, uint64_t room,
                                uint64_t smem)
{
    constexpr uint64_t kSeedCost = 48;
    // Threads that build a CTA's tables in good time: one solution of 16 words at an
    // index of 60 bits takes 8.3 us, with 32 of them 18.6.
    constexpr uint64_t kFew = 256;
    // The seed tables bind small CTAs of wide rows: at W = 16 an SM holds five of them,
    // not the eight of 64 threads that its registers would. Cut as if they fitted, 1000
    // windows of 5000 took 153 us (now 125), 1216 of 5000 168 (128).
    const uint64_t most = kSmShared / (smem + kCtaShared);
    auto fit = [&](uint64_t threads) { return room / threads < most ? room / threads : most; };
    const uint64_t runs = ((chunk - 1) >> U) + 2;  // Gray blocks the window touches, at most
    ReduceShape sh{};
    uint64_t want;  // threads for the window
    if (n_chunks == 1) {
        want = runs < sms * room ? runs : sms * room;
        uint64_t bd = want <= T ? want : (want + sms - 1) / sms;
        bd = (bd + 31) / 32 * 32;
        const uint64_t least = want > T ? 128 : kFew;
        bd = bd > T ? T : (bd < least ? least : bd);
        sh.threads = (unsigned)bd;
        sh.parts = (uint32_t)((want + bd - 1) / bd);
    } else {
        // CTAs of T threads down to 64, 1 to 64 of them a window: the fewest steps of
        // the busiest SM. Smaller CTAs only where that saves 1/16: each builds its own
        // tables (64 windows of 2^24 in CTAs of 64 threads 813 us, of 1024 792, though
        // the former fill the wave 3% better; 64 of 1239596 78 us against 82).
        // Of the cuts of one number of waves the finest costs least; `first` is the coarsest
        // that costs the same. Each cut tried by itself, a call's host side took up to 3 us
        // more; this takes 0.1 to 0.4 unless the reduce takes milliseconds.
        uint64_t best = ~0ull;
        for (uint64_t bd = T; bd >= 64; bd /= 2) {
            const uint64_t slots = sms * fit(bd);
            const uint64_t least = best - best / 16;
            const uint64_t walk = chunk * n_chunks / (slots * bd);  // a thread's share, at least, of all waves
            uint64_t finest = (runs - 1) / bd + 1;
            if (finest > 64) finest = 64;
            if (n_chunks > (~0ull >> 8)) finest = 1;  // a window each is enough
            for (uint64_t k = 1; k <= finest;) {
                const uint64_t waves = (n_chunks * k + slots - 1) / slots;
                if (waves * kSeedCost + walk >= best) break;  // nor can a finer cut cost less
                uint64_t last = waves * slots / n_chunks;
                if (last > finest) last = finest;
                const uint64_t steps = (((chunk - 1) / (last * bd)) | ((1ull << U) - 1)) + 1;
                const uint64_t cost = waves * (kSeedCost + steps);
                if (cost < best && (bd == T || cost < least)) {
                    best = cost;
                    const uint64_t first = (chunk - 1) / (steps * bd) + 1;
                    sh.parts = (uint32_t)(first > k ? first : k);
                    sh.threads = (unsigned)bd;
                }
                k = last + 1;
            }
        }
    }
    const uint64_t slots = sms * fit(sh.threads), items = n_chunks * sh.parts;
    sh.blocks = (unsigned)(items < slots ? items : slots);
    if (sh.parts == 1) {
        // Where all windows run at once a CTA needs no more threads than its window has
        // Gray blocks: 100 of 2000 at W = 4 6.5 us with 256, 8.4 with 1024.
        const bool at_once = items <= slots;
        const uint64_t use = runs < kFew ? kFew : (runs + 31) / 32 * 32;
        if (at_once && use < sh.threads) sh.threads = (unsigned)use;
        // A window with too few blocks for the threads at hand, a CTA's if all windows run
        // at once, else those of a warp, is dealt to them by the index: idle lanes cost
        // as much as walking ones. With a block a thread instead, 10^5 windows of 10 at
        // W = 11 took 1207 us (now 421), 20000 of 100 at W = 2 129 (47), 152 of 10 at W = 16
        // 13.4 (8.3). Lanes that would walk more than about a third of a block do no better
        // so: 608 of 300 at W = 11, three a lane, 14.5 us, in blocks of four 12.3.
        const uint64_t lanes = !at_once ? 32 : (sh.threads < kFew ? sh.threads : kFew);
        if (chunk <= lanes * (at_once ? ((1ull << U) + 2) / 3 : (1ull << U) - 1)) {
            if (at_once) sh.threads = (unsigned)lanes;
            sh.per = (chunk + lanes - 1) / lanes;
            sh.runs = (chunk + sh.per - 1) / sh.per;
            return sh;
        }
    }
    want = (uint64_t)sh.parts * sh.threads;
    // chunk + 2^U - 1 indices at most, counted from the window's first block;
    // past 2^63 that count could wrap, so such windows start their runs at the
    // window's own start
    sh.align = chunk <= 1ull << 63 ? (1ull << U) - 1 : 0;
    sh.per = chunk / want + (chunk % want + sh.align + want - 1) / want;
    sh.per = (sh.per + (1ull << U) - 1) & ~((1ull << U) - 1);
    sh.runs = sh.align ? want : (chunk - 1) / sh.per + 1;
    return sh;
}

}  // namespace hlf
