// Planes per chunk of the z-march kernels on grids of a few waves of CTAs.
#pragma once

#include <cstdint>

namespace psd {

// A chunk of c planes costs its CTA c + extra; a wave with q of the per_sm CTAs that an SM holds
// costs `one` (q = 1) to 1 (q = per_sm, linear between) of a full one; a march of more than one
// wave costs `later` less, as its waves overlap.  least, most: range of c.
struct WaveCost {
    double extra, one, later;
    int least, most;
};

// The chunk whose waves end soonest on `sms` SMs.  The last chunk of every tile may be shorter
// (nz % c planes); it runs in the slots that the last wave leaves free, or after it.
static inline int wave_chunk_of(int64_t nz64, int64_t tiles, int sms, int per_sm, const WaveCost &w) {
    const int nz = nz64 < 65536 ? (int)nz64 : 65536;
    // one CTA per SM at most, whatever the chunk: the shortest
    if (tiles * ((nz + w.least - 1) / w.least) <= sms) return w.least;
    const double slots = (double)sms * per_sm, inv_slots = 1.0 / slots, inv_sms = 1.0 / sms;
    const double slope = per_sm > 1 ? (1.0 - w.one) / (per_sm - 1) : 0.0, t = (double)tiles;
    auto wave = [&](double ctas) {  // ctas in [0, slots], whole
        if (ctas <= 0.0) return 0.0;
        const int q = (int)((ctas - 0.5) * inv_sms);  // CTAs per SM less one
        return q + 1 >= per_sm ? 1.0 : w.one + slope * q;
    };
    int chunk = w.least;
    double best = -1.0;
    for (int c = w.least; c <= w.most && c <= nz; ++c) {
        const int n = nz / c, rem = nz - n * c;
        const double full = t * n, waves = (double)(int64_t)((full + 0.5) * inv_slots), r = full - waves * slots;
        double last = wave(r) * (c + w.extra);
        if (rem) {
            const double over = t - (r > 0.0 ? slots - r : 0.0);  // short chunks past the free slots
            if (over > 0.0) {  // waves of their own, as many as it takes
                const double more = (double)(int64_t)((over - 0.5) * inv_slots);
                last = (r > 0.0 ? c + w.extra : 0.0) + (more + wave(over - more * slots)) * (rem + w.extra);
            } else {
                last = wave(r + t) * (rem + w.extra) + wave(r) * (c - rem);
            }
        }
        const double cost = (waves * (c + w.extra) + last) * (waves > 0.0 ? 1.0 - w.later : 1.0);
        if (best < 0.0 || cost < best) {
            best = cost;
            chunk = c;
        }
    }
    return chunk;
}

// The same, remembering a thread's last grids (the search takes a microsecond or two of host
// time, a tenth of a call).
inline int wave_chunk(int64_t nz, int64_t tiles, int sms, int per_sm, const WaveCost &w) {
    struct Entry {
        int64_t nz = -1, tiles = 0;
        int sms = 0, per_sm = 0, chunk = 0;
        WaveCost w{};
    };
    thread_local Entry seen[4];
    Entry &e = seen[(nz ^ tiles ^ per_sm) & 3];
    if (e.nz != nz || e.tiles != tiles || e.sms != sms || e.per_sm != per_sm || e.w.extra != w.extra ||
        e.w.one != w.one || e.w.later != w.later || e.w.least != w.least || e.w.most != w.most) {
        e.chunk = wave_chunk_of(nz, tiles, sms, per_sm, w);
        e.nz = nz;
        e.tiles = tiles;
        e.sms = sms;
        e.per_sm = per_sm;
        e.w = w;
    }
    return e.chunk;
}

// A chunk long enough for the planes to fit the 65535 CTAs that a grid has along z (a few nodes
// in x and y, over half a million in z).
inline int grid_chunk(int64_t nz, int chunk) {
    const int64_t least = (nz + 65534) / 65535;
    return chunk < least ? (int)least : chunk;
}

}  // namespace psd
