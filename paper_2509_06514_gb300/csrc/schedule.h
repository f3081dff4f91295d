// schedule.h — the work schedule of a batch: which kernel takes which records for which queries.
//
// A tile is covered by every group whose DB prefix min(N, 2^m) reaches it, so the schedule is a
// handful of segments (one per distinct domain size). Tiles that enough queries reach are scheduled
// for the tensor-core kernel, the rest for the warp kernels. The setup kernel builds it with one
// thread; the same code compiles for the host, where it can be checked for every (query, record).
#pragma once

#include "impir_internal.h"

#ifdef __CUDACC__
#include "bounds.cuh"
#define IMPIR_HD __host__ __device__ __forceinline__
#else
#define IMPIR_HD inline
#endif

namespace impir {

IMPIR_HD uint32_t lowest_bit(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return uint32_t(__ffsll((long long)v) - 1);
#else
    return uint32_t(__builtin_ctzll(v));
#endif
}

IMPIR_HD uint32_t highest_bit(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return uint32_t(63 - __clzll((long long)v));
#else
    return uint32_t(63 - __builtin_clzll(v));
#endif
}

// Room for segment `nseg` in the workspace (a failed check is recorded by the debug build).
IMPIR_HD bool segment_fits(uint32_t nseg) {
#ifdef __CUDA_ARCH__
    return IMPIR_IN_BOUNDS(nseg < kMaxSegments, kSiteWorkspace, nseg);
#else
    return nseg < kMaxSegments;
#endif
}

// Sorts the domain sizes (bit m of `present`: hist[m] queries have domain bits m) into buckets, largest
// first (bstart), groups of at most qpw queries (gstart, ngrp) and tile-major segments (a tile is
// 32 << lane_bits leaves for m >= 5 + lane_bits, otherwise the whole domain is one tile), and fills the
// schedule's fields of the header. Returns the number of groups.
IMPIR_HD uint32_t make_schedule(const SetupParams& S, unsigned long long present, const uint32_t* hist, uint32_t* bstart,
                                uint32_t* gstart, uint32_t* ngrp, SegDesc* segs, WsHeader* hdr) {
    // f(m) for the domain sizes that occur, ascending, until it returns false
    const auto ascending = [&](auto f) {
        for (unsigned long long p = present; p; p &= p - 1)
            if (!f(lowest_bit(p))) break;
    };
    uint32_t pos = 0;
    for (unsigned long long p = present; p;) {
        const uint32_t m = highest_bit(p);
        p ^= 1ull << m;
        bstart[m] = pos;
        pos += hist[m];
    }
    uint32_t nseg = 0;
    // Tensor-core kernel: the tiles of the prefix that at least tc_min_queries queries reach
    // (queries are sorted by domain, so that is all records below `split`), if they make enough
    // units. The split is a multiple of both kernels' tiles (a domain of 2^m >= tmax records, or
    // the database's end): the first tile that is not the tensor-core kernel's starts there. Warp tiles
    // can be the smaller ones (2^2 leaves per lane for 4 KiB records).
    unsigned long long split = 0, tc_units = 0;
    constexpr unsigned long long tc_tile = 32ull << kTcLaneBits;
    const unsigned long long tmax = 32ull << (S.lane_bits > kTcLaneBits ? S.lane_bits : kTcLaneBits);
    const auto covered = [&](uint32_t m) { return S.n_records < (1ull << m) ? S.n_records : 1ull << m; };
    if (S.group_cap) {
        unsigned long long prev = 0, units = 0;
        ascending([&](uint32_t m) {
            const unsigned long long end = covered(m);
            const uint32_t active = bstart[m] + hist[m];  // queries with domain bits >= m
            if (active < S.tc_min_queries) return false;
            const unsigned long long lo = (prev > S.rec_lo ? prev : S.rec_lo) / tc_tile;
            const unsigned long long hi = ((S.rec_hi && S.rec_hi < end ? S.rec_hi : end) + tc_tile - 1) / tc_tile;
            if (hi > lo) units += (hi - lo) * ((active + S.group_cap - 1) / S.group_cap);
            if (end > prev) prev = end;
            // (a domain that ends inside a tile is no place to split at; if too few queries go on from
            // there, the line stays at the last one that is)
            if (units >= S.tc_min_units && (prev % tmax == 0 || prev == S.n_records)) split = prev;
            return true;
        });
    }
    // segs[nseg ...]: tiles of `tile` records from tile `prev` on (clipped to the records of this
    // launch), for each domain size the tiles it adds; groups(m) of them cover such a tile
    const auto cut = [&](unsigned long long tile, unsigned long long prev, unsigned long long end_rec, auto skip,
                         auto groups, auto active) {
        unsigned long long unit = 0;
        const unsigned long long wlo = S.rec_lo / tile, whi = (S.rec_hi + tile - 1) / tile;
        ascending([&](uint32_t m) {
            if (skip(m)) return true;
            const unsigned long long tiles = (covered(m) + tile - 1) / tile;
            if (tiles > prev) {
                if (!segment_fits(nseg)) return false;
                const unsigned long long lo = prev > wlo ? prev : wlo;
                const unsigned long long hi = (S.rec_hi == 0 || tiles < whi) ? tiles : whi;
                if (hi > lo) {
                    const uint32_t g = groups(m);
                    segs[nseg++] = SegDesc{lo, unit, g, active(m), 0};
                    unit += (hi - lo) * g;
                }
                prev = tiles;
            }
            return prev * tile < end_rec;
        });
        return unit;
    };
    const auto reach = [&](uint32_t m) { return bstart[m] + hist[m]; };  // queries with domain bits >= m
    if (split)
        tc_units = cut(tc_tile, 0, split, [](uint32_t) { return false; },
                       [&](uint32_t m) { return (reach(m) + S.group_cap - 1) / S.group_cap; }, reach);
    hdr->tc_counter = 0;
    hdr->tc_units = tc_units;
    hdr->tc_segs = nseg;
    hdr->first_seg = nseg;
    const uint32_t first_seg = nseg;

    // Warp kernels, from record `split` on. Queries whose domains end early leave fewer units than
    // the launch shape was chosen for: smaller lane subtrees then make up for it (37 queries of
    // 2^14 .. 2^20 leaves on 10^6 records: 981 us with the shape for 37 of 2^20).
    uint32_t lb = S.lane_bits;
    for (; lb > 2; --lb) {
        unsigned long long units = 0, prev = (split + (32ull << lb) - 1) >> (lb + 5);
        ascending([&](uint32_t m) {
            const unsigned long long tiles = (covered(m) + (32ull << lb) - 1) >> (lb + 5);
            if (tiles > prev) units += (tiles - prev) * ((reach(m) + S.qpw - 1) / S.qpw), prev = tiles;
            return true;
        });
        if (units >= S.want_units) break;
    }
    // The XOR answer's groups mix domains of at least one tile: group g of a segment is the queries
    // at sorted positions [g qpw, (g + 1) qpw) of its `active` ones. Domains smaller than a tile (on
    // tile 0) and the additive answer's queries keep groups of one domain size, listed in group
    // descriptors.
    const unsigned long long tbig = 32ull << lb;
    const uint32_t m_mix = 5 + lb;
    uint32_t g = 0;
    for (unsigned long long p = present; p;) {
        const uint32_t m = highest_bit(p);
        p ^= 1ull << m;
        gstart[m] = g;
        ngrp[m] = S.mixed && m >= m_mix ? 0 : (hist[m] + S.qpw - 1) / S.qpw;
        g += ngrp[m];
    }
    unsigned long long unit = 0;
    const unsigned long long prev = (split + tbig - 1) / tbig;
    if (S.mixed) {
        const bool small = g && prev == 0 && S.rec_lo == 0;
        if (small) segs[nseg++] = SegDesc{0, 0, g, 0, 0};
        const uint32_t from = nseg;
        unit = cut(tbig, prev, ~0ull, [&](uint32_t m) { return m < m_mix; },
                   [&](uint32_t m) { return (reach(m) + S.qpw - 1) / S.qpw; }, reach);
        if (small) {
            for (uint32_t i = from; i < nseg; ++i) segs[i].unit_lo += g;
            unit += g;
        }
    } else {
        unit = cut(tbig, prev, ~0ull, [](uint32_t) { return false; }, [&](uint32_t m) { return gstart[m] + ngrp[m]; },
                   [](uint32_t) { return 0u; });
    }
    hdr->lane_bits = lb;
    hdr->counter = 0;
    hdr->n_units = unit;
    hdr->n_groups = g;
    hdr->n_segs = nseg - first_seg;
    return g;
}

}  // namespace impir
