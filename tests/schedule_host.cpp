// Host copy of what the setup kernel schedules, checked for every query and record: compiled by
// test_schedule_cpu.py from the headers the library is built from.
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../paper_2509_06514_gb300/csrc/schedule.h"

using namespace impir;

namespace {

struct Span {
    uint64_t lo, hi;
};

std::string g_what;

int bad(const char* what, uint64_t a, uint64_t b) {
    char buf[256];
    std::snprintf(buf, sizeof buf, "%s (%llu, %llu)", what, (unsigned long long)a, (unsigned long long)b);
    g_what = buf;
    return 1;
}

}  // namespace

struct Result {
    uint64_t tc_units, n_units;
    uint32_t lane_bits, shape_lane_bits, qpw, tc_min_active, tc_shape, pad;
};

// One launch over records [rec_lo, rec_hi) (rec_hi 0: the whole database) of hist[m] queries of 2^m
// leaves; n_launch: records the launch shape is chosen for (a shard's rows). Returns 0 if every query
// gets each record of its domain in the window exactly once and nothing else is read.
extern "C" const char* schedule_what() { return g_what.c_str(); }

extern "C" uint32_t schedule_tile_bits(uint64_t n_launch, uint32_t words, uint32_t n_queries, int sms) {
    const impir_config c = default_config(n_launch, words, n_queries, sms);
    return xor_shape(c, true, n_launch, words, n_queries, sms).tile_bits();
}

extern "C" int schedule_check(uint64_t n_records, uint64_t n_launch, uint32_t words, const uint32_t* hist, int sms,
                              uint64_t rec_lo, uint64_t rec_hi, int add, Result* out) {
    uint32_t n = 0;
    unsigned long long present = 0;
    for (uint32_t m = 1; m <= kMaxDomainBits; ++m) {
        n += hist[m];
        if (hist[m]) present |= 1ull << m;
    }
    impir_config c = default_config(n_launch, words, n, sms);
    if (add) c.queries_per_warp = std::min(c.queries_per_warp, 2u);
    const XorShape shape = xor_shape(c, true, n_launch, words, n, sms, add != 0);
    SetupParams S{};
    S.n_records = n_records;
    S.n_queries = n;
    S.words = words;
    apply_shape(shape, sms, &S);
    S.mixed = add ? 0 : 1;
    S.rec_lo = rec_lo;
    S.rec_hi = rec_hi;
    uint32_t bstart[kMaxDomainBits + 1] = {}, gstart[kMaxDomainBits + 1] = {}, ngrp[kMaxDomainBits + 1] = {};
    std::vector<SegDesc> segs(kMaxSegments);
    WsHeader hdr{};
    const uint32_t n_groups = make_schedule(S, present, hist, bstart, gstart, ngrp, segs.data(), &hdr);
    *out = Result{hdr.tc_units, hdr.n_units, hdr.lane_bits, c.lane_bits, c.queries_per_warp, n, shape.tc, 0};
    if (hdr.first_seg + hdr.n_segs > kMaxSegments) return bad("segments", hdr.first_seg, hdr.n_segs);

    std::vector<Span> got[kMaxDomainBits + 1];
    const auto domain = [&](uint32_t m) { return std::min<uint64_t>(n_records, 1ull << m); };
    const auto window = [&](uint64_t lo, uint64_t hi) { return lo >= rec_lo && (rec_hi == 0 || hi <= rec_hi || hi <= n_records); };
    // tiles [t0, t1) of T records for the queries at sorted positions [0, active)
    const auto take = [&](uint64_t T, uint64_t t0, uint64_t t1, uint32_t active, bool small_ok) {
        for (uint32_t m = 1; m <= kMaxDomainBits; ++m) {
            if (!hist[m] || bstart[m] >= active) continue;
            if (bstart[m] + hist[m] > active) return bad("a bucket is cut", m, active);
            uint64_t lo = t0 * T, hi = std::min(t1 * T, n_records);
            if (lo >= n_records) return bad("tile past the database", t0, T);
            if ((1ull << m) < T) {  // a domain below a tile: tile 0 only, its leaves only
                if (!small_ok || t0 != 0) return bad("a small domain in a tile", m, t0);
                hi = std::min(hi, domain(m));
            } else if (hi > domain(m)) {
                return bad("a tile past the domain", m, hi);
            }
            if (!window(lo, hi)) return bad("records outside the launch", lo, hi);
            got[m].push_back({lo, hi});
        }
        return 0;
    };
    uint64_t unit = 0;
    for (uint32_t j = 0; j < hdr.first_seg; ++j) {
        const SegDesc& s = segs[j];
        const uint64_t end = j + 1 < hdr.first_seg ? segs[j + 1].unit_lo : hdr.tc_units;
        if (s.unit_lo != unit || s.count == 0 || (end - unit) % s.count) return bad("units of a tensor segment", j, end);
        const uint32_t size = (s.active + s.count - 1) / s.count;
        if (size > kTcQueries) return bad("rows of a unit", size, s.active);
        out->tc_min_active = std::min(out->tc_min_active, s.active);
        if (int e = take(32u << kTcLaneBits, s.tile_lo, s.tile_lo + (end - unit) / s.count, s.active, true)) return e;
        unit = end;
    }
    if (unit != hdr.tc_units) return bad("tensor units", unit, hdr.tc_units);
    unit = 0;
    for (uint32_t j = hdr.first_seg; j < hdr.first_seg + hdr.n_segs; ++j) {
        const SegDesc& s = segs[j];
        const uint64_t end = j + 1 < hdr.first_seg + hdr.n_segs ? segs[j + 1].unit_lo : hdr.n_units;
        if (s.unit_lo != unit || s.count == 0 || (end - unit) % s.count) return bad("units of a segment", j, end);
        const uint64_t t1 = s.tile_lo + (end - unit) / s.count;
        if (s.active) {
            if (s.count != (s.active + S.qpw - 1) / S.qpw) return bad("groups of a segment", s.count, s.active);
            if (int e = take(32ull << hdr.lane_bits, s.tile_lo, t1, s.active, false)) return e;
        } else {
            if (s.count > n_groups) return bad("group count", s.count, n_groups);
            uint32_t groups = 0;
            for (uint32_t m = kMaxDomainBits; m >= 1 && groups < s.count; --m) {
                if (!hist[m] || !ngrp[m]) continue;
                if (gstart[m] != groups || ngrp[m] != (hist[m] + S.qpw - 1) / S.qpw) return bad("groups of a domain", m, groups);
                groups += ngrp[m];
                const uint64_t T = m >= 5 ? 32ull << std::min(hdr.lane_bits, m - 5) : 1ull << m;
                if (s.tile_lo * T >= domain(m)) return bad("tile past the domain", m, s.tile_lo);
                const uint64_t lo = s.tile_lo * T, hi = std::min(t1 * T, domain(m));
                if ((t1 - 1) * T >= domain(m)) return bad("last tile past the domain", m, t1);
                if (!window(lo, hi)) return bad("records outside the launch", lo, hi);
                got[m].push_back({lo, hi});
            }
            if (groups != s.count) return bad("a domain's groups are cut", groups, s.count);
        }
        unit = end;
    }
    if (unit != hdr.n_units) return bad("units", unit, hdr.n_units);

    for (uint32_t m = 1; m <= kMaxDomainBits; ++m) {
        if (!hist[m]) continue;
        const uint64_t hi = rec_hi ? std::min(rec_hi, domain(m)) : domain(m);
        std::sort(got[m].begin(), got[m].end(), [](const Span& a, const Span& b) { return a.lo < b.lo; });
        uint64_t at = rec_lo;
        for (const Span& s : got[m]) {
            if (s.lo < at) return bad("records scheduled twice", m, s.lo);
            if (s.lo > at) return bad("records left out", m, at);
            at = s.hi;
        }
        if (hi > rec_lo && at != hi) return bad("records left out at the end", m, at);
    }
    return 0;
}

// Warps that a launch in this shape has.
extern "C" uint32_t launched_warps(uint32_t lane_bits, uint32_t qpw, uint32_t warps) {
    const impir_config c{lane_bits, qpw, warps, 0};
    return split_smem(warps, size_t(qpw) * bits_words(c) * 4).warps;
}
