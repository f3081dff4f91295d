// impir_internal.h — types shared by the host runtime and the CUDA kernels of libimpir.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "../../include/impir.h"

namespace impir {

constexpr uint32_t kMaxDomainBits = 40;
constexpr uint32_t kMaxLaneBits = 10;     // 2^10 leaves per lane at most
constexpr uint32_t kMaxSegments = 48;     // one per distinct domain size (<= 41) + slack
constexpr uint32_t kTableBytes = 128 * 1024;
// Shared-memory addresses of the kernels: the T-tables at 64 KiB, the rest below and above them. The
// dynamic shared memory begins behind the 1 KiB the system reserves and the kernel's static shared
// memory (none, or the debug build's check context).
constexpr uint32_t kTableAt = 0x10000, kHighAt = kTableAt + kTableBytes;
constexpr uint32_t kSmemBase = 1024, kSmemStatic = 128;

// Largest byte count of a database, a workspace or an answer buffer the library accepts
// (1 PiB): products of record counts and strides are checked against it before any
// allocation or launch, so they never wrap.
constexpr uint64_t kMaxBytes = 1ull << 50;
inline bool bytes_ok(uint64_t count, uint64_t unit) { return unit == 0 || count <= kMaxBytes / unit; }

// Workspace header at the start of the device workspace (256 bytes).
struct WsHeader {
    unsigned long long counter;   // next work unit to hand out
    unsigned long long n_units;   // total work units of this launch
    uint32_t n_bad;               // malformed keys seen by the setup kernel
    uint32_t first_bad;           // smallest malformed query index (UINT32_MAX if none)
    uint32_t n_groups;
    uint32_t n_segs;
    uint32_t bounds_failed;       // failed index checks of this launch (debug build only)
    uint32_t timed_out;           // a wait ran out or the tables had no place: the answers are not valid
    // the tensor-core kernel's share of the batch (fused_tc.cu): its segments come first
    unsigned long long tc_counter, tc_units;
    uint32_t tc_segs;
    uint32_t first_seg;           // the warp kernel's first segment (it has n_segs of them)
    uint32_t lane_bits;           // of the warp kernels' tiles: at most the launch shape's
    uint32_t pad[47];
};
static_assert(sizeof(WsHeader) == 256, "header is 256 bytes");

// A group of up to queries_per_warp queries with one domain size, evaluated together on
// a warp tile and scanned once: [first, first + count) indexes the sorted query list.
struct GroupDesc {
    uint32_t first;
    uint32_t count;
    uint32_t m;
    uint32_t pad;
};

// Work units u in [unit_lo, next segment's unit_lo) cover warp tiles
// tile_lo + (u - unit_lo) / count with groups (u - unit_lo) % count. `active` is the number of
// sorted queries whose domains reach these tiles, which the kernels cut into `count` groups by
// themselves (0: the groups are listed in descriptors).
struct SegDesc {
    unsigned long long tile_lo;
    unsigned long long unit_lo;
    uint32_t count;
    uint32_t active;
    unsigned long long pad2;
};
static_assert(sizeof(SegDesc) == 32, "segment descriptors are 32 bytes");
// A warp's unit, for the other warps of its block (they expand the tops of the block's first units together).
struct UnitInfo {
    unsigned long long tile;
    uint32_t first, count;  // sorted positions of its queries; 0: no unit, or one without the cooperative walk
    uint32_t sq, pad[3];
};
static_assert(sizeof(UnitInfo) == 32, "unit descriptors are 32 bytes");
constexpr uint32_t kMaxWarps = 20;
// segment table and the warps' unit descriptors, at the start of the warp kernels' shared memory
constexpr uint32_t kSegSmemBytes = kMaxSegments * sizeof(SegDesc) + kMaxWarps * sizeof(UnitInfo);

// Failed index checks of the debug build (compiled with IMPIR_BOUNDS), one record per device:
// how many failed since the record was last cleared, and the site and index of the first.
struct BoundsRecord {
    unsigned int n_failed;
    unsigned int first_site;
    unsigned long long first_index;
};

// Site codes of the index checks.
enum BoundsSite : uint32_t {
    kSiteTable = 1,      // T-table offset in shared memory
    kSiteBits = 2,       // selection-bit / node / share buffer in shared memory
    kSiteRecord = 3,     // database word
    kSiteKey = 4,        // key byte (inside the key, and inside the key buffer when its size is known)
    kSiteQuery = 5,      // query index (sorted permutation, key offsets)
    kSiteSchedule = 6,   // group or segment index
    kSiteAcc = 7,        // accumulator word
    kSiteStack = 8,      // a lane's stack of pending right children
    kSiteWorkspace = 9,  // schedule written by the setup kernel
    kSiteOut = 10,       // answer byte
};

struct WsLayout {
    size_t off_perm, off_qm, off_groups, off_segs, off_acc, total;
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

inline WsLayout ws_layout(uint32_t n_queries, uint32_t stride_bytes) {
    WsLayout L;
    size_t o = sizeof(WsHeader);
    L.off_perm = o;
    o = align256(o + size_t(n_queries) * 4);
    L.off_qm = o;
    o = align256(o + size_t(n_queries) * 4);
    L.off_groups = o;
    o = align256(o + (size_t(n_queries) + kMaxDomainBits + 8) * sizeof(GroupDesc));
    L.off_segs = o;
    o = align256(o + kMaxSegments * sizeof(SegDesc));
    L.off_acc = o;
    o = align256(o + size_t(n_queries) * stride_bytes);
    L.total = o;
    return L;
}

// ---- launch shape of the XOR answer (shared by every answer path) ----

constexpr size_t kSmemMax = 227 * 1024;

// uint4 words per lane and pass that cover a record in one pass (1, 2, 4 or 8)
inline uint32_t nk_need(uint32_t words) {
    if (words <= 32) return 1;
    const uint32_t need = (words + 31) / 32;
    return need <= 2 ? 2 : need <= 4 ? 4 : 8;
}

// uint4 words per lane and pass of the XOR scan for qpw queries per warp: records above 512 B
// are scanned in column passes of nk words per lane, with qpw * nk <= 16 accumulators per lane,
// so that more queries share every tile read (records of 1 KiB: one pass at 8 queries per warp;
// 4 KiB: four)
inline uint32_t nk_xor(uint32_t words, uint32_t qpw) {
    if (words <= 32) return 1;
    return std::min(nk_need(words), std::max(2u, 16u / qpw));
}

// Widest CTA the fused kernel is built for (its launch bounds): 20 warps for the XOR answer
// with one column pass (records of at most 512 bytes) and at most 8 queries per warp, else 16.
inline uint32_t max_warps(uint32_t qpw, uint32_t words) { return nk_need(words) == 1 && qpw <= 8 ? 20u : 16u; }

// 32-bit words of a query's slot in a warp's bit area: its selection bits, or the 16 nodes that the
// cooperative walk (at most 8 queries per warp) keeps there before.
inline uint32_t bits_words(const impir_config& c) {
    return std::max(1u << c.lane_bits, c.queries_per_warp <= 8 ? 64u : 1u);
}

// Dynamic shared memory of the XOR kernels: T-tables, segment table, per-warp selection bits.
inline size_t smem_for(const impir_config& c) {
    return kTableBytes + kSegSmemBytes + size_t(c.warps_per_cta) * c.queries_per_warp * bits_words(c) * 4;
}

// Where the warps' slices of the bit area go: as many as fit between the segment table and the
// T-tables, the others above the tables; the launch's dynamic shared memory. Warps whose slices fit
// neither place (12 warps of 8 KiB, 6 of 16 KiB: one each) are left out of the launch.
struct SmemSplit {
    uint32_t low, warps, bytes;
};
inline SmemSplit split_smem(uint32_t warps, size_t slice) {
    constexpr size_t below = kTableAt - kSmemBase - kSmemStatic - kSegSmemBytes;
    constexpr size_t above = kSmemMax + kSmemBase - kHighAt;
    SmemSplit s;
    s.low = uint32_t(std::min<size_t>(warps, below / slice));
    const uint32_t high = uint32_t(std::min<size_t>(warps - s.low, above / slice));
    s.warps = s.low + high;
    s.bytes = uint32_t(kHighAt - kSmemBase + high * slice);
    return s;
}

// Estimated time of a batch in the shape c, in SM clocks: which shape is best, not how long it takes.
// The form follows the kernel; the constants, in clocks unless said, are measured where a figure is named
// here and were else adjusted by hand until the order of timed shapes came out:
//   pair      2000 alone (a chain of ten rounds of dependent lookups; a single child 1750), 330 of the
//             lookups' shared-memory port each when an SM's warps share it (329 lookups), and a warp waits
//             for the port behind the others, at least 700 more than that; in the steady state 320, 40 %
//             more by a lone warp (1 + 0.4 / w), and 2000 for the last units. 1.04 - 0.005 s: the walk's
//             loop per subtree; slow: 1 % per query slot (registers)
//   walk      top levels, 200 for 32 of them that share the port; four cooperative levels of 2500, 330 of
//             the port for 32 nodes (1.3 pairs' time each in the steady state); the fifth level 0.8 pairs
//             per query and lane. The additive answer's lanes walk all five (0.65 each for the four more)
//   scan      per 16-byte word 4.3 operations for each query and 4 (additive: 14, with its share loads) for
//             all of them, in pairs of 560 ALU operations; 900 for a round of record loads
//   memory    3300 bytes a clock from HBM (6.8 TB/s), of which n warps per SM draw 400 n, twice that where
//             the reads of one unit pass under another's lookups; 5000 from L2, where groups read a tile
//             again; L2 holds the tiles in work up to 64 MB, none of them from 256 MB
// Where every unit finds a warp at once, the block's warps share the walk and the cooperative levels if
// it has more than four units (fused.cuh); else the port is busy throughout.
inline double shape_clocks(const impir_config& c, uint64_t n_records, uint32_t words, uint32_t n_queries, int sms,
                           bool add = false) {
    const double slots = c.queries_per_warp, s = c.lane_bits, w = c.warps_per_cta;
    const double groups = std::ceil(n_queries / slots), tiles = std::ceil(double(n_records) / double(32ull << c.lane_bits));
    const double q = n_queries / groups, m = std::ceil(std::log2(double(n_records)));
    const double units = groups * tiles, top = std::max(0.0, m - s - 5);
    const double scan = std::exp2(s) * words * (4.3 * slots + (add ? 14 : 4)) / 560;
    const double lanes = q * (0.8 + (add ? 4 * 0.65 : 0) + std::exp2(s) - 1), slow = 1 + 0.010 * slots;
    const uint32_t nk = nk_xor(words, c.queries_per_warp);
    const double per_load = nk == 1 ? (slots == 1 ? 16 : slots == 2 ? 8 : 4) * std::max(1u, 32 / words) : nk <= 2 ? 4 : nk == 4 ? 2 : 1;
    const double loads = std::ceil(32 * std::exp2(s) / per_load) * std::ceil(words / (32.0 * nk));
    double clocks, hbm = 3300;
    if (units <= sms * w) {
        const double n = std::ceil(units / sms);
        const bool cta = n > 4 && !add;
        const double shared = cta ? n : 1;  // warps whose levels are expanded together
        clocks = top * std::max(1750.0, 200 * std::ceil(shared * q / 32) * (cta ? 1 : n)) +
                 slow * lanes * std::max(2000.0, 330 * n + 700) +
                 std::max(slow * scan * std::max(2000.0, 330 * n + 700), 900 * loads);
        hbm = std::min(hbm, 400 * n);
        for (int k = 0; k < 4 && !add; ++k)
            clocks += std::max(2500.0, 330 * std::ceil(shared * q * double(1 << k) / 32) * (cta ? 1 : n));
    } else {
        double coop = 0;
        for (int k = 0; k < 4 && !add; ++k) coop += 1.3 * std::ceil(q * double(1 << k) / 32);
        clocks = (1.3 * (top + coop) + lanes + scan) * slow * (1.04 - 0.005 * s) * (320 * (1 + 0.4 / w) * units / sms + 2000);
        hbm *= 2;  // (reads of one unit pass under another's lookups)
    }
    const double record = words * 16.0 * (c.queries_per_warp == 1 && !add ? 0.5 : 1.0), pass = double(n_records) * record;
    const double live = std::min(units, sms * w) / groups * double(32ull << c.lane_bits) * record;
    const double passes = 1 + (groups - 1) * std::min(1.0, std::max(0.0, (live - 64e6) / 192e6));
    return clocks + pass * passes / hbm + pass * groups / 5000;
}

// The shape with the smallest estimate (lane subtrees of at most 2^8 leaves).
inline impir_config default_config(uint64_t n_records, uint32_t words, uint32_t n_queries, int sms) {
    impir_config best{};
    double best_t = 0;
    for (uint32_t qpw = 1; qpw <= 8; qpw *= 2) {
        if (qpw * nk_xor(words, qpw) > 16 || (qpw > 1 && qpw / 2 >= n_queries)) continue;
        // as many warps as the kernel is built for (16 were never more than 1 % faster than 20, and 50 %
        // slower where the units just fill 20)
        for (uint32_t b = 0; b <= 8; ++b) {
            const impir_config c{b, qpw, max_warps(qpw, words), 0};
            if (smem_for(c) > kSmemMax) continue;
            // groups that share a database above L2's size: tiles of at most 512 KiB, read again while
            // they are there (18 queries on 2^21 x 256 B: 1395 us with tiles of 1 MiB, 1086 with 256 KiB)
            if (b > 0 && n_queries > qpw && uint64_t(n_records) * words > (64u << 20) / 16 && (uint64_t(words) << (b + 9)) > (512u << 10))
                continue;
            const double t = shape_clocks(c, n_records, words, n_queries, sms);
            if (best_t == 0 || t < best_t) {
                best_t = t;
                best = c;
            }
        }
    }
    return best;
}

// ---- the tensor-core form of the XOR answer (fused_tc.cu) ----

constexpr uint32_t kTcQueries = 128;   // most rows of a unit (rows of the tensor product)
constexpr uint32_t kTcThreads = 768;   // 4 scan warps and 20 AES warps
constexpr uint32_t kTcTasks = 32;      // AES tasks of a unit: 4 rows each
constexpr uint32_t kTcLaneBits = 5;    // tiles of 32 << 5 = 1024 records

// Fewest queries that must reach a tile for the tensor-core kernel to take it. Its scan costs the
// same for 1 query as for 128, the warp kernels' grows with every query: measured on 2^22 records,
// time of the default warp shape over the tensor-core kernel's at 64 / 80 / 96 / 128 queries: 1.00 /
// 1.01 / 1.03 / 1.02 for 64-byte records, 1.02 / 1.04 / 1.06 / 1.06 for 256 bytes, 1.04 / 1.08 / 1.10 /
// 1.13 for 512 bytes; for 1 KiB 1.21 / 1.28 at 96 / 128 (4 KiB on 2^20: 1.17 / 1.42). At 48 queries it
// was 0.94 to 0.95 up to 512 bytes, at 64 of 1 KiB 0.98.
inline uint32_t tc_min_queries(uint32_t words) { return words <= 32 ? 64u : 96u; }

// Fewest units, of at most `rows` queries, for the tensor-core kernel to take any: units of 1024 records
// go to SMs whole, and with fewer than four per SM the last round costs more than the scan gains for
// records up to 256 bytes (0.92 to 0.97 at 2^18 records and 64 or 128 queries). Wider ones are taken from
// one and a half on: full units gain (4 KiB on 2^18, 128 queries 1.13; 512 bytes on 2^18, 96 queries 1.04),
// units of 64 or 80 rows lose to the default warp shape (512 bytes on 2^19 0.90 and 0.94) though not to
// the shapes that ran before there was a choice. Above 3 KiB they did lose to those with fewer than 104
// rows (4 KiB on 2^19, 96 queries 6240 us against 6115): four per SM there too.
inline uint64_t tc_min_units(uint32_t words, uint32_t rows, int sms) {
    return uint64_t(sms) * (words <= 16 || (words > 192 && rows < 104) ? 8 : 3) / 2;
}

// How a batch is launched: the warp kernels of fused.cuh in the shape `c`, and with tc, behind them, the
// tensor-core kernel, which takes the tiles that enough queries reach (the setup kernel draws the
// line: the keys' domains are on the device) in groups of at most tc_cap queries.
struct XorShape {
    impir_config c;
    bool tc;
    uint32_t tc_cap;
    uint64_t want_units;  // see SetupParams
    // tiles of both kernels divide 32 << tile_bits() records
    uint32_t tile_bits() const { return tc ? std::max(kTcLaneBits, c.lane_bits) : c.lane_bits; }
};

// free_shape: the caller set no launch shape of its own; warps_only: the additive answer, or a tuned shape
// that was faster without the tensor-core kernel.
inline XorShape xor_shape(const impir_config& c, bool free_shape, uint64_t n_records, uint32_t words,
                          uint32_t n_queries, int sms, bool warps_only = false) {
    XorShape s{c, false, 0, 0};
    // as many units as a batch that covers the database has, but 40 per SM are enough
    const uint64_t T = 32ull << c.lane_bits;
    if (free_shape)
        s.want_units = std::min<uint64_t>(40ull * sms, ((n_records + T - 1) / T) *
                                                           ((n_queries + c.queries_per_warp - 1) / c.queries_per_warp));
    if (!free_shape || warps_only || c.queries_per_launch != 0 || n_queries < tc_min_queries(words)) return s;
    const uint64_t groups = (n_queries + kTcQueries - 1) / kTcQueries;
    const uint32_t rows = uint32_t((n_queries + groups - 1) / groups);
    if (groups * ((n_records + (32u << kTcLaneBits) - 1) >> (kTcLaneBits + 5)) < tc_min_units(words, rows, sms)) return s;
    s.tc = true;
    s.tc_cap = rows;
    return s;
}

struct SetupParams {
    const uint8_t* keys;
    const uint32_t* key_off;
    uint8_t* ws;
    uint4* acc;              // the per-query accumulators (in the workspace, or the caller's answers)
    WsLayout lay;
    uint64_t n_records;
    uint32_t n_queries;
    uint32_t words;          // stride / 16
    uint32_t lane_bits;
    uint32_t qpw;            // queries per warp (group size)
    uint32_t mixed;          // groups mix domain sizes (the XOR answer)
    unsigned long long want_units;  // units the launch shape was chosen for (0: lane_bits as it is)
    uint32_t group_cap;      // most queries of a tensor-core unit (0: the warp kernels take the whole batch)
    uint32_t tc_min_queries; // see tc_min_queries() and tc_min_units()
    unsigned long long tc_min_units;
    // A chunk of a streamed database or a row shard: only tiles of records [rec_lo, rec_hi) are
    // scheduled (whole tiles; rec_hi == 0: no upper limit), and keep_acc != 0 keeps the accumulators
    // of the previous chunks instead of zeroing them. Zero values give the whole-database
    // launch.
    unsigned long long rec_lo, rec_hi;
    uint32_t keep_acc;
    uint32_t keep_status;             // keeps the header's timed_out too: its earlier launches belong to the call
    BoundsRecord* bounds;             // debug build: where failed checks are recorded
    unsigned long long keys_bytes;    // size of the key buffer (0: unknown)
};

// Sets the launch shape's fields of the setup parameters.
inline void apply_shape(const XorShape& s, int sms, SetupParams* sp) {
    sp->lane_bits = s.c.lane_bits;
    sp->qpw = s.c.queries_per_warp;
    sp->mixed = 1;
    sp->want_units = s.want_units;
    sp->group_cap = s.tc ? s.tc_cap : 0;
    sp->tc_min_queries = tc_min_queries(sp->words);
    sp->tc_min_units = tc_min_units(sp->words, s.tc_cap, sms);
}

struct FusedParams {
    const uint4* db;
    const uint8_t* keys;
    const uint32_t* key_off;
    uint8_t* ws;
    uint4* acc;              // as in SetupParams
    const uint32_t* te0;     // 256-entry AES T-table (global memory), see host_aes.cpp
    WsLayout lay;
    uint64_t n_records;
    uint32_t n_queries;
    uint32_t words;          // uint4 words per record (stride / 16)
    uint32_t bits_words;     // 32-bit words of selection bits (additive: shares) per (warp, query slot)
    uint32_t with_tc;        // the tensor-core kernel takes part of the batch: nothing may be left here
    unsigned long long wait_ns;  // limit of the tensor-core kernel's waits
    uint32_t slices_low;     // warps whose slice of those lies below the tables
    unsigned long long rec_lo;  // global index of the record at db[0] (0 unless a chunk or a row shard)
    // extents for the debug build's index checks
    BoundsRecord* bounds;
    unsigned long long db_words;    // uint4 words of db[] the launch may read
    unsigned long long keys_bytes;  // size of the key buffer (0: unknown)
    uint32_t smem_bytes;            // dynamic shared memory of the launch
};

struct FinalizeParams {
    const uint8_t* ws;
    WsLayout lay;
    uint8_t* out;
    uint32_t n_queries;
    uint32_t record_bytes;
    uint32_t stride;
    BoundsRecord* bounds;
};

// Kernel launchers (defined in the .cu files). Each fused launcher first sets the kernel's
// dynamic shared-memory limit on the current device (once per device).
cudaError_t launch_setup(const SetupParams& p, cudaStream_t s);
// The current device's record of failed index checks in the debug build, else nullptr.
BoundsRecord* bounds_record();
// uint4 words of a database the index checks allow the kernels to read: n_words, less the
// records a debug-build test withholds (IMPIR_BOUNDS_TEST_WITHHOLD_RECORDS) to see a check fire.
unsigned long long bounds_db_words(unsigned long long n_words, uint32_t words_per_record);
// The T-table as the kernels get it: a debug-build test (IMPIR_BOUNDS_TEST_NO_TABLES) has them refuse to run,
// as they do where their shared memory does not begin at the address that the tables' place assumes.
const uint32_t* bounds_te0(const uint32_t* te0);
// Nanoseconds after which a wait between the tensor-core kernel's warps gives up: 20 s, where a unit takes
// milliseconds. A debug-build test shortens it (IMPIR_BOUNDS_TEST_WAIT_NS) to see a wait run out.
unsigned long long wait_limit_ns();
// follows: nothing but the fused kernel's launch came before it in the stream (a dependent launch).
cudaError_t launch_finalize(const FinalizeParams& p, cudaStream_t s, bool follows);
// The XOR answer's fused launch in the given shape.
cudaError_t launch_xor(const XorShape& s, int sms, cudaStream_t st, FusedParams& fp);
cudaError_t launch_fused_tc(int sms, cudaStream_t s, const FusedParams& p);
cudaError_t prepare_fused_tc();
uint32_t tc_smem_bytes();
// qpw in {1,2,4,8,16}, nk in {1,2,4,8} with qpw * nk <= 16.
cudaError_t launch_fused(uint32_t qpw, uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                         const FusedParams& p);
cudaError_t launch_fused_q1(uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const FusedParams& p);
cudaError_t launch_fused_q2(uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const FusedParams& p);
cudaError_t launch_fused_q4(uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const FusedParams& p);
cudaError_t launch_fused_add(uint32_t qc, uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             const FusedParams& p);
cudaError_t launch_fused_q16(uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const FusedParams& p);
cudaError_t launch_fused_q8(uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const FusedParams& p);
// Sets the dynamic shared-memory limit of every instantiation of the XOR answer's kernels on
// the current device and loads their code there (with lazy module loading the first launch of
// a kernel otherwise does this, which may allocate device memory).
cudaError_t prepare_xor_kernels();
cudaError_t prepare_fused_q1();
cudaError_t prepare_fused_q2();
cudaError_t prepare_fused_q4();
cudaError_t prepare_fused_q8();
cudaError_t prepare_fused_q16();

// Host AES pieces of the product (independent of the oracle): T-table and key schedule.
void host_aes_te0(uint32_t te0[256]);
void host_aes_expand(const uint8_t key[16], uint32_t rk[44]);
void host_aes_encrypt(const uint32_t rk[44], const uint8_t in[16], uint8_t out[16]);

}  // namespace impir
