// fused_tc.cu — the fused DPF evaluation + dpXOR kernel whose scan runs on the tensor cores.
//
// It computes what fused.cuh's XOR kernel computes, for batches of many queries. dpXOR of a tile
// of K records for up to 128 queries is a product over GF(2): (128 x K selection bits) times
// (K x 8B record bits). The register scan of fused.cuh spends one 32-bit XOR per record word and
// query on the ALU pipe that the AES engine's address permutes and XORs fill; here a record word
// costs 9 ALU operations for all 128 queries and the sums run on the tensor cores.
//
// The product in numbers (tcgen05.mma kind::f8f6f4, fp32 accumulators):
//   * a selection bit is the byte 0 or 1, read as e4m3: 0 or 2^-9 (operand A, in tensor memory);
//   * a record byte becomes eight bytes, one per bit, by masking alone: byte & (1 << i) read as
//     e4m3 is 0 or the power of two 2^e(i), e = -9 -8 -7 -6 -5 -3 1 for i = 0..6; bit 7, e4m3's sign,
//     is first shifted to bit 6 (operand B, in shared memory). Each bit has a column of its own, so
//     the columns' different scales never meet;
//   * a sum is a whole number of at most K = 1024 times 2^(e-9): exact in fp32 in any order (the
//     accumulators were compared with integer counts up to 2^16 on this GPU). Its parity
//     is the answer bit: adding 2^23 (scaled) puts the count's lowest bit at a fixed mantissa bit.
//
// Structure of a CTA (persistent, one per SM), 20 AES warps and 4 scan warps:
//   * unit = (tile of K = 32 << S records, group of at most 128 queries of the sorted batch);
//     units come from the launch's global counter. Domain sizes mix freely inside a group. Tiles that
//     few queries reach are left to the warp kernel, which is launched before (schedule.h, launch_xor).
//   * scan warps, thread n for query n: walk the root -> the tile's node and expand 3 levels
//     below it (8 nodes per query), for the unit after next; all lanes are busy, where a warp of
//     fused.cuh walks for its 8 queries with 8 lanes.
//   * AES warps: tasks of 4 queries: the 4 queries' level 3 -> 4 pairs fill the warp once, then
//     every lane takes its 2^S-leaf subtree depth first for each query and leaves a word of
//     selection bits in shared memory. Tasks come from a shared counter across units, so warps
//     run on into the next unit while the scan warps work on the last one.
//   * scan warps: selection bits -> tensor memory (256 columns, the whole tile), then per 32
//     bytes of the records: 64 records at a time into a ring of operand tiles (each lane masks one
//     16-byte load into 128 bytes), two MMAs of 128 x 256 x 32 each, and at the tile's end the
//     parities are read back and XORed into the per-query accumulators in global memory.
// No selection bit leaves the SM.
#define IMPIR_TABLE_POINTER
#include "fused.cuh"

namespace impir {

namespace {

constexpr uint32_t kScanThreads = 128;  // the 4 scan warps: one thread per tensor-memory lane
constexpr uint32_t kTaskQ = 4;          // queries of an AES task
constexpr uint32_t S = kTcLaneBits;     // a lane's subtree has 2^S = 32 leaves: one selection word
constexpr uint32_t K = 32u << S;        // records of a tile
constexpr uint32_t LG = S + 5;          // its levels
constexpr uint32_t kStages = 2;         // operand tiles in flight
constexpr uint32_t kStageBytes = 64 * 256;
struct UnitDesc {
    unsigned long long tile;
    uint32_t first, count;  // its queries: sorted positions [first, first + count)
    uint32_t stop, pad;     // stop: no unit, the launch is done
};

struct Ctl {
    unsigned long long ready[2];         // unit's nodes are there (scan warps -> AES warps)
    unsigned long long full[2];          // unit's selection bits are there (AES warps -> scan warps)
    unsigned long long empty[kStages];   // operand tile read by its MMAs
    unsigned long long dfull;            // accumulators of a pass complete
    unsigned long long wait_ns;          // a wait that outlasts this is an error
    UnitDesc unit[2];
    uint32_t done[2];        // finished tasks of the unit
    uint32_t task;           // next AES task
    uint32_t tmem;           // base of the 512 tensor-memory columns
    uint32_t abort;          // a wait ran out
    uint32_t pad;
};
static_assert(sizeof(Ctl) <= 256, "control block");
// Shared memory, by address: below the T-tables the operand tiles and 15 of the 16 node arrays, above
// them the last node array, the selection bits, the units' key offsets and the control block.
constexpr uint32_t kNodeArray = kTcQueries * 16;
constexpr uint32_t kAtStage = kSmemBase + kSmemStatic;
constexpr uint32_t kAtNodes = kAtStage + kStages * kStageBytes;  // [2][8][128] nodes, the last array at kHighAt
constexpr uint32_t kAtBits = kHighAt + kNodeArray;               // [2][128][32] words
constexpr uint32_t kAtKey = kAtBits + 2 * kTcQueries * 32 * 4; // [2][128] key offsets
constexpr uint32_t kAtCtl = kAtKey + 2 * kTcQueries * 4;
constexpr uint32_t kTcSmem = kAtCtl + 256 - kSmemBase;
static_assert(kAtNodes + 15 * kNodeArray <= kTableAt && kTcSmem <= kSmemMax, "shared memory");

__device__ __forceinline__ void mbar_init(unsigned long long* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem32(b)), "r"(n) : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem32(b)) : "memory");
}

__device__ __forceinline__ bool mbar_try(unsigned long long* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Waits for the phase of the given parity; false when the limit passes or another wait of this
// CTA gave up (the caller then leaves its loop; no thread waits for ever).
// `nap` (nanoseconds): pause between polls of the waits that are expected to be long, whose polling
// would otherwise take issue slots from the AES warps.
__device__ __forceinline__ bool mbar_wait(unsigned long long* b, uint32_t parity, Ctl* ctl, uint32_t nap = 0) {
    if (mbar_try(b, parity)) return true;
    const unsigned long long t0 = now_ns();
#pragma unroll 1
    for (;;) {
        if (nap) __nanosleep(nap);
        if (mbar_try(b, parity)) return true;
        if (*reinterpret_cast<volatile uint32_t*>(&ctl->abort)) return false;
        if (now_ns() - t0 > ctl->wait_ns) {
            *reinterpret_cast<volatile uint32_t*>(&ctl->abort) = 1;
            return false;
        }
    }
}

// Barrier of the scan warps; true if `bad` holds for any of them.
__device__ __forceinline__ bool scan_bar_or(bool bad) {
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, 128, p;\nselp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"(uint32_t(bad))
        : "memory");
    return r != 0;
}

// Debug build: n bytes at shared-memory address o lie inside [lo, hi).
__device__ __forceinline__ bool smem_ok(uint32_t o, uint32_t n, uint32_t lo, uint32_t hi) {
    return IMPIR_IN_BOUNDS(o >= lo && o + n <= hi, kSiteBits, o);
}

// Word w (32 records) of query row q in bits buffer b: rows of 32 words, swizzled so that both a
// warp writing one row and a warp reading one word of 32 rows touch 32 banks.
__device__ __forceinline__ uint32_t bits_at(uint32_t b, uint32_t q, uint32_t w) {
    return kAtBits + ((b * kTcQueries + q) * 32 + (w ^ (q & 31))) * 4;
}

// The key offsets of a unit's queries.
__device__ __forceinline__ uint32_t* unit_keys(uint32_t b) {
    return reinterpret_cast<uint32_t*>(smem_at(kAtKey)) + b * kTcQueries;
}

__device__ __forceinline__ uint32_t node_at(uint32_t b, uint32_t i, uint32_t q) {
    const uint32_t array = b * 8 + i;
    return (array < 15 ? kAtNodes + array * kNodeArray : kHighAt) + q * 16;
}

__device__ __forceinline__ bool node_ok(uint32_t o) {
    return IMPIR_IN_BOUNDS((o >= kAtNodes && o + 16 <= kTableAt) || (o >= kHighAt && o + 16 <= kAtBits), kSiteBits, o);
}

__device__ __forceinline__ Blk ld_node(uint32_t o) {
    if (!node_ok(o)) return {0, 0, 0, 0};
    const uint4 v = *reinterpret_cast<const uint4*>(smem_at(o));
    return {v.x, v.y, v.z, v.w};
}

__device__ __forceinline__ void st_node(uint32_t o, const Blk v) {
    if (node_ok(o)) *reinterpret_cast<uint4*>(smem_at(o)) = make_uint4(v.x, v.y, v.z, v.w);
}

// Selection bits of a domain smaller than a tile, every leaf by its own walk from the root: lane r
// gets the word of leaves 32 r .. 32 r + 31. Rare (tile 0 of queries below 2^(S + 5) leaves only):
// kept out of line, away from the hot loop's instructions.
__device__ __noinline__ uint32_t small_domain_bits(const FusedParams& P, const uint8_t* kq, uint32_t prf, uint32_t m,
                                                   uint32_t lane, uint32_t L) {
    const uint32_t leaves = 1u << m;
    uint32_t word = 0;
#pragma unroll 1
    for (uint32_t r = 0; r * 32 < leaves; ++r) {
        const uint32_t j = r * 32 + lane;
        Blk n = cw_load(kq, m, 0, 0, 0);
#pragma unroll 1
        for (uint32_t d = 1; d <= m; ++d) {
            const uint32_t x = (j >> (m - d)) & 1u;
            n = child_node(prf, kq, m, n, x, d, L);
        }
        const uint32_t w = __ballot_sync(0xffffffffu, j < leaves && (n.x & 1u));
        if (lane == r) word = w;
    }
    return word;
}

// The left (a) or right (c) child that lane src holds.
__device__ __forceinline__ Blk shfl_child(const Blk& a, const Blk& c, uint32_t src, uint32_t right) {
    const Blk l{__shfl_sync(0xffffffffu, a.x, src), __shfl_sync(0xffffffffu, a.y, src),
                __shfl_sync(0xffffffffu, a.z, src), __shfl_sync(0xffffffffu, a.w, src)};
    const Blk r{__shfl_sync(0xffffffffu, c.x, src), __shfl_sync(0xffffffffu, c.y, src),
                __shfl_sync(0xffffffffu, c.z, src), __shfl_sync(0xffffffffu, c.w, src)};
    return right ? r : l;
}

// One AES task: the selection bits of up to 4 queries of a unit.
__device__ __forceinline__ void aes_task(const FusedParams& P, uint32_t b, uint32_t q0, uint32_t nq,
                                         unsigned long long tile, uint32_t lane, uint32_t L) {
    const uint32_t* query = unit_keys(b);
    Blk a{0, 0, 0, 0}, c{0, 0, 0, 0};
    if ((lane >> 3) < nq) {  // level 3 -> 4 below the tile's node, 8 lanes per query
        const uint32_t q = q0 + (lane >> 3);
        const uint8_t* kq = P.keys + query[q];
        const uint32_t m = kq[2];
        if (m >= LG) {
            const NodePair p = child_nodes(kq[1], kq, m, ld_node(node_at(b, lane & 7, q)), m - LG + 4, L);
            a = p.a;
            c = p.b;
        }
    }
    __syncwarp();
#pragma unroll 1
    for (uint32_t i = 0; i < nq; ++i) {
        const uint32_t q = q0 + i;
        const uint8_t* kq = P.keys + query[q];
        const uint32_t prf = kq[1], m = kq[2];
        uint32_t word = 0;
        if (m >= LG) {
            // lane l's parent at level 4 is node l >> 1: child (l >> 1) & 1 of level-3 node l >> 2
            Blk n = shfl_child(a, c, i * 8 + (lane >> 2), (lane >> 1) & 1);
            if (tile * K + (lane << S) < P.n_records) {
                n = child_node(prf, kq, m, n, lane & 1u, m - S, L);
                word = subtree_bits(prf, kq, m, S, n, L);
            }
            __syncwarp();
        } else {
            // a domain smaller than a tile (tile 0 only): every leaf by its own walk from the root
            word = small_domain_bits(P, kq, prf, m, lane, L);
        }
        const uint32_t o = bits_at(b, q, lane);
        if (smem_ok(o, 4, kAtBits, kAtKey)) *reinterpret_cast<uint32_t*>(smem_at(o)) = word;
    }
}

__device__ __forceinline__ void aes_role(const FusedParams& P, Ctl* ctl, uint32_t lane, uint32_t L) {
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&ctl->task, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        const uint32_t i = t / kTcTasks, k = t % kTcTasks, b = i & 1;
        if (__any_sync(0xffffffffu, !mbar_wait(&ctl->ready[b], (i >> 1) & 1, ctl, 200))) return;
        const UnitDesc u = ctl->unit[b];
        if (u.stop) return;
        const uint32_t q0 = k * kTaskQ;
        if (q0 < u.count) aes_task(P, b, q0, min(kTaskQ, u.count - q0), u.tile, lane, L);
        __syncwarp();
        if (lane == 0) {
            // the fences order the words of all the unit's tasks, through the count, before the one arrival
            __threadfence_block();
            if (atomicAdd(&ctl->done[b], 1u) + 1 == kTcTasks) {
                __threadfence_block();
                mbar_arrive(&ctl->full[b]);
            }
        }
    }
}

// Takes the launch's next unit (the CTA's i-th) and prepares its nodes; all scan threads.
__device__ __forceinline__ void prepare_unit(const FusedParams& P, Ctl* ctl, uint32_t i, uint32_t tid, uint32_t L) {
    const uint32_t b = i & 1;
    if (tid == 0) {
        WsHeader* hdr = reinterpret_cast<WsHeader*>(P.ws);
        const SegDesc* segs = reinterpret_cast<const SegDesc*>(P.ws + P.lay.off_segs);
        UnitDesc d{0, 0, 0, 1, 0};
        const unsigned long long u = atomicAdd(&hdr->tc_counter, 1ull);
        if (u < hdr->tc_units) {
            uint32_t j = 0, n_segs = hdr->tc_segs;
            if (!IMPIR_IN_BOUNDS(n_segs <= kMaxSegments, kSiteSchedule, n_segs)) n_segs = kMaxSegments;
            while (j + 1 < n_segs && segs[j + 1].unit_lo <= u) ++j;
            const SegDesc sg = segs[j];
            const unsigned long long off = u - sg.unit_lo;
            const uint32_t g = uint32_t(off % sg.count), size = (sg.active + sg.count - 1) / sg.count;
            d.tile = sg.tile_lo + off / sg.count;
            d.first = g * size;
            d.count = d.first < sg.active ? min(size, sg.active - d.first) : 0u;
            d.stop = 0;
            if (!IMPIR_IN_BOUNDS(d.count <= kTcQueries && d.first + d.count <= P.n_queries, kSiteSchedule, d.first)) d.count = 0;
        }
        ctl->unit[b] = d;
        ctl->done[b] = 0;
    }
    scan_bar_or(false);
    const UnitDesc d = ctl->unit[b];
    if (tid < d.count) {
        const uint32_t qi = query_at(P, reinterpret_cast<const uint32_t*>(P.ws + P.lay.off_perm) + d.first, tid);
        const uint8_t* kq = query_key(P, qi);
        unit_keys(b)[tid] = uint32_t(kq - P.keys);
        const uint32_t prf = kq[1], m = kq[2];
        if (m >= LG) {
            const uint32_t Dt = m - LG;
            Blk n = cw_load(kq, m, 0, 0, 0);  // R(0,0) = C_0[0][0], Eq. (2)
#pragma unroll 1
            for (uint32_t e = 1; e <= Dt; ++e) {
                n = child_node(prf, kq, m, n, uint32_t(d.tile >> (Dt - e)) & 1u, e, L);
            }
            st_node(node_at(b, 0, tid), n);
            // 3 levels: parents 0 | 1 0 | 3 2 1 0; children 2p, 2p + 1 overwrite only nodes already expanded
#pragma unroll 1
            for (uint32_t e = 1; e < 8; ++e) {
                const uint32_t k = 31 - __clz(int(e)), p = (2u << k) - 1 - e;
                const NodePair c = child_nodes(prf, kq, m, ld_node(node_at(b, p, tid)), Dt + k + 1, L);
                st_node(node_at(b, 2 * p, tid), c.a);
                st_node(node_at(b, 2 * p + 1, tid), c.b);
            }
        }
    }
    mbar_arrive(&ctl->ready[b]);
}

// tcgen05.mma: D (128 lanes x n columns, fp32) = or += A (tensor memory, 128 x 32 bytes) times B
// (shared memory, 32 records x n columns, columns innermost).
__device__ __forceinline__ void mma_f8(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
        "r"(a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(unsigned long long* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem32(b)) : "memory");
}

// The parities of the 128 columns of 16 record bytes (plane i = bits i of the 16 bytes) of this
// thread's query row, as the 16 bytes.
__device__ __forceinline__ uint4 read_parities(uint32_t taddr) {
    // plane i's unit is 2^(e(i) - 9); adding 2^(23 - i) units leaves the count's lowest bit at mantissa bit i
    constexpr int kExp[8] = {-9, -8, -7, -6, -5, -3, 1, 1};
    uint32_t acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0;
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        uint32_t r[32];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
            "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
              "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
              "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
            : "r"(taddr + i * 16));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float magic = __uint_as_float(uint32_t(127 + 23 - (i + e) + kExp[i + e] - 9) << 23);
#pragma unroll
            for (int k = 0; k < 16; ++k)
                acc[k] |= __float_as_uint(__uint_as_float(r[e * 16 + k]) + magic) & (1u << (i + e));
        }
    }
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        w[k] = __byte_perm(__byte_perm(acc[4 * k], acc[4 * k + 1], 0x0040), __byte_perm(acc[4 * k + 2], acc[4 * k + 3], 0x0040), 0x5410);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void scan_role(const FusedParams& P, Ctl* ctl, uint32_t tid, uint32_t L) {
    const uint32_t lane = tid & 31, warp = tid >> 5, W = P.words;
    const uint32_t dcol = ctl->tmem, acol = ctl->tmem + 256, lanes = (warp * 32) << 16;
    uint4* acc_out = P.acc;
    // this thread's place in an operand tile of 64 records x 2 words: record row k (k groups of 8
    // rows: 8 lanes fill 128 contiguous bytes) and word h. Row p = 4 i + j of 32 holds record 8 j + i,
    // the order in which masking a selection word by bytes leaves its bits.
    const uint32_t k = warp * 16 + (lane >> 4) * 8 + (lane & 7), h = (lane >> 3) & 1;
    const uint32_t rec = (k & 32) + (k & 3) * 8 + ((k & 31) >> 2);
    const uint32_t dst = h * 8 * 1024 + (k >> 3) * 128 + (k & 7) * 16;
    uint32_t use = 0, dpar = 0;  // operand tiles used so far; parity of the next dfull phase

    // step i takes the bits of unit i - 2, prepares unit i in the buffers that frees, and scans unit i - 2
#pragma unroll 1
    for (uint32_t i = 0;; ++i) {
        const uint32_t b = i & 1;
        UnitDesc u{0, 0, 0, 0, 0};
        uint32_t qi = 0;
        bool bad = false;
        if (i >= 2) {
            u = ctl->unit[b];
            if (u.stop) return;
            bad = !mbar_wait(&ctl->full[b], ((i - 2) >> 1) & 1, ctl, 1000);
            if (scan_bar_or(bad)) return;
            if (tid < u.count)
                qi = query_at(P, reinterpret_cast<const uint32_t*>(P.ws + P.lay.off_perm) + u.first, tid);
            // selection bits -> operand A: byte 4 i + j of a 32-record chunk is bit 8 j + i of its word
#pragma unroll 1
            for (uint32_t w = 0; w < K / 32; ++w) {
                const uint32_t o = bits_at(b, tid, w);
                const uint32_t s = smem_ok(o, 4, kAtBits, kAtKey) ? *reinterpret_cast<const uint32_t*>(smem_at(o)) : 0u;
                asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(acol + lanes + w * 8),
                             "r"(s & 0x01010101u), "r"((s >> 1) & 0x01010101u), "r"((s >> 2) & 0x01010101u),
                             "r"((s >> 3) & 0x01010101u), "r"((s >> 4) & 0x01010101u), "r"((s >> 5) & 0x01010101u),
                             "r"((s >> 6) & 0x01010101u), "r"((s >> 7) & 0x01010101u)
                             : "memory");
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            scan_bar_or(false);  // operand A complete; bits, nodes and descriptor of this buffer are free
        }
        prepare_unit(P, ctl, i, tid, L);
        if (i < 2) continue;

        const unsigned long long base = u.tile * K;
        const uint32_t nrec = uint32_t(min((unsigned long long)K, P.n_records - base));
        const uint32_t chunks = (nrec + 63) / 64;
        const uint4* src = P.db + (base - P.rec_lo + rec) * W + h;
        // the thread's word of the next chunk (zero past the database or the record); two chunks are in
        // flight ahead of the one being masked, across passes
        uint32_t lw = 0, lc = 0;
        auto load = [&]() {
            if (lc == chunks) lc = 0, lw += 2;
            const uint4 v = (lc * 64 + rec < nrec && lw + h < W) ? ld_db(src + size_t(lc) * 64 * W + lw) : make_uint4(0, 0, 0, 0);
            ++lc;
            return v;
        };
        uint4 v = load(), v1 = load();
#pragma unroll 1
        for (uint32_t w0 = 0; w0 < W; w0 += 2) {
            const bool two = w0 + 1 < W;
            // fp32 accumulators, e4m3 operands, B with its columns innermost, 128 rows
            const uint32_t idesc = (1u << 4) | (1u << 16) | ((two ? 256u : 128u) >> 3 << 17) | ((128u >> 4) << 24);
#pragma unroll 1
            for (uint32_t c = 0; c < chunks; ++c, ++use) {
                const uint4 v2 = load();
                const uint32_t st = use % kStages;
                bad = use >= kStages && !mbar_wait(&ctl->empty[st], ((use / kStages) - 1) & 1, ctl);
                const uint32_t so = kAtStage + st * kStageBytes;
                if (!bad && (two || h == 0) && smem_ok(so + dst + 7 * 1024, 16, kAtStage, kAtNodes)) {
                    uint8_t* o = smem_at(so + dst);
#pragma unroll
                    for (int j = 0; j < 7; ++j) {
                        const uint32_t msk = 0x01010101u << j;
                        *reinterpret_cast<uint4*>(o + j * 1024) = make_uint4(v.x & msk, v.y & msk, v.z & msk, v.w & msk);
                    }
                    const uint32_t msk = 0x40404040u;
                    *reinterpret_cast<uint4*>(o + 7 * 1024) =
                        make_uint4((v.x >> 1) & msk, (v.y >> 1) & msk, (v.z >> 1) & msk, (v.w >> 1) & msk);
                }
                v = v1;
                v1 = v2;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                if (scan_bar_or(bad)) return;
                if (tid == 0) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (uint32_t j = 0; j < 2; ++j) {
                        // 128 B between groups of 8 records, 1024 B between blocks of 16 columns, no swizzle
                        const uint64_t desc = uint64_t(((so + j * 512) >> 4) & 0x3fff) |
                                              (uint64_t(128 >> 4) << 16) | (uint64_t(1024 >> 4) << 32) | (1ull << 46);
                        mma_f8(dcol, acol + (c * 2 + j) * 8, desc, idesc, (c | j) ? 1u : 0u);
                    }
                    mma_commit(&ctl->empty[st]);
                    if (c + 1 == chunks) mma_commit(&ctl->dfull);
                }
            }
            bad = !mbar_wait(&ctl->dfull, dpar, ctl);
            dpar ^= 1;
            if (scan_bar_or(bad)) return;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (uint32_t e = 0; e < (two ? 2u : 1u); ++e) {
                const uint4 r = read_parities(dcol + lanes + e * 128);
                if (tid < u.count) acc_xor(P, acc_out, qi, w0 + e, r);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
    }
}

__global__ void __launch_bounds__(kTcThreads, 1) fused_tc_kernel(const __grid_constant__ FusedParams P) {
    const uint32_t tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
    WsHeader* hdr = reinterpret_cast<WsHeader*>(P.ws);
    const bool tables = fill_tables(P.te0, tid, nthr);
    grid_wait();
    if (hdr->tc_units == 0) return;  // every tile is the warp kernel's
    if (!tables) {
        hdr->timed_out = 1;
        return;
    }
    Ctl* ctl = reinterpret_cast<Ctl*>(smem_at(kAtCtl));
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem32(&ctl->tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
#ifdef IMPIR_BOUNDS
        s_bctx.rec = P.bounds;
        s_bctx.hdr = hdr;
        s_bctx.keys = P.keys;
        s_bctx.keys_bytes = P.keys_bytes;
        s_bctx.db = P.db;
        s_bctx.db_words = P.db_words;
        s_bctx.smem_bytes = P.smem_bytes;
        s_bctx.warp_slice_bytes = 0;
        s_bctx.slices_low = 0;
#endif
        for (int j = 0; j < 2; ++j) {
            mbar_init(&ctl->ready[j], kScanThreads);
            mbar_init(&ctl->full[j], 1);
        }
        for (uint32_t j = 0; j < kStages; ++j) mbar_init(&ctl->empty[j], 1);
        mbar_init(&ctl->dfull, 1);
        ctl->task = 0;
        ctl->abort = 0;
        ctl->wait_ns = P.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = ctl->tmem;

    const uint32_t L = lane_base(lane);
    if (warp < kScanThreads / 32)
        scan_role(P, ctl, tid, L);
    else
        aes_role(P, ctl, lane, L);

    __syncthreads();
    if (ctl->abort && tid == 0) {
        // a wait ran out: give the MMAs in flight time to end before the tensor memory is given back
        const unsigned long long t0 = now_ns();
        while (now_ns() - t0 < 1000 * 1000) {
        }
        atomicExch(&hdr->timed_out, 1u);
    }
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

}  // namespace

uint32_t tc_smem_bytes() { return kTcSmem; }

// The dynamic shared-memory limit belongs to the device: set once per device (a bit per device
// below 64; devices beyond that set it at every call).
cudaError_t prepare_fused_tc() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev >= 0 && dev < 64 ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(fused_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kTcSmem));
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

cudaError_t launch_fused_tc(int sms, cudaStream_t s, const FusedParams& p) {
    const cudaError_t e = prepare_fused_tc();
    if (e != cudaSuccess) return e;
    return launch_after(fused_tc_kernel, dim3(sms), dim3(kTcThreads), kTcSmem, s, p);
}

}  // namespace impir
