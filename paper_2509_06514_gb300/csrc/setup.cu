// setup.cu — per-batch scheduling and answer write-out kernels.
//
// setup_kernel (one CTA) reads the key headers on the device, validates them, sorts the
// queries by domain size (largest first), forms query groups (the paper's queries handled
// together, §3.4), and builds the tile-major work-unit schedule the fused kernels walk (schedule.h).
// It also zeroes the per-query accumulators and the work counters.
//
// finalize_kernel copies each query's accumulator (record stride) into the caller's
// answer buffer (record_bytes per query) where the answers were not accumulated there.
#include <algorithm>
#include <cstdlib>

#include "bounds.cuh"
#include "impir_internal.h"
#include "launch.cuh"
#include "schedule.h"

namespace impir {

#ifdef IMPIR_BOUNDS
// The per-device record of failed index checks (debug build).
static __device__ BoundsRecord g_bounds_rec;
#endif

__global__ void __launch_bounds__(1024) setup_kernel(const SetupParams S) {
    __shared__ uint32_t hist[kMaxDomainBits + 1], cursor[kMaxDomainBits + 1];
    __shared__ uint32_t bstart[kMaxDomainBits + 1], gstart[kMaxDomainBits + 1], ngrp[kMaxDomainBits + 1];
    __shared__ uint32_t s_nbad, s_first_bad, s_ngroups;
    __shared__ unsigned long long s_present;  // bit m: some query has domain bits m
    const uint32_t tid = threadIdx.x, nthr = blockDim.x;
    grid_launch_next();
    WsHeader* hdr = reinterpret_cast<WsHeader*>(S.ws);
    uint32_t* perm = reinterpret_cast<uint32_t*>(S.ws + S.lay.off_perm);
    uint32_t* qm = reinterpret_cast<uint32_t*>(S.ws + S.lay.off_qm);
    GroupDesc* groups = reinterpret_cast<GroupDesc*>(S.ws + S.lay.off_groups);
    SegDesc* segs = reinterpret_cast<SegDesc*>(S.ws + S.lay.off_segs);
    uint4* acc = S.acc;

    if (tid <= kMaxDomainBits) hist[tid] = cursor[tid] = 0;
    if (tid == 0) {
        s_nbad = 0;
        s_first_bad = 0xffffffffu;
        hdr->bounds_failed = 0;
        if (!S.keep_status) hdr->timed_out = 0;
#ifdef IMPIR_BOUNDS
        s_bctx = BoundsCtx{S.bounds, hdr, S.keys, S.keys_bytes, nullptr, 0, 0, 0, 0};
#endif
    }
    __syncthreads();

    // 1. validate each key's header and column 0 (a1 key intake)
    for (uint32_t q = tid; q < S.n_queries; q += nthr) {
        const uint32_t off = S.key_off[q];
        bool ok = (off & 7u) == 0;
        uint32_t m = 0;
        if (ok && !IMPIR_IN_BOUNDS(S.keys_bytes == 0 || off + 8ull <= S.keys_bytes, kSiteKey, off)) ok = false;
        if (ok) {
            const uint8_t* k = S.keys + off;
            const uint2 h = *reinterpret_cast<const uint2*>(k);
            const uint32_t ver = h.x & 0xffu, prf = (h.x >> 8) & 0xffu;
            m = (h.x >> 16) & 0xffu;
            ok = ver == 1 && prf <= 1 && m >= 1 && m <= kMaxDomainBits && (h.x >> 24) <= 1 && h.y == 0;
            if (ok) {
                const size_t z[3] = {8 + size_t(m + 1) * 16, 8 + size_t(m + 1) * 32, 8 + size_t(m + 1) * 48};
                for (int i = 0; i < 3; ++i) {
                    if (!IMPIR_IN_BOUNDS(S.keys_bytes == 0 || off + z[i] + 16 <= S.keys_bytes, kSiteKey, off + z[i])) {
                        ok = false;
                        break;
                    }
                    const uint2* p = reinterpret_cast<const uint2*>(k + z[i]);
                    const uint2 a = p[0], b = p[1];
                    ok = ok && (a.x | a.y | b.x | b.y) == 0;
                }
            }
        }
        qm[q] = ok ? m : 0;
        if (ok) {
            atomicAdd(&hist[m], 1u);
        } else {
            atomicAdd(&s_nbad, 1u);
            atomicMin(&s_first_bad, q);
        }
    }
    __syncthreads();

    if (tid < 32) {
        const uint32_t lo = __ballot_sync(0xffffffffu, hist[tid] != 0);
        const uint32_t hi = __ballot_sync(0xffffffffu, tid + 32 <= kMaxDomainBits && hist[min(tid + 32, kMaxDomainBits)] != 0);
        if (tid == 0) s_present = lo | (unsigned long long)hi << 32;
    }
    __syncthreads();

    // 2. the schedule. One thread, over the domain sizes that occur.
    if (tid == 0) {
        s_ngroups = make_schedule(S, s_present, hist, bstart, gstart, ngrp, segs, hdr);
        hdr->n_bad = s_nbad;
        hdr->first_bad = s_first_bad;
    }
    __syncthreads();

    // 3. scatter queries into their buckets (order inside a bucket does not matter: XOR
    //    answers are independent of which queries share a group)
    for (uint32_t q = tid; q < S.n_queries; q += nthr) {
        const uint32_t m = qm[q];
        if (m) {
            const uint32_t i = bstart[m] + atomicAdd(&cursor[m], 1u);
            if (IMPIR_IN_BOUNDS(i < S.n_queries, kSiteWorkspace, i)) perm[i] = q;
        }
    }
    // 4. group descriptors (the tensor-core kernel takes its groups from the sorted list itself)
    for (uint32_t gi = tid; gi < s_ngroups; gi += nthr) {
        uint32_t m = 0;
        for (unsigned long long p = s_present; p; p &= p - 1) {
            const uint32_t k = uint32_t(__ffsll((long long)p) - 1);
            if (gi >= gstart[k] && gi < gstart[k] + ngrp[k]) m = k;
        }
        const uint32_t k = gi - gstart[m];
        GroupDesc d;
        d.first = bstart[m] + k * S.qpw;
        d.count = min(S.qpw, hist[m] - k * S.qpw);
        d.m = m;
        d.pad = 0;
        if (IMPIR_IN_BOUNDS(gi < S.n_queries + kMaxDomainBits + 8, kSiteWorkspace, gi)) groups[gi] = d;
    }
    // 5. zero the accumulators (kept across the chunks of a streamed database)
    if (!S.keep_acc) {
        const size_t nacc = size_t(S.n_queries) * S.words;
        for (size_t i = tid; i < nacc; i += nthr) acc[i] = make_uint4(0, 0, 0, 0);
    }
}

__global__ void finalize_kernel(const FinalizeParams F) {
    grid_wait();
#ifdef IMPIR_BOUNDS
    if (threadIdx.x == 0) s_bctx = BoundsCtx{F.bounds, nullptr, nullptr, 0, nullptr, 0, 0, 0, 0};
    __syncthreads();
#endif
    const uint8_t* acc = F.ws + F.lay.off_acc;
    const size_t n = size_t(F.n_queries) * F.record_bytes;
    for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
        const size_t q = i / F.record_bytes, b = i - q * F.record_bytes;
        const size_t a = q * F.stride + b;
        if (IMPIR_IN_BOUNDS(b < F.stride && a < size_t(F.n_queries) * F.stride, kSiteAcc, a)) F.out[i] = acc[a];
    }
}

BoundsRecord* bounds_record() {
#ifdef IMPIR_BOUNDS
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_bounds_rec) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return static_cast<BoundsRecord*>(p);
#else
    return nullptr;
#endif
}

unsigned long long bounds_db_words(unsigned long long n_words, uint32_t words_per_record) {
#ifdef IMPIR_BOUNDS
    // a debug-build test withholds the last records of every database from the checked extent
    // (the memory stays valid), so that the checks on record reads fire
    if (const char* w = std::getenv("IMPIR_BOUNDS_TEST_WITHHOLD_RECORDS")) {
        const unsigned long long k = std::strtoull(w, nullptr, 10) * words_per_record;
        return k < n_words ? n_words - k : 0;
    }
#else
    (void)words_per_record;
#endif
    return n_words;
}

const uint32_t* bounds_te0(const uint32_t* te0) {
#ifdef IMPIR_BOUNDS
    if (std::getenv("IMPIR_BOUNDS_TEST_NO_TABLES")) return nullptr;
#endif
    return te0;
}

unsigned long long wait_limit_ns() {
#ifdef IMPIR_BOUNDS
    if (const char* w = std::getenv("IMPIR_BOUNDS_TEST_WAIT_NS")) return std::strtoull(w, nullptr, 10);
#endif
    return 20ull * 1000 * 1000 * 1000;
}

cudaError_t launch_setup(const SetupParams& p, cudaStream_t s) {
    // one CTA, no larger than the queries and accumulator words it has to pass over
    const size_t work = std::max(size_t(p.n_queries), p.keep_acc ? size_t(0) : size_t(p.n_queries) * p.words / 4);
    setup_kernel<<<1, unsigned(std::min(size_t(1024), std::max(size_t(128), (work + 31) / 32 * 32))), 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalizeParams& p, cudaStream_t s, bool follows) {
    const size_t n = size_t(p.n_queries) * p.record_bytes;
    const unsigned blocks = unsigned(n / 256 + 1 < 1024 ? n / 256 + 1 : 1024);
    if (follows) return launch_after(finalize_kernel, dim3(blocks), dim3(256), 0, s, p);
    finalize_kernel<<<blocks, 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_fused(uint32_t qpw, uint32_t nk, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                         const FusedParams& p) {
    switch (qpw) {
        case 1: return launch_fused_q1(nk, grid, block, smem, s, p);
        case 2: return launch_fused_q2(nk, grid, block, smem, s, p);
        case 4: return launch_fused_q4(nk, grid, block, smem, s, p);
        case 8: return launch_fused_q8(nk, grid, block, smem, s, p);
        case 16: return launch_fused_q16(nk, grid, block, smem, s, p);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_xor(const XorShape& s, int sms, cudaStream_t st, FusedParams& fp) {
    // The warp kernel's share, often none, goes first: behind the tensor-core kernel it would wait for an
    // SM while another stream's launch fills the chip (a streamed database's next chunk, another batch of
    // a server), and with it everything that waits for this batch: 416 uneven queries on 8 GiB streamed
    // in 2 GiB chunks 302-308 ms behind it, 286 before it.
    fp.with_tc = s.tc ? 1u : 0u;
    fp.bits_words = bits_words(s.c);
    const SmemSplit sp = split_smem(s.c.warps_per_cta, size_t(s.c.queries_per_warp) * fp.bits_words * 4);
    fp.slices_low = sp.low;
    fp.smem_bytes = sp.bytes;
    const cudaError_t e = launch_fused(s.c.queries_per_warp, nk_xor(fp.words, s.c.queries_per_warp), dim3(sms),
                                       dim3(sp.warps * 32), sp.bytes, st, fp);
    if (e != cudaSuccess || !s.tc) return e;
    fp.smem_bytes = tc_smem_bytes();
    fp.wait_ns = wait_limit_ns();
    return launch_fused_tc(sms, st, fp);
}

cudaError_t prepare_xor_kernels() {
    cudaError_t e = prepare_fused_q1();
    if (e == cudaSuccess) e = prepare_fused_tc();
    if (e == cudaSuccess) e = prepare_fused_q2();
    if (e == cudaSuccess) e = prepare_fused_q4();
    if (e == cudaSuccess) e = prepare_fused_q8();
    if (e == cudaSuccess) e = prepare_fused_q16();
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, setup_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, finalize_kernel);
    return e;
}

}  // namespace impir
