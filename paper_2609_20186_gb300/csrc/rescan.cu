// rescan.cu -- the rescan kernel: switchsd_step / switchsd_verify_step / switchsd_verify_sampled_step and the
// candidate entry points, with the linear probe (Eq. 3) or the two-layer probe's finish, laid out for a
// short chain of dependent phases after the grid-dependency wait.
//
// Paper: §3.3 (kappa-gram gate, recency-ranked copy candidates, Eq. 4 decision rule, parallel
// verification), Eq. 3 (linear probe), Fig. 1 (three cases).
//
// Row b is handled by a cluster of C CTAs of kRescanThreads threads (grid = C x B).  The row's old
// candidate ends [0, L_old - 1) are split into C contiguous 16-byte-aligned ranges; each CTA stages its
// range (plus kHalo tokens of look-back and kFwd of look-ahead) with one bulk copy, and the row's last
// kHalo tokens with another, as soon as it has read the row length -- before the grid-dependency wait
// when the caller allows it -- and, in the hash instance, warps 1.. hash every staged old end into one
// byte once the copy lands.  The CTAs are small (four warps, at most 64 registers a thread) so that the
// next launch's CTAs are resident, with their copies in flight, while this launch finishes.
//
// After the wait no cluster-wide barrier is on the path, and no CTA-wide one outside candidate mode
// (the hash instance's barrier on the hash bytes completes before the wait when the context is
// prefetched):
//  * every warp verifies the previous draft itself (the draft and the target are a few L2 lines), and
//    keeps its own window of the row's last kHalo old tokens followed by the appended tokens: the new
//    suffix and the appended positions come from it, so the staged tile is never patched;
//  * every warp scans its share of the CTA's old ends (a hash filter on the last F tokens -- computed
//    from the tokens, or the pre-wait hash bytes -- then an exact test and a backward compare against
//    its suffix window), and the leader's warp 0 also tests the a+1 ends the append creates;
//  * every warp ships its best key, its share of the probe's dot product and its best match's
//    continuation (from the staged tile, or from its window past the old length) to the row's leader CTA
//    (the last one) with asynchronous DSMEM stores completing on the leader's mbarrier, and is done.
// The leader's warp 0 writes the appended tokens, waits (bounded) for the C x kRescanWarps messages, reduces
// them in a fixed order and writes the outputs and the new length.  The only cluster barrier is arrived on
// right after the length read and waited on beside the verification's loads, so the leader's message barrier
// is initialised before anyone ships to it; the messages order every read of the length before its rewrite.
#include <mutex>
#include <type_traits>

#include "mlp.cuh"
#include "step.cuh"

namespace switchsd {

// Per-warp window of y = old context followed by the append: s_y[w][j] = y[L_old - kHalo + j].
constexpr int kYLen = kHalo + SWITCHSD_KMAX + 4;
// 32-bit match keys: m << kKeyShift | e with m <= SWITCHSD_NMAX (bits 25..30) and e < 2^25; bit 31 alone
// marks a copy that did not land.
constexpr int kKeyShift = 25;
constexpr uint32_t kKeyEndMask = (1u << kKeyShift) - 1u;
constexpr uint32_t kKeyTimeout = 1u << 31;
static_assert(SWITCHSD_NMAX < (1 << (31 - kKeyShift)), "m must fit below the timeout bit");
static_assert(SWITCHSD_WMAX * SWITCHSD_KMAX <= 1024 && SWITCHSD_KMAX <= 64, "the candidates' division by D");
// The scan: kScanWords words per thread per round; a thread's words of a CTA range fit the 32 bits of its
// pass mask.
constexpr int kScanWords = 4;
static_assert(kRescanTileMax / 4 / kRescanThreads <= 32, "a thread's words fit its pass mask");

// The scan of a CTA's old ends [e_lo, e_end) against the new suffix (suf[-q] = its q-th token from the end)
// for the longest-then-most-recent match: the largest key m << kKeyShift | e over the ends with
// m(e) >= n_min, 0 if none.  stage[kHalo + p - e_lo] = x[p] over [e_lo - kHalo, e_end + kFwd).
//
// Filter depth F = min(n_min, 3): end e can match only if its last F tokens equal the suffix's.  Pass 1
// tests a hash of them, h(e) = x[e] + x[e-1] A + x[e-2] B (the first F terms, mod 2^32), against the
// suffix's: equal tokens give equal hashes, so no end that matches is missed, and the few that collide
// are dropped by pass 2's exact test.  Two multiply-adds per end and two mins a word of four ends; the
// shared-memory reads, not the arithmetic, set the pace.
//
// Pass 1: rounds of kScanWords words per thread (word tid + i kT for i = 0, 1, ...: consecutive lanes read
// consecutive words), each with the two tokens before it (unset before position 0, where lim < F drops the
// end); a word with an end that passes sets bit i.  No branch and no backward compare in the hot loop.
// Pass 2 (rare): the words that passed, in warp-synchronous steps (each step every lane with a word left
// takes its next one, so the compares of a hot suffix run side by side), reloaded from shared memory;
// their ends that pass the exact test (x[e-i] = suf[-i] for i < F) take the backward compare from m = F,
// eight positions per step with independent loads.  (A bit a round of four words instead made every step
// of pass 2 test sixteen ends: 16 launches on the 32K rows 73.6 us against 69.7 us, 8 on the 128K rows 46.3
// against 43.2 us.)
constexpr uint32_t kHashA = 0x9E3779B1u, kHashB = 0x85EBCA77u;  // odd multipliers

// The F-token hash of end e (x0 = x[e], x1 = x[e-1], x2 = x[e-2]; the first F terms, mod 2^32).
template <int F>
__device__ __forceinline__ uint32_t end_hash(int32_t x0, int32_t x1, int32_t x2) {
    uint32_t h = uint32_t(x0);
    if (F >= 2) h += uint32_t(x1) * kHashA;
    if (F >= 3) h += uint32_t(x2) * kHashB;
    return h;
}
// One byte of it for the pre-wait table (multiplicative: the top byte of an odd multiple).
__device__ __forceinline__ uint32_t hash_byte(uint32_t h) { return (h * 0x2C1B3C6Du) >> 24; }
// Nonzero iff some byte of v is zero (exact as a whole-word test).
__device__ __forceinline__ uint32_t has_zero_byte(uint32_t v) { return (v - 0x01010101u) & ~v & 0x80808080u; }

// Pre-wait hashing: hb[g] holds the hash bytes of the ends e_lo + 4g .. + 3 (byte j = end e_lo + 4g + j),
// for the words g < n4 of this CTA's old ends; threads t, t + nt, ... of the caller take one word each.
template <int F>
__device__ __forceinline__ void hash_ends(const int32_t *stage, uint32_t *hb, int32_t n4, int t, int nt) {
    const int4 *g4 = reinterpret_cast<const int4 *>(stage + kHalo);
    for (int32_t g = t; g < n4; g += nt) {
        const int4 v = g4[g];
        const int2 pv = F >= 2 ? *reinterpret_cast<const int2 *>(stage + kHalo + 4 * g - 2) : make_int2(0, 0);
        hb[g] = hash_byte(end_hash<F>(v.x, pv.y, pv.x)) | hash_byte(end_hash<F>(v.y, v.x, pv.y)) << 8 |
                hash_byte(end_hash<F>(v.z, v.y, v.x)) << 16 | hash_byte(end_hash<F>(v.w, v.z, v.y)) << 24;
    }
}

//
// Candidate mode (kCand): every end whose common suffix reaches kappa_c is also marked in the CTA's bitmap
// bm (bit e - e_lo; F <= kappa_c, so the filter passes every such end).
//
// kPre: the hashes were taken before the grid-dependency wait (hash_ends into hb); pass 1 then compares
// one byte per end against the suffix's (four ends a 4-byte load), and pass 2 takes only the ends whose
// byte matches.  The byte filter passes every end that matches and about 1 in 256 of the others, which
// the exact test drops.
//
// The key holds e - key0, the bitmap starts at end bm_lo (a ring of tiles scans one tile at a time: e_lo is
// then the tile's first end).
template <int F, bool kCand, bool kPre>
__device__ __forceinline__ uint32_t scan_ends(const int32_t *stage, int32_t e_lo, int32_t e_end, const int32_t *suf,
                                              int32_t n_min, int32_t n_max, int tid, int lane, uint32_t *bm,
                                              int32_t kappa_c, const uint32_t *hb, int32_t key0, int32_t bm_lo,
                                              bool *marked) {
    const int32_t s0 = suf[0], s1 = F >= 2 ? suf[-1] : 0, s2 = F >= 3 ? suf[-2] : 0;
    const uint32_t hs = end_hash<F>(s0, s1, s2);
    const uint32_t hs4 = hash_byte(hs) * 0x01010101u;
    const int32_t n4 = (e_end - e_lo + 3) >> 2;
    const int4 *g4 = reinterpret_cast<const int4 *>(stage + kHalo);
    const int32_t off = kHalo - e_lo;
    constexpr int kWords = kPre ? 2 * kScanWords : kScanWords;  // a round's words a thread: 4-byte or 16-byte loads
    uint32_t passed = 0u;  // bit i: word tid + i * kRescanThreads holds an end that passes
    int rnd = 0;
    int32_t g0 = tid;
    // One round: words g0, g0 + kT, ...; kAll: every lane's words lie in the range (the hot rounds: no
    // predicates, one base address), else the words past it read as no match.
    auto round = [&](auto all) {
        constexpr bool kAll = decltype(all)::value;
        uint32_t hit = 0u;
        if constexpr (kPre) {
            const uint32_t *w = hb + g0;
#pragma unroll
            for (int u = 0; u < kWords; ++u)
                if ((kAll || g0 + u * kRescanThreads < n4) && has_zero_byte(w[u * kRescanThreads] ^ hs4) != 0u) hit |= 1u << u;
        } else {
            const int4 *w = g4 + g0;
            int4 v[kWords];
            int2 pv[kWords];  // x[4g - 2], x[4g - 1]
#pragma unroll
            for (int u = 0; u < kWords; ++u) {
                const bool in = kAll || g0 + u * kRescanThreads < n4;
                v[u] = in ? w[u * kRescanThreads] : make_int4(0, 0, 0, 0);
                pv[u] = (F >= 2 && in) ? reinterpret_cast<const int2 *>(w + u * kRescanThreads)[-1] : make_int2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < kWords; ++u) {
                const uint32_t h0 = end_hash<F>(v[u].x, pv[u].y, pv[u].x), h1 = end_hash<F>(v[u].y, v[u].x, pv[u].y);
                const uint32_t h2 = end_hash<F>(v[u].z, v[u].y, v[u].x), h3 = end_hash<F>(v[u].w, v[u].z, v[u].y);
                if ((h0 == hs) | (h1 == hs) | (h2 == hs) | (h3 == hs)) hit |= 1u << u;
            }
        }
        passed |= hit << (rnd & 31);
        g0 += kWords * kRescanThreads;
        rnd += kWords;
    };
    while (g0 - lane + (kWords - 1) * kRescanThreads + kWarp <= n4) round(std::true_type{});
    while (g0 - lane < n4) round(std::false_type{});
    uint32_t mine = 0u;
    // m(e) from F for an end whose last F tokens match: x[e - q] against suf[-q], eight positions per step,
    // every load issued unconditionally (q clamped to lim - 1; the sentinel bit ends the run at the count).  With
    // n_min = 1 every end of the suffix's last token comes here, up to a seventh of a Zipf text, and most differ in
    // the token before: that one is compared first (a launch, without and with: 60 rows of 34K tokens 7.69 and 6.31
    // us, 10 of 159K 13.99 and 11.79, 29 of 292K 37.5 and 29.5; rare last tokens +2 %).
    auto match_len = [&](int32_t e, int32_t lim) {
        int32_t m = F;
        if (F == 1 && lim > 1 && stage[off + e - 1] != suf[-1]) return m;
#pragma unroll 1
        while (m < lim) {
            const int32_t cnt = min(8, lim - m);
            unsigned miss = 1u << cnt;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int32_t q = min(m + i, lim - 1);
                miss |= unsigned(stage[off + e - q] != suf[-q]) << i;
            }
            const int32_t run = __ffs(miss) - 1;
            m += run;
            if (run < cnt) break;
        }
        return m;
    };
    auto take = [&](int32_t e, int32_t m) {
        if (m >= n_min) {
            const uint32_t key = (uint32_t(m) << kKeyShift) | uint32_t(e - key0);
            mine = key > mine ? key : mine;
        }
        if (kCand && m >= kappa_c) {
            atomicOr(&bm[(e - bm_lo) >> 5], 1u << ((e - bm_lo) & 31));
            *marked = true;
        }
    };
    while (__any_sync(kFull, passed != 0u)) {
        if (passed == 0u) continue;
        const int32_t g = tid + (__ffs(passed) - 1) * kRescanThreads;
        passed &= passed - 1u;
        if (g >= n4) continue;  // (a lane past the range read zeros)
        if constexpr (kPre) {
            // the word's ends whose hash byte matches: the lowest byte flagged is an exact match, and is then
            // made nonzero
            uint32_t x = hb[g] ^ hs4;
            for (uint32_t z = has_zero_byte(x); z != 0u; z = has_zero_byte(x)) {
                const int j = (__ffs(z) - 1) >> 3;
                x |= 1u << (8 * j);
                const int32_t e = e_lo + 4 * g + j;
                if (e >= e_end) break;
                const int32_t lim = min(n_max, e + 1);
                const int32_t x0 = stage[off + e], x1 = F >= 2 ? stage[off + e - 1] : s1, x2 = F >= 3 ? stage[off + e - 2] : s2;
                // (lim < F: the hash read a token before position 0)
                if (((x0 ^ s0) | (x1 ^ s1) | (x2 ^ s2)) == 0 && lim >= F) take(e, match_len(e, lim));
            }
        } else {
            const int4 v = g4[g];
            const int2 pv = *reinterpret_cast<const int2 *>(stage + kHalo + 4 * g - 2);
            // exact test of the last F tokens of each end
            const int32_t x[6] = {pv.x, pv.y, v.x, v.y, v.z, v.w};
            uint32_t hall = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                bool ok = x[j + 2] == s0;
                if (F >= 2) ok = ok && x[j + 1] == s1;
                if (F >= 3) ok = ok && x[j] == s2;
                hall |= uint32_t(ok) << j;
            }
            while (hall) {
                const int j = __ffs(hall) - 1;
                hall &= hall - 1;
                const int32_t e = e_lo + 4 * g + j;
                if (e >= e_end) break;
                const int32_t lim = min(n_max, e + 1);
                if (lim < F) continue;  // the test read a token before position 0
                take(e, match_len(e, lim));
            }
        }
    }
    return mine;
}

constexpr int kVerifyLoads = 4;  // candidate verification: staging loads a thread has in flight at once

// Candidate mode's shared memory beyond the single-draft layout: per CTA one candidate message of cslot
// bytes -- a 16-byte header (count), the ends (W, most recent first), their continuations [W][D] (not from
// a ring, whose tiles are gone by then: the leader reads them from the row) -- the
// leader receiving C of them and every CTA staging its own; a bitmap of the CTA's marked ends; the
// verification's staging of the previous candidates (drafts [W][D], targets [W][D+1]).
struct CandLayout {
    uint32_t cslot;  // bytes of a candidate message
    int bm_words;    // bitmap words (a multiple of 4)
    int v_ints;      // verification staging (a multiple of 4)
};
__host__ __device__ inline CandLayout cand_layout(int range, int W, int D, bool ring) {
    CandLayout c;
    c.cslot = 16u * uint32_t(1 + (W + 3) / 4 + (ring ? 0 : (W * D + 3) / 4));
    c.bm_words = ((range + 31) / 32 + 3) & ~3;
    c.v_ints = (W * D + W * (D + 1) + 3) & ~3;
    return c;
}

// kScan: how a CTA's old ends are staged and scanned -- one copy, filtered on the tokens (kScanTokens) or on
// the pre-wait hash bytes (kScanHashed, a.hash_words > 0); or, for ranges above kRescanTileMax ends, a ring
// of a.stages tiles filtered on the tokens (kScanRing).  kMlp: the two-layer probe's finish (a.z1_part set).
// Separate instances, so that each carries only its own scan and its own probe code and registers.
//
// The ring: every warp scans its share of each tile as it lands, keeps its best match's continuation while
// that tile is staged, and counts itself out of the stage; the last warp out refills it.  No CTA barrier and
// no producer warp: the warps drift by up to the ring's depth.  Its CTAs are sized for rows that stream from memory, a
// few warps an SM; where the compares weigh more than the stream -- n_min = 1 and a last token that fills a seventh
// of the row -- a ring of 256-thread CTAs, 16 a row, was faster (29 rows of 292K Zipf tokens 18.4 us a launch, 29.4 here;
// 33 rows of random ids 16.3 and 7.2).
enum { kScanTokens = 0, kScanHashed = 1, kScanRing = 2 };
template <bool kSampled, bool kCand, int kScan, bool kMlp>
__global__ void __launch_bounds__(kRescanThreads, kScan == kScanRing ? kRingLaunchBlocks : kRescanLaunchBlocks)
    rescan_kernel(const StepArgs a) {
    constexpr bool kPre = kScan == kScanHashed, kRing = kScan == kScanRing;
    extern __shared__ __align__(128) int32_t dsm[];
    __shared__ __align__(8) uint64_t ring[kRing ? kRingStages : 1];  // a tile of the ring landed
    __shared__ int s_out_of[kRing ? kRingStages : 1];                // warps done with a stage, counted on and on
    __shared__ __align__(8) uint64_t bars[5];              // tile, tail, probe slices, messages (leader),
                                                           // pre-wait hashes
    __shared__ __align__(16) int32_t s_tail[kHalo + 8];    // x[tail_lo .. L_old), tail_lo = roundown4(L_old - kHalo)
    __shared__ int32_t s_y[kRescanWarps][kYLen];
    __shared__ int32_t s_sel[kMaxCand];                    // candidate mode: the CTA's selected ends / the
                                                           // leader's merged candidates' sources
    __shared__ int32_t s_wtot[kRescanWarps];               // candidate mode: marks per warp in a pass
    __shared__ int32_t s_miss[kMaxCand];                   // candidate mode: the first position of each previous
                                                           // candidate that differs from the target

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();
    const uint32_t C = cluster_nctarank();
    const uint32_t lead = C - 1;
    const int b = blockIdx.y;
    const int stage_ints = kHalo + a.tile + kFwd;
    int32_t *stage = dsm;
    uint32_t *hb = reinterpret_cast<uint32_t *>(dsm + (kRing ? a.stages : 1) * ((stage_ints + 3) & ~3));  // [hash_words]
    uint4 *s_pw = reinterpret_cast<uint4 *>(hb + a.hash_words);
    uint4 *s_ph = s_pw + a.probe_words;
    unsigned char *msgs = reinterpret_cast<unsigned char *>(s_ph + a.probe_words);
    const bool verifying = a.pv_len != nullptr;
    const int kw = kCand ? 0 : (a.k + 3) >> 2;             // 16-byte words of a message's continuation
    const uint32_t slot_bytes = 16u * uint32_t(1 + kw);
    const int nmsg = int(C) * kRescanWarps;
    const CandLayout cl = cand_layout(kCand ? a.range : 0, kCand ? a.W : 0, kCand ? a.D : 0, kRing);
    unsigned char *cmsgs = msgs + size_t(nmsg) * slot_bytes;                  // [C][cslot] (leader)
    unsigned char *cstage = cmsgs + size_t(C) * cl.cslot;                     // this CTA's message
    uint32_t *bm = reinterpret_cast<uint32_t *>(cstage + cl.cslot);           // [bm_words]
    int32_t *vc = reinterpret_cast<int32_t *>(bm + cl.bm_words);              // previous drafts [W][D]
    int32_t *vt = vc + a.W * a.D;                                             // their targets [W][D+1]

    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_init(&bars[2], 1);
        mbar_init(&bars[4], kRescanThreads - kWarp);
        if (kRing)
            for (int s = 0; s < a.stages; ++s) {
                mbar_init(&ring[s], 1);
                s_out_of[s] = 0;
            }
        if (rank == lead) {
            mbar_init(&bars[3], 1);
            mbar_arrive_expect_tx(&bars[3], slot_bytes * uint32_t(nmsg) + (kCand ? cl.cslot * C : 0u));
        }
        fence_mbar_init();
    }
    // Candidate mode: i / D for i < W D <= 1024 as (i inv_d) >> 16 (inv_d D - 2^16 < 64, so the error term stays
    // below 2^16): the divisions leave the chain after the wait.
    const uint32_t inv_d = kCand ? (65536u + uint32_t(a.D) - 1u) / uint32_t(a.D) : 0u;
    auto over_d = [&](int i) { return int((uint32_t(i) * inv_d) >> 16); };
    if (kCand) {
        for (int i = tid; i < cl.bm_words; i += kRescanThreads) bm[i] = 0u;
        if (tid < kMaxCand) s_miss[tid] = SWITCHSD_KMAX;
    }
    __syncthreads();  // the barriers are initialised (and the bitmap cleared) before any thread uses them

    const bool pf_ctx = (a.prefetch & SWITCHSD_PREFETCH_CONTEXT) != 0;
    const bool gather = verifying && a.hidden_rows > 1;
    // Two-layer probe: the first layer's split-K partial sums come from the probe kernel just before this
    // one (read after the wait); this CTA finishes units [u0, u1) (b1, ReLU, w2).
    constexpr bool mlp = kMlp;
    const bool pf_probe = (a.prefetch & SWITCHSD_PREFETCH_PROBE) != 0 && !gather && !mlp;
    // Two-layer probe: every input but the partial sums was written by kernels that completed before the
    // first-layer kernel released this launch (it does so only after its own wait), so verification and
    // scan run while it computes; the warps wait just before reading the sums.  Reads before that wait
    // go through L2 (bulk copies, ld.global.cg).
    const bool late = mlp && a.wait_late != 0;
    if (!pf_ctx && !late) pdl_wait();
    int32_t *row = a.ctx + size_t(b) * size_t(a.cap);
    // The CTA's ends are split on the row's old length, or, with a length bound, on the bound: its tile
    // copy then leaves before the length is read, and a row longer than the bound is a bad length.
    const bool bounded = a.len_bound > 0;
    auto range_of = [&](int32_t E, int32_t &e_lo_, int32_t &e_hi_) {
        int32_t chunk = (E + int32_t(C) - 1) / int32_t(C);
        chunk = (chunk + 3) & ~3;
        e_lo_ = min(E, int32_t(rank) * chunk);
        e_hi_ = min(E, e_lo_ + chunk);
    };
    int32_t e_lo = 0, e_hi = 0, lo = 0;
    if (bounded) {
        range_of(a.len_bound - 1, e_lo, e_hi);
        lo = max(0, e_lo - kHalo);
    }
    auto tile_hi = [&]() { return e_hi > e_lo ? min((e_hi + kFwd + 3) & ~3, a.cap) : lo; };
    const uint64_t pol = l2_evict_first_policy();
    // Ring: tile t of the range (ends [t0, t0 + a.tile)) into stage s = t mod a.stages, x[p] at [kHalo + p - t0].
    auto issue_ring = [&](int t, int s) {
        const int32_t t0 = e_lo + t * a.tile, t1 = min(e_hi, t0 + a.tile);
        const int32_t lo_t = max(0, t0 - kHalo), hi_t = min((t1 + kFwd + 3) & ~3, a.cap);
        const uint32_t bytes = uint32_t(hi_t - lo_t) * 4u;
        mbar_expect_tx_relaxed(&ring[s], bytes);
        bulk_g2s_hint(stage + s * stage_ints + (kHalo + lo_t - t0), row + lo_t, bytes, &ring[s], pol);
    };
    auto ring_tiles = [&]() { return e_hi > e_lo ? (e_hi - e_lo - 1) / a.tile + 1 : 0; };
    auto issue_tile = [&](int32_t hi_) {  // positions [lo, hi_) land at stage[kHalo + p - e_lo]
        if (kRing) {
            for (int t = 0; t < min(ring_tiles(), a.stages); ++t) issue_ring(t, t);
            return;
        }
        const uint32_t bytes = uint32_t(hi_ - lo) * 4u;
        mbar_expect_tx_relaxed(&bars[0], bytes);
        if (bytes > 0) bulk_g2s_hint(stage + (kHalo + lo - e_lo), row + lo, bytes, &bars[0], pol);
    };
    if (bounded && tid == 0) issue_tile(tile_hi());
    // The verification's inputs (lane i: positions i and i + 32) are loaded as soon as the wait allows -- before
    // the length when that is read after the wait too, so that the two round trips overlap (8 launches on 37
    // ragged rows of 9K tokens: 38.9 -> 37.6 us).
    int32_t pv_n = 0, d_lo = 0, d_hi = 0, t_lo = 0, t_hi = 0, t_top = 0;
    float pv_lo[3] = {0.f, 1.f, 0.f}, pv_hi[3] = {0.f, 1.f, 0.f};  // sampled: u, q, p
    auto load_draft = [&]() {
        if (kCand || !verifying) return;
        const int32_t *dr = a.pv_draft + size_t(b) * a.k;
        const int32_t *tg = a.pv_target + size_t(b) * (a.k + 1);
        pv_n = __ldcg(a.pv_len + b);
        if (lane < a.k) d_lo = __ldcg(dr + lane);
        if (lane + 32 < a.k) d_hi = __ldcg(dr + lane + 32);
        if (lane <= a.k) t_lo = __ldcg(tg + lane);
        if (lane + 32 <= a.k) t_hi = __ldcg(tg + lane + 32);
        if (lane == 0 && a.k >= 64) t_top = __ldcg(tg + 64);
        if (kSampled) {
            const size_t o = size_t(b) * a.k + lane;
            if (lane < a.k) {
                pv_lo[0] = __ldcg(a.pv_u + o);
                if (a.pv_q) pv_lo[1] = __ldcg(a.pv_q + o);
                pv_lo[2] = __ldcg(a.pv_p + o);
            }
            if (lane + 32 < a.k) {
                pv_hi[0] = __ldcg(a.pv_u + o + 32);
                if (a.pv_q) pv_hi[1] = __ldcg(a.pv_q + o + 32);
                pv_hi[2] = __ldcg(a.pv_p + o + 32);
            }
        }
    };
    if (!pf_ctx) load_draft();
    // Every thread reads the length itself (one L2 request per warp), then arrives on the cluster
    // barrier.  The arrive is relaxed: the barrier only has to publish the leader's message barrier (its
    // initialisation fence is a release).  It does not order this read against the leader's store of the new
    // length (a relaxed arrive need not wait for a load in flight); the data does: a warp's message is computed
    // from the length it read, and the leader stores the new one after its wait for all the messages.
    const int32_t L_old = __ldcg(a.lens + b);
    cluster_arrive_relaxed();
    const bool len_ok = L_old >= 1 && L_old <= (bounded ? a.len_bound : a.cap);
    const int32_t E_old = len_ok ? L_old - 1 : 0;
    if (!bounded) {
        range_of(E_old, e_lo, e_hi);
        lo = max(0, e_lo - kHalo);
    }
    const int32_t hi = tile_hi();                       // the staged positions end here
    const int32_t e_end = max(e_lo, min(e_hi, E_old));  // the old ends scanned: [e_lo, e_end)
    const int32_t tail_lo = max(0, (L_old - kHalo) & ~3);
    const int32_t tail_hi = len_ok ? (L_old + 3) & ~3 : tail_lo;  // <= cap since cap % 4 == 0

    // Linear probe: this CTA's slice is words [v0, v1) of 8 bf16; the first probe_words of w and h are
    // staged by bulk copies, the rest read directly.  Warps 1.. compute it (warp 0 issues the copies and
    // releases the next launch).
    const int nv = a.d >> 3;
    const int vper = (nv + int(C) - 1) / int(C);
    const int v0 = min(nv, int(rank) * vper), v1 = min(nv, v0 + vper);
    const int v_staged = mlp ? 0 : min(v1 - v0, a.probe_words);
    const uint4 *w4 = reinterpret_cast<const uint4 *>(a.probe_w);
    const uint4 *h4 = reinterpret_cast<const uint4 *>(a.hidden + size_t(b) * size_t(gather ? a.hidden_rows : 1) *
                                                                  size_t(a.d));
    auto issue_probe = [&]() {
        const uint32_t pb = uint32_t(v_staged) * 16u;
        mbar_expect_tx_relaxed(&bars[2], 2u * pb);
        if (pb > 0) {
            bulk_g2s(s_pw, w4 + v0, pb, &bars[2]);
            bulk_g2s(s_ph, h4 + v0, pb, &bars[2]);
        }
    };
    if (tid == 0) {
        const uint32_t tb = uint32_t(tail_hi - tail_lo) * 4u;
        mbar_expect_tx_relaxed(&bars[1], tb);
        if (tb > 0) bulk_g2s_hint(s_tail, row + tail_lo, tb, &bars[1], pol);
        if (pf_probe) issue_probe();
        if (!bounded) issue_tile(hi);
        // The parameters only the leader's last phase reads are fetched now, so that phase does not wait
        // on the constant cache.
        asm volatile("" ::"l"(a.out_mode), "l"(a.out_len), "l"(a.out_score), "l"(a.out_match_n), "l"(a.out_match_end),
                     "l"(a.status), "l"(a.out_draft), "l"(a.out_accept), "r"(a.kappa), "f"(a.logit_tau));
    }
    float zp = 0.f;
    bool probe_ok = true;
    auto probe_dot = [&](const uint4 *h) {  // warps 1..: thread j = tid - 32 takes words j, j + kT - 32, ...
        if (v_staged > 0) {
            probe_ok = mbar_wait(&bars[2], 0);
            if (probe_ok)
                for (int i = tid - kWarp; i < v_staged; i += kRescanThreads - kWarp) zp = dot8_bf16(s_pw[i], s_ph[i], zp);
        }
        for (int v = v0 + v_staged + tid - kWarp; v < v1; v += kRescanThreads - kWarp)
            zp = dot8_bf16(w4[v], h[v], zp);
    };
    // A prefetched probe is finished before the wait by warps 1.. (its inputs are not written by the
    // preceding kernel); warp 0 goes straight to the wait and releases the next launch.  The sum over the warp
    // stands at the message: taken here it made every warp wait for the products before its verification (a
    // launch without verification, 17 rows of 98 tokens 2.71 us here, 2.46 there; 66 of 572, context not
    // prefetched, 3.86 and 3.60; 16 launches on the 32K rows 69.3 and 66.9 us).
    if (pf_probe && warp >= 1) probe_dot(h4);
    // Warps 1.. hash this CTA's old ends once the tile has landed -- before the wait when the context is
    // prefetched -- so that the scan after it compares one byte per end (scan_ends, kPre).
    constexpr bool pre = kPre;
    // the filter depth F (in candidate mode no deeper than the gate length kappa)
    auto filter_depth = [&]() {
        return min(kCand ? min(a.n_min, a.kappa > 0 ? a.kappa : a.n_min) : a.n_min, 3);
    };
    if (pre && warp >= 1) {
        const int fdepth = filter_depth();
        if (len_ok && (hi == lo || mbar_wait(&bars[0], 0))) {
            const int32_t n4 = (e_end - e_lo + 3) >> 2;
            if (fdepth >= 3) hash_ends<3>(stage, hb, n4, tid - kWarp, kRescanThreads - kWarp);
            else if (fdepth == 2) hash_ends<2>(stage, hb, n4, tid - kWarp, kRescanThreads - kWarp);
            else hash_ends<1>(stage, hb, n4, tid - kWarp, kRescanThreads - kWarp);
        }
        mbar_arrive(&bars[4]);  // every thread of warps 1.., whether or not it hashed
    }
    if (pf_ctx && !late) pdl_wait();
    if (pf_ctx) load_draft();
    pdl_trigger();
    // The leader's message barrier is initialised once this returns; the arrive was long before, so it costs little
    // beside the loads in flight (on the way out it cost the row's chain).
    cluster_wait_acquire();
    if (!pf_probe && !gather && !mlp && tid == 0) issue_probe();

    // Two-layer probe: this CTA finishes units [u0m, u1m) (the S partial sums in order, b1, ReLU, w2);
    // thread j takes units u0m + j, u0m + j + kT, ...  When this launch's
    // wait already covers the first-layer kernel (not late), the first unit's partial sums are loaded
    // now, so that their round trip overlaps the verification's; the sums are taken after it.
    const int uper = mlp ? (a.H1 + int(C) - 1) / int(C) : 0;
    const int u0m = min(a.H1, int(rank) * uper), u1m = min(a.H1, u0m + uper);
    auto mlp_unit = [&](int u, const float *pz, float acc) {
        float z1 = 0.f;
#pragma unroll
        for (int sp = 0; sp < kMaxMlpSplit; ++sp)
            if (sp < a.mlp_S) z1 += pz[sp];
        if (a.b1) z1 += a.b1[u];
        return fmaf(bf16_lo(uint32_t(a.w2[u])), fmaxf(z1, 0.f), acc);
    };
    auto mlp_load = [&](int u, float *pz) {
#pragma unroll
        for (int sp = 0; sp < kMaxMlpSplit; ++sp)
            pz[sp] = sp < a.mlp_S ? __ldcg(a.z1_part + (size_t(sp) * a.B + size_t(b)) * a.H1p + u) : 0.f;
    };
    // every partial sum of a unit is loaded before the first add (independent L2 reads), then added in
    // order; the same threads and order either way, so the logit does not depend on when this runs
    auto mlp_finish = [&](int from) {
        for (int u = from; u < u1m; u += kRescanThreads) {
            float pz[kMaxMlpSplit];
            mlp_load(u, pz);
            zp = mlp_unit(u, pz, zp);
        }
    };
    const bool mlp_early = mlp && !late;
    float pz0[kMaxMlpSplit];
    const int u_first = u0m + tid;
    if (mlp_early && u_first < u1m) mlp_load(u_first, pz0);

    // ---- verification of the previous draft (every warp) ----
    int32_t acc = -1, L = L_old, vst = len_ok ? SWITCHSD_ROW_OK : SWITCHSD_ROW_BAD_LEN;
    int32_t t_acc = 0;
    int32_t choice = 0;  // candidate mode: the kept candidate
    if (kCand && verifying) {
        // The W previous candidates verified at once (§3.3): thread i takes the positions i, i + kRescanThreads, ... of the
        // candidates laid end to end, stages their draft and target tokens and notes the first position of each
        // candidate that differs; each warp then takes the accepted lengths with lane w on candidate w.  The
        // longest is kept, the lowest index on a tie.  A count of 0 (a neural draft) uses slot 0 with length 0.
        const int W = a.W, D = a.D;
        const size_t o = size_t(b) * size_t(W);
        const int n_d = W * D;
        const int32_t ncv = __ldcg(a.pv_len + b);
        const int32_t lenv = lane < W ? __ldcg(a.pv_cand_len + o + lane) : 0;
        const int32_t topv = tid < W ? __ldcg(a.pv_target + (o + tid) * (D + 1) + D) : 0;  // after a whole candidate
        // each thread issues its loads before its first store, so they share one round trip
        for (int base = tid; base < n_d; base += kVerifyLoads * kRescanThreads) {
            int32_t c[kVerifyLoads], t[kVerifyLoads];
#pragma unroll
            for (int u = 0; u < kVerifyLoads; ++u) {
                const int i = base + u * kRescanThreads;
                c[u] = t[u] = 0;
                if (i < n_d) {
                    c[u] = __ldcg(a.pv_draft + o * D + i);
                    t[u] = __ldcg(a.pv_target + o * (D + 1) + i + over_d(i));
                }
            }
#pragma unroll
            for (int u = 0; u < kVerifyLoads; ++u) {
                const int i = base + u * kRescanThreads;
                if (i < n_d) {
                    const int w = over_d(i);
                    vc[i] = c[u];
                    vt[i + w] = t[u];
                    if (c[u] != t[u]) atomicMin(&s_miss[w], i - w * D);
                }
            }
        }
        if (tid < W) vt[tid * (D + 1) + D] = topv;
        __syncthreads();
        const int32_t nc = ncv;
        if (len_ok) {
            const bool nc_ok = nc >= 0 && nc <= W;
            const int ncx = !nc_ok ? 0 : (nc > 0 ? nc : 1);
            const int32_t len = nc > 0 ? lenv : 0;
            const bool used = lane < ncx;
            const bool len_bad = used && (len < 0 || len > D);
            const bool badlen = __any_sync(kFull, len_bad) || !nc_ok;
            const int32_t acc_w = used && !len_bad ? min(s_miss[lane], len) : 0;
            const uint32_t rank_w = __reduce_max_sync(kFull, used ? (uint32_t(acc_w) << 5 | uint32_t(31 - lane)) + 1u : 0u);
            const int32_t best = rank_w != 0u ? int32_t((rank_w - 1u) >> 5) : -1;
            choice = rank_w != 0u ? 31 - int32_t((rank_w - 1u) & 31u) : 0;
            if (badlen) {
                vst = SWITCHSD_ROW_BAD_LEN;
            } else if (L_old + best + 1 > a.cap) {
                vst = SWITCHSD_ROW_CAPACITY;
            } else {
                acc = best;
                L = L_old + acc + 1;
            }
        }
    }
    if (!kCand && verifying && len_ok) {
        if (pv_n < 0 || pv_n > a.k) {
            vst = SWITCHSD_ROW_BAD_LEN;
        } else {
            bool rej_lo, rej_hi;
            if (kSampled) {
                // T > 0: draft token i is rejected when u_i * q_i (binary32) is not below p_i
                rej_lo = lane < pv_n && !(__fmul_rn(pv_lo[0], pv_lo[1]) < pv_lo[2]);
                rej_hi = lane + 32 < pv_n && !(__fmul_rn(pv_hi[0], pv_hi[1]) < pv_hi[2]);
            } else {
                rej_lo = lane < pv_n && d_lo != t_lo;
                rej_hi = lane + 32 < pv_n && d_hi != t_hi;
            }
            const unsigned m_lo = __ballot_sync(kFull, rej_lo);
            const unsigned m_hi = __ballot_sync(kFull, rej_hi);
            const int32_t at = m_lo ? __ffs(m_lo) - 1 : (m_hi ? 32 + __ffs(m_hi) - 1 : pv_n);
            if (L_old + at + 1 > a.cap) {
                vst = SWITCHSD_ROW_CAPACITY;
            } else {
                acc = at;
                t_acc = __shfl_sync(kFull, acc < 32 ? t_lo : (acc < 64 ? t_hi : t_top), acc & 31);
                L = L_old + acc + 1;
            }
        }
    }
    if (mlp_early && u_first < u1m) {
        zp = mlp_unit(u_first, pz0, zp);
        mlp_finish(u_first + kRescanThreads);
    }
    // The probed state of a fused verification with hidden_rows = k + 1: row a_b (row 0 when nothing was
    // appended).  Its slice is staged now and used after the scan.
    if (gather) {
        h4 += size_t(acc > 0 ? acc : 0) * size_t(nv);
        if (tid == 0) issue_probe();
    }

    // ---- this warp's window: y[L_old - kHalo + j], the old tail then the appended tokens ----
    const bool tail_in = tail_hi == tail_lo || mbar_wait(&bars[1], 0);
    int32_t *y = s_y[warp];
    {
        const int32_t p = L_old - kHalo + lane;
        y[lane] = (len_ok && p >= 0 && tail_in) ? s_tail[p - tail_lo] : 0;
        if (acc >= 0) {
            if (kCand) {  // the kept candidate's accepted tokens, then its target's next token
                for (int i = lane; i < acc; i += kWarp) y[kHalo + i] = vc[choice * a.D + i];
                if (lane == 0) y[kHalo + acc] = vt[choice * (a.D + 1) + acc];
            } else {
                if (lane < acc) y[kHalo + lane] = d_lo;
                if (lane + 32 < acc) y[kHalo + 32 + lane] = d_hi;
                if (lane == 0) y[kHalo + acc] = t_acc;
            }
        }
    }
    __syncwarp();
    const int32_t *suf = y + kHalo + acc;  // suf[-m] = the m-th token from the end of the new context
    const int32_t n_max = a.n_max, n_min = a.n_min;

    // ---- scan of this warp's share of the CTA's old ends ----
    const int32_t kappa_c = a.kappa > 0 ? a.kappa : a.n_min;  // candidate mode: the gate length
    uint32_t new_c[3] = {0u, 0u, 0u};                         // candidate mode: appended ends (leader)
    // key = m << kKeyShift | e (e < 2^kKeyShift, m <= 32): the largest key is the longest match, then the
    // most recent; 0 = no match; kKeyTimeout marks a copy that did not land.
    uint32_t mine = 0;
    const bool tile_in = kRing || hi == lo || mbar_wait(&bars[0], 0);
    const bool hashed = !pre || mbar_wait(&bars[4], 0);
    bool timed_out = !tail_in || !tile_in || !hashed;
    const int32_t off = kHalo - e_lo;  // stage[off + p] = x[p] over the staged range
    // (n_min and kappa are uniform over the launch: one instance runs)
    // the filter depth may test no more than a candidate needs (fdepth <= kappa in candidate mode)
    bool marked = false;  // candidate mode: this thread marked an end
    auto scan = [&](const int32_t *st, int32_t lo_e, int32_t end_e, int32_t key0) {
        const int fdepth = filter_depth();
        return fdepth >= 3
                   ? scan_ends<3, kCand, kPre>(st, lo_e, end_e, suf, n_min, n_max, tid, lane, bm, kappa_c, hb, key0, e_lo, &marked)
                   : (fdepth == 2 ? scan_ends<2, kCand, kPre>(st, lo_e, end_e, suf, n_min, n_max, tid, lane, bm, kappa_c,
                                                              hb, key0, e_lo, &marked)
                                  : scan_ends<1, kCand, kPre>(st, lo_e, end_e, suf, n_min, n_max, tid, lane, bm, kappa_c,
                                                              hb, key0, e_lo, &marked));
    };
    // the continuation of a match ending at e: lane j (1..kw) gathers tokens 4(j-1) .. +3, from the staged
    // tile (tl[o_ + p] = x[p]) or past the old length from this warp's window
    uint4 cw = make_uint4(0, 0, 0, 0);
    auto gather_next = [&](int32_t e, const int32_t *tl, int32_t o_) {
        if (lane < 1 || lane > kw) return;
        const int32_t len = min(a.k, L - 1 - e);
        int32_t t4[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int32_t i = 4 * (lane - 1) + q;
            const int32_t p = e + 1 + i;
            t4[q] = i < len ? (p < L_old ? tl[o_ + p] : y[kHalo + p - L_old]) : 0;
        }
        cw = make_uint4(uint32_t(t4[0]), uint32_t(t4[1]), uint32_t(t4[2]), uint32_t(t4[3]));
    };
    // ring: this warp's best match so far (m_b = 0: none), warp-uniform; its continuation is in cw
    int32_t m_b = 0, e_b = -1;
    if constexpr (kRing) {
        const int nt = ring_tiles();
        int s = 0;
        uint32_t phase = 0u;
        for (int t = 0; t < nt; ++t) {
            if (!__all_sync(kFull, mbar_wait(&ring[s], phase))) {
                timed_out = true;
                // copies still in flight get a second bounded wait before the CTA's memory goes away
                if (lane == 0)
                    for (int u = t; u < min(nt, t + a.stages); ++u)
                        (void)mbar_wait(&ring[u % a.stages], uint32_t(u / a.stages) & 1u);
                break;
            }
            const int32_t t0 = e_lo + t * a.tile;
            const int32_t *tl = stage + s * stage_ints;
            uint32_t k_t = 0u;
            if (tail_in && len_ok && t0 < e_end) k_t = scan(tl, t0, min(e_end, t0 + a.tile), t0);
            k_t = __reduce_max_sync(kFull, k_t);
            if (k_t != 0u && int32_t(k_t >> kKeyShift) >= m_b) {  // a later tile's ends are the more recent
                m_b = int32_t(k_t >> kKeyShift);
                e_b = t0 + int32_t(k_t & kKeyEndMask);
                gather_next(e_b, tl, kHalo - t0);
            }
            __syncwarp();
            if (lane == 0 && t + a.stages < nt) {
                __threadfence_block();  // this warp's reads of the stage, before the last warp out refills it
                if ((atomicAdd(&s_out_of[s], 1) + 1) % kRescanWarps == 0) {
                    __threadfence_block();
                    fence_proxy_async();
                    issue_ring(t + a.stages, s);
                }
            }
            if (++s == a.stages) {
                s = 0;
                phase ^= 1u;
            }
        }
    }
    if (!timed_out && len_ok && L >= 2) {
        if (!kRing) mine = scan(stage, e_lo, e_end, 0);
        // The ends the append creates, [L_old - 1, L - 1), lie in the window: the leader's warp 0.  In
        // candidate mode new_c[t] bit i marks end L_old - 1 + 32 t + i as a candidate (warp-uniform).
        if (kCand && rank == lead && warp == 0 && acc >= 0) {
#pragma unroll 1
            for (int t = 0; 32 * t <= acc; ++t) {
                const int32_t j = lane + 32 * t;
                bool qual = false;
                if (j <= acc) {
                    const int32_t e = L_old - 1 + j;
                    const int32_t lim = min(n_max, e + 1);
                    int32_t m = 0;
#pragma unroll 1
                    while (m < lim && y[kHalo - 1 + j - m] == suf[-m]) ++m;
                    if (m >= n_min) {
                        const uint32_t key = (uint32_t(m) << kKeyShift) | uint32_t(kRing ? j : e);
                        mine = key > mine ? key : mine;
                    }
                    qual = m >= kappa_c;
                }
                new_c[t] = __ballot_sync(kFull, qual);
            }
        } else if (rank == lead && warp == 0 && acc >= 0) {
#pragma unroll 1
            for (int32_t j = lane; j <= acc; j += kWarp) {
                const int32_t e = L_old - 1 + j;
                const int32_t lim = min(n_max, e + 1);
                int32_t m = 0;
#pragma unroll 1
                while (m < lim && y[kHalo - 1 + j - m] == suf[-m]) ++m;
                if (m >= n_min) {
                    const uint32_t key = (uint32_t(m) << kKeyShift) | uint32_t(kRing ? j : e);
                    mine = key > mine ? key : mine;
                }
            }
        }
    }
    uint32_t key = __reduce_max_sync(kFull, mine);
    if constexpr (kRing) {
        // the appended ends (the leader's warp 0) are more recent than every old one
        if (key != 0u && int32_t(key >> kKeyShift) >= m_b) {
            m_b = int32_t(key >> kKeyShift);
            e_b = L_old - 1 + int32_t(key & kKeyEndMask);
            gather_next(e_b, stage, 0);  // every token of it is in the window
        }
        key = uint32_t(m_b) << kKeyShift;  // the message carries the end beside it
    }
    if (timed_out) key = kKeyTimeout;

    // ---- candidate mode: this CTA's W most recent marked ends and their continuations (warp 0) ----
    if constexpr (kCand) {
        // every warp's marks are in the bitmap after this barrier; most CTAs have none to rank
        const bool any_marked = __syncthreads_or(marked);
        // Bitmap words from the top, kRescanThreads per pass: thread t holds word top - t; prefix sums of
        // the popcounts (within the warp, then over the warps) rank its bits after those of higher words.
        // `found` is CTA-uniform.
        const int nwords = any_marked ? (e_end - e_lo + 31) >> 5 : 0;
        int found = 0;
        for (int top = nwords - 1; top >= 0 && found < a.W; top -= kRescanThreads) {
            const int idx = top - tid;
            const uint32_t wd = idx >= 0 ? bm[idx] : 0u;
            const int c = __popc(wd);
            int incl = c;
#pragma unroll
            for (int o_ = 1; o_ < kWarp; o_ <<= 1) {
                const int t_ = __shfl_up_sync(kFull, incl, o_);
                if (lane >= o_) incl += t_;
            }
            if (lane == kWarp - 1) s_wtot[warp] = incl;
            __syncthreads();
            int r = found, total = 0;
#pragma unroll
            for (int w = 0; w < kRescanWarps; ++w) {
                r += w < warp ? s_wtot[w] : 0;
                total += s_wtot[w];
            }
            r += incl - c;
            uint32_t w2 = wd;
            while (w2 != 0u && r < a.W) {
                const int bit = 31 - __clz(w2);
                w2 &= ~(1u << bit);
                s_sel[r++] = e_lo + idx * 32 + bit;
            }
            found += total;
            __syncthreads();  // s_wtot is rewritten by the next pass; s_sel is complete after the last
        }
        if (warp == 0) {
            const int nsel = min(found, a.W);
            // the message: header (count), the ends, then candidate w's D tokens at w D -- from the staged
            // tile, or past the old length from this warp's window (an end e continues for
            // min(D, L - 1 - e) tokens, all below L)
            int32_t *ce = reinterpret_cast<int32_t *>(cstage + 16);
            int32_t *ct = reinterpret_cast<int32_t *>(cstage + 16 + 16 * ((a.W + 3) / 4));
            if (lane == 0) *reinterpret_cast<int4 *>(cstage) = make_int4(nsel, 0, 0, 0);
            if (lane < nsel) ce[lane] = s_sel[lane];
            const int dw = over_d(kWarp), di = kWarp - dw * a.D;  // (candidate, token) step of 32 slots
            int w = over_d(lane), i = lane - w * a.D;
            for (int t = lane; !kRing && t < nsel * a.D; t += kWarp) {  // (the ring's tiles are gone)
                const int32_t ew = s_sel[w];
                const int32_t p = ew + 1 + i;
                ct[t] = i < min(a.D, L - 1 - ew) ? (p < L_old ? stage[off + p] : y[kHalo + p - L_old]) : 0;
                w += dw;
                i += di;
                if (i >= a.D) {
                    i -= a.D;
                    ++w;
                }
            }
            fence_proxy_async();  // the bulk copy below reads the message through the async proxy
            __syncwarp();
        }
    }

    // ---- probe share (unless finished before the wait) ----
    if (late) {  // the partial sums only now: this launch waits for the first-layer kernel here
        pdl_wait();
        mlp_finish(u0m + tid);
    } else if (warp >= 1) {
        if (mlp) {
            // finished after the verification (mlp_early)
        } else if (!pf_probe) {
            probe_dot(h4);
        }
    }
    if (!probe_ok) key = kKeyTimeout;
    const float z_w = warp_sum_f32(zp);

    // ---- the continuation of this warp's best match (the ring has it already) ----
    if (!kRing && key != 0u && key != kKeyTimeout) gather_next(int32_t(key & kKeyEndMask), stage, off);

    // ---- ship to the leader ----
    const uint32_t done_addr = map_to_rank(&bars[3], lead);
    unsigned char *slot = msgs + size_t(rank * kRescanWarps + warp) * slot_bytes;
    if (lane == 0) {
        uint4 h;
        h.x = key;
        h.y = __float_as_uint(z_w);
        h.z = uint32_t(e_b);
        h.w = 0u;
        st_async_v4(map_to_rank(slot, lead), h, done_addr);
    } else if (lane <= kw) {
        st_async_v4(map_to_rank(slot + 16 * lane, lead), cw, done_addr);
    }
    // This CTA's candidates, in one bulk copy (a launch without verification; a store a word a lane instead, and so: 4
    // candidates of 8 tokens on 287 rows of 223 tokens 3.99 and 3.60 us, 14 of 20 on 146 of 177 4.77 and 4.50; 10 of
    // 20 on the 32K rows, 8 fused launches, 50.5 and 49.3 us).
    const bool ships_cand = kCand && warp == 0 && lane == 0;
    if (ships_cand) bulk_s2c(map_to_rank(cmsgs + size_t(rank) * cl.cslot, lead), cstage, cl.cslot, done_addr);
    if (rank != lead || warp != 0) {
        if (ships_cand) bulk_wait_read();  // the message has been read out
        if (timed_out && lane == 0) {  // copies still in flight get a second bounded wait
            if (!kRing) (void)mbar_wait(&bars[0], 0);
            (void)mbar_wait(&bars[1], 0);
        }
        if (!probe_ok && lane == 0) (void)mbar_wait(&bars[2], 0);
        return;
    }

    // ---- leader, warp 0: the append, then the row's answer ----
    // (the appended positions are past every end the other CTAs scan; what their copies hold there is not used)
    if (verifying)
        for (int32_t i = lane; i <= acc; i += kWarp) row[L_old + i] = y[kHalo + i];
    const bool all_in = __all_sync(kFull, mbar_wait_polls(&bars[3], 0, a.msg_wait_polls));
    // messages still in flight get a second bounded wait: before the new length goes out, and before the CTA's
    // memory goes away
    if (!all_in && lane == 0) (void)mbar_wait(&bars[3], 0);
    uint32_t k_r = 0u, e_r = 0u;
    int32_t i_r = 0;
    float z_r = 0.f;
    if (all_in) {
        for (int i = lane; i < nmsg; i += kWarp) {  // lane j: messages j, j + 32, ... in order
            const uint4 hv = *reinterpret_cast<const uint4 *>(msgs + size_t(i) * slot_bytes);
            z_r += __uint_as_float(hv.y);
            if (hv.x > k_r || (kRing && hv.x == k_r && hv.x != 0u && hv.z > e_r)) {
                k_r = hv.x;
                e_r = hv.z;
                i_r = i;
            }
        }
    }
    const uint32_t best = all_in ? __reduce_max_sync(kFull, k_r) : kKeyTimeout;
    // ring: the keys hold the lengths alone, the most recent end decides among them
    const uint32_t best_e = kRing ? __reduce_max_sync(kFull, k_r == best ? e_r : 0u) : 0u;
    const unsigned at = __ballot_sync(kFull, k_r == best && (!kRing || e_r == best_e));
    const int32_t win = __shfl_sync(kFull, i_r, at != 0u ? __ffs(at) - 1 : 0);
    // The winner's continuation is read beside the logit's sum (8K rows 3.54 -> 3.45 us a launch; not in the hash
    // instance, whose register file is full: 32K rows 4.20 -> 4.22).
    constexpr bool kDraftEarly = !kCand && !kPre && !kMlp;
    const int32_t *wd = reinterpret_cast<const int32_t *>(msgs + size_t(win) * slot_bytes + 16);
    const int32_t w_lo = kDraftEarly && lane < 4 * kw ? wd[lane] : 0;
    const int32_t w_hi = kDraftEarly && lane + kWarp < 4 * kw ? wd[lane + kWarp] : 0;
    const float z = warp_sum_f32(z_r) + (mlp ? a.b2 : 0.f);
    const bool timeout = best == kKeyTimeout;
    const bool hit = len_ok && !timeout && best != 0u;
    const int32_t n = hit ? int32_t(best >> kKeyShift) : 0;
    const int32_t e = hit ? int32_t(kRing ? best_e : best & kKeyEndMask) : -1;
    if constexpr (kCand) {
        // The row's candidates, most recent first: the appended ends (highest first), then the CTAs' lists
        // from the leader's (the most recent range) down to CTA 0's.  s_sel[w] is merged candidate w's
        // source: -1 - j for the appended end L_old - 1 + j, else r kMaxCand + i for entry i of CTA r.
        // Lane r holds CTA r's count; a suffix sum places its entries after those of the more recent CTAs.
        const int n_new = hit ? __popc(new_c[0]) + __popc(new_c[1]) + __popc(new_c[2]) : 0;
        int cnt = 0;
        if (hit && lane < int(C)) cnt = min(*reinterpret_cast<const int32_t *>(cmsgs + size_t(lane) * cl.cslot), a.W);
        int after = cnt;
#pragma unroll
        for (int o_ = 1; o_ < kMaxSplit; o_ <<= 1) {
            const int t_ = __shfl_down_sync(kFull, after, o_);
            if (lane + o_ < kWarp) after += t_;
        }
        const int first = n_new + after - cnt;  // the rank of CTA `lane`'s first entry
        const int ncand = min(n_new + __shfl_sync(kFull, after, 0), a.W);
        int32_t mode = SWITCHSD_MODE_NO_REP;
        if (hit) mode = (ncand > 0 && z >= a.logit_tau) ? SWITCHSD_MODE_COPY : SWITCHSD_MODE_REP_NO_COPY;
        const int nc = mode == SWITCHSD_MODE_COPY ? ncand : 0;
        if (lane < nc) {
            if (lane < n_new) {
                int k = lane, j = -1;
                for (int t = 2; t >= 0 && j < 0; --t) {
                    const int pc = __popc(new_c[t]);
                    if (k < pc) {
                        uint32_t mm = new_c[t];
                        for (int q = 0; q < k; ++q) mm &= ~(1u << (31 - __clz(mm)));
                        j = 32 * t + 31 - __clz(mm);
                    } else {
                        k -= pc;
                    }
                }
                s_sel[lane] = -1 - j;
            }
        }
        for (int i = 0; i < cnt && first + i < nc; ++i) s_sel[first + i] = lane * kMaxCand + i;
        __syncwarp();
        const int cwE = (a.W + 3) / 4;
        auto cand_end = [&](int src) -> int32_t {
            if (src < 0) return L_old - 2 - src;  // L_old - 1 + j with j = -1 - src
            const int r = src / kMaxCand;
            return reinterpret_cast<const int32_t *>(cmsgs + size_t(r) * cl.cslot + 16)[src - r * kMaxCand];
        };
        if (lane < nc) a.out_cand_len[size_t(b) * a.W + lane] = min(a.D, L - 1 - cand_end(s_sel[lane]));
        const int dw = over_d(kWarp), di = kWarp - dw * a.D;  // (candidate, token) step of 32 slots
        int w = over_d(lane), i = lane - w * a.D;
        for (int t = lane; t < nc * a.D; t += kWarp, w += dw, i += di) {
            if (i >= a.D) {
                i -= a.D;
                ++w;
            }
            const int src = s_sel[w];
            const int32_t ew = cand_end(src);
            if (i < min(a.D, L - 1 - ew)) {
                int32_t tok;
                if (src < 0) {
                    tok = y[kHalo + ew + 1 + i - L_old];
                } else if (kRing) {
                    const int32_t p = ew + 1 + i;
                    tok = p < L_old ? __ldcg(row + p) : y[kHalo + p - L_old];
                } else {
                    const int r = src / kMaxCand;
                    tok = reinterpret_cast<const int32_t *>(cmsgs + size_t(r) * cl.cslot + 16 + 16 * cwE)
                        [(src - r * kMaxCand) * a.D + i];
                }
                a.out_cand[(size_t(b) * a.W + w) * a.D + i] = tok;
            }
        }
        if (lane == 0) {
            a.out_mode[b] = mode;
            a.out_score[b] = z;
            a.out_ncand[b] = nc;
            if (a.out_match_n) a.out_match_n[b] = n;
            if (a.out_match_end) a.out_match_end[b] = e;
            if (verifying) {
                a.out_accept[b] = acc;          // -1: nothing appended
                if (len_ok) a.lens[b] = L;      // every warp of the row has read the old one: its message is in
            }
            if (verifying && a.out_choice) a.out_choice[b] = len_ok ? choice : 0;
            if (a.status) {
                int32_t st = vst;
                if (st == SWITCHSD_ROW_OK && timeout) st = SWITCHSD_ROW_TIMEOUT;
                a.status[b] = st;
            }
        }
    } else {
        const int32_t kappa = a.kappa > 0 ? a.kappa : a.n_min;
        int32_t mode = SWITCHSD_MODE_NO_REP;
        if (hit) mode = (n >= kappa && z >= a.logit_tau) ? SWITCHSD_MODE_COPY : SWITCHSD_MODE_REP_NO_COPY;
        const int32_t len = mode == SWITCHSD_MODE_COPY ? min(a.k, L - 1 - e) : 0;
        if (lane == 0) {
            if (a.counters) count_row(a.counters, mode, verifying, a.out_mode[b], acc);  // out_mode: the previous mode
            a.out_mode[b] = mode;
            a.out_len[b] = len;
            a.out_score[b] = z;
            if (a.out_match_n) a.out_match_n[b] = n;
            if (a.out_match_end) a.out_match_end[b] = e;
            if (verifying) {
                a.out_accept[b] = acc;          // -1: nothing appended
                if (len_ok) a.lens[b] = L;      // every warp of the row has read the old one: its message is in
            }
            if (a.status) {
                int32_t st = vst;
                if (st == SWITCHSD_ROW_OK && timeout) st = SWITCHSD_ROW_TIMEOUT;
                a.status[b] = st;
            }
        }
        int32_t *out = a.out_draft + size_t(b) * a.k;
        if (lane < len) out[lane] = kDraftEarly ? w_lo : wd[lane];
        if (lane + kWarp < len) out[lane + kWarp] = kDraftEarly ? w_hi : wd[lane + kWarp];
    }
    if (ships_cand) bulk_wait_read();  // the leader's own message has been read out
    if (timed_out && lane == 0) {
        if (!kRing) (void)mbar_wait(&bars[0], 0);
        (void)mbar_wait(&bars[1], 0);
    }
    if (!probe_ok && lane == 0) (void)mbar_wait(&bars[2], 0);
}

size_t rescan_smem_bytes(const StepArgs &args, int split) {
    const bool cand = args.W > 0;
    const size_t stage = size_t(args.stages) * size_t((kHalo + args.tile + kFwd + 3) & ~3) * sizeof(int32_t);
    const size_t probe = 2 * size_t(args.probe_words) * 16 + size_t(args.hash_words) * 4;
    const size_t msgs = size_t(split) * kRescanWarps * 16 * size_t(1 + (cand ? 0 : ((args.k + 3) >> 2)));
    if (!cand) return stage + probe + msgs;
    const CandLayout c = cand_layout(args.range, args.W, args.D, args.ring != 0);
    return stage + probe + msgs + size_t(split + 1) * c.cslot + size_t(c.bm_words + c.v_ints) * sizeof(int32_t);
}

template <bool kSampled, bool kCand, int kScan, bool kMlp>
static cudaError_t rescan_attrs() {
    static bool attr_done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(rescan_kernel<kSampled, kCand, kScan, kMlp>,
                                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(rescan_kernel<kSampled, kCand, kScan, kMlp>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(kScan == kScanRing ? kRingSmemBudget : kRescanSmemBudget));
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
    return cudaSuccess;
}

template <bool kSampled, bool kCand, int kScan, bool kMlp>
static cudaError_t launch_rescan(const StepArgs &args, int split, cudaStream_t stream) {
    const cudaError_t e = rescan_attrs<kSampled, kCand, kScan, kMlp>();
    if (e != cudaSuccess) return e;
    return launch_pdl(rescan_kernel<kSampled, kCand, kScan, kMlp>, dim3(unsigned(split), unsigned(args.B), 1),
                      dim3(kRescanThreads, 1, 1), rescan_smem_bytes(args, split), stream, unsigned(split), args);
}

// Resident CTAs per SM of an instance at a dynamic shared-memory size (cached: the occupancy calculator
// runs once per instance, device and size).
template <bool kSampled, bool kCand, int kScan, bool kMlp>
static cudaError_t rescan_per_sm(size_t smem, int &out) {
    struct Entry {
        int dev;
        size_t smem;
        int n;
    };
    static std::mutex mu;
    static Entry cache[32];
    static int used = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(mu);
        for (int i = 0; i < used; ++i)
            if (cache[i].dev == dev && cache[i].smem == smem) {
                out = cache[i].n;
                return cudaSuccess;
            }
    }
    cudaError_t e = rescan_attrs<kSampled, kCand, kScan, kMlp>();
    if (e != cudaSuccess) return e;
    int n = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, rescan_kernel<kSampled, kCand, kScan, kMlp>, kRescanThreads, smem);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (used < 32) cache[used++] = Entry{dev, smem, n};
    out = n;
    return cudaSuccess;
}

template <bool kSampled, bool kCand, bool kMlp>
static cudaError_t choose_hash(StepArgs &args, int split, int sms) {
    const int32_t words = int32_t(((args.tile + 3) / 4 + 3) & ~3);  // one byte an end; 16-byte multiple
    args.hash_words = 0;
    // The hashing overlaps the preceding launch only when this launch's CTAs are resident early, which a
    // grid of fewer CTAs than SMs is not, measured: the 8K rows (two CTAs a row, 128 CTAs) lose 0.1 us a
    // launch with it, the 32K rows (512 CTAs) gain 0.1 us and the 128K rows (256 CTAs of 8.5K ends) 0.8 us.
    if (int64_t(split) * args.B < int64_t(sms)) return cudaSuccess;
    // Without the context prefetch the tiles land after the wait, and the hashing would only stand before the
    // scan: one batch of 64 rows of 32K tokens takes 6.20 us a launch without it and 7.00 with it, 16 of 128K
    // 8.55 and 9.69, 768 of 4K with the two-layer probe 18.4 and 19.3.
    if ((args.prefetch & SWITCHSD_PREFETCH_CONTEXT) == 0) return cudaSuccess;
    int without = 0, with = 0;
    cudaError_t e = rescan_per_sm<kSampled, kCand, kScanTokens, kMlp>(rescan_smem_bytes(args, split), without);
    if (e != cudaSuccess) return e;
    StepArgs h = args;
    h.hash_words = words;
    const size_t bytes = rescan_smem_bytes(h, split);
    if (bytes > kRescanSmemBudget) return cudaSuccess;
    e = rescan_per_sm<kSampled, kCand, kScanHashed, kMlp>(bytes, with);
    if (e != cudaSuccess) return e;
    if (with >= 1 && with >= (without < kRescanMinBlocks ? without : kRescanMinBlocks)) args.hash_words = words;
    return cudaSuccess;
}

template <bool kSampled, bool kCand>
static cudaError_t choose_hash2(StepArgs &args, int split, int sms) {
    return args.z1_part != nullptr ? choose_hash<kSampled, kCand, true>(args, split, sms)
                                   : choose_hash<kSampled, kCand, false>(args, split, sms);
}

cudaError_t rescan_choose_hash(StepArgs &args, int split, int sms) {
    if (args.W > 0) return choose_hash2<false, true>(args, split, sms);
    return args.pv_p != nullptr ? choose_hash2<true, false>(args, split, sms)
                                : choose_hash2<false, false>(args, split, sms);
}

template <bool kSampled, bool kCand, bool kMlp>
static cudaError_t launch_rescan3(const StepArgs &args, int split, cudaStream_t stream) {
    if (args.ring) return launch_rescan<kSampled, kCand, kScanRing, kMlp>(args, split, stream);
    return args.hash_words > 0 ? launch_rescan<kSampled, kCand, kScanHashed, kMlp>(args, split, stream)
                               : launch_rescan<kSampled, kCand, kScanTokens, kMlp>(args, split, stream);
}

template <bool kSampled, bool kCand>
static cudaError_t launch_rescan2(const StepArgs &args, int split, cudaStream_t stream) {
    return args.z1_part != nullptr ? launch_rescan3<kSampled, kCand, true>(args, split, stream)
                                 : launch_rescan3<kSampled, kCand, false>(args, split, stream);
}

cudaError_t launch_rescan_kernel(const StepArgs &args, int split, cudaStream_t stream) {
    // candidate verification is greedy (the candidates' targets are compared token by token)
    if (args.W > 0) return launch_rescan2<false, true>(args, split, stream);
    return args.pv_p != nullptr ? launch_rescan2<true, false>(args, split, stream)
                                : launch_rescan2<false, false>(args, split, stream);
}

}  // namespace switchsd
