// index.cu -- incremental n-gram index: the same (n*, e*) as the rescan, from hash chains.
//
// For every row b and every n in [n_min, n_max] the index keeps
//   heads[n][b][bucket]  the most recent end position e whose n-gram x[e-n+1..e] hashes to bucket,
//   prev[n][b][e]        the previous end position with the same bucket (-1 at the end of a chain).
// Contexts only grow and positions are inserted in increasing order, so every chain lists end
// positions in decreasing order.  Looking up the suffix n-gram walks its bucket's chain from the head,
// skips the suffix's own end (L-1) and compares candidates token by token; the first exact match is
// the most recent earlier occurrence (§3.3's recency ranking).  n* is the largest n with a match and
// e* its end: exactly the rescan's answer, hash collisions included (they only lengthen the walk).
//
// index_kernel runs one CTA per row with one warp per n and does, in order:
//   verification of the previous draft (as switchsd_verify) and its append, when verifying;
//   insertion of the appended end positions (all lanes at once; positions of one run that fall into
//   the same bucket are linked through __match_any_sync, so one read of the old heads suffices);
//   the lookup, the probe and the switch / copy draft (as switchsd_step), when stepping.
// What bounds it is the chain of dependent L2 round trips, three after the wait: the verification's inputs
// (all loads at once), the heads (with the link of a position inserted before), then per chain entry the
// tokens compared, the next link and the tokens that follow it.  The lookup starts from the link that the
// insert of the suffix's own end found, and the draft is written from the registers of the n that wins.  16
// rows of 128K tokens, n = 2..12, 16 launches: 82.6 us with the heads and links read again for the lookup and
// the draft gathered at the end (seven round trips), 71.7 us so, over positions that the index held already (the lengths
// were rewound between passes).  With every append new (the index rebuilt before each pass; medians of 12 texts, one
// pass at a time): 111.7 us against 74.9, and 124.1 against 85.2 with the seven round trips.
// Candidate mode (W > 0, as switchsd_step_candidates / switchsd_verify_candidates): the previous W
// candidates are verified and the longest accepted one appended; the warp of n = kappa walks its
// chain on past the first match and lists the W most recent ends whose kappa-gram equals the
// suffix's -- exactly the ends whose common suffix with the current one reaches kappa.
#include <new>

#include "common.cuh"
#include "index.cuh"
#include "mlp.cuh"

struct switchsd_index {
    int32_t B, cap, n_min, n_max, nn, log2_buckets;
    int32_t *heads;  // [nn][B][1 << log2_buckets]
    int32_t *prev;   // [nn][B][cap]
    int device;
};

namespace switchsd {

constexpr int kIdxMaxWarps = SWITCHSD_NMAX;
constexpr int kIdxTail = SWITCHSD_NMAX + SWITCHSD_KMAX + 1;  // staged context tail: old end +- the append

// Hash of the n tokens ending at the last one (`tok(i)` = token i steps back): the sum of their products with
// the powers of an odd multiplier, whose terms are independent (one multiply-add each, no chain through a
// mixer), in 64 bits so that tokens that differ in their high bits alone still spread, then one
// multiply-xorshift round; the bucket is its top bits.
constexpr uint32_t kGramMul = 0x9E3779B1u;
__device__ __forceinline__ uint32_t gram_bucket(uint64_t sum, int n, int log2_buckets) {
    uint32_t h = uint32_t(sum) + uint32_t(sum >> 32) * 0x7FEB352Du + uint32_t(n) * 0x85EBCA77u;
    h ^= h >> 15;
    h *= 0x2C1B3C6Du;
    return h >> (32 - log2_buckets);
}
template <typename Tok>
__device__ __forceinline__ uint32_t gram_hash(int n, Tok tok, int log2_buckets) {
    uint64_t h = 0u;
    uint32_t pw = 1u;
    for (int i = 0; i < n; ++i) {
        h += uint64_t(uint32_t(tok(i))) * pw;
        pw *= kGramMul;
    }
    return gram_bucket(h, n, log2_buckets);
}

struct IndexArgs {
    int32_t *ctx, *lens;
    const uint16_t *hidden, *probe_w;
    const float *z1_part;  // two-layer probe: split-K partial sums of W1 h [mlp_S][B][H1p], else null
    const float *b1;       // two-layer probe: first-layer biases (null = zero) and output weights
    const uint16_t *w2;
    int32_t mlp_S, H1, H1p;
    float b2;
    const int32_t *pv_draft, *pv_target, *pv_len;  // verification inputs (null: no verification)
    const float *pv_p, *pv_q, *pv_u;               // sampled verification (null p: greedy)
    int32_t hidden_rows;                           // > 1: the probe reads row a_b of [B, hidden_rows, d]
    int32_t *out_accept;
    int32_t *out_draft, *out_len, *out_mode;
    float *out_score;
    int32_t *out_match_n, *out_match_end, *status;
    int32_t *heads, *prev;
    int32_t B, cap, d, k, n_min, n_max, kappa, log2_buckets, stepping;
    float logit_tau;
    // candidate mode (W > 0): W candidates of up to D tokens; pv_draft / pv_target / pv_len then hold
    // the previous candidates [B][W][D], their targets [B][W][D+1] and counts [B]
    int32_t W, D;
    const int32_t *pv_cand_len;  // [B][W]
    int32_t *out_choice, *out_cand, *out_cand_len, *out_ncand;
    int32_t prefetch;  // SWITCHSD_PREFETCH_* bits: the inputs they name are read before the wait
    unsigned long long *counters;  // optional per-mode tallies (switchsd_params.counters), else null
};

// This thread's share of the linear probe's dot product over row b's hidden state (threads stride the
// d/8 words; the same partition wherever it is computed, so the logit is the same).
__device__ __forceinline__ float index_probe_partial(const IndexArgs &a, int b, int32_t hrow) {
    const uint4 *h4 = reinterpret_cast<const uint4 *>(
        a.hidden + (size_t(b) * size_t(a.hidden_rows > 1 ? a.hidden_rows : 1) + size_t(hrow)) * a.d);
    const uint4 *w4 = reinterpret_cast<const uint4 *>(a.probe_w);
    float zp = 0.f;
    for (int v = threadIdx.x; v < (a.d >> 3); v += blockDim.x) {
        const uint4 w = w4[v], h = h4[v];
        zp = fmaf(bf16_lo(w.x), bf16_lo(h.x), zp);
        zp = fmaf(bf16_hi(w.x), bf16_hi(h.x), zp);
        zp = fmaf(bf16_lo(w.y), bf16_lo(h.y), zp);
        zp = fmaf(bf16_hi(w.y), bf16_hi(h.y), zp);
        zp = fmaf(bf16_lo(w.z), bf16_lo(h.z), zp);
        zp = fmaf(bf16_hi(w.z), bf16_hi(h.z), zp);
        zp = fmaf(bf16_lo(w.w), bf16_lo(h.w), zp);
        zp = fmaf(bf16_hi(w.w), bf16_hi(h.w), zp);
    }
    return zp;
}

__global__ void __launch_bounds__(kIdxMaxWarps * kWarp) index_kernel(const IndexArgs a) {
    __shared__ int32_t s_tail[kIdxTail];     // x[L_old - NMAX .. L_old + KMAX]
    __shared__ int32_t s_ver[3];             // accepted, new length, status
    __shared__ int32_t s_found[kIdxMaxWarps];
    __shared__ float s_wz[kIdxMaxWarps];
    __shared__ int32_t s_cend[SWITCHSD_WMAX];  // candidate mode: the listed ends, most recent first
    __shared__ int32_t s_ncf;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;
    const int b = blockIdx.x;
    const bool verifying = a.pv_len != nullptr;
    // With the prefetch bits (the caller's promise that the preceding kernel writes neither) the row's
    // length and tail, and the linear probe of row 0 of its state, are read before the wait.
    const bool pf_ctx = (a.prefetch & SWITCHSD_PREFETCH_CONTEXT) != 0;
    const bool pf_probe = (a.prefetch & SWITCHSD_PREFETCH_PROBE) != 0 && a.stepping && a.z1_part == nullptr &&
                          a.hidden_rows <= 1;
    float zp_early = 0.f;
    if (pf_probe) zp_early = index_probe_partial(a, b, 0);
    if (!pf_ctx) pdl_wait();

    if (tid == 0) s_ncf = 0;
    // The previous draft, the target (and the sampled rule's numbers), lane i positions i and i + 32: one round
    // of independent loads, after the wait.
    int32_t pv_n = 0, d_lo = 0, d_hi = 0, t_lo = 0, t_hi = 0, t_top = 0;
    float u_lo = 0.f, u_hi = 0.f, q_lo = 1.f, q_hi = 1.f, p_lo = 0.f, p_hi = 0.f;
    auto load_draft = [&]() {
        if (!verifying || a.W > 0 || warp != 0) return;
        const int32_t *dr = a.pv_draft + size_t(b) * a.k;
        const int32_t *tg = a.pv_target + size_t(b) * (a.k + 1);
        pv_n = __ldcg(a.pv_len + b);
        if (lane < a.k) d_lo = __ldcg(dr + lane);
        if (lane + 32 < a.k) d_hi = __ldcg(dr + lane + 32);
        if (lane <= a.k) t_lo = __ldcg(tg + lane);
        if (lane + 32 <= a.k) t_hi = __ldcg(tg + lane + 32);
        if (a.k >= 64) t_top = __ldcg(tg + 64);
        if (a.pv_p != nullptr) {
            const size_t o = size_t(b) * a.k + lane;
            if (lane < a.k) {
                u_lo = __ldcg(a.pv_u + o);
                p_lo = __ldcg(a.pv_p + o);
                if (a.pv_q) q_lo = __ldcg(a.pv_q + o);
            }
            if (lane + 32 < a.k) {
                u_hi = __ldcg(a.pv_u + o + 32);
                p_hi = __ldcg(a.pv_p + o + 32);
                if (a.pv_q) q_hi = __ldcg(a.pv_q + o + 32);
            }
        }
    };
    if (!pf_ctx) load_draft();
    int32_t *row = a.ctx + size_t(b) * a.cap;
    const int32_t L_old = __ldcg(a.lens + b);  // (rewritten each step: not from an L1 line of an earlier grid)
    const bool len_ok = L_old >= 1 && L_old <= a.cap;
    const int32_t tail0 = L_old - SWITCHSD_NMAX;  // s_tail[i] = x[tail0 + i]
    for (int i = tid; i < SWITCHSD_NMAX; i += blockDim.x) {
        const int32_t p = tail0 + i;
        s_tail[i] = (len_ok && p >= 0) ? __ldcg(row + p) : 0;
    }
    if (pf_ctx) {
        pdl_wait();  // the previous draft, the target and the index tables come after this
        load_draft();
    }
    pdl_trigger();
    if (warp == 0) {
        int32_t acc = -1, L = L_old, vst = len_ok ? SWITCHSD_ROW_OK : SWITCHSD_ROW_BAD_LEN;
        int32_t choice = 0;
        if (verifying && len_ok && a.W > 0) {
            // The previous W candidates: lane i tests positions i and i + 32 of each; the longest
            // accepted one is kept (the lowest index on a tie).  ncand = 0 is one empty candidate.
            const int32_t nc = a.pv_len[b];
            bool badlen = nc < 0 || nc > a.W;
            const int ncx = badlen ? 0 : (nc > 0 ? nc : 1);
            int32_t best = -1;
            for (int w = 0; w < ncx; ++w) {
                const size_t o = size_t(b) * a.W + w;
                const int32_t *c = a.pv_draft + o * a.D;
                const int32_t *t = a.pv_target + o * (a.D + 1);
                const int32_t c_lo = lane < a.D ? c[lane] : 0, c_hi = lane + 32 < a.D ? c[lane + 32] : 0;
                const int32_t t_lo = lane < a.D ? t[lane] : 0, t_hi = lane + 32 < a.D ? t[lane + 32] : 0;
                const int32_t len = nc > 0 ? a.pv_cand_len[o] : 0;
                badlen |= len < 0 || len > a.D;
                const unsigned m_lo = __ballot_sync(kFull, lane < len && c_lo != t_lo);
                const unsigned m_hi = __ballot_sync(kFull, lane + 32 < len && c_hi != t_hi);
                const int32_t acc_w = m_lo ? __ffs(m_lo) - 1 : (m_hi ? 32 + __ffs(m_hi) - 1 : len);
                if (acc_w > best) {
                    best = acc_w;
                    choice = w;
                }
            }
            if (badlen) {
                vst = SWITCHSD_ROW_BAD_LEN;
                choice = 0;
            } else if (L_old + best + 1 > a.cap) {
                vst = SWITCHSD_ROW_CAPACITY;
            } else {
                const size_t o = size_t(b) * a.W + choice;
                const int32_t *c = a.pv_draft + o * a.D;
                const int32_t tb = a.pv_target[o * (a.D + 1) + best];
                for (int i = lane; i <= best; i += kWarp) {
                    const int32_t t = i < best ? c[i] : tb;
                    s_tail[SWITCHSD_NMAX + i] = t;
                    row[L_old + i] = t;
                }
                acc = best;
                L = L_old + best + 1;
            }
        } else if (verifying && len_ok) {
            if (pv_n < 0 || pv_n > a.k) {
                vst = SWITCHSD_ROW_BAD_LEN;
            } else {
                // greedy: a draft token is rejected when it differs from the target's; sampled: when u * q
                // (binary32) is not below p
                bool rej_lo = lane < pv_n && d_lo != t_lo, rej_hi = lane + 32 < pv_n && d_hi != t_hi;
                if (a.pv_p != nullptr) {
                    rej_lo = lane < pv_n && !(__fmul_rn(u_lo, q_lo) < p_lo);
                    rej_hi = lane + 32 < pv_n && !(__fmul_rn(u_hi, q_hi) < p_hi);
                }
                const unsigned m_lo = __ballot_sync(kFull, rej_lo);
                const unsigned m_hi = __ballot_sync(kFull, rej_hi);
                acc = m_lo ? __ffs(m_lo) - 1 : (m_hi ? 32 + __ffs(m_hi) - 1 : pv_n);
                if (L_old + acc + 1 > a.cap) {
                    vst = SWITCHSD_ROW_CAPACITY;
                    acc = -1;
                } else {
                    const int32_t t_acc = __shfl_sync(kFull, acc < 32 ? t_lo : (acc < 64 ? t_hi : t_top), acc & 31);
                    for (int i = lane; i <= acc; i += kWarp) {
                        const int32_t t = i == acc ? t_acc : (i < 32 ? d_lo : d_hi);
                        s_tail[SWITCHSD_NMAX + i] = t;
                        row[L_old + i] = t;
                    }
                    L = L_old + acc + 1;
                }
            }
        }
        if (lane == 0) {
            s_ver[0] = acc;
            s_ver[1] = L;
            s_ver[2] = vst;
            if (verifying) a.out_accept[b] = acc;  // -1: nothing appended
            if (verifying && a.W > 0 && a.out_choice) a.out_choice[b] = choice;
            if (!a.stepping && a.status) a.status[b] = vst;
        }
    }
    __syncthreads();
    const int32_t L = s_ver[1];
    if (tid == 0 && verifying && len_ok) a.lens[b] = L;  // every warp has read the old length: behind the barrier
    const int n = a.n_min + warp;  // this warp's gram length
    const bool has_n = warp < a.n_max - a.n_min + 1;
    const size_t nb = size_t(1) << a.log2_buckets;
    int32_t *heads = a.heads + (size_t(warp) * a.B + b) * nb;
    int32_t *prev = a.prev + (size_t(warp) * a.B + b) * a.cap;
    auto tail_tok = [&](int32_t p) { return s_tail[p - tail0]; };  // valid for p in [tail0, L)

    // Insert the appended end positions p in [L_old, L) (lanes over p, chained through match_any).  The last of
    // them ends the suffix, so its link is where the lookup starts.
    int32_t e = -1;         // the chain of the suffix n-gram, the suffix's own end skipped
    bool linked = false;    // e is known from the insert
    if (has_n && L > L_old) {
        for (int32_t base = L_old; base < L; base += kWarp) {
            const int32_t p = base + lane;
            const bool valid = p < L && p >= n - 1;
            uint32_t bucket = 0xffffffffu;
            if (valid) bucket = gram_hash(n, [&](int i) { return tail_tok(p - i); }, a.log2_buckets);
            int32_t old_head = -1, old_link = -1;
            if (valid) {
                old_head = __ldcg(heads + bucket);
                if (p == L - 1) old_link = __ldcg(prev + p);  // p's link, if p was inserted before
            }
            const unsigned peers = __match_any_sync(kFull, bucket) & __ballot_sync(kFull, valid);
            __syncwarp();  // every lane has read its head before any lane replaces one
            // A head at or past p means these positions were inserted before (the same tokens appended
            // again after the lengths were rewound): the chains already hold them, so leave them be.
            // This keeps prev[p] < p, so every chain stays acyclic.
            int32_t link = old_head == p ? old_link : old_head;
            const bool fresh = valid && old_head < p;
            if (fresh) {
                const unsigned earlier = peers & ((1u << lane) - 1u);
                link = earlier ? base + (31 - __clz(earlier)) : old_head;
                prev[p] = link;
                if ((peers >> lane) == 1u) heads[bucket] = p;  // the latest position of the run
            }
            const unsigned last = __ballot_sync(kFull, valid && p == L - 1);
            if (last) {
                e = __shfl_sync(kFull, link, __ffs(last) - 1);
                linked = true;
            }
            __syncwarp();
        }
    }
    if (!a.stepping) return;

    // Lookup: the most recent earlier occurrence of the suffix n-gram, if any.  Candidate mode: the
    // warp of n = kappa lists the W most recent.  Per entry, the tokens compared, the next link and the
    // tokens that follow (the draft, should it match) are loaded at once: one round trip an entry.
    const int32_t kappa_c = a.kappa > 0 ? a.kappa : a.n_min;
    const bool collect = a.W > 0 && has_n && n == kappa_c;
    int32_t found = -1, nfound = 0;
    int32_t f_lo = 0, f_hi = 0;  // the tokens after `found`: e + 1 + lane, e + 33 + lane
    if (has_n && len_ok && L >= n + 1) {
        const int32_t mine = lane < n ? tail_tok(L - 1 - lane) : 0;
        if (!linked) {
            const uint32_t bucket = gram_hash(n, [&](int i) { return tail_tok(L - 1 - i); }, a.log2_buckets);
            const int32_t own = __ldcg(prev + L - 1);  // (an unbuilt index may hold anything here: used below only as a link)
            e = __ldcg(heads + bucket);
            if (e == L - 1) e = own;
        }
        auto tok = [&](int32_t p) { return p >= L_old ? tail_tok(p) : __ldcg(row + p); };
        // A valid chain strictly decreases and ends at -1 within L hops; the bounds keep a stale or
        // unbuilt index from reading outside its tables.
        for (int32_t hops = 0; e >= 0 && e < a.cap && hops < a.cap; ++hops) {
            const int32_t next = __ldcg(prev + e);
            if (e <= L - 2 && e >= n - 1) {
                const int32_t x = lane < n ? tok(e - lane) : 0;
                const int32_t lo = e + 1 + lane, hi = lo + 32;
                const int32_t y_lo = lane < a.k && lo < L ? tok(lo) : 0;
                const int32_t y_hi = lane + 32 < a.k && hi < L ? tok(hi) : 0;
                if (__all_sync(kFull, x == mine)) {
                    if (found < 0) {
                        found = e;
                        f_lo = y_lo;
                        f_hi = y_hi;
                    }
                    if (!collect) break;
                    if (lane == 0) s_cend[nfound] = e;
                    if (++nfound >= a.W) break;
                }
            }
            e = next;
        }
    }
    if (lane == 0 && warp < kIdxMaxWarps) s_found[warp] = found;
    if (collect && lane == 0) s_ncf = nfound;

    // Probe partial over the whole hidden vector (linear probe), or over every unit of the two-layer
    // probe: the S split-K partial sums in order, then b1, ReLU and w2.
    float zp = 0.f;
    if (a.z1_part != nullptr) {
        for (int u = tid; u < a.H1; u += blockDim.x) {
            float z1 = 0.f;
            for (int s = 0; s < a.mlp_S; ++s) z1 += a.z1_part[(size_t(s) * a.B + size_t(b)) * a.H1p + u];
            const float bias = a.b1 ? a.b1[u] : 0.f;
            zp = fmaf(bf16_lo(uint32_t(a.w2[u])), fmaxf(z1 + bias, 0.f), zp);
        }
    } else if (pf_probe) {
        zp = zp_early;
    } else {
        const int32_t hrow = a.hidden_rows > 1 && s_ver[0] > 0 ? s_ver[0] : 0;  // row a_b when gathering
        zp = index_probe_partial(a, b, hrow);
    }
    zp = warp_sum_f32(zp);
    if (lane == 0) s_wz[warp] = zp;
    __syncthreads();

    // Every thread takes the decision from shared memory (the same sums in the same order); thread 0 writes
    // it, and the winning n's warp its draft.
    float z = 0.f;
    for (int w = 0; w < nwarps; ++w) z += s_wz[w];
    if (a.z1_part != nullptr) z += a.b2;
    int win = a.n_max - a.n_min;
    while (win >= 0 && s_found[win] < 0) --win;
    const bool hit = len_ok && win >= 0;
    const int32_t nstar = win >= 0 ? a.n_min + win : 0, estar = win >= 0 ? s_found[win] : -1;
    const bool gate = a.W > 0 ? s_ncf > 0 : nstar >= kappa_c;
    int32_t mode = SWITCHSD_MODE_NO_REP;
    if (hit) mode = (gate && z >= a.logit_tau) ? SWITCHSD_MODE_COPY : SWITCHSD_MODE_REP_NO_COPY;
    const int32_t len = (a.W == 0 && mode == SWITCHSD_MODE_COPY) ? min(a.k, L - 1 - estar) : 0;
    const int32_t nc = mode == SWITCHSD_MODE_COPY ? s_ncf : 0;  // candidate mode: candidates written
    if (tid == 0) {
        if (a.W == 0 && a.counters)  // out_mode still holds the previous step's mode
            count_row(a.counters, mode, verifying, a.out_mode[b], s_ver[0]);
        a.out_mode[b] = mode;
        if (a.W == 0) a.out_len[b] = len;
        else a.out_ncand[b] = nc;
        a.out_score[b] = z;
        if (a.out_match_n) a.out_match_n[b] = nstar;
        if (a.out_match_end) a.out_match_end[b] = estar;
        if (a.status) a.status[b] = s_ver[2];
    }
    if (a.W > 0) {
        // The candidates' continuations x[e_w+1 .. e_w+len_w], len_w = min(D, L-1-e_w).
        for (int t = tid; t < nc * a.D; t += blockDim.x) {
            const int w = t / a.D, i = t - w * a.D;
            const int32_t ew = s_cend[w];
            const int32_t lw = min(a.D, L - 1 - ew);
            const int32_t p = ew + 1 + i;
            if (i == 0) a.out_cand_len[size_t(b) * a.W + w] = lw;
            if (i < lw) a.out_cand[(size_t(b) * a.W + w) * a.D + i] = p >= L_old ? tail_tok(p) : row[p];
        }
        return;
    }
    if (warp == win) {  // the copy draft x[e+1 .. e+len], loaded with the match
        int32_t *out = a.out_draft + size_t(b) * a.k;
        if (lane < len) out[lane] = f_lo;
        if (lane + 32 < len) out[lane + 32] = f_hi;
    }
}

// ------------------------------------------------------------------------------------------------
// Build.  One item = one (row, n); its buckets are split over P CTAs (part = the bucket's top bits; a few calls take
// index_walk_kernel below).  A CTA goes over the row in chunks of kChunk positions; per chunk, warp w owns a contiguous segment:
//   1. hash and rank: every position's bucket, positions of other parts dropped, and its rank within the
//      segment's positions of its bin (the next 6 to 8 bits of the bucket), kept in registers; the lanes of a bin
//      find each other through a mask per bin in shared memory (an atomicOr, a read), and the segment's counts
//      per bin run along;
//   2. scan: offsets of every (bin, warp), so that a bin's entries lie in position order;
//   3. scatter: (position, key) into a queue in shared memory, key = the bucket's remaining bits (<= 9);
//   4. link: warp w takes the bins w, w + kW, ... on its own (no barrier): the bin's heads (<= 512, 16-bit
//      chunk positions) live in shared memory, the entries are linked 32 at a time in order (entries of one key
//      in a round find each other through the head that one of them holds), and the bin's heads go out in one
//      coalesced write, the empty ones included (so nothing clears the table first);
//   5. the links, held in shared memory as 16-bit chunk positions, go out coalesced (P = 1; with P > 1 a
//      part's positions are scattered and step 4 stores them).
// Steps 1 to 3 are one stable radix pass, so the time does not depend on how the tokens repeat, except that
// one bucket's entries are linked by one warp.  A later chunk takes the head of a bucket it has not seen
// from the table its own bins' warp wrote (same warp, earlier chunk) and updates only the heads it moved.
//
// Why: one warp per item walking its row 32 positions at a time (a dependent head read and write each) took
// 1210 us for 64 rows of 32K tokens, n = 3..8 (build and one step); this takes 120 us, and 144 with 256 bins
// instead of 128.  With 256: ranks by eight ballots a position, counted in a pass of their own 177 us; the groups
// of equal keys in a round of step 4 by nine ballots
// (six rounds in ten hold one) 155 us.  The tokens staged in shared memory by one copy made no difference.  The
// table written sets the floor (101 MB of heads + 50 MB of links: 22 us at the measured copy bandwidth); what
// bounds it is the shared-memory pipe (random accesses, three to four wavefronts each: 70 % of its peak while a
// CTA runs) and the issue rate, at one 1024-thread CTA an SM, 2.5 waves of them here.
// ------------------------------------------------------------------------------------------------
// A bucket within its part: bin (at most 8 bits) and key (at most 9).  A position's rank within its segment and bin
// (below 1024), and in the queue its place in the chunk (15 bits), stand above it.
constexpr int kLocalBits = 17;
constexpr uint32_t kNone16 = 0xffffu;  // no earlier entry; kDone16: the link is in global memory already
constexpr uint32_t kDone16 = 0xfffeu;

struct BuildArgs {
    const int32_t *ctx, *lens;
    int32_t *heads, *prev;
    int32_t B, cap, n_min, nn, log2_buckets, log2_parts;
};

template <int kT, int kChunk, int kBinBits, int kKeyBits>
struct BuildLayout {
    static constexpr int kW = kT / kWarp, kBins = 1 << kBinBits;
    static constexpr size_t queue = size_t(kChunk) * 4;
    static constexpr size_t counts = size_t(kW) * (kBins + 1) * 4;
    static constexpr size_t links = ((size_t(kChunk) * 2 > counts ? size_t(kChunk) * 2 : counts) + 15) & ~size_t(15);  // then links
    static constexpr int warp_heads = (2 << kKeyBits) > 4 * kBins ? 2 << kKeyBits : 4 * kBins;
    static constexpr size_t heads = size_t(kW) * warp_heads;  // per warp step 1's masks, then a bin's heads
    static constexpr size_t bytes = queue + links + heads;
};

template <int kT, int kChunk, int kBinBits, int kKeyBits>
__global__ void __launch_bounds__(kT, 1024 / kT) index_build_kernel(const BuildArgs a) {
    using Lay = BuildLayout<kT, kChunk, kBinBits, kKeyBits>;
    static_assert(kBinBits + kKeyBits <= kLocalBits, "a bucket's bits");
    constexpr int kW = Lay::kW, kBins = Lay::kBins;
    constexpr int kIts = kChunk / kT;  // positions a thread holds
    static_assert(kIts % 8 == 0 && kChunk <= 32768, "15-bit chunk positions, rounds of eight");
    extern __shared__ __align__(16) unsigned char build_smem[];
    uint32_t *q = reinterpret_cast<uint32_t *>(build_smem);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(build_smem + Lay::queue);     // [kW][kBins + 1]
    uint16_t *links = reinterpret_cast<uint16_t *>(build_smem + Lay::queue);   // [kChunk]
    uint16_t *heads16 = reinterpret_cast<uint16_t *>(build_smem + Lay::queue + Lay::links);
    __shared__ uint32_t s_bin[kBins + 1];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = int(blockIdx.x) & ((1 << a.log2_parts) - 1);
    const int item = int(blockIdx.x) >> a.log2_parts;
    const int w = item / a.B, b = item - w * a.B;
    const int n = a.n_min + w;
    const int lg = a.log2_buckets, lgp = lg - a.log2_parts;  // bucket bits, and those within the part
    const int binbits = lgp < kBinBits ? lgp : kBinBits, keybits = lgp - binbits;
    const uint32_t keymask = (1u << keybits) - 1u, localmask = (1u << lgp) - 1u;
    pdl_wait();
    pdl_trigger();
    int32_t *heads = a.heads + (size_t(w) * a.B + b) * (size_t(1) << lg) + (size_t(part) << lgp);
    int32_t *prev = a.prev + (size_t(w) * a.B + b) * size_t(a.cap);
    const int32_t *row = a.ctx + size_t(b) * size_t(a.cap);
    int32_t L = a.lens[b];
    if (L < 0 || L > a.cap) L = 0;
    uint16_t *H = heads16 + warp * (Lay::warp_heads / 2);

    for (int32_t c0 = 0; c0 == 0 || c0 < L; c0 += kChunk) {
        const int32_t clen = min(kChunk, L - c0);
        const int32_t seg = ((clen + kW - 1) / kW + 31) & ~31;  // a warp's positions: <= kChunk / kW
        const int32_t p_seg = c0 + warp * seg;
        for (int i = tid; i < kW * (kBins + 1); i += kT) cnt[i] = 0u;
        for (int i = tid; i < int(Lay::heads / 4); i += kT) reinterpret_cast<uint32_t *>(heads16)[i] = 0u;
        __syncthreads();

        // 1. hash and rank
        uint32_t *mask = reinterpret_cast<uint32_t *>(H), *my = cnt + warp * (kBins + 1);
        uint32_t code[kIts];  // rank << kLocalBits | the bucket in the part, all ones for a dropped position
        const int32_t p_end = min(L, p_seg + seg);
#pragma unroll
        for (int r = 0; r < kIts / 8; ++r) {
            uint64_t h[8];
            const int32_t p0 = p_seg + 256 * r;
#pragma unroll
            for (int u = 0; u < 8; ++u) h[u] = 0u;
            if (256 * r < seg && p0 < L) {  // warp-uniform
                uint32_t pw = 1u;
                if (p0 >= n - 1 && p0 + 256 <= L) {
                    const int32_t *x = row + p0 + lane;
                    for (int i = 0; i < n; ++i, --x, pw *= kGramMul)
#pragma unroll
                        for (int u = 0; u < 8; ++u) h[u] += uint64_t(uint32_t(x[32 * u])) * pw;
                } else {
                    for (int i = 0; i < n; ++i, pw *= kGramMul)
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            h[u] += uint64_t(uint32_t(row[min(max(p0 + lane + 32 * u - i, 0), L - 1)])) * pw;
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int32_t p = p0 + 32 * u + lane;
                const uint32_t bucket = gram_bucket(h[u], n, lg);
                const bool mine = p >= n - 1 && p < p_end && int(bucket >> lgp) == part;
                const uint32_t local = bucket & localmask;
                const uint32_t bin = local >> keybits;
                if (mine) atomicOr(&mask[bin], 1u << lane);
                __syncwarp();
                const uint32_t peers = mine ? mask[bin] : 0u, at = mine ? my[bin] : 0u;
                const uint32_t below = peers & ((1u << lane) - 1u);
                __syncwarp();  // every lane has read its bin before the bin's first lane moves it on
                if (mine && below == 0u) {
                    my[bin] = at + uint32_t(__popc(peers));
                    mask[bin] = 0u;
                }
                code[8 * r + u] = mine ? (at + uint32_t(__popc(below))) << kLocalBits | local : 0xffffffffu;
                __syncwarp();
            }
        }
        __syncthreads();

        // 2. offsets: within a bin over the warps, then over the bins
        for (int bin = warp; bin < kBins; bin += kW) {
            const uint32_t v = lane < kW ? cnt[lane * (kBins + 1) + bin] : 0u;
            uint32_t incl = v;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane < kW) cnt[lane * (kBins + 1) + bin] = incl - v;
            if (lane == kWarp - 1) s_bin[bin + 1] = incl;
        }
        if (tid == 0) s_bin[0] = 0u;
        __syncthreads();
        if (warp == 0) {
            uint32_t v[kBins / kWarp], sum = 0u;
#pragma unroll
            for (int j = 0; j < kBins / kWarp; ++j) {
                sum += s_bin[1 + lane * (kBins / kWarp) + j];
                v[j] = sum;
            }
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
#pragma unroll
            for (int j = 0; j < kBins / kWarp; ++j)
                s_bin[1 + lane * (kBins / kWarp) + j] = incl - sum + v[j];
        }
        __syncthreads();
        for (int i = tid; i < kW * kBins; i += kT)  // a (bin, warp)'s place in the queue
            cnt[(i >> kBinBits) * (kBins + 1) + (i & (kBins - 1))] += s_bin[i & (kBins - 1)];
        __syncthreads();

        // 3. scatter into the queue, in position order within a bin
#pragma unroll
        for (int i = 0; i < kIts; ++i) {
            const uint32_t c = code[i];
            if (c != 0xffffffffu) {
                const uint32_t local = c & ((1u << kLocalBits) - 1u), bin = local >> keybits;
                const uint32_t lp = uint32_t(p_seg - c0 + 32 * i + lane);
                q[my[bin] + (c >> kLocalBits)] = lp << kLocalBits | local;
            }
        }
        __syncthreads();  // the counters are dead from here on: the links take their place

        // 4. link each bin's entries in order
        const int nbins = 1 << binbits, kb = 1 << keybits;
        for (int bin = warp; bin < nbins; bin += kW) {
            for (int i = lane; i < (kb + 7) / 8; i += kWarp)  // H holds 1 << kKeyBits entries
                reinterpret_cast<uint4 *>(H)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
            __syncwarp();
            int32_t *hb = heads + (size_t(bin) << keybits);
            const uint32_t end = s_bin[bin + 1];
            // one round of 32 entries: (position, link), the link kNone16 when the bin holds no earlier entry
            auto round = [&](uint32_t base, bool live, uint32_t &key, uint32_t &lp) {
                const uint32_t ent = live ? q[base + lane] : 0u;
                key = ent & keymask;
                lp = ent >> kLocalBits;
                uint32_t l16 = live ? uint32_t(H[key]) : kNone16;
                __syncwarp();  // every lane has read its head before any lane replaces one
                if (live) H[key] = uint16_t(lp);
                __syncwarp();
                // Entries of one key in a round: one of them holds H now, the others see it.  Such a group
                // (one a round, mostly two entries) links each entry to the one before it; the last is the head.
                for (unsigned todo = __ballot_sync(kFull, live && uint32_t(H[key]) != lp); todo != 0u;) {
                    const uint32_t k = __shfl_sync(kFull, key, __ffs(todo) - 1);
                    const bool in = live && key == k;
                    const unsigned peers = __ballot_sync(kFull, in);
                    const unsigned earlier = peers & ((1u << lane) - 1u);
                    const uint32_t before = __shfl_sync(kFull, lp, earlier ? 31 - __clz(earlier) : lane);
                    if (in && earlier) l16 = before;
                    if (in && (peers >> lane) == 1u) H[key] = uint16_t(lp);
                    todo &= ~peers;
                }
                __syncwarp();
                return l16;
            };
            uint32_t key, lp;
            if (c0 == 0 && a.log2_parts == 0) {
                for (uint32_t base = s_bin[bin]; base < end; base += kWarp) {
                    const bool live = base + lane < end;
                    const uint32_t l16 = round(base, live, key, lp);
                    if (live) links[lp] = uint16_t(l16);
                }
            } else {
                for (uint32_t base = s_bin[bin]; base < end; base += kWarp) {
                    const bool live = base + lane < end;
                    uint32_t l16 = round(base, live, key, lp);
                    if (live) {
                        if (a.log2_parts > 0 || l16 == kNone16) {
                            // an earlier chunk's head: from the table, where this warp left it
                            prev[c0 + int32_t(lp)] = l16 != kNone16 ? c0 + int32_t(l16) : (c0 > 0 ? hb[key] : -1);
                            l16 = kDone16;
                        }
                        if (a.log2_parts == 0) links[lp] = uint16_t(l16);
                    }
                }
            }
            __syncwarp();
            if (c0 == 0 && kb >= 4) {
                for (int i = lane; i < kb / 4; i += kWarp) {
                    const short4 h = reinterpret_cast<const short4 *>(H)[i];  // kNone16 widens to -1
                    reinterpret_cast<int4 *>(hb)[i] = make_int4(h.x, h.y, h.z, h.w);
                }
            } else {
                for (int i = lane; i < kb; i += kWarp) {
                    const uint32_t h = H[i];
                    if (h != kNone16) hb[i] = c0 + int32_t(h);
                    else if (c0 == 0) hb[i] = -1;
                }
            }
            __syncwarp();
        }
        __syncthreads();

        // 5. the links, four positions a thread (positions below n - 1 belong to no chain)
        if (a.log2_parts == 0) {
            for (int i = tid; 4 * i < clen; i += kT) {
                const short4 l = reinterpret_cast<const short4 *>(links)[i];
                int32_t *dst = prev + c0 + 4 * i;
                if (c0 == 0) {  // kNone16 widens to -1, and no link is in global memory yet
                    *reinterpret_cast<int4 *>(dst) = make_int4(l.x, l.y, l.z, l.w);
                } else {  // every link here is to an entry of this chunk, or in global memory already
                    if (uint16_t(l.x) != kDone16) dst[0] = c0 + l.x;
                    if (uint16_t(l.y) != kDone16) dst[1] = c0 + l.y;
                    if (uint16_t(l.z) != kDone16) dst[2] = c0 + l.z;
                    if (uint16_t(l.w) != kDone16) dst[3] = c0 + l.w;
                }
            }
        }
        __syncthreads();  // the queue and the counters' space are free for the next chunk
    }
}

// The same tables from one warp per item, which inserts its row's positions in increasing order, 32 at a time, into
// heads that were set to -1 before (a dependent head read and write per 32 positions: about 1.4 us, whatever the
// number of items up to a thousand or so).  For many short rows, where a CTA per item costs its fixed steps, and for
// many rows so long that index_build_kernel would go over each of them once per part (index_walks).
constexpr int kWalkWarps = 8;
__global__ void __launch_bounds__(kWalkWarps * kWarp) index_walk_kernel(const BuildArgs a) {
    const int lane = threadIdx.x & 31;
    const int item = int(blockIdx.x) * kWalkWarps + int(threadIdx.x >> 5);
    pdl_wait();
    pdl_trigger();
    if (item >= a.nn * a.B) return;
    const int w = item / a.B, b = item - w * a.B;
    const int n = a.n_min + w;
    int32_t *heads = a.heads + (size_t(w) * a.B + b) * (size_t(1) << a.log2_buckets);
    int32_t *prev = a.prev + (size_t(w) * a.B + b) * size_t(a.cap);
    const int32_t *row = a.ctx + size_t(b) * size_t(a.cap);
    int32_t L = a.lens[b];
    if (L < 0 || L > a.cap) L = 0;
    for (int32_t base = n - 1; base < L; base += kWarp) {
        const int32_t p = base + lane;
        const bool valid = p < L;
        uint32_t bucket = 0xffffffffu;
        if (valid) bucket = gram_hash(n, [&](int i) { return row[p - i]; }, a.log2_buckets);
        const unsigned peers = __match_any_sync(kFull, bucket) & __ballot_sync(kFull, valid);
        const int32_t old_head = valid ? heads[bucket] : -1;
        __syncwarp();  // every lane has read its head before any lane replaces one
        if (valid) {
            const unsigned earlier = peers & ((1u << lane) - 1u);
            prev[p] = earlier ? base + (31 - __clz(earlier)) : old_head;
            if ((peers >> lane) == 1u) heads[bucket] = p;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------------
// Host side.
// ------------------------------------------------------------------------------------------------
// The build's parts per item: enough that a part's buckets fit 1 << kBinBits bins of 1 << kKeyBits heads,
// and more (up to 8) while the grid leaves SMs idle -- every part hashes the whole row, so more parts only
// pay while they add CTAs.
//
// The instance by the row's capacity: the smallest chunk that takes it whole, with as many CTAs an SM as make 1024
// threads (four, two, one), and the fewest bins whose heads fit (a bin costs its round trips whatever it holds).
// Build and one step, n = 3..8 unless given, us (the warp-per-item walk; 512 threads, 16384, 8 bin bits up to 16K
// rows and 1024, 32768, 8 above; now):
//   44 rows of 1.4K, n = 2..9   57.8, 65.6, 23.2      64 of 4K, n = 2..12   158.6, about 95, 48.6
//   64 rows of 8K, n = 2..12    305.6, 160.4, 91.0    64 of 16K             567.8, 124.5, 77.5    64 of 32K  1203, 144, 120
// (With 8 bin bits two CTAs of 512 threads do not fit an SM.)  Where the repeats fall on few buckets, more bins would
// be a little quicker: 64 rows of 32K tokens of code 219 with 8 bits, 232 with 7.  Past 2^16 buckets 7 bits would
// need twice the parts: 16 rows of 128K, n = 2..5, 188 with 8, 219 with 7.  Chunks of 16384 for 32K rows: 179.
template <int kT, int kChunk, int kBinBits, int kKeyBits>
static cudaError_t launch_index_build(BuildArgs a, cudaStream_t stream) {
    constexpr auto kernel = index_build_kernel<kT, kChunk, kBinBits, kKeyBits>;
    constexpr size_t smem = BuildLayout<kT, kChunk, kBinBits, kKeyBits>::bytes;
    static int sms[64] = {0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int n_sm = dev >= 0 && dev < 64 ? sms[dev] : 0;
    if (n_sm == 0) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) sms[dev] = n_sm;
    }
    const int64_t items = int64_t(a.nn) * a.B;
    int lp = a.log2_buckets > kBinBits + kKeyBits ? a.log2_buckets - kBinBits - kKeyBits : 0;
    while (lp < 3 && (items << (lp + 1)) <= n_sm && a.log2_buckets - lp > 8) ++lp;
    a.log2_parts = lp;
    return launch_pdl(kernel, dim3(unsigned(items << lp)), dim3(kT), smem, stream, 0u, a);
}

// Parts that an item's buckets need (log2): a part has at most 8 bits of bins and 9 of keys.
static int index_parts_needed(int log2_buckets) { return log2_buckets > 17 ? log2_buckets - 17 : 0; }

// Whether the build takes the warp-per-item walk.  Measured, us, zipf text (walk, index_build_kernel; items = rows x n):
//   short rows  items of 64: 1 6.1, 9.6   96 6.3, 9.9   24,576 18.6, 463      256: 6 8.9, 11.2   384 11.2, 17.3
//               512: 6 13.2, 11.2   384 17.3, 17.6   1,536 19.1, 43.4      1K: 384 30.1, 19.4   1,536 33.2, 47.5
//               1.5K: 384 43.7, 20.4   1,536 49.6, 50.6   6,144 150, 175   2K: 2,400 87, 92   6,144 193, 198   24,576 818, 769
//   long rows   (ms) 300K (8 parts): 1,024 14.8, 16.3   2,048 24.9, 32.5       600K (16): 384 23.5, 22.1   768 27.0, 44.0
//               1M (16): 384 48.5, 37.1   660 45.1, 64.3      2M (32): 192 104, 71   240 90, 89   288 84, 107
//               4M (64): 48 183, 67   144 177, 204      8M (128): 24 372, 128   72 375, 373
// The long rows' line is where items x parts pass about 8,192 (index_build_kernel's time per token goes by it, the
// walk's does not); with 4 parts and fewer the walk is never ahead (2,048 items of 256K: 21.1 and 15.3).  Rows of few
// distinct n-grams, whose heads stay in L2, would take the walk earlier (64 rows of 600K, period 64: 14.5 and 22.3).
static bool index_walks(int32_t cap, int64_t items, int log2_buckets) {
    const int lp = index_parts_needed(log2_buckets);
    const bool short_rows = cap <= 256 || (cap <= 1536 && items >= cap) || (cap <= 2048 && items >= cap && items <= 8192);
    return short_rows || (lp >= 3 && (items << lp) > 8192);
}

static cudaError_t launch_index_walk(const BuildArgs &a, cudaStream_t stream) {
    const size_t items = size_t(a.nn) * size_t(a.B);
    const cudaError_t e = cudaMemsetAsync(a.heads, 0xff, items * (size_t(1) << a.log2_buckets) * sizeof(int32_t), stream);
    if (e != cudaSuccess) return e;  // (every head -1)
    return launch_pdl(index_walk_kernel, dim3(unsigned((items + kWalkWarps - 1) / kWalkWarps)), dim3(kWalkWarps * kWarp), 0,
                      stream, 0u, a);
}

int index_n_min(const switchsd_index *idx) { return idx->n_min; }
int index_n_max(const switchsd_index *idx) { return idx->n_max; }

int index_launch(switchsd_index *idx, int32_t *ctx, int32_t *lens, const uint16_t *hidden, const uint16_t *probe_w,
                 const float *z1_part, const float *b1, const uint16_t *w2, int mlp_S, int H1, int H1p, float b2,
                 const int32_t *pv_draft, const int32_t *pv_target, const int32_t *pv_len, int32_t *out_accept,
                 int32_t *out_draft, int32_t *out_len, int32_t *out_mode, float *out_score, int32_t *out_match_n,
                 int32_t *out_match_end, int32_t *status, int B, int cap, int d, int k, int n_min, int n_max, int kappa,
                 float logit_tau, bool stepping, cudaStream_t stream, const float *pv_p, const float *pv_q,
                 const float *pv_u, int hidden_rows, const IndexCandidates *cand, int prefetch,
                 unsigned long long *counters) {
    if (idx->B != B || idx->cap != cap || idx->n_min != n_min || idx->n_max != n_max) return SWITCHSD_ERR_SHAPE;
    // Candidate mode lists the ends of the kappa-gram chain: kappa must be one of the index's n, or
    // above n_max (no end can then reach it: no candidate, as for the rescan).
    if (cand != nullptr && (kappa > 0 ? kappa : n_min) < n_min) return SWITCHSD_ERR_SHAPE;
    IndexArgs a;
    a.W = cand ? cand->W : 0;
    a.D = cand ? cand->D : 0;
    a.pv_cand_len = cand ? cand->pv_cand_len : nullptr;
    a.out_choice = cand ? cand->out_choice : nullptr;
    a.out_cand = cand ? cand->out_cand : nullptr;
    a.out_cand_len = cand ? cand->out_cand_len : nullptr;
    a.out_ncand = cand ? cand->out_ncand : nullptr;
    a.prefetch = prefetch;
    a.counters = stepping ? counters : nullptr;
    a.pv_p = pv_p;
    a.pv_q = pv_q;
    a.pv_u = pv_u;
    a.hidden_rows = hidden_rows;
    a.ctx = ctx;
    a.lens = lens;
    a.hidden = hidden;
    a.probe_w = probe_w;
    a.z1_part = z1_part;
    a.b1 = b1;
    a.w2 = w2;
    a.mlp_S = mlp_S;
    a.H1 = H1;
    a.H1p = H1p;
    a.b2 = b2;
    a.pv_draft = pv_draft;
    a.pv_target = pv_target;
    a.pv_len = pv_len;
    a.out_accept = out_accept;
    a.out_draft = out_draft;
    a.out_len = out_len;
    a.out_mode = out_mode;
    a.out_score = out_score;
    a.out_match_n = out_match_n;
    a.out_match_end = out_match_end;
    a.status = status;
    a.heads = idx->heads;
    a.prev = idx->prev;
    a.B = B;
    a.cap = cap;
    a.d = d;
    a.k = k;
    a.n_min = n_min;
    a.n_max = n_max;
    a.kappa = kappa;
    a.log2_buckets = idx->log2_buckets;
    a.stepping = stepping ? 1 : 0;
    a.logit_tau = logit_tau;
    const cudaError_t e = launch_pdl(index_kernel, dim3(unsigned(B)), dim3(unsigned(idx->nn * kWarp)), 0, stream, 0u, a);
    return e == cudaSuccess ? SWITCHSD_OK : SWITCHSD_ERR_CUDA;
}

}  // namespace switchsd

using namespace switchsd;

extern "C" int switchsd_index_create(const switchsd_params *p, switchsd_index **out) {
    if (!p || !out) return SWITCHSD_ERR_ARG;
    *out = nullptr;
    if (p->B < 1 || p->B > 65535 || p->cap < 4 || (p->cap & 3) != 0) return SWITCHSD_ERR_SHAPE;
    if (p->n_min < 1 || p->n_max > SWITCHSD_NMAX || p->n_min > p->n_max) return SWITCHSD_ERR_SHAPE;
    switchsd_index *idx = new (std::nothrow) switchsd_index();
    if (!idx) return SWITCHSD_ERR_CUDA;
    idx->B = p->B;
    idx->cap = p->cap;
    idx->n_min = p->n_min;
    idx->n_max = p->n_max;
    idx->nn = p->n_max - p->n_min + 1;
    int lg = 4;
    while ((int64_t(1) << lg) < 2 * int64_t(p->cap) && lg < 30) ++lg;  // load factor <= 1/2
    idx->log2_buckets = lg;
    cudaGetDevice(&idx->device);
    const size_t heads = size_t(idx->nn) * size_t(p->B) * (size_t(1) << lg) * sizeof(int32_t);
    const size_t prev = size_t(idx->nn) * size_t(p->B) * size_t(p->cap) * sizeof(int32_t);
    if (cudaMalloc(&idx->heads, heads) != cudaSuccess) {
        delete idx;
        return SWITCHSD_ERR_CUDA;
    }
    if (cudaMalloc(&idx->prev, prev) != cudaSuccess) {
        cudaFree(idx->heads);
        delete idx;
        return SWITCHSD_ERR_CUDA;
    }
    *out = idx;
    return SWITCHSD_OK;
}

extern "C" int switchsd_index_build(switchsd_index *idx, const int32_t *ctx_tokens, const int32_t *ctx_lens,
                                    void *stream) {
    if (!idx || !ctx_tokens || !ctx_lens) return SWITCHSD_ERR_ARG;
    BuildArgs a;
    a.ctx = ctx_tokens;
    a.lens = ctx_lens;
    a.heads = idx->heads;
    a.prev = idx->prev;
    a.B = idx->B;
    a.cap = idx->cap;
    a.n_min = idx->n_min;
    a.nn = idx->nn;
    a.log2_buckets = idx->log2_buckets;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    a.log2_parts = 0;
    const cudaError_t e =
        index_walks(a.cap, int64_t(a.nn) * a.B, a.log2_buckets) ? launch_index_walk(a, st)
        : idx->cap <= 4096         ? launch_index_build<256, 4096, 6, 7>(a, st)
        : idx->cap <= 8192         ? launch_index_build<256, 8192, 7, 8>(a, st)
        : idx->cap <= 16384        ? launch_index_build<512, 16384, 7, 8>(a, st)
        : idx->log2_buckets <= 16  ? launch_index_build<1024, 32768, 7, 9>(a, st)
                                   : launch_index_build<1024, 32768, 8, 9>(a, st);
    return e == cudaSuccess ? SWITCHSD_OK : SWITCHSD_ERR_CUDA;
}

extern "C" size_t switchsd_index_bytes(const switchsd_index *idx) {
    if (!idx) return 0;
    return size_t(idx->nn) * size_t(idx->B) * ((size_t(1) << idx->log2_buckets) + size_t(idx->cap)) * sizeof(int32_t);
}

extern "C" void switchsd_index_destroy(switchsd_index *idx) {
    if (!idx) return;
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != idx->device) cudaSetDevice(idx->device);
    cudaFree(idx->heads);
    cudaFree(idx->prev);
    if (cur != idx->device) cudaSetDevice(cur);
    delete idx;
}
