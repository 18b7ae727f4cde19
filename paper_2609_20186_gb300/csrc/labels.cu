// labels.cu -- switchsd_copy_labels: copy-mode labels of every position of B rows (§3.2).
//
// Position j of a row is labelled 1 when it lies in a window of n consecutive tokens that also occurs
// starting at an earlier position of the row (the paper trains its probe on these labels with
// n = n_train = 5).
//
// Short rows, and longer ones where the batch fills the chip (label_one_kernel): one kernel, a cluster of P CTAs
// per row.  The windows are split over the CTAs by hash; each CTA hashes every window of the row and inserts its own into an
// open-addressing table in its shared memory.  A slot holds hash bits above the smallest start so far of one
// window: an empty slot is claimed with an atomicCAS, a slot whose bits and tokens agree takes an atomicMin,
// and whichever of the two starts is the larger is marked in the CTA's bitmap -- every start but the smallest
// of its window is marked exactly once, in whatever order they come.  Each warp keeps its windows in two
// stacks, those to try at a slot and those to compare, and takes 32 of one at a time: a window that has to go
// on to the next slot goes back on the stack, so no lane waits for another's probe sequence.
// The cluster then ORs the P bitmaps through distributed shared memory, and position j takes the OR of the n
// marks that cover it.  No global table, no clear and no second pass.
//
// What bounds it is the issue rate of the hashing (P times a row) and of the inserts.  64 rows of 16K..32K
// tokens, n = 5: 55.9 us with the two kernels below and their table in memory (a chain of dependent random L2
// atomics a window), 36.5 us with each lane following its own probe sequence, 27.5 us with the stacks, 29.1 us
// with hash sums of 64 bits instead of 32 (kept, so that ids that differ in their high bits alone still spread).
//
// Other long rows: two kernels over a per-row table in the caller's workspace, which spread a row's windows over
// the whole chip.
//   insert  thread per window start s: hash the n tokens, probe linearly; an empty slot is claimed with
//           atomicCAS, a slot whose window holds the same tokens takes atomicMin(slot, s).  Every slot
//           then holds the smallest start among the windows with its tokens -- the same value whatever
//           order the inserts ran in.  The slot of s is recorded in where[s].
//   label   CTA per 256 positions: for the window starts s in [j0 - n + 1, j0 + 256) it reads the slot
//           of s and marks s when the slot's smallest start is below s (the window repeats); position
//           j is then the OR of the marks of the n windows that cover it.
// That table has a power of two >= 2 * cap slots per row (load factor <= 1/2), so every probe sequence
// ends within the table.  Windows are compared token by token, so hash collisions cost time only.
#include "common.cuh"

namespace switchsd {

constexpr int kLabelThreads = 256;

struct LabelArgs {
    const int32_t *ctx, *lens;
    int32_t *table;     // [B][T]
    int32_t *where;     // [B][cap]: the slot of each window start
    uint8_t *labels;    // [B][cap]
    int32_t B, cap, n;
    uint32_t tmask;     // T - 1
};

__device__ __forceinline__ uint32_t window_hash(const int32_t *w, int n, uint32_t tmask) {
    uint64_t h = 0x9E3779B97F4A7C15ull ^ uint64_t(n);
    for (int i = 0; i < n; ++i) {
        h = (h ^ uint64_t(uint32_t(w[i]))) * 0xBF58476D1CE4E5B9ull;
        h ^= h >> 31;
    }
    return uint32_t(h ^ (h >> 32)) & tmask;
}

__device__ __forceinline__ bool same_window(const int32_t *a, const int32_t *b, int n) {
    for (int i = 0; i < n; ++i)
        if (a[i] != b[i]) return false;
    return true;
}

__device__ __forceinline__ int32_t row_length(const LabelArgs &a, int b) {
    const int32_t L = a.lens[b];
    return (L >= 0 && L <= a.cap) ? L : 0;  // a length outside [0, cap] labels nothing
}

__global__ void __launch_bounds__(kLabelThreads) label_insert_kernel(const LabelArgs a) {
    const int b = blockIdx.y;
    const int32_t s = int32_t(blockIdx.x) * kLabelThreads + threadIdx.x;
    pdl_wait();
    pdl_trigger();
    const int32_t L = row_length(a, b);
    if (s + a.n > L) return;
    const int32_t *x = a.ctx + size_t(b) * size_t(a.cap);
    int32_t *tab = a.table + size_t(b) * (size_t(a.tmask) + 1);
    int32_t *where = a.where + size_t(b) * size_t(a.cap);
    uint32_t h = window_hash(x + s, a.n, a.tmask);
    for (uint32_t probe = 0; probe <= a.tmask; ++probe, h = (h + 1) & a.tmask) {
        // Claim the slot if empty; otherwise the CAS returns its start (one round trip either way).
        const int32_t v = atomicCAS(&tab[h], -1, s);
        if (v < 0) {
            where[s] = int32_t(h);
            return;
        }
        if (same_window(x + v, x + s, a.n)) {
            atomicMin(&tab[h], s);
            where[s] = int32_t(h);
            return;
        }
    }
}

__global__ void __launch_bounds__(kLabelThreads) label_mark_kernel(const LabelArgs a) {
    __shared__ uint8_t s_rep[kLabelThreads + SWITCHSD_NMAX];  // window repeats, for starts j0 - n + 1 ..
    const int b = blockIdx.y;
    const int32_t j0 = int32_t(blockIdx.x) * kLabelThreads;
    pdl_wait();
    pdl_trigger();
    const int32_t L = row_length(a, b);
    const int32_t *tab = a.table + size_t(b) * (size_t(a.tmask) + 1);
    const int32_t *where = a.where + size_t(b) * size_t(a.cap);
    const int32_t first = j0 - a.n + 1;
    for (int t = threadIdx.x; t < kLabelThreads + a.n - 1; t += kLabelThreads) {
        const int32_t s = first + t;
        uint8_t rep = 0;
        if (s >= 0 && s + a.n <= L) {
            const int32_t h = where[s];  // written by the insert of s
            rep = h >= 0 && uint32_t(h) <= a.tmask && tab[h] < s;
        }
        s_rep[t] = rep;
    }
    __syncthreads();
    const int32_t j = j0 + int32_t(threadIdx.x);
    if (j >= a.cap) return;
    uint8_t y = 0;
    if (j < L)
        for (int i = 0; i < a.n; ++i) y |= s_rep[threadIdx.x + i];  // windows starting at j - n + 1 .. j
    a.labels[size_t(b) * size_t(a.cap) + j] = y;
}

// ------------------------------------------------------------------------------------------------
// One kernel: short rows, and longer ones where the batch fills the chip (label_one_kernel).
// ------------------------------------------------------------------------------------------------
constexpr int kLabelMaxParts = 8;          // CTAs a row: the portable cluster size
constexpr int kLabelPartWindows = 32768;   // windows a CTA's table is meant for
constexpr int kLabelClusterCap = 65536;    // the largest capacity of the one-kernel form
constexpr int kLabelClusterThreads = 1024;
constexpr size_t kLabelSmemMax = 224 * 1024;
// The stacks' sizes: fewer than 32 windows are left when 32 more come from the hash or a round of tries, and a
// round of compares can return 32 in between.
constexpr int kLabelTries = 96, kLabelCompares = 64;
constexpr uint32_t kSlotEmpty = 0xffffffffu;
constexpr uint32_t kLabelProbes = 512;     // slots a window tries in a pass
constexpr uint32_t kLabelMul = 0x9E3779B1u;

struct ClusterLabelArgs {
    const int32_t *ctx, *lens;
    uint8_t *labels;
    int32_t cap, n, pos_bits;  // cap < 1 << pos_bits: a slot's low bits hold a start, the rest hash bits
    uint32_t slots;            // of a CTA's table
    int32_t bm_words;          // of each of a CTA's two bitmaps: ceil(cap / 32)
};

__device__ __forceinline__ uint32_t label_mix(uint64_t sum) {
    uint32_t h = uint32_t(sum) + uint32_t(sum >> 32) * 0x7FEB352Du;
    h ^= h >> 15;
    h *= 0x2C1B3C6Du;
    h ^= h >> 12;
    h *= 0x297A2D39u;
    return h ^ (h >> 15);
}

__device__ __forceinline__ uint32_t ld_cluster_u32(const uint32_t *p, uint32_t rank) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(v) : "r"(map_to_rank(p, rank)) : "memory");
    return v;
}

__global__ void __launch_bounds__(kLabelClusterThreads, 1) label_cluster_kernel(const ClusterLabelArgs a) {
    extern __shared__ __align__(16) uint32_t lsm[];
    uint32_t *tab = lsm;                          // [slots]
    uint32_t *bm = lsm + ((a.slots + 3) & ~3u);   // [bm_words]: starts whose window occurs earlier
    uint32_t *left = bm + ((a.bm_words + 3) & ~3);  // [bm_words]: starts left for the next pass
    uint2 *stacks = reinterpret_cast<uint2 *>(left + ((a.bm_words + 3) & ~3));

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthreads = blockDim.x;
    const uint32_t part = cluster_ctarank(), P = cluster_nctarank();
    const int b = blockIdx.y;
    uint2 *stack_t = stacks + (kLabelTries + kLabelCompares) * warp, *stack_c = stack_t + kLabelTries;
    for (uint32_t i = tid; i < a.slots; i += nthreads) tab[i] = kSlotEmpty;
    for (int i = tid; i < a.bm_words; i += nthreads) bm[i] = left[i] = 0u;
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    int32_t L = a.lens[b];
    if (L < 0 || L > a.cap) L = 0;  // a length outside [0, cap] labels nothing
    const int32_t *x = a.ctx + size_t(b) * size_t(a.cap);
    const int32_t n = a.n, nw = L - n + 1;  // windows start at [0, nw)
    const uint32_t pos_mask = (1u << a.pos_bits) - 1u;

    auto same = [&](int32_t p, int32_t s) {
        for (int i0 = 0; i0 < n; i0 += 8) {  // eight tokens of each a round: their loads are independent
            bool eq = true;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = min(i0 + u, n - 1);
                eq &= x[p + i] == x[s + i];
            }
            if (!eq) return false;
        }
        return true;
    };
    auto mark = [&](int32_t s) { atomicOr(&bm[s >> 5], 1u << (s & 31)); };
    // A window on a stack: its slot entry, and slot | probes << 16.
    int tries = 0, compares = 0;  // the stacks' sizes, warp-uniform
    const unsigned below = (1u << lane) - 1u;
    auto push = [&](uint2 *stack, int &size, bool on, uint2 e) {
        const unsigned who = __ballot_sync(kFull, on);
        if (on) stack[size + __popc(who & below)] = e;
        size += __popc(who);
        __syncwarp();
    };
    // The next slot of a window.  After kLabelProbes of them it is left for a pass over the emptied table with another
    // hash: only tokens built against the hash, or a part with far more windows than its share, fill a table so (a row
    // of 32K tokens with 17K or 32K distinct windows in a part of 16K slots takes 0.7 or 3.5 ms; 206 ms or 4 s when they
    // tried every slot and were then compared with every earlier window).  Equal
    // windows go the same way, since they try the same slots in the same order and nothing leaves the table: a slot
    // that one of them found taken by another window is so for all that come later.
    bool leaves = false;  // this thread left a window
    auto next_slot = [&](uint2 &e) {
        uint32_t slot = e.y & 0xffffu, probes = (e.y >> 16) + 1u;
        if (probes >= kLabelProbes) {
            const int32_t s = int32_t(e.x & pos_mask);
            atomicOr(&left[s >> 5], 1u << (s & 31));
            leaves = true;
            return false;
        }
        if (++slot == a.slots) slot = 0u;
        e.y = probes << 16 | slot;
        return true;
    };
    auto try_round = [&]() {  // up to 32 windows of the try stack at their slots
        const int take = min(tries, kWarp);
        tries -= take;
        const bool on = lane < take;
        uint2 e = make_uint2(0u, 0u);
        if (on) e = stack_t[tries + lane];
        __syncwarp();
        bool cmp = false, again = false;
        if (on) {
            const uint32_t v = atomicCAS(&tab[e.y & 0xffffu], kSlotEmpty, e.x);
            if (v != kSlotEmpty) {
                cmp = ((v ^ e.x) & ~pos_mask) == 0u;
                again = !cmp && next_slot(e);
            }
        }
        push(stack_c, compares, cmp, e);
        push(stack_t, tries, again, e);
    };
    auto compare_round = [&]() {  // up to 32 windows of the compare stack with the window of their slot
        const int take = min(compares, kWarp);
        compares -= take;
        const bool on = lane < take;
        uint2 e = make_uint2(0u, 0u);
        if (on) e = stack_c[compares + lane];
        __syncwarp();
        bool again = false;
        if (on) {
            const int32_t s = int32_t(e.x & pos_mask);
            uint32_t *slot = &tab[e.y & 0xffffu];
            // (the slot's start can only move to a smaller start of the same window)
            if (same(int32_t(*reinterpret_cast<volatile uint32_t *>(slot) & pos_mask), s))
                mark(max(int32_t(atomicMin(slot, e.x) & pos_mask), s));
            else
                again = next_slot(e);
        }
        push(stack_t, tries, again, e);
    };

    // The slot entry of window s with hash m, and its first slot: the slot from another multiple than the part's, the
    // entry's tag from the low bits.
    auto entry = [&](uint32_t m, int32_t s) {
        return make_uint2((m << a.pos_bits) | uint32_t(s), __umulhi(m * 0x85EBCA77u, a.slots));
    };
    auto full_rounds = [&]() {
        while (tries >= kWarp) {
            try_round();
            if (compares >= kWarp) compare_round();
        }
    };
    auto drain = [&]() {
        while (tries > 0 || compares > 0) {
            if (tries > 0) try_round();
            if (compares >= kWarp || tries == 0) compare_round();
        }
    };

    constexpr int kW4 = 4;  // windows a lane hashes at once
    for (int32_t s0 = warp * (kWarp * kW4); s0 < nw; s0 += nthreads * kW4) {
        uint64_t h[kW4];  // 64-bit sums, so that tokens that differ in their high bits alone still spread
#pragma unroll
        for (int u = 0; u < kW4; ++u) h[u] = 0u;
        uint32_t pw = 1u;
        if (s0 + kWarp * kW4 + n <= L) {
            const int32_t *at = x + s0 + lane;
            for (int i = 0; i < n; ++i, ++at, pw *= kLabelMul)
#pragma unroll
                for (int u = 0; u < kW4; ++u) h[u] += uint64_t(uint32_t(at[kWarp * u])) * pw;
        } else {
            for (int i = 0; i < n; ++i, pw *= kLabelMul)
#pragma unroll
                for (int u = 0; u < kW4; ++u) h[u] += uint64_t(uint32_t(x[min(s0 + kWarp * u + lane + i, L - 1)])) * pw;
        }
#pragma unroll
        for (int u = 0; u < kW4; ++u) {
            const int32_t s = s0 + kWarp * u + lane;
            const uint32_t m = label_mix(h[u]);
            push(stack_t, tries, s < nw && __umulhi(m, P) == part, entry(m, s));  // the part from the top bits
            full_rounds();
        }
    }
    drain();
    // The windows left, if any: each pass empties the table, where at least kLabelProbes of them then find a slot.
    // (Word w of `left` is read and written by its warp alone within a pass.)
    uint64_t seed = 0u;
    while (__syncthreads_or(leaves)) {
        leaves = false;
        seed += 0x9E3779B97F4A7C15ull;
        for (uint32_t i = tid; i < a.slots; i += nthreads) tab[i] = kSlotEmpty;
        __syncthreads();
        for (int w = warp; w < a.bm_words; w += nthreads / kWarp) {
            const uint32_t word = left[w];
            if (word == 0u) continue;
            __syncwarp();
            if (lane == 0) left[w] = 0u;
            __syncwarp();
            const int32_t s = 32 * w + lane;
            const bool on = (word >> lane & 1u) != 0u;
            uint64_t sum = 0u;
            uint32_t pw = 1u;
            if (on)
                for (int i = 0; i < n; ++i, pw *= kLabelMul) sum += uint64_t(uint32_t(x[s + i])) * pw;
            push(stack_t, tries, on, entry(label_mix(sum ^ seed), s));
            full_rounds();
        }
        drain();
    }
    // every CTA's marks are in (P = 1: the cluster is this CTA)
    cluster_arrive_release();
    cluster_wait_acquire();

    // Labels: CTA `part` takes a contiguous P-th of the row's groups of 16 positions.
    uint8_t *out = a.labels + size_t(b) * size_t(a.cap);
    const int groups = (a.cap + 15) >> 4;
    const int per = (groups + int(P) - 1) / int(P);
    const int g1 = min(groups, (int(part) + 1) * per);
    const bool wide = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
    for (int g = int(part) * per + tid; g < g1; g += nthreads) {
        const int w = g >> 1;
        uint32_t cur = 0u, before = 0u;
        for (uint32_t r = 0; r < P; ++r) {
            cur |= ld_cluster_u32(&bm[w], r);
            if (w > 0) before |= ld_cluster_u32(&bm[w - 1], r);
        }
        // bit j of the label word: the OR of the marks j - n + 1 .. j, by doubling
        uint64_t m = (uint64_t(cur) << 32) | before;
        int have = 1;
        for (; 2 * have <= n; have *= 2) m |= m << have;
        m |= m << (n - have);
        const uint32_t bits = uint32_t(m >> 32) >> (16 * (g & 1));
        // four bits to four bytes: the multiplier puts bit i at bit 8 i
        auto bytes = [](uint32_t v) { return ((v & 15u) * 0x00204081u) & 0x01010101u; };
        const uint4 v = make_uint4(bytes(bits), bytes(bits >> 4), bytes(bits >> 8), bytes(bits >> 12));
        if (wide && 16 * g + 16 <= a.cap) {
            reinterpret_cast<uint4 *>(out)[g] = v;
        } else {
            for (int i = 0; i < 16 && 16 * g + i < a.cap; ++i) out[16 * g + i] = uint8_t(bits >> i & 1u);
        }
    }
    cluster_arrive_relaxed();
    cluster_wait_acquire();  // no CTA leaves while another reads its bitmap
}

// CTAs a row: enough that a CTA's windows fit its table, and more while the grid leaves SMs idle (every CTA
// hashes the whole row, so more only pay while they add SMs).  SMs that do not fill a cluster in their part of
// the chip stay idle, the more the larger the cluster: 5 clusters' worth is left for them.
static int label_parts(int32_t B, int32_t cap, int sms) {
    int P = 1;
    while (int64_t(P) * kLabelPartWindows < cap) P *= 2;
    while (P < kLabelMaxParts && 2 * int64_t(P) * (B + 5) <= sms && cap / (2 * P) >= 512) P *= 2;
    return P;
}

// The one-kernel form costs what its longest row does -- a CTA hashes the whole row, n tokens a window -- and the two
// kernels what the batch does, spread over the chip, least where few windows are distinct.  Measured on Zipf text and on
// tiles of code, the worse of the two counts (two kernels / one kernel, of the time; above 1 the one kernel is faster):
//   rows of   8K  n = 3..32  1 row 1.13 and more
//             9K  n = 5, 8   6 rows 0.99 1.01   14 rows 1.03 0.79   18 rows 0.95 0.87   22 rows 1.13 1.03   24 rows 0.98 1.13
//            16K  n = 5, 8   1 row 0.96 0.85    4 rows 1.06 1.01    8 rows 1.08 1.05    16 rows 1.12 1.05
//                 n = 12, 32 4 rows 0.85 0.82   16 rows 1.00 0.97   20 rows 1.16 1.13
//            32K  n = 5, 8   16 rows 0.86 0.86  20 rows 1.03 1.02   24 rows 1.11 1.11   34 rows 0.99 1.01   80 rows 1.17 1.22
//                 n = 12, 32 24 rows 0.96 0.94  33 rows 1.16 1.20   34 rows 0.84 0.91   52 rows 1.14 1.29   72 rows 0.94 1.12
//            64K  n = 5, 8   28 rows 1.07 1.00  33 rows 1.23 1.17   34 rows 0.81 0.80   52 rows 1.14 1.13   80 rows 0.88 0.89
//                 n = 12, 32 33 rows 0.96 0.99  60 rows 1.01 1.12   71 rows 1.18 1.31   80 rows 0.70 0.76   152 rows 1.35 1.43
// (A row just past a multiple of the 4,096 windows that a CTA hashes at once costs one more round: 9K.)  Past 16K or
// 32K the time goes by whole waves of CTAs (an SM holds one) and the CTAs a row halve as the rows grow
// (33 and 34), so the rule asks how much of its waves the grid fills: three quarters, and seven eighths where both the
// rows and the windows are long.
static bool label_one_kernel(int32_t B, int32_t cap, int32_t n, int P, int sms) {
    const bool short_windows = n <= 8;
    if (cap <= 8192) return true;
    if (cap <= 16384) return B >= (short_windows && cap > 12288 ? 4 : 22);
    if (cap <= 32768 && short_windows) return B >= 24;
    if (cap > kLabelClusterCap) return false;
    const int64_t ctas = int64_t(B) * P, waves = (ctas + sms - 1) / sms;
    return 8 * ctas >= (cap > 32768 && !short_windows ? 7 : 6) * waves * sms;
}

// SMs of the current device; sets the cluster kernel's shared-memory limit on its first call for the device.
static cudaError_t label_sms(int &sms) {
    static int sm_counts[64] = {0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    sms = dev >= 0 && dev < 64 ? sm_counts[dev] : 0;
    if (sms == 0) {
        e = cudaFuncSetAttribute(label_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kLabelSmemMax));
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) sm_counts[dev] = sms;
    }
    return cudaSuccess;
}

static cudaError_t launch_label_cluster(const int32_t *ctx, const int32_t *lens, int32_t B, int32_t cap, int32_t n,
                                        uint8_t *labels, int P, cudaStream_t stream) {
    ClusterLabelArgs a;
    a.ctx = ctx;
    a.lens = lens;
    a.labels = labels;
    a.cap = cap;
    a.n = n;
    a.pos_bits = 1;
    while ((int64_t(1) << a.pos_bits) <= cap) ++a.pos_bits;
    a.bm_words = (cap + 31) / 32;
    // twice the windows a CTA expects, as far as the shared memory goes (load 1/2 to 3/4)
    const int windows = (cap + P - 1) / P;
    // threads by the row, which every CTA hashes: four windows each
    int threads = 128;
    while (threads < kLabelClusterThreads && 4 * threads < cap) threads *= 2;
    const size_t fixed = 2 * size_t((a.bm_words + 3) & ~3) * 4 + size_t(threads / kWarp) * (kLabelTries + kLabelCompares) * sizeof(uint2) + 16;
    const size_t most = (kLabelSmemMax - fixed) / 4;
    const size_t want = size_t(2) * size_t(windows) + 64;
    a.slots = uint32_t(want < most ? want : most);
    const size_t smem = fixed + size_t((a.slots + 3) & ~3u) * 4;
    return launch_pdl(label_cluster_kernel, dim3(unsigned(P), unsigned(B)), dim3(unsigned(threads)), smem, stream,
                      unsigned(P), a);
}

static uint32_t table_slots(int32_t cap) {
    uint32_t t = 16;
    while (t < 2u * uint32_t(cap)) t <<= 1;
    return t;
}

}  // namespace switchsd

using namespace switchsd;

extern "C" size_t switchsd_labels_workspace_bytes(int32_t B, int32_t cap) {
    if (B < 1 || cap < 1) return 0;
    return size_t(B) * (size_t(table_slots(cap)) + size_t(cap)) * sizeof(int32_t);
}

extern "C" int switchsd_copy_labels(const int32_t *ctx_tokens, const int32_t *ctx_lens, int32_t B, int32_t cap,
                                    int32_t n, uint8_t *out_labels, void *workspace, size_t workspace_bytes,
                                    void *stream) {
    if (!ctx_tokens || !ctx_lens || !out_labels || !workspace) return SWITCHSD_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(workspace) & 3) != 0) return SWITCHSD_ERR_ARG;
    if (B < 1 || B > 65535 || cap < 1 || cap > (1 << 30) || n < 1 || n > SWITCHSD_NMAX) return SWITCHSD_ERR_SHAPE;
    if (workspace_bytes < switchsd_labels_workspace_bytes(B, cap)) return SWITCHSD_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int sms = 0;
    if (label_sms(sms) != cudaSuccess) return SWITCHSD_ERR_CUDA;
    const int P = label_parts(B, cap, sms);
    if (label_one_kernel(B, cap, n, P, sms))
        return launch_label_cluster(ctx_tokens, ctx_lens, B, cap, n, out_labels, P, s) == cudaSuccess ? SWITCHSD_OK
                                                                                                      : SWITCHSD_ERR_CUDA;
    const uint32_t T = table_slots(cap);
    if (cudaMemsetAsync(workspace, 0xff, size_t(B) * T * sizeof(int32_t), s) != cudaSuccess) return SWITCHSD_ERR_CUDA;
    LabelArgs a;
    a.ctx = ctx_tokens;
    a.lens = ctx_lens;
    a.table = static_cast<int32_t *>(workspace);
    a.where = a.table + size_t(B) * T;
    a.labels = out_labels;
    a.B = B;
    a.cap = cap;
    a.n = n;
    a.tmask = T - 1;
    const dim3 grid(unsigned((cap + kLabelThreads - 1) / kLabelThreads), unsigned(B));
    if (launch_pdl(label_insert_kernel, grid, dim3(kLabelThreads), 0, s, 0u, a) != cudaSuccess)
        return SWITCHSD_ERR_CUDA;
    if (launch_pdl(label_mark_kernel, grid, dim3(kLabelThreads), 0, s, 0u, a) != cudaSuccess)
        return SWITCHSD_ERR_CUDA;
    return SWITCHSD_OK;
}
