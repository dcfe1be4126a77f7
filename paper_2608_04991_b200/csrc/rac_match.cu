// Exact-token span retrieval for prefill uplinks (Sec. IV-B.1, Eq. 3) on the GPU.
//
// Index: a hash table with one slot per DISTINCT w-token window of the history, in buckets of four slots (32 bytes, one
// trip to L2).  A slot holds 32 bits of the window's hash beside one representative start position; where the hash bits
// agree the key is verified token by token, so hash collisions can never change the result.  Beside the slot stand the K
// largest start positions of that window, as a set that does not depend on the order in which threads run (set_insert).
// Query: one thread per query position looks its window up and extends each of the <= K candidates forward to the longest
// exact match; long matches are finished by the warp together.  lexargmax(length, start) is kept.
// Selection: the left-to-right scan of Eq. 3 visits a position, jumps by the span length if it has a candidate and by one
// otherwise.  Positions are cut into chunks; every chunk works out, for each of its positions, where a scan that enters there
// leaves the chunk and how many spans it selects on the way (pointer doubling in shared memory).  What is left is one hop per
// chunk; then every chunk is walked from the position where the scan enters it, and writes its spans and rows.  Up to eight
// chunks are the CTAs of one cluster, and all of the query is one launch; more take three.
//
// All of it is bound by the latency of dependent trips to L2 and of launches, not by the bytes: the forms above were chosen
// to make fewer of both, and every kernel lets the next one be set up while it runs.  32768 history and 2048 query tokens:
// 18 us in three launches (52 us in nine before: sorted lists, a thread per match, a suffix scan and a serial walk; 23.5 us
// with selection and emission in two launches and a test before every load of the extension), 131072 / 131072 tokens 35.5 us
// (99 us, 43.6 us), a query of 2048 tokens against an index of 16384 12 us (60 us, 22 us), with intra-sequence references 14.3 us
// (28 us), eight appends of 2048 tokens behind a reset 36 us (54 us; 38 us in CTAs of 128 threads).  Of the query's 12 us, 5 are
// the slowest warp's candidates: up to eight of them, two at a time, two trips each (one at a time 9 of 16 us).
#include <cooperative_groups.h>

#include <mutex>

#include "rac_common.cuh"

namespace rac {

namespace cg = cooperative_groups;

typedef unsigned long long u64;
constexpr u64 kEmptySlot = ~0ull;
constexpr int kBucket = 4;             // slots per bucket
constexpr int kChunk = 512;            // query positions per chunk of the selection = threads of its CTAs
constexpr int kClusterChunks = 8;      // up to so many chunks are one cluster of CTAs (the portable limit), and the query one launch

struct MatchParams {
    const int32_t *hist;
    const int32_t *query;
    int32_t *ref_row;
    rac_span *spans_out;   // may be null
    int32_t *n_spans;
    u64 *slots;            // [M]      hash bits (high half) and representative start of the slot's window, all ones = empty
    int32_t *top;          // [n_hist*K] the K largest starts of a window, in no order, -1 = none, at its representative start
    int32_t *next;         // [nwin]   unlimited hits (max_hits = 0) only: another start of the same window, -1 = none;
                           //          top[representative] is then the head of the window's chain (K = 1)
    int2 *best;            // [N]      (length, history start) of the best candidate, length 0 = none
    int2 *jump;            // [N]      where a scan that enters the chunk here leaves it, and the spans it selects until then
    int2 *entry;           // [chunks] where the scan enters the chunk, and the spans selected before
    int n_hist, n_query, nwin, w, K;
    unsigned int bmask;    // buckets - 1
    const int32_t *end_of; // [n_hist] end of the request that holds each history position; null = one request
    const int32_t *indexed;// [1]      tokens the index holds (a query may name more or fewer); null = n_hist
    int first_live;        // only windows that start at or after this history position are candidates (0 = all)
    // intra-sequence references: a table of the prompt's tokens (TokenTable).  One cluster keeps it in shared memory.
    unsigned int *tok;     // [tmask + 1] else null
    unsigned int tmask;
    int intra;
    int ahead;             // the launch before this one is of the same call and began after everything before the call had ended
};

// Four tokens of a window (or what is left of it) per step, loaded before any is used: a chain of one or two trips to memory, not
// one per token.  Kernels that may read the call's tokens ahead of their turn stage them in shared memory.
__device__ __forceinline__ u64 hash_step(u64 h, int32_t t) {
    h ^= (u64)(uint32_t)t;
    h *= 0xff51afd7ed558ccdull;
    return h ^ (h >> 32);
}
constexpr u64 kHashStart = 0x9E3779B97F4A7C15ull;
__device__ __forceinline__ u64 window_hash(const int32_t *win, int w) {
    u64 h = kHashStart;
    for (int m = 0; m < w; m += 4) {
        int32_t t[4];
#pragma unroll
        for (int u = 0; u < 4; u++) t[u] = m + u < w ? win[m + u] : 0;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (m + u < w) h = hash_step(h, t[u]);
    }
    return h;
}
// tokens [lo, lo + n) of src, as far as they lie before `end`, into shared memory; the caller synchronises
__device__ __forceinline__ void stage_tokens(int32_t *dst, const int32_t *src, int lo, int n, int end) {
    for (int t = threadIdx.x; t < n; t += blockDim.x) dst[t] = lo + t < end ? __ldcg(src + lo + t) : 0;
}
// the window at `win` (staged) is the one at `a` (history): eight tokens of it per trip
__device__ __forceinline__ bool same_window(const int32_t *a, const int32_t *win, int w) {
    for (int m = 0; m < w; m += 8) {
        int32_t x[8];
#pragma unroll
        for (int u = 0; u < 8; u++) x[u] = m + u < w ? a[m + u] : 0;
        int32_t ne = 0;
#pragma unroll
        for (int u = 0; u < 8; u++) ne |= m + u < w ? x[u] ^ win[m + u] : 0;
        if (ne) return false;
    }
    return true;
}
// a bucket as the L2 holds it (other SMs may be filling it)
__device__ __forceinline__ void load_bucket(const u64 *slots, unsigned int b, u64 (&e)[kBucket]) {
    const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(slots + (size_t)b * kBucket);
    const ulonglong2 lo = __ldcg(q), hi = __ldcg(q + 1);
    e[0] = lo.x; e[1] = lo.y; e[2] = hi.x; e[3] = hi.y;
}

// First slot of a bucket, from slot `from` on, that is empty or carries the hash bits (kBucket if none), and what it holds.
// Selects, not branches: the lanes of a warp then look at whatever slot each of them is at in ONE trip, where a branch per
// slot made a trip of each (the two trips per slot took most of the table's time).
__device__ __forceinline__ int find_in_bucket(const u64 (&e)[kBucket], uint32_t tag, int from, u64 &held) {
    int at = kBucket;
    held = kEmptySlot;
#pragma unroll
    for (int s = kBucket - 1; s >= 0; s--) {
        const bool hit = s >= from && (e[s] == kEmptySlot || (uint32_t)(e[s] >> 32) == tag);
        at = hit ? s : at;
        held = hit ? e[s] : held;
    }
    return at;
}

// a set as the L2 holds it, `none` beyond its K entries
__device__ __forceinline__ void load_set(const int32_t *set, int K, int none, int (&v)[16]) {
#pragma unroll
    for (int m = 0; m < 4; m++) {
        if ((K & 3) == 0) {       // whole 16-byte pieces (the table's sections are 16-byte aligned)
            int4 q = make_int4(none, none, none, none);
            if (4 * m < K) q = __ldcg(reinterpret_cast<const int4 *>(set) + m);
            v[4 * m] = q.x; v[4 * m + 1] = q.y; v[4 * m + 2] = q.z; v[4 * m + 3] = q.w;
        } else {
#pragma unroll
            for (int u = 0; u < 4; u++) v[4 * m + u] = 4 * m + u < K ? __ldcg(set + 4 * m + u) : none;
        }
    }
}

// Start c enters a window's set of the K largest starts (-1 = empty entry).  An atomicMax puts it into one entry, and the smaller
// of it and what stood there is carried on, until that is -1 or every entry is larger.  Entries only grow, so what a thread has
// seen of an entry is never more than it holds, and a value is dropped only when K larger ones exist: the set ends as the K
// largest values ever offered, whatever the interleaving; the order of its entries is of no meaning.  Every swap either puts a
// value in or shows an entry that the value need not try again.
// The first swap goes to an entry picked by position, together with the look at the set: one trip for a window that occurs once,
// as most do, and threads with the same window at different entries.  (Look, then compare-and-swap of the smallest entry: two
// trips, and one winner per trip among such threads.  131072 tokens hold one window 65
// times: 40.7 us for the match, 35.7 so; 32768 tokens 20.5 and 17.9.)
__device__ __forceinline__ void set_insert(int32_t *set, int K, int c) {
    const unsigned int first = (unsigned int)c % (unsigned int)K, behind = ~((1u << first) - 1u);
    int at = (int)first;
    for (bool spread = false;; spread = true) {
        const int old = atomicMax(&set[at], c);
        int v[16];
        load_set(set, K, 0x7fffffff, v);
        if (old < 0) return;
        const int held = max(old, c);
        c = min(old, c);
        int low = 0x7fffffff, low_at = 0;
        unsigned int empty = 0, less = 0;
#pragma unroll
        for (int r = 0; r < 16; r++) {
            const int x = r == at ? held : v[r];
            if (x < low) { low = x; low_at = r; }
            empty |= x < 0 ? (1u << r) : 0u;
            less |= x < c ? (1u << r) : 0u;
        }
        if (!less) return;
        at = low_at;
        if (empty | (spread ? less : 0u)) {      // several threads are at this set: each at an entry of its own
            const unsigned int m = empty ? empty : less;
            at = __ffs(m & behind ? m & behind : m) - 1;
        }
    }
}
// Start j enters the index, h = the hash of its window `win`.  Its window's slot holds a representative start; the first empty slot
// of the probe sequence is claimed where there is none.  Slots fill in probe order and are never emptied, so two threads with the
// same window end at one slot.  The window's set of starts stands at the place of its representative in `top`.
// A claim goes out together with j's place in the set that j heads if the claim succeeds (else nobody reads that set), and beside
// the verification of the lanes that found a slot taken: a window that occurs once, as most do, is the trip for its bucket and
// one more.  (One after another 18.4 us for a match of 32768 tokens, so 17.9.)
// Unlimited hits: every start goes onto its window's chain.  The order of a chain depends on which thread came first; the query
// looks at ALL of it and keeps lexargmax(length, start), so the result does not.
__device__ __forceinline__ void index_start(u64 *slots, int32_t *top, int32_t *next, unsigned int bmask, const int32_t *hist,
                                            int j, const int32_t *win, int w, int K, u64 h) {
    const uint32_t tag = (uint32_t)(h >> 32);
    unsigned int b = (unsigned int)h & bmask, probes = 0;
    u64 e[kBucket];
    load_bucket(slots, b, e);
    int from = 0, rep = -1, carry = j, old = -1;
    bool placed = next != nullptr;
    while (probes <= bmask) {     // (the table has at least twice as many slots as windows: ends before)
        u64 held;
        const int s = find_in_bucket(e, tag, from, held);
        if (s == kBucket) {                   // full of other windows: the next bucket
            b = (b + 1) & bmask;
            probes++;
            load_bucket(slots, b, e);
            from = 0;
            continue;
        }
        const bool claim = held == kEmptySlot;
        u64 found = kEmptySlot;
        if (claim) {
            found = atomicCAS(slots + (size_t)b * kBucket + s, kEmptySlot, ((u64)tag << 32) | (uint32_t)j);
            if (!placed) {      // once: from then on the value is in the set, wherever others may have moved it
                old = atomicMax(&top[(size_t)j * K + (unsigned int)j % (unsigned int)K], j);
                placed = true;
            }
        }
        const int r = claim ? j : (int)(uint32_t)held;
        const bool same = same_window(hist + r, win, w);
        if (claim && found != kEmptySlot) {   // another thread was faster: look at what it put there
#pragma unroll
            for (int u = 0; u < kBucket; u++) e[u] = u == s ? found : e[u];
            from = s;
        } else if (same) {
            rep = r;
            if (claim && !next) carry = min(old, j);
            break;
        } else from = s + 1;
    }
    if (rep < 0 || carry < 0) return;
    if (next) next[j] = atomicExch(&top[rep], j);
    else set_insert(top + (size_t)rep * K, K, carry);
}

// All ones in n16 pieces of 16 bytes; with zero, also *zero = 0.  The kernel after it may begin once the work before this call
// has ended (not at once): it then reads the call's tokens while the fill is under way.
__global__ void fill_ones_kernel(uint4 *dst, long long n16, int32_t *zero) {
    grid_dependency_wait();
    grid_launch_dependents();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (long long k = i; k < n16; k += (long long)gridDim.x * blockDim.x) dst[k] = make_uint4(~0u, ~0u, ~0u, ~0u);
    if (zero && i == 0) *zero = 0;
}

// Tokens and hashes before the wait for the fill: the tokens are of before the call, and the fill let this kernel begin only
// once that had ended.  (The query kernel does the same behind this one.)
__global__ void __launch_bounds__(256) match_insert_kernel(const MatchParams p) {
    __shared__ int32_t s_tok[256 + 32];
    // the latest starts first: once a set is full of them the earlier ones are done with one look
    const int j = p.nwin - 1 - (int)(blockIdx.x * 256 + threadIdx.x), lo = p.nwin - 256 - (int)(blockIdx.x * 256);
    for (int t = threadIdx.x; t < 256 + p.w - 1; t += 256) s_tok[t] = lo + t >= 0 ? __ldcg(p.hist + lo + t) : 0;
    __syncthreads();
    const int32_t *win = s_tok + (255 - threadIdx.x);
    const u64 h = window_hash(win, p.w);
    grid_dependency_wait();
    grid_launch_dependents();
    if (j >= 0) index_start(p.slots, p.top, p.next, p.bmask, p.hist, j, win, p.w, p.K, h);
}

// first position at or after this thread's position in its chunk that has a candidate (`limit` if none)
__device__ __forceinline__ int next_candidate(bool has, int i, int limit) {
    __shared__ int s_first[kChunk / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned int b = __ballot_sync(0xffffffffu, has);
    if (lane == 0) s_first[warp] = b ? i + __ffs(b) - 1 : limit;
    __syncthreads();
    if (b >> lane) return i + __ffs(b >> lane) - 1;
    for (int w = warp + 1; w < kChunk / 32; w++)
        if (s_first[w] < limit) return s_first[w];
    return limit;
}

// The tokens of a prompt: open addressing, a slot holds the smallest position so far of the token that claimed it (positions of
// one token only ever replace each other), all ones = empty.  In global memory, or spread over the shared memories of a cluster.
constexpr int kTokSlots = 2 * kChunk;     // per CTA of a cluster
struct TokenTable {
    const int32_t *query;
    unsigned int *base;
    unsigned int mask;
    bool spread;
    __device__ __forceinline__ unsigned int *at(unsigned int s) const {
        return spread ? cg::this_cluster().map_shared_rank(base, s / kTokSlots) + s % kTokSlots : base + s;
    }
    // slots: a power of two in global memory, any multiple of kTokSlots in a cluster
    __device__ __forceinline__ unsigned int start(int32_t tok) const {
        const unsigned int h = (unsigned int)hash_step(kHashStart, tok);
        return spread ? __umulhi(h, mask + 1u) : h & mask;
    }
    __device__ __forceinline__ unsigned int after(unsigned int s) const { return s == mask ? 0u : s + 1u; }
    __device__ __forceinline__ void insert(int32_t tok, unsigned int i) const {
        unsigned int s = start(tok);
        for (unsigned int probe = 0; probe <= mask; probe++, s = after(s)) {
            unsigned int *slot = at(s);
            unsigned int cur = *(volatile unsigned int *)slot;
            if (cur == ~0u) cur = atomicCAS(slot, ~0u, i);
            if (cur == ~0u) return;
            if (query[cur] == tok) {
                if (i < cur) atomicMin(slot, i);
                return;
            }
        }
    }
    // first position of the token (it is in the table)
    __device__ __forceinline__ unsigned int first(int32_t tok) const {
        unsigned int s = start(tok);
        for (unsigned int probe = 0; probe <= mask; probe++, s = after(s)) {
            const unsigned int cur = *(volatile unsigned int *)at(s);
            if (cur == ~0u || query[cur] == tok) return cur;
        }
        return ~0u;
    }
};

// What a chunk hands out: the scan through it from its entry.  Every position at or after the entry belongs to this CTA alone,
// and so does the part of its last span that reaches into later chunks (their entries lie behind it).
struct EmitSmem {
    int next[kChunk], len[kChunk], start[kChunk], row[kChunk], list[kChunk];
    int entry, before, n;
};
__device__ __forceinline__ void emit_chunk(const MatchParams &p, EmitSmem &m, int base, const int32_t *tokens, const TokenTable &tt) {
    const int N = p.n_query, limit = min(base + kChunk, N), i = base + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        int pos = m.entry, n = 0;
        while (pos < limit) {
            const int s = m.next[pos - base];
            if (s >= limit) break;
            m.list[n++] = s - base;
            pos = s + m.len[s - base];
        }
        m.n = n;
        if (limit == N) *p.n_spans = m.before + n;
    }
    m.row[threadIdx.x] = -1;
    __syncthreads();
    const int n = m.n;
    for (int k = warp; k < n; k += kChunk / 32) {        // a warp per span, up to the end of the chunk
        const int at = m.list[k], len = m.len[at], s = base + at, h = m.start[at];
        if (lane == 0 && p.spans_out) {
            rac_span sp;
            sp.q_start = s;
            sp.h_start = h;
            sp.len = len;
            p.spans_out[m.before + k] = sp;
        }
        const int in = min(len, limit - s);
        for (int q = lane; q < in; q += 32) m.row[at + q] = h + q;
    }
    if (n > 0) {                                         // the last span's part in later chunks: the whole CTA
        const int at = m.list[n - 1], s = base + at, end = s + m.len[at], h = m.start[at];
        for (int q = limit + threadIdx.x; q < end; q += kChunk) p.ref_row[q] = h + (q - s);
    }
    __syncthreads();
    if (i < N && i >= m.entry) {
        int row = m.row[threadIdx.x];
        if (row < 0 && p.intra) {
            // intra-sequence reference: the first occurrence of this token, if it is an earlier one
            const unsigned int f = tt.first(tokens[threadIdx.x]);
            if (f < (unsigned int)i) row = p.n_hist + (int)f;
        }
        p.ref_row[i] = row;
    }
}

// Lookup, extension, and the chunk's jumps.  One CTA per chunk, one thread per position.
// Extension: a thread compares eight tokens at its candidate by itself; what is still open after that is finished by the
// warp, 256 tokens per trip, or 128 each at two distances.  Neighbouring positions inside one copied stretch have the same (history - query) distance and
// so the same end: one comparison closes them all.  A thread by itself took a trip per eight tokens, for every position
// of a long match (2048-token prompt: 21 us, with copies of copies 55 us).
// ONE: the chunks are the CTAs of one cluster, which hands out spans and rows as well: a cluster barrier and jumps read from the
// neighbours' shared memory in place of a launch, a table of tokens in shared memory in place of one that a launch has to fill.
template <bool ONE>
__global__ void __launch_bounds__(kChunk, ONE ? 1 : 2) match_query_kernel(const MatchParams p) {
    __shared__ int32_t s_tok[kChunk + 40];
    __shared__ unsigned int s_slots[ONE ? kTokSlots : 1];
    grid_launch_dependents();
    const int N = p.n_query;
    const int base = blockIdx.x * kChunk, i = base + threadIdx.x, lane = threadIdx.x & 31;
    TokenTable tt{p.query, p.tok, p.tmask, false};
    if constexpr (ONE) {
        if (p.intra) {
            tt = TokenTable{p.query, s_slots, gridDim.x * kTokSlots - 1u, true};
            for (int t = threadIdx.x; t < kTokSlots; t += kChunk) s_slots[t] = ~0u;
            cg::this_cluster().barrier_arrive();
        }
    }
    int held_tokens = p.n_hist;           // no history token behind them is read
    if (!p.ahead) {
        grid_dependency_wait();
        if (p.indexed) held_tokens = __ldcg(p.indexed);
    }
    stage_tokens(s_tok, p.query, base, kChunk + p.w + 8, N);
    __syncthreads();
    const int32_t *win = s_tok + threadIdx.x;
    const u64 h = window_hash(win, p.w);
    if (p.ahead) {
        grid_dependency_wait();
        if (p.indexed) held_tokens = __ldcg(p.indexed);
    }
    if (p.intra) {
        if constexpr (ONE) cg::this_cluster().barrier_wait();
        if (i < N) tt.insert(win[0], i);
    }
    int rep = -1;      // representative start of the window at i, -1: not in the history
    int v[16];         // its set
#pragma unroll
    for (int r = 0; r < 16; r++) v[r] = -1;
    if (i < N && i + p.w <= N && p.nwin > 0) {
        const uint32_t tag = (uint32_t)(h >> 32);
        unsigned int b = (unsigned int)h & p.bmask;
        u64 e[kBucket];
        load_bucket(p.slots, b, e);
        int from = 0;
        for (unsigned int probe = 0; probe <= p.bmask;) {
            u64 held;
            const int s = find_in_bucket(e, tag, from, held);
            if (s == kBucket) {
                b = (b + 1) & p.bmask;
                probe++;
                load_bucket(p.slots, b, e);
                from = 0;
                continue;
            }
            if (held == kEmptySlot) break;      // ends the probe sequence: the window is not in the history
            if (same_window(p.hist + (int)(uint32_t)held, win, p.w)) {
                rep = (int)(uint32_t)held;
                break;
            }
            from = s + 1;
        }
    }
    int bestL = 0, bestj = -1;
    // Up to two candidates per lane (-1: none), all lanes of the warp together.  One replaces the best so far only with a longer
    // match, or with one as long and a larger start, so its token at has_to_match has to be equal.  That token, the first eight
    // behind the window and the end of the request come in one trip (no test stands before a load: it would make a trip of each).
    // What is still open goes on to the extension, two distances at a time, one per half of the warp.
    auto has_to_match = [&](int j) { return max(bestL - (j > bestj ? 1 : 0), 0); };
    struct Candidate {
        int j, L, room;
        bool can_win, open;
    };
    auto begin = [&](int j) {
        const int jj = max(j, 0), at = has_to_match(j);
        int32_t hh[8];
#pragma unroll
        for (int u = 0; u < 8; u++) hh[u] = p.hist[min(jj + p.w + u, held_tokens - 1)];
        const int32_t h_at = p.hist[min(jj + at, held_tokens - 1)], q_at = p.query[min(i + at, N - 1)];
        const int end_j = p.end_of ? p.end_of[jj] : p.n_hist;
        Candidate c;
        c.j = j;
        c.room = min(N - i, end_j - jj);          // the longest the match can be, inside its request
        uint32_t ne = 0;
#pragma unroll
        for (int u = 0; u < 8; u++) ne |= win[p.w + u] != hh[u] ? (1u << u) : 0u;
        c.can_win = j >= 0 && (bestL == 0 || (at < c.room && h_at == q_at));
        c.L = min(p.w + (ne ? __ffs(ne) - 1 : 8), c.room);
        c.open = c.can_win && ne == 0u && p.w + 8 < c.room;
        return c;
    };
    auto consider = [&](int j1, int j2) {
        Candidate c = begin(j1), e = begin(ONE ? j2 : -1);
        while (true) {
            // The leads: the lowest lane with an open candidate, and the lowest with one at another distance.  A lane's second
            // candidate counts as its first does: nobody below a lead may be open at the lead's distance (see close()).
            const unsigned int mc = __ballot_sync(0xffffffffu, c.open), me = ONE ? __ballot_sync(0xffffffffu, e.open) : 0u;
            if (!(mc | me)) break;
            const int la = __ffs(mc | me) - 1;
            const bool a_is_c = (mc >> la) & 1u;
            const int da = __shfl_sync(0xffffffffu, (a_is_c ? c.j : e.j) - i, la);
            const unsigned int oc = __ballot_sync(0xffffffffu, c.open && c.j - i != da);
            const unsigned int oe = ONE ? __ballot_sync(0xffffffffu, e.open && e.j - i != da) : 0u;
            const int lb = oc | oe ? __ffs(oc | oe) - 1 : la;
            const bool b_is_c = oc | oe ? ((oc >> lb) & 1u) != 0u : a_is_c;
            const bool mine_c = lane < 16 ? a_is_c : b_is_c;      // which of its lead's candidates this half extends
            const int lead = lane < 16 ? la : lb;
            const int jc = __shfl_sync(0xffffffffu, c.j, lead), je = ONE ? __shfl_sync(0xffffffffu, e.j, lead) : 0;
            const int rc = __shfl_sync(0xffffffffu, c.room, lead), re = ONE ? __shfl_sync(0xffffffffu, e.room, lead) : 0;
            const int i0 = __shfl_sync(0xffffffffu, i, lead), j0 = mine_c ? jc : je, room0 = mine_c ? rc : re;
            // one distance only: the second half takes the tokens behind the first half's (131072 query tokens 37.5 -> 35.7 us; in
            // the cluster's form it cost the query 4 of 16 us)
            const bool one = !ONE && !(oc | oe);
            const int mine = (lane & 15) + (one && lane >= 16 ? 128 : 0), step = one ? 256 : 128;
            int len = p.w + 8;
            bool more = true;
            while (__any_sync(0xffffffffu, more)) {
                int32_t q[8], hh[8];
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    const int at = min(len + 16 * u + mine, room0 - 1);
                    q[u] = p.query[i0 + at];
                    hh[u] = p.hist[j0 + at];
                }
                int first = 0x7fffffff;              // this lane's first position that differs or lies outside
#pragma unroll
                for (int u = 7; u >= 0; u--) {
                    const int at = len + 16 * u + mine;
                    first = at >= room0 || q[u] != hh[u] ? at : first;
                }
                const int fa = __reduce_min_sync(0xffffffffu, lane < 16 ? first : 0x7fffffff);
                const int fb = __reduce_min_sync(0xffffffffu, lane < 16 ? 0x7fffffff : first);
                const int f = one ? min(fa, fb) : lane < 16 ? fa : fb;
                if (more) {
                    more = f == 0x7fffffff;
                    len = more ? len + step : f;
                }
            }
            // Every open position of the same distance that lies before the end has the same end: it lies at or behind the lead, and
            // what the lead compared reaches from there to the end.  (Not so before the lead: between a lower lane's own first
            // eight tokens and the lead there may be tokens that nobody has compared.)
            const int sa = __shfl_sync(0xffffffffu, i0 + len, 0), sb = __shfl_sync(0xffffffffu, i0 + len, 16);
            const int db = __shfl_sync(0xffffffffu, j0 - i0, 16);
            auto close = [&](Candidate &x) {
                const int d = x.j - i, stop = d == da ? sa : sb;
                if (x.open && (d == da || d == db) && i < stop) {
                    x.L = stop - i;
                    x.open = false;
                }
            };
            close(c);
            if (ONE) close(e);
        }
        auto keep = [&](const Candidate &x) {
            if (x.can_win && (x.L > bestL || (x.L == bestL && x.j > bestj))) {
                bestL = x.L;
                bestj = x.j;
            }
        };
        keep(c);
        if (ONE) keep(e);
    };
    if (p.next) {
        // every occurrence of the window (at most nwin of them: the walk is bounded by construction)
        int chain = rep >= 0 ? p.top[rep] : -1, n = 0;
        while (true) {
            while (chain >= 0 && chain < p.first_live && n < p.nwin) { chain = p.next[chain]; n++; }
            const int j = n < p.nwin ? chain : -1;
            if (!__any_sync(0xffffffffu, j >= 0)) break;
            if (j >= 0) { chain = p.next[j]; n++; }
            consider(j, -1);
        }
    } else {
        // The K most recent starts.  After the first candidate, one trip for all the others rules most of them out (the end of
        // a request is left to consider()).
        if (rep >= 0) load_set(p.top + (size_t)rep * p.K, p.K, -1, v);
#pragma unroll
        for (int r = 0; r < 16; r++) v[r] = v[r] >= p.first_live ? v[r] : -1;     // first_live >= 0: no empty ones
        bool first = true;
        while (true) {
            // largest starts first: neighbours inside one copied stretch then look at the same distances at the same time
            auto take = [&]() {
                int j = v[0];
#pragma unroll
                for (int r = 1; r < 16; r++) j = max(j, v[r]);
#pragma unroll
                for (int r = 0; r < 16; r++) v[r] = v[r] == j ? -1 : v[r];
                return j;
            };
            const int j = take();
            if (!__any_sync(0xffffffffu, j >= 0)) break;
            consider(j, ONE ? take() : -1);
            if (first && bestL > 0) {
                const int32_t q_last = p.query[i + bestL - 1], q_beyond = p.query[min(i + bestL, N - 1)];
#pragma unroll
                for (int r0 = 0; r0 < 16; r0 += 8) {
                    if (r0 < p.K) {
                        int32_t tok[8];
#pragma unroll
                        for (int r = 0; r < 8; r++)
                            tok[r] = p.hist[min(max(v[r0 + r], 0) + has_to_match(v[r0 + r]), held_tokens - 1)];
#pragma unroll
                        for (int r = 0; r < 8; r++)
                            if (tok[r] != (v[r0 + r] > bestj ? q_last : q_beyond)) v[r0 + r] = -1;
                    }
                }
            }
            first = false;
        }
    }

    // ---- where a scan that is at position i leaves the chunk, by pointer doubling
    __shared__ int s_nxt[kChunk], s_cnt[kChunk];
    const int limit = min(base + kChunk, N);
    const int cand = next_candidate(bestL > 0, i, limit);
    int nxt = cand, cnt = 0;
    if (bestL > 0) { nxt = i + bestL; cnt = 1; }
    if (i >= limit) { nxt = limit; cnt = 0; }
    while (true) {
        s_nxt[threadIdx.x] = nxt;
        s_cnt[threadIdx.x] = cnt;
        if (!__syncthreads_or(nxt < limit)) break;
        if (nxt < limit) {
            const int k = nxt - base;
            nxt = s_nxt[k];
            cnt += s_cnt[k];
        }
        __syncthreads();
    }
    if constexpr (ONE) {
        __shared__ EmitSmem s_emit;
        s_emit.next[threadIdx.x] = cand;
        s_emit.len[threadIdx.x] = bestL;
        s_emit.start[threadIdx.x] = bestj;
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        if (threadIdx.x == 0) {          // a hop per chunk before this one
            int e = 0, before = 0;
            for (unsigned int k = 0; k < blockIdx.x; k++) {
                if (e >= (int)(k + 1) * kChunk) continue;
                const int at = e - (int)k * kChunk;
                e = cluster.map_shared_rank(s_nxt, k)[at];
                before += cluster.map_shared_rank(s_cnt, k)[at];
            }
            s_emit.entry = e;
            s_emit.before = before;
        }
        emit_chunk(p, s_emit, base, s_tok, tt);
        cluster.sync();                  // nobody leaves while its shared memory may be read
    } else if (i < N) {
        p.best[i] = make_int2(bestL, bestj);
        p.jump[i] = make_int2(nxt, cnt);
    }
}

// Where the scan enters every chunk: entry of chunk c+1 = where a scan that enters chunk c at ITS entry leaves it.  All
// chunks guess their first position and exchange exits until nothing changes; scans that enter a chunk at different
// positions usually leave it at the same one, so two or three exchanges do (at most one per chunk, as in the serial walk).
// One CTA, 1024 chunks at a time.
__global__ void __launch_bounds__(1024) match_resolve_kernel(const MatchParams p, int nchunks) {
    __shared__ int s_exit[1024], s_warp[32];
    grid_launch_dependents();
    grid_dependency_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int carry = 0, carry_cnt = 0;
    for (int c0 = 0; c0 < nchunks; c0 += 1024) {
        const int c = c0 + tid;
        const int start = c * kChunk, end = min(start + kChunk, p.n_query);
        const bool live = c < nchunks;
        int e = tid == 0 ? carry : start, exit = e, cnt = 0;
        while (true) {
            exit = e;
            cnt = 0;
            if (live && e < end) {
                const int2 j = __ldcg(p.jump + e);
                exit = j.x;
                cnt = j.y;
            }
            s_exit[tid] = exit;
            __syncthreads();
            const int ne = tid == 0 ? carry : s_exit[tid - 1];
            const bool changed = live && ne != e;
            e = ne;
            if (!__syncthreads_or(changed)) break;
        }
        // spans selected before the chunk
        int incl = live ? cnt : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, incl, o);
            incl += lane >= o ? up : 0;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        int before = carry_cnt, total = 0;
        for (int w = 0; w < 32; w++) {
            before += w < warp ? s_warp[w] : 0;
            total += s_warp[w];
        }
        if (live) p.entry[c] = make_int2(e, before + incl - cnt);
        carry = s_exit[min(1024, nchunks - c0) - 1];
        carry_cnt += total;
        __syncthreads();
    }
}

// Spans and rows (emit_chunk) of more chunks than a cluster holds.
__global__ void __launch_bounds__(kChunk) match_emit_kernel(const MatchParams p) {
    __shared__ EmitSmem s_emit;
    __shared__ int32_t s_tok[kChunk];
    grid_launch_dependents();
    grid_dependency_wait();
    const int base = blockIdx.x * kChunk, i = base + threadIdx.x;
    const int2 mine = i < p.n_query ? __ldcg(p.best + i) : make_int2(0, -1);
    if (p.intra && i < p.n_query) s_tok[threadIdx.x] = p.query[i];
    if (threadIdx.x == 0) {
        const int2 e = __ldcg(p.entry + blockIdx.x);
        s_emit.entry = e.x;
        s_emit.before = e.y;
    }
    s_emit.next[threadIdx.x] = next_candidate(mine.x > 0, i, min(base + kChunk, p.n_query));
    s_emit.len[threadIdx.x] = mine.x;
    s_emit.start[threadIdx.x] = mine.y;
    __syncthreads();
    emit_chunk(p, s_emit, base, s_tok, TokenTable{p.query, p.tok, p.tmask, false});
}

__global__ void spans_to_rows_kernel(const rac_span *spans, const int32_t *n_spans, long long n_query, int32_t *ref_row) {
    grid_launch_dependents();
    grid_dependency_wait();
    const int ns = *n_spans;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    for (int s = gw; s < ns; s += warps) {
        long long q0 = spans[s].q_start, len = spans[s].len;
        int h0 = spans[s].h_start;
        for (long long m = lane; m < len; m += 32) {
            long long i = q0 + m;
            if (i >= 0 && i < n_query) ref_row[i] = h0 + (int)m;
        }
    }
}

// The same in one launch: a CTA owns kSpanRows positions, looks at all spans and keeps what reaches into its own.  A piece of up to
// kSpanShort positions is written by the thread that sees it, longer ones wait in a list and are written by whole warps (a list of
// more than kSpanList -- only overlapping spans make one -- goes the short way).  Bound by launches and two trips to L2 where spans
// have the usual length (132 tokens, gaps of 56: 2.2 us up to 98304 positions, 2.8 at 262144; 4.1 in the two launches of a fill and
// the kernel above), by reading the list where they are as short as they get: 4 tokens, no gaps, 2.2 us at 4096 positions (3.7), 6.3 at
// 65536 (11.3), 19.9 at 262144 (20.4).  Every CTA reads every span, so that beyond kSpanRowsQuery the two launches are the better
// ones.
constexpr int kSpanRows = 1024, kSpanShort = 8, kSpanList = 128;
constexpr long long kSpanRowsQuery = 262144;
static_assert(kSpanList > kSpanRows / (kSpanShort + 1), "spans that do not overlap fit the list");
__global__ void __launch_bounds__(kSpanRows) span_rows_kernel(const rac_span *spans, const int32_t *n_spans, int n_query, int32_t *ref_row) {
    __shared__ int s_row[kSpanRows], s_n;
    __shared__ rac_span s_span[kSpanList];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lo = blockIdx.x * kSpanRows, hi = min(lo + kSpanRows, n_query);
    grid_launch_dependents();
    s_row[tid] = -1;
    if (tid == 0) s_n = 0;
    __syncthreads();
    grid_dependency_wait();
    const int ns = *n_spans;
    for (long long base = tid; base < ns; base += 4 * kSpanRows) {
        rac_span sp[4];
#pragma unroll
        for (int u = 0; u < 4; u++) sp[u] = spans[base + u * kSpanRows < ns ? base + u * kSpanRows : base];   // loads without a branch
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (base + u * kSpanRows >= ns) continue;
            const long long q0 = sp[u].q_start, q1 = q0 + sp[u].len;
            if (q0 >= hi || q1 <= lo || q1 <= q0) continue;
            const int a = (int)(q0 > lo ? q0 : lo), b = (int)(q1 < hi ? q1 : hi);
            const int at = b - a > kSpanShort ? atomicAdd(&s_n, 1) : kSpanList;
            if (at < kSpanList) {
                s_span[at] = sp[u];
            } else {
                for (int q = a; q < b; q++) s_row[q - lo] = sp[u].h_start + (int)(q - q0);
            }
        }
    }
    __syncthreads();
    const int n = min(s_n, kSpanList);
    for (int k = warp; k < n; k += kSpanRows / 32) {
        const rac_span sp = s_span[k];
        const long long q0 = sp.q_start, q1 = q0 + sp.len;
        const int b = (int)(q1 < hi ? q1 : hi);
        for (int q = (int)(q0 > lo ? q0 : lo) + lane; q < b; q += 32) s_row[q - lo] = sp.h_start + (int)(q - q0);
    }
    __syncthreads();
    if (lo + tid < hi) ref_row[lo + tid] = s_row[tid];
}

// Spans and the gaps between them as segments: boundaries in ascending order, empty pieces dropped, the unused
// tail of seg_off filled with T (empty segments).  One CTA; thread k looks at span k.
__global__ void __launch_bounds__(1024) spans_to_segments_kernel(const rac_span *spans, const int32_t *n_spans, int T,
                                                                 int max_seg, int32_t *seg_off, int32_t *n_seg) {
    __shared__ int s_scan[1024];
    __shared__ int s_base;
    grid_launch_dependents();
    grid_dependency_wait();
    const int ns = min(*n_spans, (max_seg - 1) / 2);
    const int tid = threadIdx.x;
    if (tid == 0) { s_base = 1; seg_off[0] = 0; }   // boundary 0 always; every span adds its start (if a gap precedes) and its end
    __syncthreads();
    for (int k0 = 0; k0 < ns; k0 += 1024) {
        const int k = k0 + tid;
        int q0 = 0, q1 = 0, prev_end = 0, cnt = 0;
        if (k < ns) {
            q0 = spans[k].q_start;
            q1 = q0 + spans[k].len;
            prev_end = k > 0 ? spans[k - 1].q_start + spans[k - 1].len : 0;
            cnt = (q0 > prev_end ? 1 : 0) + (q1 > q0 ? 1 : 0);   // boundaries q0 (new only after a gap) and q1
        }
        s_scan[tid] = cnt;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {
            const int v = tid >= o ? s_scan[tid - o] : 0;
            __syncthreads();
            s_scan[tid] += v;
            __syncthreads();
        }
        int at = s_base + s_scan[tid] - cnt;
        if (k < ns) {
            if (q0 > prev_end) seg_off[at++] = q0;
            if (q1 > q0) seg_off[at] = q1;
        }
        __syncthreads();
        if (tid == 1023) s_base += s_scan[1023];
        __syncthreads();
    }
    int nb = s_base;                      // boundaries written so far, the last one is the end of the last span
    __syncthreads();
    if (tid == 0) {
        if (seg_off[nb - 1] < T) seg_off[nb++] = T;   // the gap behind the last span
        *n_seg = nb - 1;
        s_base = nb;
    }
    __syncthreads();
    for (int i = s_base + tid; i <= max_seg; i += 1024) seg_off[i] = T;
}

__global__ void fill_i32_kernel(int32_t *dst, long long n, int32_t v) {
    grid_launch_dependents();
    grid_dependency_wait();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long stride = (long long)gridDim.x * blockDim.x;
    for (; i < n; i += stride) dst[i] = v;
}

// ---------------------------------------------------------------------------------------------
// Persistent index over a growing list of requests
// ---------------------------------------------------------------------------------------------
struct IndexParams {
    const int32_t *hist;
    u64 *slots;         // [M]
    int32_t *top;       // [capacity*K]
    int32_t *end_of;    // [capacity]
    int32_t *next;      // [capacity]  no cap on the hits: another start of the same window (chain link), else null
    int32_t *indexed;   // [1]         tokens the index holds
    int a, b;           // the request: tokens [a, b)
    int w, K;
    unsigned int bmask;
};

// Appending a request: every position learns the end of its request; every window of the request finds or claims
// its slot and enters the slot's set.  The request's starts are larger than everything already there, so the oldest
// entries fall out as a by-product.  One launch, any request size.
__global__ void __launch_bounds__(64) index_append_kernel(const IndexParams p) {
    grid_launch_dependents();
    grid_dependency_wait();
    const int j = p.b - 1 - (int)(blockIdx.x * blockDim.x + threadIdx.x);   // the latest starts first
    if (j < p.a) return;
    p.end_of[j] = p.b;
    if (j == p.b - 1) atomicMax(p.indexed, p.b);
    if (j + p.w <= p.b)      // else the window would leave the request
        index_start(p.slots, p.top, p.next, p.bmask, p.hist, j, p.hist + j, p.w, p.K, window_hash(p.hist + j, p.w));
}

static size_t align16(size_t v) { return (v + 15) / 16 * 16; }

// SMs of the current device (grids of the grid-stride kernels are sized from it); looked up once per device
static int sm_count() {
    static int cache[64];
    static std::mutex m;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    std::lock_guard<std::mutex> lock(m);
    if (cache[dev] == 0) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 148;
        cache[dev] = sms;
    }
    return cache[dev];
}

static int fill_blocks(long long n16) {
    const long long b = (n16 + 255) / 256, most = (long long)sm_count() * 8;
    return (int)(b < 1 ? 1 : b > most ? most : b);
}
// Slots for n windows: at least `per` each, but no more than 2^31 in all, which leaves two for each of up to 2^30 windows.  Four
// per window leave one bucket in 250 full, two one in seven, and the slowest of a warp's lanes sets its pace.
static unsigned int table_slots(long long n, unsigned long long per) {
    unsigned long long M = 1024;
    while (M < per * (unsigned long long)(n > 0 ? n : 1) && M < (1ull << 31)) M <<= 1;
    return (unsigned int)M;
}

// lookup and extension, the chunks' entries, spans and rows: one cluster does all of it for up to kClusterChunks chunks
static bool query_in_one(long long n_query) { return n_query <= (long long)kClusterChunks * kChunk; }
static void launch_query(const MatchParams &p, cudaStream_t st) {
    const int nchunks = (p.n_query + kChunk - 1) / kChunk;
    if (query_in_one(p.n_query)) {
        launch_cluster_after(match_query_kernel<true>, nchunks, nchunks, kChunk, 0, st, p);
        return;
    }
    launch_after(match_query_kernel<false>, nchunks, kChunk, 0, st, p);
    launch_after(match_resolve_kernel, 1, 1024, 0, st, p, nchunks);
    launch_after(match_emit_kernel, nchunks, kChunk, 0, st, p);
}

constexpr int kSlotsPerWindow = 4;
struct MatchLayout {
    size_t slots, top, filled, best, jump, entry, next, total;
    unsigned int M;
};
// K = 0 (unlimited hits): one entry per window (the head of its chain) and a chain link per history position.  per: table slots
// per window.
static MatchLayout match_layout(long long n_hist, long long n_query, int K, int per) {
    MatchLayout L;
    const bool chains = K == 0;
    if (chains) K = 1;
    const size_t n = (size_t)(n_query > 0 ? n_query : 1);
    const size_t h = (size_t)(n_hist > 0 ? n_hist : 1);
    L.M = table_slots(n_hist, per);
    size_t o = 0;
    L.slots = o;    o += (size_t)L.M * 8;                      // slots and top must stay contiguous (one fill)
    L.top = o;      o = align16(o + h * K * 4);
    L.filled = o;
    L.best = o;     o = align16(o + n * 8);
    L.jump = o;     o = align16(o + n * 8);
    L.entry = o;    o = align16(o + (n / kChunk + 1) * 8);
    L.next = o;     if (chains) o = align16(o + h * 4);
    L.total = o;
    return L;
}

// ---------------------------------------------------------------------------------------------
// Scratch for rac_match_spans_static: lives in the library image, so every GPU that loads the library
// holds these bytes until the process exits.  Host code must not pass the symbol itself to a kernel (on
// the host it is only a stand-in); the device address is looked up once per device below.
constexpr size_t kStaticMatchBytes = RAC_MATCH_STATIC_BYTES;  // 3 MiB: a 32768-token history, 8192 query tokens, 8 hits
static __device__ __align__(256) unsigned char g_match_scratch[kStaticMatchBytes];

static std::mutex g_match_scratch_mutex;
static void *g_match_scratch_addr[64];  // device address of g_match_scratch, per device ordinal; null = not looked up yet

// Device address of the scratch array on the CURRENT device (first call per device does the lookup).
static int static_match_scratch(void **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return RAC_ECUDA;
    std::lock_guard<std::mutex> lock(g_match_scratch_mutex);
    if (!g_match_scratch_addr[dev]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_match_scratch) != cudaSuccess || !ptr) return RAC_ECUDA;
        g_match_scratch_addr[dev] = ptr;
    }
    *out = g_match_scratch_addr[dev];
    return RAC_OK;
}

}  // namespace rac

using namespace rac;

extern "C" {

size_t rac_match_workspace_bytes(int64_t n_hist, int64_t n_query, int32_t max_hits) {
    if (n_hist < 0 || n_query < 0 || max_hits < 0 || max_hits > 16) return 0;
    if (n_hist >= (1ll << 30) || n_query >= (1ll << 30)) return 0;
    return match_layout(n_hist, n_query, max_hits, kSlotsPerWindow).total;
}

static int match_spans(const int32_t *hist_tok, int64_t n_hist, const int32_t *query_tok, int64_t n_query,
                       int32_t min_ngram, int32_t max_hits, int32_t *ref_row, rac_span *spans, int32_t *n_spans,
                       void *workspace, size_t workspace_bytes, int per, void *stream) {
    if (n_hist < 0 || n_query < 0 || !n_spans) return RAC_EINVAL;
    if (n_hist >= (1ll << 30) || n_query >= (1ll << 30)) return RAC_EUNSUPPORTED;
    if (min_ngram < 1 || min_ngram > 32) return RAC_EUNSUPPORTED;
    if (max_hits < 0 || max_hits > 16) return RAC_EUNSUPPORTED;
    if ((n_hist > 0 && !hist_tok) || (n_query > 0 && (!query_tok || !ref_row))) return RAC_EINVAL;
    if (!workspace) return RAC_EINVAL;
    if (reinterpret_cast<uintptr_t>(workspace) & 15u) return RAC_EALIGN;
    MatchLayout L = match_layout(n_hist, n_query, max_hits, per);
    if (workspace_bytes < L.total) return RAC_ESIZE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    MatchParams p = {};
    p.hist = hist_tok;
    p.query = query_tok;
    p.ref_row = ref_row;
    p.spans_out = spans;
    p.n_spans = n_spans;
    p.slots = reinterpret_cast<u64 *>(ws + L.slots);
    p.top = reinterpret_cast<int32_t *>(ws + L.top);
    p.best = reinterpret_cast<int2 *>(ws + L.best);
    p.jump = reinterpret_cast<int2 *>(ws + L.jump);
    p.entry = reinterpret_cast<int2 *>(ws + L.entry);
    p.n_hist = (int)n_hist;
    p.n_query = (int)n_query;
    p.nwin = (int)(n_hist - min_ngram + 1 > 0 ? n_hist - min_ngram + 1 : 0);
    p.w = min_ngram;
    p.K = max_hits > 0 ? max_hits : 1;
    p.next = max_hits == 0 ? reinterpret_cast<int32_t *>(ws + L.next) : nullptr;
    p.bmask = L.M / kBucket - 1;

    // three launches, five when there are many chunks; the times are in the head of this file
    p.ahead = 1;
    const long long n16 = n_query > 0 ? (long long)(L.filled / 16) : 0;
    launch_after(fill_ones_kernel, fill_blocks(n16), 256, 0, st, reinterpret_cast<uint4 *>(ws + L.slots), n16, n_spans);
    if (n_query > 0) {
        if (p.nwin > 0) launch_after(match_insert_kernel, (p.nwin + 255) / 256, 256, 0, st, p);
        launch_query(p, st);
    }
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

int rac_match_spans(const int32_t *hist_tok, int64_t n_hist, const int32_t *query_tok, int64_t n_query,
                    int32_t min_ngram, int32_t max_hits, int32_t *ref_row, rac_span *spans, int32_t *n_spans,
                    void *workspace, size_t workspace_bytes, void *stream) {
    return match_spans(hist_tok, n_hist, query_tok, n_query, min_ngram, max_hits, ref_row, spans, n_spans, workspace,
                       workspace_bytes, kSlotsPerWindow, stream);
}

int rac_spans_to_rows(const rac_span *spans, const int32_t *n_spans, int64_t n_query, int32_t *ref_row, void *stream) {
    if (n_query < 0 || !n_spans) return RAC_EINVAL;
    if (n_query == 0) return RAC_OK;
    if (!spans || !ref_row) return RAC_EINVAL;
    if (n_query >= (1ll << 30)) return RAC_EUNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n_query <= kSpanRowsQuery) {
        launch_after(span_rows_kernel, (unsigned)((n_query + kSpanRows - 1) / kSpanRows), kSpanRows, 0, st, spans, n_spans, (int)n_query,
                     ref_row);
        return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
    }
    int blocks = (int)((n_query + 255) / 256);
    if (blocks > sm_count() * 8) blocks = sm_count() * 8;
    launch_after(fill_i32_kernel, blocks, 256, 0, st, ref_row, (long long)n_query, -1);
    launch_after(spans_to_rows_kernel, sm_count(), 256, 0, st, spans, n_spans, (long long)n_query, ref_row);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

int rac_match_spans_static(const int32_t *hist_tok, int64_t n_hist, const int32_t *query_tok, int64_t n_query,
                           int32_t min_ngram, int32_t max_hits, int32_t *ref_row, rac_span *spans, int32_t *n_spans,
                           void *stream) {
    // size check first, with the same layout function the caller-workspace entry point uses
    const size_t need = rac_match_workspace_bytes(n_hist, n_query, max_hits);
    if (need == 0) return (n_hist < 0 || n_query < 0) ? RAC_EINVAL : RAC_EUNSUPPORTED;
    // where few hits per window leave most of the memory to the table (65536 tokens, four hits), half the table still fits
    const int per = need <= kStaticMatchBytes ? kSlotsPerWindow : kSlotsPerWindow / 2;
    if (match_layout(n_hist, n_query, max_hits, per).total > kStaticMatchBytes) return RAC_ESIZE;  // too large for the scratch
    void *scratch = nullptr;
    int rc = static_match_scratch(&scratch);
    if (rc != RAC_OK) return rc;
    // every launch of the matcher re-initialises the table, the rows and the span count, so whatever the
    // previous call left in the scratch is harmless
    return match_spans(hist_tok, n_hist, query_tok, n_query, min_ngram, max_hits, ref_row, spans, n_spans, scratch,
                       kStaticMatchBytes, per, stream);
}

}  // extern "C"

// ---- persistent index ------------------------------------------------------------------------
namespace {
struct IndexLayout {
    size_t slots, top, filled, end_of, next, indexed, total;
    unsigned int M;
};
bool index_cfg_ok(const rac_index_cfg *c) {
    return c && c->capacity >= 1 && c->capacity < (1ll << 30) && c->min_ngram >= 1 && c->min_ngram <= 32 &&
           c->max_hits >= 0 && c->max_hits <= 16;   // 0 = no cap: chains instead of K-lists
}
IndexLayout index_layout(const rac_index_cfg *c) {
    IndexLayout L;
    L.M = table_slots(c->capacity, 4);
    size_t o = 0;
    L.slots = o;    o += (size_t)L.M * 8;                      // slots and top contiguous: one fill
    L.top = o;      o = align16(o + (size_t)c->capacity * (c->max_hits > 0 ? c->max_hits : 1) * 4);
    L.filled = o;
    L.end_of = o;   o = align16(o + (size_t)c->capacity * 4);
    L.next = o;     o = align16(o + (size_t)c->capacity * 4);
    L.indexed = o;  o = align16(o + 4);
    L.total = o;
    return L;
}
struct QueryLayout {
    size_t best, jump, entry, tok, total;
    unsigned int Mq;
};
QueryLayout query_layout(long long n_query) {
    QueryLayout L;
    const size_t n = (size_t)(n_query > 0 ? n_query : 1);
    L.Mq = table_slots(n_query, 2);
    size_t o = 0;
    L.best = o;    o = align16(o + n * 8);
    L.jump = o;    o = align16(o + n * 8);
    L.entry = o;   o = align16(o + (n / kChunk + 1) * 8);
    L.tok = o;     o += (size_t)L.Mq * 4;
    L.total = o;
    return L;
}
}  // namespace

extern "C" {

size_t rac_index_bytes(const rac_index_cfg *cfg) { return index_cfg_ok(cfg) ? index_layout(cfg).total : 0; }

int rac_index_reset(const rac_index_cfg *cfg, void *index, size_t index_bytes, void *stream) {
    if (!index_cfg_ok(cfg)) return cfg ? RAC_EUNSUPPORTED : RAC_EINVAL;
    if (!index) return RAC_EINVAL;
    if (reinterpret_cast<uintptr_t>(index) & 15u) return RAC_EALIGN;
    const IndexLayout L = index_layout(cfg);
    if (index_bytes < L.total) return RAC_ESIZE;
    const long long n16 = (long long)(L.filled / 16);
    unsigned char *ix = static_cast<unsigned char *>(index);
    launch_after(fill_ones_kernel, fill_blocks(n16), 256, 0, static_cast<cudaStream_t>(stream),
                 reinterpret_cast<uint4 *>(ix + L.slots), n16, reinterpret_cast<int32_t *>(ix + L.indexed));
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

int rac_index_append(const rac_index_cfg *cfg, void *index, size_t index_bytes, const int32_t *hist_tok,
                     int64_t n_before, int64_t n_after, void *stream) {
    if (!index_cfg_ok(cfg)) return cfg ? RAC_EUNSUPPORTED : RAC_EINVAL;
    if (!index || n_before < 0 || n_after < n_before) return RAC_EINVAL;
    if (n_after > cfg->capacity) return RAC_ESIZE;
    if (reinterpret_cast<uintptr_t>(index) & 15u) return RAC_EALIGN;
    const IndexLayout L = index_layout(cfg);
    if (index_bytes < L.total) return RAC_ESIZE;
    if (n_after == n_before) return RAC_OK;
    if (!hist_tok) return RAC_EINVAL;
    unsigned char *ix = static_cast<unsigned char *>(index);
    IndexParams p;
    p.hist = hist_tok;
    p.slots = reinterpret_cast<u64 *>(ix + L.slots);
    p.top = reinterpret_cast<int32_t *>(ix + L.top);
    p.end_of = reinterpret_cast<int32_t *>(ix + L.end_of);
    p.next = cfg->max_hits == 0 ? reinterpret_cast<int32_t *>(ix + L.next) : nullptr;
    p.indexed = reinterpret_cast<int32_t *>(ix + L.indexed);
    p.a = (int)n_before;
    p.b = (int)n_after;
    p.w = cfg->min_ngram;
    p.K = cfg->max_hits > 0 ? cfg->max_hits : 1;
    p.bmask = L.M / kBucket - 1;
    launch_after(index_append_kernel, (unsigned)((n_after - n_before + 63) / 64), 64, 0, static_cast<cudaStream_t>(stream), p);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

size_t rac_index_query_workspace_bytes(int64_t n_query) {
    if (n_query < 0 || n_query >= (1ll << 30)) return 0;
    return query_layout(n_query).total;
}

int rac_index_query(const rac_index_cfg *cfg, const void *index, size_t index_bytes, const int32_t *hist_tok,
                    int64_t n_hist, const int32_t *query_tok, int64_t n_query, int32_t intra, int32_t *ref_row,
                    rac_span *spans, int32_t *n_spans, void *workspace, size_t workspace_bytes, void *stream) {
    return rac_index_query_live(cfg, index, index_bytes, hist_tok, n_hist, 0, query_tok, n_query, intra, ref_row, spans,
                                n_spans, workspace, workspace_bytes, stream);
}

int rac_index_query_live(const rac_index_cfg *cfg, const void *index, size_t index_bytes, const int32_t *hist_tok,
                         int64_t n_hist, int64_t first_live, const int32_t *query_tok, int64_t n_query, int32_t intra,
                         int32_t *ref_row, rac_span *spans, int32_t *n_spans, void *workspace, size_t workspace_bytes,
                         void *stream) {
    if (!index_cfg_ok(cfg)) return cfg ? RAC_EUNSUPPORTED : RAC_EINVAL;
    if (!index || !n_spans || n_hist < 0 || n_query < 0 || !workspace) return RAC_EINVAL;
    if (first_live < 0 || first_live > n_hist) return RAC_EINVAL;
    if (n_hist > cfg->capacity) return RAC_ESIZE;
    if (n_query >= (1ll << 30) || n_hist + n_query >= (1ll << 31)) return RAC_EUNSUPPORTED;
    if ((n_hist > 0 && !hist_tok) || (n_query > 0 && (!query_tok || !ref_row))) return RAC_EINVAL;
    if ((reinterpret_cast<uintptr_t>(index) & 15u) || (reinterpret_cast<uintptr_t>(workspace) & 15u)) return RAC_EALIGN;
    const IndexLayout L = index_layout(cfg);
    if (index_bytes < L.total) return RAC_ESIZE;
    const QueryLayout Q = query_layout(n_query);
    if (workspace_bytes < Q.total) return RAC_ESIZE;
    const unsigned char *ix = static_cast<const unsigned char *>(index);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    MatchParams p = {};
    p.hist = hist_tok;
    p.query = query_tok;
    p.ref_row = ref_row;
    p.spans_out = spans;
    p.n_spans = n_spans;
    p.slots = const_cast<u64 *>(reinterpret_cast<const u64 *>(ix + L.slots));
    p.top = const_cast<int32_t *>(reinterpret_cast<const int32_t *>(ix + L.top));
    p.best = reinterpret_cast<int2 *>(ws + Q.best);
    p.jump = reinterpret_cast<int2 *>(ws + Q.jump);
    p.entry = reinterpret_cast<int2 *>(ws + Q.entry);
    p.n_hist = (int)n_hist;
    p.n_query = (int)n_query;
    p.nwin = (int)(n_hist - cfg->min_ngram + 1 > 0 ? n_hist - cfg->min_ngram + 1 : 0);
    p.w = cfg->min_ngram;
    p.K = cfg->max_hits > 0 ? cfg->max_hits : 1;
    p.bmask = L.M / kBucket - 1;
    p.next = cfg->max_hits == 0 ? const_cast<int32_t *>(reinterpret_cast<const int32_t *>(ix + L.next)) : nullptr;
    p.first_live = (int)first_live;
    p.end_of = reinterpret_cast<const int32_t *>(ix + L.end_of);
    p.indexed = reinterpret_cast<const int32_t *>(ix + L.indexed);
    if (n_query == 0) {
        launch_after(fill_ones_kernel, 1, 32, 0, st, (uint4 *)nullptr, 0ll, n_spans);
        return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
    }
    p.intra = intra != 0;
    if (intra && !query_in_one(n_query)) {     // the token table starts empty
        p.tok = reinterpret_cast<unsigned int *>(ws + Q.tok);
        p.tmask = Q.Mq - 1;
        const long long n16 = (long long)Q.Mq / 4;
        launch_after(fill_ones_kernel, fill_blocks(n16), 256, 0, st, reinterpret_cast<uint4 *>(ws + Q.tok), n16, (int32_t *)nullptr);
        p.ahead = 1;
    }
    launch_query(p, st);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

}  // extern "C"

extern "C" int rac_spans_to_segments(const rac_span *spans, const int32_t *n_spans, int64_t T, int64_t max_seg,
                                     int32_t *seg_off, int32_t *n_seg, void *stream) {
    if (!n_spans || !seg_off || !n_seg || T < 0 || max_seg < 1) return RAC_EINVAL;
    if (T >= (1ll << 30) || max_seg >= (1ll << 30)) return RAC_EUNSUPPORTED;
    if (!spans) return RAC_EINVAL;
    launch_after(spans_to_segments_kernel, 1, 1024, 0, static_cast<cudaStream_t>(stream), spans, n_spans, (int)T, (int)max_seg,
                 seg_off, n_seg);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}
