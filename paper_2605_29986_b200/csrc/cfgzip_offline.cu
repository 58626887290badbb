// Offline step of CFGzip behind the C ABI (declarations and contracts: include/cfgzip.h).
//   host: grammars in Greibach normal form, the stack-adjacency relation (Appendix C), the displacement of every
//         token (Algorithm 1) serialised into fixed-width signature rows;
//   GPU : grouping of tokens with equal signature into classes, representatives, class lists (Section 3.1,
//         "Pre-Computation").
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstring>
#include <new>
#include <thread>
#include <vector>
#ifdef __SSE2__
#include <emmintrin.h>
#endif

#include "cfgzip.h"
#include "class_sort.cuh"
#include "workspace.h"

struct cfgzip_grammar {
    int32_t n = 0, start = 0;
    struct Prod {
        int32_t head;
        uint8_t term;
        std::vector<int32_t> rhs;
    };
    std::vector<Prod> prods;
    std::vector<std::vector<int32_t>> by_term;  // production indices by terminal byte, ascending by head
    uint8_t byte_class[256] = {};               // bytes with the same productions have the same number
    std::vector<uint8_t> adj;                   // n * n, adj[y * n + z] = 1: z may be popped right after y left nothing
};

namespace {

// Appendix C: edge A -> B for every production whose right-most non-terminal is B; for every production
// A -> a B_1 .. B_n Z beta a breadth-first search from B_n collects the reachable Y with a production Y -> y.
void build_adjacency(cfgzip_grammar& g) {
    const int32_t n = g.n;
    std::vector<std::vector<int32_t>> edges(static_cast<size_t>(n));
    std::vector<uint8_t> unary(static_cast<size_t>(n), 0);
    for (const auto& p : g.prods) {
        if (p.rhs.empty())
            unary[size_t(p.head)] = 1;
        else
            edges[size_t(p.head)].push_back(p.rhs.back());
    }
    g.adj.assign(size_t(n) * size_t(n), 0);
    std::vector<int32_t> queue;
    std::vector<uint8_t> seen;
    for (const auto& p : g.prods) {
        for (size_t i = 1; i < p.rhs.size(); ++i) {
            const int32_t z = p.rhs[i];
            seen.assign(size_t(n), 0);
            queue.clear();
            queue.push_back(p.rhs[i - 1]);
            seen[size_t(p.rhs[i - 1])] = 1;
            for (size_t q = 0; q < queue.size(); ++q) {
                const int32_t x = queue[q];
                if (unary[size_t(x)]) g.adj[size_t(x) * size_t(n) + size_t(z)] = 1;
                for (int32_t y : edges[size_t(x)])
                    if (!seen[size_t(y)]) {
                        seen[size_t(y)] = 1;
                        queue.push_back(y);
                    }
            }
        }
    }
}

// Two bytes whose productions have the same heads and right-hand sides can stand for one another in every token.
void number_bytes(cfgzip_grammar& g) {
    auto less = [&](int32_t x, int32_t y) {
        const auto &a = g.prods[size_t(x)], &b = g.prods[size_t(y)];
        return a.head != b.head ? a.head < b.head : a.rhs < b.rhs;
    };
    std::vector<std::vector<int32_t>> known;  // sorted production lists, one per class
    for (int b = 0; b < 256; ++b) {
        std::vector<int32_t> list = g.by_term[size_t(b)];
        std::sort(list.begin(), list.end(), less);
        size_t k = 0;
        for (; k < known.size(); ++k)
            if (known[k].size() == list.size() &&
                std::equal(list.begin(), list.end(), known[k].begin(), [&](int32_t x, int32_t y) { return !less(x, y) && !less(y, x); }))
                break;
        if (k == known.size()) known.push_back(std::move(list));
        g.byte_class[b] = uint8_t(k);  // (at most 256 classes)
    }
}

constexpr size_t padded(size_t words) { return (words + 15) & ~size_t(15); }  // to whole lines of 64 bytes

// Signature rows one worker has already built in this call, by the token's string of byte classes: most tokens of a vocabulary
// (words, runs of digits) read the same to the grammar as another token. Only the words a row uses are kept, as rows may be wide
// and mostly zeros. Bounded; what does not fit is built anew. (128256 tokens on one core, ms without / with: a JSON grammar without
// literals and escapes, 99 in 100 tokens known, rows of 64 words 15 / 6.1, of 256 words 21 / 12; with them, 6 in 10 known, 29 / 23
// and 34 / 29. Whole rows kept, the wide ones took 42.)
class RowCache {
  public:
    struct Entry {
        uint64_t hash;
        size_t key, row;     // start in keys_, in rows_
        int32_t len, words;  // words: of the signature, -1: too many pairs
        int32_t used;        // words in front of the row's zeros
        bool fits;
    };
    RowCache(const cfgzip_grammar& g, int32_t V) : g_(g), most_(std::min(size_t(8192), size_t(V))) {
        size_t n = 16;
        while (n < 4 * most_) n *= 2;
        slots_.assign(n, -1);
    }
    // The entry of a token, null if it is not known (then `add` takes what is built for it).
    const Entry* find(const uint8_t* bytes, int32_t len) {
        token_.resize(size_t(len));
        uint64_t h = 0x9E3779B97F4A7C15ull + uint64_t(len);
        for (int32_t i = 0; i < len; ++i) {
            token_[size_t(i)] = g_.byte_class[bytes[i]];
            h = (h ^ token_[size_t(i)]) * 0x100000001B3ull;
        }
        h ^= h >> 29;
        hash_ = h;
        for (at_ = size_t(h) & (slots_.size() - 1); slots_[at_] >= 0; at_ = (at_ + 1) & (slots_.size() - 1)) {
            const Entry& e = entries_[size_t(slots_[at_])];
            if (e.hash == h && e.len == len && std::memcmp(keys_.data() + e.key, token_.data(), size_t(len)) == 0) return &e;
        }
        return nullptr;
    }
    const int32_t* row(const Entry& e) const { return rows_.data() + e.row; }
    void add(const int32_t* row, int32_t used, int32_t words, bool fits) {  // for the token last looked for
        if (entries_.size() >= most_ || rows_.size() + size_t(used) > kMostWords) return;
        slots_[at_] = int32_t(entries_.size());
        entries_.push_back(Entry{hash_, keys_.size(), rows_.size(), int32_t(token_.size()), words, used, fits});
        keys_.insert(keys_.end(), token_.begin(), token_.end());
        rows_.insert(rows_.end(), row, row + used);
        rows_.resize(padded(rows_.size()), 0);  // (every row starts a line, as the one before it does)
    }

  private:
    static constexpr size_t kMostWords = size_t(1) << 22;
    const cfgzip_grammar& g_;
    const size_t most_;
    std::vector<int32_t> slots_;  // four times as many as entries: an empty one always ends a search
    std::vector<Entry> entries_;
    std::vector<uint8_t> keys_, token_;
    std::vector<int32_t> rows_;
    uint64_t hash_ = 0;
    size_t at_ = 0;
};

// Algorithm 1 as a depth-first enumeration with explicit stacks. `prev` is the symbol popped last (-1: none yet). The
// pairs found are kept flat in one growing array ([n_in, in .., n_out, out (top first) ..] each) that is reused from
// token to token, so that a token allocates nothing; they are sorted and made unique at the end. (A std::set of pairs of
// vectors took 260 ns per token on one core, this 118.)
struct Displacer {
    const cfgzip_grammar& g;
    int64_t max_pairs;
    const uint8_t* t = nullptr;
    int32_t len = 0;
    bool overflow = false;
    std::vector<int32_t> s_in, s_out;  // s_out: top at the back
    std::vector<int32_t> flat;
    std::vector<size_t> pairs;         // where each pair starts in `flat`
    size_t compact_at = 0;             // pairs are made unique when this many have piled up

    Displacer(const cfgzip_grammar& grammar, int64_t most) : g(grammar), max_pairs(most) {}

    // order and equality of std::pair<std::vector, std::vector> on (input stack, output stack)
    int compare(size_t x, size_t y) const {
        const int32_t *a = flat.data() + x, *b = flat.data() + y;
        for (int part = 0; part < 2; ++part) {
            const int32_t na = *a++, nb = *b++;
            const int32_t n = std::min(na, nb);
            for (int32_t i = 0; i < n; ++i)
                if (a[i] != b[i]) return a[i] < b[i] ? -1 : 1;
            if (na != nb) return na < nb ? -1 : 1;
            a += na;
            b += nb;
        }
        return 0;
    }
    void make_unique() {
        std::sort(pairs.begin(), pairs.end(), [&](size_t x, size_t y) { return compare(x, y) < 0; });
        pairs.erase(std::unique(pairs.begin(), pairs.end(), [&](size_t x, size_t y) { return compare(x, y) == 0; }), pairs.end());
        if (int64_t(pairs.size()) > max_pairs) overflow = true;
    }

    void displace(const uint8_t* bytes, int32_t n) {
        t = bytes;
        len = n;
        overflow = false;
        s_in.clear();
        s_out.clear();
        flat.clear();
        pairs.clear();
        compact_at = 4096;
        run(0, -1);  // (an empty token moves no stack: its only pair is (empty, empty))
        if (!overflow) make_unique();
    }

    void found() {
        pairs.push_back(flat.size());
        flat.push_back(int32_t(s_in.size()));
        flat.insert(flat.end(), s_in.begin(), s_in.end());
        flat.push_back(int32_t(s_out.size()));
        flat.insert(flat.end(), s_out.rbegin(), s_out.rend());
        if (pairs.size() >= compact_at) {  // many derivations, perhaps of few pairs
            make_unique();
            std::vector<int32_t> kept;
            for (size_t& at : pairs) {
                const size_t from = at, n_in = size_t(flat[from]), n = 2 + n_in + size_t(flat[from + 1 + n_in]);
                at = kept.size();
                kept.insert(kept.end(), flat.begin() + long(from), flat.begin() + long(from + n));
            }
            flat.swap(kept);
            compact_at = std::max(size_t(4096), 2 * pairs.size());
        }
    }

    void run(int32_t pos, int32_t prev) {
        if (overflow) return;
        if (pos == len) return found();
        const auto& cands = g.by_term[t[pos]];  // ascending by head
        if (s_out.empty()) {  // stack backtrack: the next symbol of the input stack is guessed
            for (int32_t pi : cands) {
                const auto& p = g.prods[size_t(pi)];
                if (prev >= 0 && !g.adj[size_t(prev) * size_t(g.n) + size_t(p.head)]) continue;
                s_in.push_back(p.head);
                s_out.insert(s_out.end(), p.rhs.rbegin(), p.rhs.rend());
                run(pos + 1, p.head);
                s_out.resize(s_out.size() - p.rhs.size());
                s_in.pop_back();
            }
        } else {
            const int32_t top = s_out.back();
            auto it = cands.begin();
            if (cands.size() > 8)
                it = std::lower_bound(it, cands.end(), top, [&](int32_t pi, int32_t h) { return g.prods[size_t(pi)].head < h; });
            for (; it != cands.end(); ++it) {
                const auto& p = g.prods[size_t(*it)];
                if (p.head > top) break;
                if (p.head < top) continue;
                s_out.pop_back();
                s_out.insert(s_out.end(), p.rhs.rbegin(), p.rhs.rend());
                run(pos + 1, top);
                s_out.resize(s_out.size() - p.rhs.size());
                s_out.push_back(top);
            }
        }
    }
};

// Tokens are independent: worker threads take them in runs of this many from a shared counter. A run is some tens of
// microseconds of work, so a thread is started for every few of them only, and never more than the machine has cores.
constexpr int32_t kTokenRun = 256;
constexpr int32_t kRunsPerThread = 8;

// A finished row goes out with stores that pass the caches by, where the row's alignment allows it: rows left dirty in
// the caches of a dozen cores make the copy to the GPU that usually follows two and a half times slower (33 MB: 1.5 ms
// against 0.6). `used` words, zeros behind them; `from` has zeros up to the next whole line of 16 words:
// by lines the loops' lengths differ little from token to token.
void write_row(int32_t* row, const int32_t* from, size_t used, size_t words) {
#ifdef __SSE2__
    if (words % 4 == 0 && (reinterpret_cast<uintptr_t>(row) & 15u) == 0) {
        size_t i = 0;
        used = std::min(padded(used), words);
        for (; i < used; i += 4)
            _mm_stream_si128(reinterpret_cast<__m128i*>(row + i), _mm_loadu_si128(reinterpret_cast<const __m128i*>(from + i)));
        for (; i < words; i += 4) _mm_stream_si128(reinterpret_cast<__m128i*>(row + i), _mm_setzero_si128());
        return;
    }
#endif
    std::memcpy(row, from, used * 4);
    std::memset(row + used, 0, (words - used) * 4);
}
void rows_written() {  // such stores are ordered before whatever tells another thread that the rows are there
#ifdef __SSE2__
    _mm_sfence();
#endif
}

int worker_count(int32_t V) {
    const int64_t wanted = V / (kTokenRun * kRunsPerThread);
    if (wanted <= 1) return 1;
    return int(std::min({int64_t(std::max(1u, std::thread::hardware_concurrency())), int64_t(32), wanted}));
}

}  // namespace

extern "C" {

int cfgzip_grammar_create(int32_t n_nonterminals, int32_t start, const int32_t* prod_head, const uint8_t* prod_terminal,
                          const int32_t* prod_rhs_off, const int32_t* prod_rhs, int32_t n_prod, cfgzip_grammar** out) {
    if (!out) return CFGZIP_E_ARG;
    *out = nullptr;
    if (n_nonterminals <= 0 || start < 0 || start >= n_nonterminals || n_prod < 0) return CFGZIP_E_ARG;
    if (n_prod > 0 && (!prod_head || !prod_terminal || !prod_rhs_off)) return CFGZIP_E_ARG;
    cfgzip_grammar* g = new (std::nothrow) cfgzip_grammar();
    if (!g) return CFGZIP_E_NOMEM;
    g->n = n_nonterminals;
    g->start = start;
    g->by_term.resize(256);
    for (int32_t i = 0; i < n_prod; ++i) {
        const int32_t lo = prod_rhs_off[i], hi = prod_rhs_off[i + 1];
        bool ok = prod_head[i] >= 0 && prod_head[i] < n_nonterminals && lo >= 0 && hi >= lo && (hi == lo || prod_rhs);
        cfgzip_grammar::Prod p{prod_head[i], prod_terminal[i], {}};
        for (int32_t j = lo; ok && j < hi; ++j) {
            ok = prod_rhs[j] >= 0 && prod_rhs[j] < n_nonterminals;
            p.rhs.push_back(prod_rhs[j]);
        }
        if (!ok) {
            delete g;
            return CFGZIP_E_RANGE;
        }
        g->by_term[p.term].push_back(int32_t(g->prods.size()));
        g->prods.push_back(std::move(p));
    }
    for (auto& list : g->by_term)
        std::stable_sort(list.begin(), list.end(), [&](int32_t x, int32_t y) { return g->prods[size_t(x)].head < g->prods[size_t(y)].head; });
    number_bytes(*g);
    build_adjacency(*g);
    cfgzip::Workspace::hold();
    *out = g;
    return CFGZIP_OK;
}

int cfgzip_grammar_destroy(cfgzip_grammar* g) {
    if (!g) return CFGZIP_E_ARG;
    delete g;
    cfgzip::Workspace::drop();
    return CFGZIP_OK;
}

int cfgzip_grammar_adjacency(const cfgzip_grammar* g, uint8_t* adjacency) {
    if (!g || !adjacency) return CFGZIP_E_ARG;
    std::memcpy(adjacency, g->adj.data(), g->adj.size());
    return CFGZIP_OK;
}

int cfgzip_displacement_signatures(const cfgzip_grammar* g, const uint8_t* token_bytes, const int64_t* token_off, int32_t V,
                                   int32_t row_words, int32_t* signatures, int32_t* signature_words, int64_t max_pairs) {
    if (!g || !token_off || V < 0 || row_words < 1 || !signatures || max_pairs < 1) return CFGZIP_E_ARG;
    if (V > 0 && !token_bytes && token_off[V] > token_off[0]) return CFGZIP_E_ARG;
    for (int32_t i = 0; i < V; ++i)
        if (token_off[i + 1] < token_off[i] || token_off[i + 1] - token_off[i] > 0x7FFFFFFF) return CFGZIP_E_ARG;
    std::atomic<int32_t> next{0};
    std::atomic<int> rc{CFGZIP_OK};
    auto work = [&]() noexcept {
        try {
            Displacer d(*g, max_pairs);
            RowCache cache(*g, V);
            std::vector<int32_t> built(padded(size_t(row_words)));
            for (;;) {
                const int32_t first = next.fetch_add(kTokenRun);
                if (first >= V || first < 0) break;
                const int32_t last = int32_t(std::min<int64_t>(int64_t(first) + kTokenRun, V));
                for (int32_t i = first; i < last; ++i) {
                    const uint8_t* token = token_bytes + token_off[i];
                    const int32_t len = int32_t(token_off[i + 1] - token_off[i]);
                    int32_t* row = signatures + int64_t(i) * row_words;
                    if (const RowCache::Entry* known = cache.find(token, len)) {
                        if (signature_words) signature_words[i] = known->words;
                        if (!known->fits) rc.store(CFGZIP_E_RANGE);
                        write_row(row, cache.row(*known), size_t(known->used), size_t(row_words));
                        continue;
                    }
                    d.displace(token, len);
                    // canonical sequence: the pairs in lexicographic order, each as len(sigma_i), sigma_i, len(sigma_o), sigma_o
                    int64_t n = 0;
                    for (size_t at : d.pairs) n += 2 + d.flat[at] + d.flat[at + 1 + size_t(d.flat[at])];
                    const bool fits = !d.overflow && n + 1 <= row_words;
                    if (signature_words) signature_words[i] = d.overflow ? -1 : int32_t(n);
                    int32_t* out = built.data();
                    if (fits) {
                        *out++ = int32_t(n);
                        for (size_t at : d.pairs) {
                            const int32_t* p = d.flat.data() + at;
                            out = std::copy(p, p + 2 + p[0] + p[1 + p[0]], out);
                        }
                    } else {
                        rc.store(CFGZIP_E_RANGE);
                    }
                    const int32_t used = int32_t(out - built.data());
                    std::fill(out, built.data() + padded(size_t(used)), 0);
                    write_row(row, built.data(), size_t(used), size_t(row_words));
                    cache.add(built.data(), used, d.overflow ? -1 : int32_t(n), fits);
                }
            }
            rows_written();
        } catch (...) {
            rc.store(CFGZIP_E_NOMEM);
            next.store(V);
        }
    };
    std::vector<std::thread> helpers;
    try {
        const int n_workers = worker_count(V);
        helpers.reserve(size_t(n_workers));
        for (int w = 1; w < n_workers; ++w) helpers.emplace_back(work);
    } catch (...) {
        // fewer helpers than wanted: the tokens are shared out among those there are
    }
    work();
    for (std::thread& h : helpers) h.join();
    return rc.load();
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------------------------
// Grouping on the GPU. Tokens whose signature rows are equal word for word form a class. An open-addressing table
// keyed by the row CONTENT (a hash only picks the first slot; a slot is shared only after the rows compared equal)
// gives every token the slot of its class; the lowest token id of a slot names the class, classes are numbered in
// the order of those lowest ids (a prefix sum over "I am the lowest id of my class" flags), the representative is
// the member with the smallest (byte length, id), and the class lists are a stable sort of the tokens by class
// (class_sort.cuh).
// What bounds it: reading the signature rows once (33 MB at V = 128256 and 64 words: 5 us from HBM) and a dozen short
// launches. Most tokens often share one class (what no rule of the grammar can use), so every atomic on a class is
// preceded by a look whether it still changes anything, or made once for the equal lanes of a warp.
// ---------------------------------------------------------------------------------------------------------------
namespace {

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

constexpr int kRowLanes = 8;       // lanes that read a signature row together
constexpr int kSeedTokens = 2048;  // tokens the first, small launch inserts

// Eight lanes per token: coalesced reads of the row, words hashed with their positions, the sums of the lanes added up.
// The slots of the big classes are taken by a first launch over the first kSeedTokens tokens: without it tens of
// thousands of tokens of one class find its slot empty at once and queue up at one compare-and-swap.
__global__ void __launch_bounds__(256) k_group_insert(const int32_t* __restrict__ sig, int W, int first, int end, int32_t* owner,
                                                      unsigned table_mask, int32_t* slot_of) {
    const int sub = threadIdx.x & (kRowLanes - 1);
    const int t = first + int((blockIdx.x * blockDim.x + threadIdx.x) / kRowLanes);
    if (t >= end) return;
    const unsigned lanes = ((1u << kRowLanes) - 1u) << (threadIdx.x & 31 & ~(kRowLanes - 1));
    const int32_t* row = sig + int64_t(t) * W;
    unsigned long long h = 0ull;
    for (int w = sub; w < W; w += kRowLanes)
        h += mix64((static_cast<unsigned long long>(unsigned(w) + 1u) << 32) ^ static_cast<unsigned>(__ldg(row + w)));
#pragma unroll
    for (int d = kRowLanes / 2; d >= 1; d >>= 1) h += __shfl_xor_sync(lanes, h, d, kRowLanes);
    unsigned slot = unsigned(mix64(h)) & table_mask;
    for (unsigned probe = 0; probe <= table_mask; ++probe) {  // the table has at least 2 V slots: a free one always turns up
        int32_t o = 0;
        if (sub == 0) {
            o = *reinterpret_cast<volatile int32_t*>(owner + slot);
            if (o == -1) o = atomicCAS(owner + slot, -1, t);
        }
        o = __shfl_sync(lanes, o, 0, kRowLanes);
        bool same = true;
        if (o != -1 && o != t) {
            const int32_t* other = sig + int64_t(o) * W;
            for (int w = sub; w < W && same; w += kRowLanes) same = __ldg(other + w) == __ldg(row + w);
        }
        if (__all_sync(lanes, same)) break;
        slot = (slot + 1) & table_mask;
    }
    if (sub == 0) slot_of[t] = int32_t(slot);
}

// The lowest token id and the smallest (length, id) of every slot. Both arrays start at all ones.
__global__ void __launch_bounds__(256) k_group_min(const int32_t* slot_of, const int32_t* __restrict__ len, int V, unsigned* min_id,
                                                   unsigned long long* rep_key) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool have = t < V;
    const int slot = have ? slot_of[t] : -1 - lane;  // lanes without a token match nobody
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, slot);
    const unsigned n = have ? unsigned(len[t]) : 0u;
    const unsigned shortest = __reduce_min_sync(peers, n);
    const unsigned of_shortest = __reduce_min_sync(peers, n == shortest ? unsigned(t) : 0xFFFFFFFFu);
    if (!have || lane != __ffs(int(peers)) - 1) return;  // the first lane of a class holds its lowest id in the warp
    if (*reinterpret_cast<volatile unsigned*>(min_id + slot) > unsigned(t)) atomicMin(min_id + slot, unsigned(t));
    const unsigned long long key = (static_cast<unsigned long long>(shortest) << 32) | of_shortest;
    if (*reinterpret_cast<volatile unsigned long long*>(rep_key + slot) > key) atomicMin(rep_key + slot, key);
}

// How many of a block's tokens are the lowest of their class.
constexpr int kNumberTile = 4096;  // tokens per block of the numbering kernels, four per thread
__global__ void __launch_bounds__(1024) k_group_count(const int32_t* slot_of, const unsigned* min_id, int V, int32_t* block_count) {
    int n = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int t = blockIdx.x * kNumberTile + q * 1024 + threadIdx.x;
        n += __syncthreads_count(t < V && min_id[slot_of[t]] == unsigned(t));
    }
    if (threadIdx.x == 0) block_count[blockIdx.x] = n;
}

// Classes numbered in token order (every block adds up the counts of the blocks in front of it), representatives.
__global__ void __launch_bounds__(1024) k_group_number(const int32_t* slot_of, const unsigned* min_id,
                                                       const unsigned long long* rep_key, int V, const int32_t* block_count,
                                                       int32_t* class_of_slot, int32_t* r, int32_t* n_classes) {
    __shared__ int s_warp[32], s_front;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_front = 0;
    __syncthreads();
    int front = 0;
    for (int b = tid; b < int(blockIdx.x); b += 1024) front += block_count[b];
    front = __reduce_add_sync(0xFFFFFFFFu, front);
    if (lane == 0 && front) atomicAdd(&s_front, front);
    const int t0 = blockIdx.x * kNumberTile + tid * 4;
    int slot[4];
    bool lowest[4];
    int mine = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        slot[q] = t0 + q < V ? slot_of[t0 + q] : -1;
        lowest[q] = slot[q] >= 0 && min_id[slot[q]] == unsigned(t0 + q);
        mine += lowest[q];
    }
    int inc = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += up;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    int k = s_front + inc - mine;
    for (int w = 0; w < warp; ++w) k += s_warp[w];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (lowest[q]) {
            class_of_slot[slot[q]] = k;
            r[k] = int32_t(rep_key[slot[q]] & 0xFFFFFFFFull);
            ++k;
        }
    if (blockIdx.x == gridDim.x - 1 && tid == 1023) *n_classes = k;  // the last thread has counted everybody
}

__global__ void __launch_bounds__(256) k_group_assign(const int32_t* slot_of, const int32_t* class_of_slot, int V, int32_t* c) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < V) c[t] = class_of_slot[slot_of[t]];
}

inline unsigned blocks_for(int64_t n, int threads) { return unsigned((n + threads - 1) / threads); }

}  // namespace

extern "C" int cfgzip_group_tokens(const int32_t* signatures, int32_t row_words, const int32_t* token_len, int32_t V,
                                   int32_t* token_to_class, int32_t* class_to_rep, int32_t* n_classes, int32_t* class_off,
                                   int32_t* class_tok, void* stream) {
    if (V < 0 || row_words < 1) return CFGZIP_E_ARG;
    if (V == 0) return CFGZIP_OK;
    if (!signatures || !token_len || !token_to_class || !class_to_rep || !n_classes) return CFGZIP_E_ARG;
    if ((class_off == nullptr) != (class_tok == nullptr)) return CFGZIP_E_ARG;
    if (V > (1 << 28)) return CFGZIP_E_RANGE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned table = 1;
    while (table < 2u * unsigned(V)) table <<= 1;
    // scratch: rep_key, min_id, owner [table], all ones to begin with; slot_of [V], block counts, the sort's own
    const unsigned number_blocks = blocks_for(V, kNumberTile);
    const size_t words = size_t(table) * 4 + size_t(V) + number_blocks + (class_off ? cfgzip::class_sort_scratch_words(V) : 0);
    cfgzip::Workspace scratch(words * 4);
    if (!scratch.ptr) return CFGZIP_E_NOMEM;
    unsigned long long* rep_key = static_cast<unsigned long long*>(scratch.ptr);
    unsigned* min_id = reinterpret_cast<unsigned*>(rep_key + table);
    int32_t* owner = reinterpret_cast<int32_t*>(min_id + table);  // later the class of a slot
    int32_t* slot_of = owner + table;
    int32_t* block_count = slot_of + V;
    bool ok = cudaMemsetAsync(rep_key, 0xFF, size_t(table) * 16, st) == cudaSuccess;
    if (ok) {
        const int T = 256, per_block = T / kRowLanes, seed = std::min(V, kSeedTokens);
        k_group_insert<<<blocks_for(seed, per_block), T, 0, st>>>(signatures, row_words, 0, seed, owner, table - 1, slot_of);
        if (V > seed)
            k_group_insert<<<blocks_for(V - seed, per_block), T, 0, st>>>(signatures, row_words, seed, V, owner, table - 1, slot_of);
        k_group_min<<<blocks_for(V, T), T, 0, st>>>(slot_of, token_len, V, min_id, rep_key);
        k_group_count<<<number_blocks, 1024, 0, st>>>(slot_of, min_id, V, block_count);
        k_group_number<<<number_blocks, 1024, 0, st>>>(slot_of, min_id, rep_key, V, block_count, owner, class_to_rep, n_classes);
        k_group_assign<<<blocks_for(V, T), T, 0, st>>>(slot_of, owner, V, token_to_class);
        if (class_off)
            cfgzip::class_sort(token_to_class, V, n_classes, 0, class_off, class_tok, block_count + number_blocks, st);
        ok = cudaGetLastError() == cudaSuccess;
    }
    ok = (cudaStreamSynchronize(st) == cudaSuccess) && ok;  // the scratch is released below
    if (!ok) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    return CFGZIP_OK;
}
