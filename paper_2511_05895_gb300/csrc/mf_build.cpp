// Host construction of the Bi-CSR graph representation (Sec. 5.1 of the
// paper: outgoing and incoming edges of every vertex in one list, zero-
// capacity entries for missing reverse edges, and an array giving the
// position of each arc's reverse in the neighbour's list, so that a push
// touches both directions in O(1)).
//
// Parallel edges u -> v share one arc (capacities add) and both directions of
// a vertex pair form one arc pair; this changes no max-flow value.
//
// Every step runs on one team of host threads (one start per build), split
// into pieces of equal numbers of entries rather than of vertices, so that
// rows of any length share out; the arrays are first touched by the threads
// that fill them.  (Measured on 16 Grace cores, against steps that counted,
// scattered and zero-filled on one thread: 2^20-vertex RMAT graph of 16.8M
// edges 650 -> 260 ms, 65,537 vertices with 1M edges 23 -> 12 ms, 2048^2 grid of
// 25M edges 505 -> 115 ms.)
#include <algorithm>
#include <atomic>
#include <climits>
#include <condition_variable>
#include <functional>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>
#include <vector>

#include "mf_internal.h"

namespace mf {
namespace {

// Threads that live for one build and run its steps one after the other.
class Team {
  public:
    explicit Team(int64_t work) {
        const unsigned hw = std::thread::hardware_concurrency();
        // a thread costs about what 16k entries cost
        n_ = int(std::max<int64_t>(1, std::min<int64_t>({int64_t(hw ? hw : 1), 64, work >> 14})));
        pool_.reserve(size_t(n_));
        try {
            for (int i = 1; i < n_; ++i) pool_.emplace_back([this] { loop(); });
        } catch (const std::system_error &) {   // fewer threads then
            n_ = int(pool_.size()) + 1;
        } catch (const std::bad_alloc &) {      // likewise
            n_ = int(pool_.size()) + 1;
        }
    }
    ~Team() {
        {
            std::lock_guard<std::mutex> lk(mu_);
            quit_ = true;
            ++round_;
        }
        go_.notify_all();
        for (auto &t : pool_) t.join();
    }
    int size() const { return n_; }

    // fn(begin, end) over pieces of [0, count), taken by the threads as they
    // get free.  fn must not throw.
    template <class F>
    void each(int64_t count, int64_t grain, F &&fn) {
        if (count <= 0) return;
        grain = std::max<int64_t>(1, grain);
        if (n_ == 1 || count <= grain) {
            fn(int64_t(0), count);
            return;
        }
        std::atomic<int64_t> next(0);
        run([&] {
            for (;;) {
                const int64_t b = next.fetch_add(grain, std::memory_order_relaxed);
                if (b >= count) return;
                fn(b, std::min(count, b + grain));
            }
        });
    }
    template <class F>
    void each(int64_t count, F &&fn) {
        each(count, std::max<int64_t>(4096, count / (int64_t(n_) * 8)), fn);
    }

    // fn(u0, u1) over vertex ranges of about equal numbers of entries, row[]
    // being the vertices' entry offsets.
    template <class T, class F>
    void rows(const T *row, int32_t n, F &&fn) {
        const int64_t total = row[n] - row[0];
        const int64_t parts = n_ == 1 ? 1 : std::min<int64_t>(int64_t(n_) * 16, total / 2048 + 1);
        each(parts, 1, [&](int64_t b, int64_t e) {
            for (int64_t p = b; p < e; ++p) fn(cut(row, n, p, parts), cut(row, n, p + 1, parts));
        });
    }

    // fn(b, e) over pieces of the edges [0, m), a long row's shared out too.
    template <class F>
    void edges(int64_t m, F &&fn) {
        each(m, std::max<int64_t>(4096, m / (int64_t(n_) * 16)), fn);
    }

  private:
    template <class T>
    static int32_t cut(const T *row, int32_t n, int64_t p, int64_t parts) {
        if (p <= 0) return 0;
        if (p >= parts) return n;
        const T at = T(row[0] + (row[n] - row[0]) / parts * p);
        return int32_t(std::lower_bound(row, row + n, at) - row);
    }
    void run(const std::function<void()> &job) {
        {
            std::lock_guard<std::mutex> lk(mu_);
            job_ = &job;
            busy_ = n_ - 1;
            ++round_;
        }
        go_.notify_all();
        job();
        std::unique_lock<std::mutex> lk(mu_);
        done_.wait(lk, [this] { return busy_ == 0; });
    }
    void loop() {
        uint64_t seen = 0;
        for (;;) {
            const std::function<void()> *job;
            {
                std::unique_lock<std::mutex> lk(mu_);
                go_.wait(lk, [&] { return round_ != seen; });
                seen = round_;
                if (quit_) return;
                job = job_;
            }
            (*job)();
            std::lock_guard<std::mutex> lk(mu_);
            if (--busy_ == 0) done_.notify_one();
        }
    }
    int n_ = 1, busy_ = 0;
    uint64_t round_ = 0;
    bool quit_ = false;
    const std::function<void()> *job_ = nullptr;
    std::mutex mu_;
    std::condition_variable go_, done_;
    std::vector<std::thread> pool_;
};

// fn(u, i0, i1) for every vertex u with edges [i0, i1) in [b, e).
template <class F>
void by_tail(const int64_t *row, int32_t n, int64_t b, int64_t e, F &&fn) {
    int32_t u = int32_t(std::upper_bound(row, row + n + 1, b) - row) - 1;
    for (int64_t i = b; i < e; ++u) {
        const int64_t end = std::min(e, row[u + 1]);
        if (end > i) fn(u, i, end);
        i = std::max(i, end);
    }
}

// A bitmap of n ids, all clear; false without memory for it.
bool clear_marks(std::vector<uint64_t> &marks, int32_t n) noexcept {
    try {
        marks.assign(size_t(n) / 64 + 1, 0);
        return true;
    } catch (const std::bad_alloc &) {
        return false;
    }
}

// Sort p[0, d) (values below n) and keep each value once; returns how many.  A
// row that holds a good part of all ids is sorted by marking them in a bitmap.
// (Runs in the team's steps, which must not throw.)
int32_t sort_unique(int32_t *p, int64_t d, int32_t n, std::vector<uint64_t> &marks) noexcept {
    if (std::is_sorted(p, p + d) || d < 4096 || d < n / 32 || !clear_marks(marks, n)) {
        if (!std::is_sorted(p, p + d)) std::sort(p, p + d);
        return int32_t(std::unique(p, p + d) - p);
    }
    for (int64_t i = 0; i < d; ++i) marks[size_t(p[i]) >> 6] |= uint64_t(1) << (p[i] & 63);
    int32_t *q = p;
    for (size_t w = 0; w < marks.size(); ++w)
        for (uint64_t x = marks[w]; x; x &= x - 1) *q++ = int32_t(w * 64 + size_t(__builtin_ctzll(x)));
    return int32_t(q - p);
}

inline int64_t find_sorted(const int32_t *a, int64_t lo, int64_t hi, int32_t key) {
    const int32_t *p = std::lower_bound(a + lo, a + hi, key);
    return (p != a + hi && *p == key) ? (p - a) : -1;
}

// Whether vertices are worth renumbering by degree: s and t aside (every arc
// of a grid or assignment graph's terminals is spread over the others), the
// vertices of more than 64 entries hold at least a quarter of all entries.
// On such a power-law graph most heads are then among the first ids: their
// heights sit in few cache lines (L1 serves part of them), the reads of a
// sorted row fall into the same sectors, and a bottom-up search meets the
// likely parents first.  Measured per batch on an RMAT-20 graph with random
// ids: 100k repair 1.61 -> 1.26 ms, push-pull 0.67 -> 0.56 ms, static solve
// 2.83 -> 2.38 ms.  Where degrees are alike, the given order may have locality
// of its own (grids) and is kept.  A power-law graph whose given order has some
// loses it: with 90 % of the edges inside blocks of 256 consecutive ids (2^18
// vertices) a repair takes 1.16 ms, push-pull 0.49, with 95 % inside blocks of
// 512 (2^20) 2.37 and 0.82, still 0.68-0.84 of what the kernel before the
// renumbering took on the same graphs.
bool skewed(const HostArray<int32_t> &deg, int32_t n, int32_t s, int32_t t) {
    int64_t total = 0, big = 0;
    for (int32_t u = 0; u < n; ++u) {
        const int64_t d = deg[size_t(u)];
        total += d;
        if (d > kBigDeg && u != s && u != t) big += d;
    }
    return big > 0 && big * 4 >= total;
}

// Vertices by descending degree, equal degrees in the given order.
void order_by_degree(const HostArray<int32_t> &deg, int32_t n, HostBiCSR &G) {
    int32_t top = 0;
    for (int32_t u = 0; u < n; ++u) top = std::max(top, deg[size_t(u)]);
    std::vector<int32_t> at(size_t(top) + 2, 0);
    for (int32_t u = 0; u < n; ++u) at[size_t(top - deg[size_t(u)]) + 1]++;
    for (int32_t d = 0; d <= top; ++d) at[size_t(d) + 1] += at[size_t(d)];
    G.ord.resize(size_t(n));
    G.inv.resize(size_t(n));
    for (int32_t u = 0; u < n; ++u) {
        const int32_t p = at[size_t(top - deg[size_t(u)])]++;
        G.ord[size_t(p)] = u;
        G.inv[size_t(u)] = p;
    }
}

}  // namespace

int build_bicsr(int32_t n, int64_t m, const int64_t *row_ptr, const int32_t *col,
                const int32_t *cap, int32_t s, int32_t t, bool renumber, HostBiCSR *out) {
    if (n < 2 || m < 0 || m >= INT32_MAX || s < 0 || t < 0 || s >= n || t >= n || s == t)
        return 1;
    if (row_ptr[0] != 0 || row_ptr[n] != m) return 1;
    for (int32_t u = 0; u < n; ++u)
        if (row_ptr[u + 1] < row_ptr[u]) return 1;
    try {
        Team team(m + n);
        std::atomic<int> bad(0);
        team.each(m, [&](int64_t b, int64_t e) {
            int wrong = 0;
            for (int64_t i = b; i < e; ++i) wrong |= col[i] < 0 || col[i] >= n || cap[i] < 0;
            if (wrong) bad.store(1);
        });
        if (bad.load()) return 1;
        HostBiCSR &G = *out;
        G.n = n; G.m = m; G.s = s; G.t = t;
        // 1. entries per vertex (out-heads and in-tails, self-loops left out)
        HostArray<int32_t> deg(static_cast<size_t>(n));
        team.each(n, [&](int64_t b, int64_t e) { std::fill(deg.data() + b, deg.data() + e, 0); });
        // (the sink, which a good part of the edges may enter, is counted per
        // piece: one atomic instead of one per edge on one word)
        team.edges(m, [&](int64_t pb, int64_t pe) {
            int32_t to_t = 0;
            by_tail(row_ptr, n, pb, pe, [&](int32_t u, int64_t b, int64_t e) {
                int32_t own = 0;
                for (int64_t i = b; i < e; ++i) {
                    if (col[i] == u) continue;
                    ++own;
                    if (col[i] == t) ++to_t;
                    else __atomic_fetch_add(&deg[size_t(col[i])], 1, __ATOMIC_RELAXED);
                }
                if (own) __atomic_fetch_add(&deg[size_t(u)], own, __ATOMIC_RELAXED);
            });
            if (to_t) __atomic_fetch_add(&deg[size_t(t)], to_t, __ATOMIC_RELAXED);
        });
        if (renumber && skewed(deg, n, s, t)) order_by_degree(deg, n, G);
        const int32_t *inv = G.inv.empty() ? nullptr : G.inv.data();
        const int32_t *ord = G.ord.empty() ? nullptr : G.ord.data();
        auto id = [inv](int32_t v) { return inv ? inv[v] : v; };
        std::vector<int64_t> at(size_t(n) + 1);   // entry offsets (from here on in the new ids)
        at[0] = 0;
        for (int32_t u = 0; u < n; ++u) at[size_t(u) + 1] = at[size_t(u)] + deg[size_t(ord ? ord[u] : u)];
        // 2. every vertex's neighbour multiset, sorted, each neighbour once
        HostArray<int32_t> nb(size_t(at[size_t(n)]));
        HostArray<int32_t> fill(static_cast<size_t>(n));
        team.each(n, [&](int64_t b, int64_t e) { std::fill(fill.data() + b, fill.data() + e, 0); });
        team.edges(m, [&](int64_t pb, int64_t pe) {
            int32_t to_t = 0;
            by_tail(row_ptr, n, pb, pe, [&](int32_t u, int64_t b, int64_t e) {
                if (u != t)
                    for (int64_t i = b; i < e; ++i) to_t += col[i] == t;
            });
            const int32_t nt = id(t);
            int64_t pt = at[size_t(nt)] + (to_t ? __atomic_fetch_add(&fill[size_t(nt)], to_t, __ATOMIC_RELAXED) : 0);
            by_tail(row_ptr, n, pb, pe, [&](int32_t u, int64_t b, int64_t e) {
                const int32_t nu = id(u);
                int32_t own = 0;
                for (int64_t i = b; i < e; ++i) own += col[i] != u;
                if (!own) return;
                int64_t p = at[size_t(nu)] + __atomic_fetch_add(&fill[size_t(nu)], own, __ATOMIC_RELAXED);
                for (int64_t i = b; i < e; ++i) {
                    if (col[i] == u) continue;
                    const int32_t nv = id(col[i]);
                    nb[size_t(p++)] = nv;
                    if (nv == nt) nb[size_t(pt++)] = nu;
                    else nb[size_t(at[size_t(nv)] + __atomic_fetch_add(&fill[size_t(nv)], 1, __ATOMIC_RELAXED))] = nu;
                }
            });
        });
        HostArray<int32_t> &uniq = fill;   // distinct neighbours
        team.rows(at.data(), n, [&](int32_t u0, int32_t u1) {
            std::vector<uint64_t> marks;
            for (int32_t u = u0; u < u1; ++u)
                uniq[size_t(u)] = sort_unique(nb.data() + at[size_t(u)], at[size_t(u) + 1] - at[size_t(u)], n, marks);
        });
        int64_t A = 0;
        for (int32_t u = 0; u < n; ++u) A += uniq[size_t(u)];
        if (A >= INT32_MAX) return 1;
        G.arcs = A;
        G.row.resize(size_t(n) + 1);
        G.row[0] = 0;
        for (int32_t u = 0; u < n; ++u) G.row[size_t(u) + 1] = G.row[size_t(u)] + uniq[size_t(u)];
        const int32_t *row = G.row.data();
        G.head.resize(size_t(A));
        G.rev.resize(size_t(A));
        G.cap.resize(size_t(A));
        HostArray<int32_t> mult(static_cast<size_t>(A));
        team.rows(row, n, [&](int32_t u0, int32_t u1) {
            for (int32_t u = u0; u < u1; ++u)
                std::copy(nb.data() + at[size_t(u)], nb.data() + at[size_t(u)] + uniq[size_t(u)], G.head.data() + row[u]);
            std::fill(G.cap.data() + row[u0], G.cap.data() + row[u1], 0);
            std::fill(mult.data() + row[u0], mult.data() + row[u1], 0);
        });
        nb.resize(0);
        // 3. reverse arcs: each pair from its lower end, whose position in the
        // other row a binary search finds
        team.rows(row, n, [&](int32_t u0, int32_t u1) {
            for (int32_t u = u0; u < u1; ++u) {
                const int32_t *p = std::upper_bound(G.head.data() + row[u], G.head.data() + row[u + 1], u);
                for (int32_t a = int32_t(p - G.head.data()); a < row[u + 1]; ++a) {
                    const int32_t v = G.head[size_t(a)];
                    const int32_t b = int32_t(find_sorted(G.head.data(), row[v], row[v + 1], u));
                    G.rev[size_t(a)] = b;
                    G.rev[size_t(b)] = a;
                }
            }
        });
        // 4. edge -> arc map, arc capacities, pair multiplicities
        G.arc_of_edge.resize(size_t(m));
        std::atomic<int> overflow(0);
        // (whole rows: the capacities of parallel edges add up on one thread; a
        // sorted row's edges lie at consecutive arcs, which are tried first)
        team.rows(row_ptr, n, [&](int32_t u0, int32_t u1) {
            for (int32_t u = u0; u < u1; ++u) {
                const int32_t nu = id(u);
                int64_t a = row[nu];
                for (int64_t i = row_ptr[u]; i < row_ptr[u + 1]; ++i) {
                    if (col[i] == u) {
                        G.arc_of_edge[size_t(i)] = -1;
                        continue;
                    }
                    const int32_t nv = id(col[i]);
                    if (a >= row[nu + 1] || G.head[size_t(a)] != nv)
                        a = find_sorted(G.head.data(), row[nu], row[nu + 1], nv);
                    G.arc_of_edge[size_t(i)] = int32_t(a);
                    int64_t c = int64_t(G.cap[size_t(a)]) + cap[i];
                    if (c > INT32_MAX) {
                        overflow.store(1);
                        c = INT32_MAX;
                    }
                    G.cap[size_t(a)] = int32_t(c);
                    mult[size_t(a)]++;
                    ++a;
                }
            }
        });
        std::mutex mu;
        int64_t maxmult = 1;
        team.each(A, [&](int64_t b, int64_t e) {
            int64_t most = 1;
            for (int64_t a = b; a < e; ++a)
                if (mult[size_t(a)]) most = std::max(most, int64_t(mult[size_t(a)]) + mult[size_t(G.rev[size_t(a)])]);
            std::lock_guard<std::mutex> lk(mu);
            maxmult = std::max(maxmult, most);
        });
        G.cap_limit = int32_t(INT32_MAX / maxmult);
        if (overflow.load()) return 1;
        team.each(m, [&](int64_t b, int64_t e) {
            int wrong = 0;
            for (int64_t i = b; i < e; ++i) wrong |= cap[i] > G.cap_limit;
            if (wrong) bad.store(1);
        });
        if (bad.load()) return 1;
        // 5. work-item bound for big vertices
        G.chunk_items = 0;
        G.hubs = 0;
        G.hub_chunk_items = 0;
        G.max_deg = 0;
        for (int32_t u = 0; u < n; ++u) {
            const int32_t d = row[u + 1] - row[u];
            G.max_deg = std::max(G.max_deg, d);
            if (d > kBigDeg) G.chunk_items += (d + kChunk - 1) / kChunk;
            if (d > kHubDeg) {
                G.hubs += 1;
                G.hub_chunk_items += (d + kPrChunk - 1) / kPrChunk;
            }
        }
        // 6. the policy's "edges out of s or into t" feature, one byte per edge
        // (0 for a self-loop, which has no arc)
        G.edge_st.resize(size_t(m));
        team.rows(row_ptr, n, [&](int32_t u0, int32_t u1) {
            for (int32_t u = u0; u < u1; ++u)
                for (int64_t i = row_ptr[u]; i < row_ptr[u + 1]; ++i)
                    G.edge_st[size_t(i)] = col[i] != u && (u == s || col[i] == t);
        });
    } catch (const std::bad_alloc &) {
        return 2;
    }
    return 0;
}

void external_arcs(int32_t n, const int32_t *row, const int32_t *head, const int32_t *ord, const int32_t *inv,
                   int32_t *ext_row, int32_t *arc_at) {
    ext_row[0] = 0;
    for (int32_t u = 0; u < n; ++u) ext_row[u + 1] = ext_row[u] + (row[inv[u] + 1] - row[inv[u]]);
    Team team(int64_t(ext_row[n]) + n);
    team.rows(ext_row, n, [&](int32_t u0, int32_t u1) {
        for (int32_t u = u0; u < u1; ++u) {
            int32_t *p = arc_at + ext_row[u], *q = arc_at + ext_row[u + 1];
            for (int32_t a = row[inv[u]], *x = p; x != q; ++x) *x = a++;
            std::sort(p, q, [&](int32_t a, int32_t b) { return ord[head[a]] < ord[head[b]]; });
        }
    });
}

void gather_i32(const int32_t *src, const int32_t *at, int64_t count, bool scatter, int32_t *dst) {
    Team team(count);
    team.each(count, [&](int64_t b, int64_t e) {
        if (scatter)
            for (int64_t i = b; i < e; ++i) dst[at[i]] = src ? src[i] : int32_t(i);
        else
            for (int64_t i = b; i < e; ++i) dst[i] = src[at[i]];
    });
}

}  // namespace mf
