// Internal declarations shared by the host graph builder (mf_build.cpp) and
// the CUDA library (mf_gpu.cu).  Not part of the public ABI (include/mf.h).
#pragma once

#include <cstddef>
#include <cstdint>
#include <memory>
#include <vector>

namespace mf {

// Frontier vertices whose Bi-CSR degree exceeds kBigDeg are expanded by the
// BFS as kChunk-arc work items spread over all warps instead of inside their
// 32-vertex group, so that no warp holds more than 32 x kBigDeg arcs of a
// level.
constexpr int kBigDeg = 64;
constexpr int kChunk = 256;
// Active vertices whose degree exceeds kHubDeg ("hubs") run PushRelabel and
// RemoveInvalidEdges cooperatively over the whole grid, in kPrChunk-arc work
// items; smaller ones are handled by one warp each.
constexpr int kHubDeg = 512;
constexpr int kPrChunk = 256;

// A host array whose elements are not touched before they are filled (a
// std::vector would zero them on one thread first).
template <class T>
class HostArray {
  public:
    HostArray() = default;
    explicit HostArray(size_t n) { resize(n); }
    void resize(size_t n) {   // the old contents are lost
        p_.reset();
        size_ = 0;
        if (n) p_.reset(new T[n]);
        size_ = n;
    }
    T *data() { return p_.get(); }
    const T *data() const { return p_.get(); }
    T &operator[](size_t i) { return p_[i]; }
    const T &operator[](size_t i) const { return p_[i]; }
    size_t size() const { return size_; }
    bool empty() const { return size_ == 0; }
    const T *begin() const { return p_.get(); }
    const T *end() const { return p_.get() + size_; }

  private:
    std::unique_ptr<T[]> p_;
    size_t size_ = 0;
};

// Host image of the Bi-CSR of Sec. 5.1.  Vertex u owns arcs row[u] ..
// row[u+1]-1, one per distinct neighbour v (u -> v edge, v -> u edge, or
// both), sorted by v.  rev[a] is the arc of the opposite direction in the
// neighbour's list.  cap[a] is the sum of the capacities of the input edges
// u -> v (0 when there is none).  arc_of_edge[e] is the arc that carries input
// edge e, or -1 for a self-loop.  A renumbered graph's rows and heads are in
// its own vertex ids: ord[u] is the input's id of vertex u, inv its inverse
// (both empty otherwise); s and t are the input's.
struct HostBiCSR {
    int32_t n = 0;
    int64_t m = 0;
    int64_t arcs = 0;
    int32_t s = 0, t = 0;
    HostArray<int32_t> row;
    HostArray<int32_t> head, rev, cap;
    HostArray<int32_t> arc_of_edge;
    HostArray<int32_t> ord, inv;
    HostArray<unsigned char> edge_st;   // per edge: 1 if it leaves s or enters t
    int32_t cap_limit = 0;      // largest capacity one edge may take
    int64_t chunk_items = 0;    // sum over big vertices of ceil(deg / kChunk)
    int64_t hubs = 0;           // vertices with degree > kHubDeg
    int64_t hub_chunk_items = 0;  // sum over hubs of ceil(deg / kPrChunk)
    int32_t max_deg = 0;
};

// Returns 0 on success, 1 (MF_EINVAL) on bad input, 2 (MF_ENOMEM) on
// allocation failure.  Inputs are host pointers.  With renumber, vertices are
// renumbered by degree where that pays (mf_build.cpp).
int build_bicsr(int32_t n, int64_t m, const int64_t *row_ptr, const int32_t *col,
                const int32_t *cap, int32_t s, int32_t t, bool renumber, HostBiCSR *out);

// The arcs of a renumbered graph in the order of the input's ids (rows by
// input id, heads within a row by input id): ext_row [n+1] their offsets,
// arc_at [arcs] the renumbered graph's arc at each place.
void external_arcs(int32_t n, const int32_t *row, const int32_t *head, const int32_t *ord, const int32_t *inv,
                   int32_t *ext_row, int32_t *arc_at);

// dst[i] = src[at[i]] (dst may be at itself), or with scatter dst[at[i]] = src[i]
// (src null: i), on several threads.
void gather_i32(const int32_t *src, const int32_t *at, int64_t count, bool scatter, int32_t *dst);

}  // namespace mf
