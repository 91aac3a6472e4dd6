// Internal host-side structures of the FE-LBM library (not part of the ABI).
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <exception>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "felbm.h"

namespace felbm {

void set_error(const std::string& msg);

// Reverse Cuthill-McKee order of a node graph given as CSR adjacency
// (no self loops); returns order[new] = old.  Components one after another.
std::vector<int32_t> rcm_order(int32_t N, const std::vector<int32_t>& adj_ptr,
                               const std::vector<int32_t>& adj);

// Most nodes in one node tile and in one block of the blocked solve (half a
// tile), most nodes of a block and the layers around it, and most layers.
constexpr int32_t kTileNodes = 1024;
constexpr int32_t kBlockCore = 512;
constexpr int32_t kBlockNodes = 1024;
constexpr int32_t kBlockSteps = 8;

// f(k, scratch) for k in [0, n) on the host's cores, at least `grain` of them a
// thread (on the calling thread alone where no other can be started); every
// thread works with its own make().  The first exception is rethrown on the
// calling thread.
template <class Make, class F>
void parallel_for(int32_t n, int32_t grain, const Make& make, const F& f) {
    const int32_t nt = std::min<int32_t>(std::max(1u, std::thread::hardware_concurrency()), n / grain);
    std::vector<std::thread> pool;
    std::atomic<int32_t> next{0};
    std::exception_ptr failed;
    std::mutex mu;
    const auto work = [&]() {
        try {
            auto scratch = make();
            for (int32_t k; (k = next.fetch_add(1)) < n;) f(k, scratch);
        } catch (...) {
            std::lock_guard<std::mutex> lock(mu);
            if (!failed) failed = std::current_exception();
        }
    };
    try {
        for (int32_t t = 1; t < nt; ++t) pool.emplace_back(work);
    } catch (...) {
    }
    work();
    for (auto& t : pool) t.join();
    if (failed) std::rethrow_exception(failed);
}

// The nodes around one block and their places in its node list: a hash table of a
// fixed size, so that what a thread of parallel_for keeps does not grow with the
// mesh.  Holds up to kBlockNodes + 1 nodes.
struct NodePlaces {
    static constexpr int kBits = 12;
    std::vector<int32_t> node, place;
    NodePlaces() : node(size_t(1) << kBits, -1), place(size_t(1) << kBits) {}
    void clear() { std::fill(node.begin(), node.end(), -1); }
    // the slot that holds node c, or the free one where it would stand
    size_t slot(int32_t c) const {
        size_t s = (uint32_t)c * 2654435761u >> (32 - kBits);
        while (node[s] >= 0 && node[s] != c) s = (s + 1) & (node.size() - 1);
        return s;
    }
    bool add(int32_t c, int32_t at) {        // false: it was there
        const size_t s = slot(c);
        if (node[s] == c) return false;
        node[s] = c;
        place[s] = at;
        return true;
    }
};
static_assert(kBlockNodes + 1 < 1 << (NodePlaces::kBits - 1), "the table of NodePlaces stays half empty");

// Host mesh after preprocessing.  Node ids are the internal ids (node tiles
// of recursive coordinate bisection, reverse Cuthill-McKee order inside a
// tile); perm[new] = caller id, iperm[caller] = new.
struct HostMesh {
    int32_t N = 0, T = 0, E = 0;
    double period[2] = {0.0, 0.0};
    std::vector<int32_t> perm, iperm;
    std::vector<double> x, y;                 // node coordinates, internal order
    // triangles, structure of arrays: vertex k of triangle t at tri[k*T + t]
    std::vector<int32_t> tri;                 // [3][T]
    std::vector<double> area;                 // [T]
    std::vector<double> grad;                 // [6][T]: bx0, by0, bx1, by1, bx2, by2
    std::vector<int32_t> nbr;                 // [3][T]: triangle across the edge opposite vertex k, -1 = wall
    std::vector<int32_t> nbr_slot;            // [3][T]: that edge's local index in the neighbour
    // node-node pattern (CSR, sorted columns, diagonal included)
    std::vector<int32_t> row_ptr, col;
    std::vector<double> mass;                 // consistent mass matrix entries
    std::vector<double> stiff;                // P1 stiffness entries sum_T A_T b_i.b_j
    std::vector<double> lumped;               // row sums of the mass matrix
    std::vector<double> patch;                // area of the vertex patch
    // node -> incident triangles (CSR) with the node's shape gradient there
    std::vector<int32_t> inc_ptr, inc_tri;
    std::vector<double> inc_bx, inc_by;
    // wall edges: end nodes, id, length, unit normal out of the fluid
    std::vector<int32_t> wall_a, wall_b, wall_id;
    std::vector<double> wall_len, wall_nx, wall_ny;
    // node -> incident wall edges (CSR)
    std::vector<int32_t> winc_ptr, winc_edge;
    double min_area = 0.0, total_area = 0.0;
    int32_t max_degree = 0, bandwidth = 0;
    // node tiles: tile k holds the internal nodes [tile_ptr[k], tile_ptr[k+1]),
    // at most kTileNodes, all in one component
    std::vector<int32_t> tile_ptr;
    int32_t max_halo = 0;                     // most nodes outside a tile that its matrix rows reference
    // blocks of the blocked solve: a tile, or each half of one of more than
    // kBlockCore nodes.  halo[halo_ptr[k] ...] lists the nodes around block k
    // layer by layer (layer 1: the nodes outside that share a matrix row entry
    // with one inside, layer 2: those that share one with layer 1, ...; each
    // layer sorted); layer_cnt[k][l] counts the block's nodes and those up to
    // layer l.  n_layers layers, the same for every block: as many as keep
    // every block's count within kBlockNodes (at most kBlockSteps; 0: none do).
    std::vector<int32_t> blk_ptr;
    std::vector<int32_t> halo_ptr, halo;
    std::vector<int32_t> layer_cnt;           // [blocks][kBlockSteps + 1]
    int32_t n_layers = 0;
    // triangles at the nodes of block k: blk_tri[blk_tri_ptr[k] ...], sorted
    std::vector<int32_t> blk_tri_ptr, blk_tri;
    int32_t max_blk_tri = 0;
    // connected components ("groups"), numbered by their lowest caller node
    // id; each occupies a contiguous range of internal nodes and triangles
    int32_t G = 0;
    std::vector<int32_t> grp_node_begin, grp_node_end, grp_tri_begin, grp_tri_end;
    std::vector<int32_t> grp_wall_ptr, grp_wall_edge;   // wall edges of each group (CSR)
    std::vector<int32_t> grp_first_caller, grp_size;
    std::vector<double> grp_period_x, grp_period_y;      // periodic lengths of each group
};

}  // namespace felbm

struct felbm_mesh {
    felbm::HostMesh h;
};
