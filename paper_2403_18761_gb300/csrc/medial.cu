// Dual medial mesh of the restricted power diagram and its thinning.
//
// Sec. 3.2: the medial mesh is the dual of the RPD: one vertex per sphere with
// a nonempty restricted power cell, an edge (i, j) per RPF, a triangle
// (i, j, k) per RPE and a tetrahedron (i, j, k, l) per RPV.
//
// Sec. 5.3 (geometry-guided thinning): a simple pair (x, y) is a simplex x and
// a face y of x that no other simplex of the complex has as a face; removing
// it keeps the complex's homotopy type.  Every triangle f_ijk gets the
// importance alpha_ijk = length(RPE_ijk) / mean(2 r_i, 2 r_j, 2 r_k).  First
// the tet-face simple pairs are removed, least important triangle first, until
// no tetrahedron is left; then the triangle-edge simple pairs whose triangle
// belonged to an original tetrahedron are removed, least important first,
// while the importance is below sigma.
//
// Ties (readings of the paper, which does not fix them): equal importances go
// to the triangle whose key (sorted sphere ids) is lexicographically
// smallest; a triangle with several free edges gives up the edge with the
// smallest key.  Runs on the host: the pruning is a sequential priority
// process over a complex of a few 10^4 simplices.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <queue>
#include <utility>
#include <vector>

#include "internal.cuh"

namespace {

// Rows of sorted keys (arity words each, ascending), indexed by their first
// word: a sub-key is found among the few rows that share its first sphere.
struct Rows {
    const int32_t* k;
    int arity;
    std::vector<int32_t> start;   // first row of each first word
    Rows(const std::vector<int32_t>& keys, int ar) : k(keys.data()), arity(ar) {
        const size_t n = keys.size() / ar;
        int32_t mx = -1;
        for (size_t i = 0; i < n; i++) mx = std::max(mx, keys[i * ar]);
        start.assign((size_t)mx + 2, 0);
        for (size_t i = 0; i < n; i++) start[keys[i * ar] + 1]++;
        for (size_t v = 1; v < start.size(); v++) start[v] += start[v - 1];
    }
    // row of (q[0], ..., q[arity-1]), or -1
    long long find(const int32_t* q) const {
        if (q[0] < 0 || (size_t)q[0] + 1 >= start.size()) return -1;
        int32_t lo = start[q[0]], hi = start[q[0] + 1];
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            const int32_t* r = k + (size_t)mid * arity;
            int c = 1;
            while (c < arity && r[c] == q[c]) c++;
            if (c == arity) return mid;
            if (r[c] < q[c]) lo = mid + 1;
            else hi = mid;
        }
        return -1;
    }
};

// Cofaces of each of n simplices in one array: list[start[x] .. start[x + 1]).
struct Cofaces {
    std::vector<int32_t> start, list;
    template <size_t W>
    Cofaces(size_t n, const std::vector<std::array<int32_t, W>>& sub) : start(n + 1, 0) {
        for (const auto& s : sub)
            for (int32_t x : s)
                if (x >= 0) start[x + 1]++;
        for (size_t v = 1; v <= n; v++) start[v] += start[v - 1];
        list.resize(start[n]);
        std::vector<int32_t> at(start.begin(), start.end() - 1);
        for (size_t i = 0; i < sub.size(); i++)
            for (int32_t x : sub[i])
                if (x >= 0) list[at[x]++] = (int32_t)i;
    }
};

// A binary heap of faces by (alpha, face index), smallest first.  A face may be
// in it more than once: whoever pops one looks whether it is still a candidate.
struct Item {
    double alpha;
    int32_t f;
};
struct After {
    bool operator()(const Item& a, const Item& b) const { return a.alpha > b.alpha || (a.alpha == b.alpha && a.f > b.f); }
};
using Queue = std::priority_queue<Item, std::vector<Item>, After>;

}  // namespace

// On the 205k-tet slab's 9 k edges, 11 k triangles and 4 k tetrahedra the form
// with a std::map per key table, a std::vector per simplex and a std::set as
// the queue took some 15 ms of rpd_medial.
int medial_thin(const std::vector<int32_t>& edges, const std::vector<int32_t>& faces,
                const std::vector<double>& alpha, const std::vector<int32_t>& tets, double sigma,
                std::vector<uint8_t>& edge_alive, std::vector<uint8_t>& face_alive, std::vector<uint8_t>& tet_alive) {
    const size_t ne = edges.size() / 2, nf = faces.size() / 3, nt = tets.size() / 4;
    edge_alive.assign(ne, 1);
    face_alive.assign(nf, 1);
    tet_alive.assign(nt, 1);
    const Rows erow(edges, 2), frow(faces, 3);
    // boundary relations (keys are sorted, so sub-keys are too)
    std::vector<std::array<int32_t, 3>> f_edges(nf);
    std::vector<std::array<int32_t, 4>> t_faces(nt);
    for (size_t f = 0; f < nf; f++) {
        const int32_t* k = &faces[3 * f];
        const int32_t sub[3][2] = {{k[0], k[1]}, {k[0], k[2]}, {k[1], k[2]}};
        for (int q = 0; q < 3; q++) f_edges[f][q] = (int32_t)erow.find(sub[q]);
    }
    std::vector<uint8_t> orig(nf, 0);
    for (size_t t = 0; t < nt; t++) {
        const int32_t* k = &tets[4 * t];
        const int32_t sub[4][3] = {{k[0], k[1], k[2]}, {k[0], k[1], k[3]}, {k[0], k[2], k[3]}, {k[1], k[2], k[3]}};
        for (int q = 0; q < 4; q++) {
            t_faces[t][q] = (int32_t)frow.find(sub[q]);
            if (t_faces[t][q] >= 0) orig[t_faces[t][q]] = 1;
        }
    }
    const Cofaces face_tet(nf, t_faces), edge_face(ne, f_edges);
    std::vector<int32_t> face_tets(nf), edge_faces(ne);
    for (size_t f = 0; f < nf; f++) face_tets[f] = face_tet.start[f + 1] - face_tet.start[f];
    for (size_t e = 0; e < ne; e++) edge_faces[e] = edge_face.start[e + 1] - edge_face.start[e];
    // priority: (alpha, face index); face indices follow key order
    std::vector<Item> first;
    for (size_t f = 0; f < nf; f++)
        if (face_tets[f] == 1) first.push_back({alpha[f], (int32_t)f});
    Queue queue(After(), std::move(first));
    auto push_tf = [&](size_t f) {
        if (face_alive[f] && face_tets[f] == 1) queue.push({alpha[f], (int32_t)f});
    };
    long long left = (long long)nt;
    while (left > 0 && !queue.empty()) {
        const size_t f = (size_t)queue.top().f;
        queue.pop();
        if (!face_alive[f] || face_tets[f] != 1) continue;
        size_t t = (size_t)-1;
        for (int32_t z = face_tet.start[f]; z < face_tet.start[f + 1]; z++)
            if (tet_alive[face_tet.list[z]]) t = (size_t)face_tet.list[z];
        if (t == (size_t)-1) continue;
        tet_alive[t] = 0;
        left--;
        face_alive[f] = 0;
        for (int q = 0; q < 3; q++)
            if (f_edges[f][q] >= 0) edge_faces[f_edges[f][q]]--;
        for (int q = 0; q < 4; q++) {
            const int32_t g = t_faces[t][q];
            if (g < 0 || (size_t)g == f) continue;
            face_tets[g]--;
            push_tf((size_t)g);
        }
    }
    // triangle-edge pairs of the original tetrahedra's triangles, alpha < sigma
    Queue q2;
    auto push_fe = [&](size_t f) {
        if (!face_alive[f] || !orig[f] || face_tets[f] != 0 || !(alpha[f] < sigma)) return;
        for (int q = 0; q < 3; q++) {
            const int32_t e = f_edges[f][q];
            if (e >= 0 && edge_alive[e] && edge_faces[e] == 1) {
                q2.push({alpha[f], (int32_t)f});
                return;
            }
        }
    };
    for (size_t f = 0; f < nf; f++) push_fe(f);
    while (!q2.empty()) {
        const size_t f = (size_t)q2.top().f;
        q2.pop();
        if (!face_alive[f] || face_tets[f] != 0) continue;
        int32_t ebest = -1;
        for (int q = 0; q < 3; q++) {   // sub-keys in order: the first free edge has the smallest key
            const int32_t e = f_edges[f][q];
            if (e >= 0 && edge_alive[e] && edge_faces[e] == 1) {
                ebest = e;
                break;
            }
        }
        if (ebest < 0) continue;
        face_alive[f] = 0;
        edge_alive[ebest] = 0;
        for (int q = 0; q < 3; q++) {
            const int32_t e = f_edges[f][q];
            if (e < 0 || e == ebest) continue;
            edge_faces[e]--;
            // the other triangle on this edge may have become prunable
            if (edge_faces[e] == 1)
                for (int32_t z = edge_face.start[e]; z < edge_face.start[e + 1]; z++)
                    push_fe((size_t)edge_face.list[z]);
        }
    }
    return 0;
}
