// Host check of the builder's walk grid, no GPU: every point of a triangle
// has to be found from the grid cell that it lies in.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "../../paper_2203_14354_gb300/csrc/lxo_internal.h"

// Builds the trees of tri_v ([nt] x 3 vertices) as lxo_build_bvh does.
// Returns -1 on a failed build, 0 if the scene has no walk grid, else 1 with
// *lost = how many of the points pts[k], each on triangle ids[k], are not in
// the tree of their cell: descending from it into every box that contains the
// point meets no leaf with that triangle.  Points of triangles outside the
// main tree (planar layers) are not looked at; *seen counts the others.
extern "C" int walk_grid_check(const float* tri_v, uint32_t nt, uint32_t leaf_size, uint32_t n_threads,
                               const float* pts, const uint32_t* ids, uint32_t n, uint32_t* lost, uint32_t* seen)
{
    *lost = *seen = 0;
    float max_abs = 0.0f;
    for (uint64_t k = 0; k < 9ull * nt; ++k) max_abs = std::max(max_abs, std::fabs(tri_v[k]));
    std::vector<int32_t> layer(nt, -1);
    const int n_layers = lxo::detect_layers(tri_v, nt, layer.data());
    lxo::BvhHost b;
    char msg[256] = {0};
    try {
        if (lxo::build_bvh(tri_v, nt, layer.data(), n_layers, leaf_size, 0, n_threads, std::ldexp(max_abs, -19), &b,
                           msg, sizeof msg))
            return -1;
    } catch (...) {
        lxo::free_bvh(&b);
        return -1;
    }
    const bool grid = !b.walk_ref.empty();
    for (uint32_t k = 0; grid && k < n; ++k) {
        if (layer[ids[k]] >= 0) continue;
        ++*seen;
        double g[3];
        int c[3];
        for (int a = 0; a < 3; ++a) {
            g[a] = ((double)pts[3 * k + a] - b.grid_org[a]) / b.grid_h;
            c[a] = std::min(std::max((int)std::floor(g[a]), 0), b.walk_n[a] - 1);
        }
        std::vector<int32_t> todo{b.walk_ref[((size_t)c[2] * b.walk_n[1] + c[1]) * b.walk_n[0] + c[0]]};
        bool found = false;
        while (!todo.empty() && !found) {
            const int32_t r = todo.back();
            todo.pop_back();
            if (r == lxo::kEmptyChild) continue;
            if (r < 0) {
                const uint32_t enc = ~(uint32_t)r, first = enc >> 3, count = (enc & 7u) + 1u;
                for (uint32_t q = first; q < first + count; ++q) {
                    uint32_t id;
                    memcpy(&id, &b.tris[3ull * q + 2].y, 4);
                    found = found || id == ids[k];
                }
                continue;
            }
            const float4* f = &b.nodes[4ull * r];
            const float box[2][6] = {{f[0].x, f[0].y, f[1].x, f[1].y, f[2].x, f[2].y},
                                     {f[0].z, f[0].w, f[1].z, f[1].w, f[2].z, f[2].w}};
            int32_t child[4];
            memcpy(child, &f[3], 16);
            for (int s = 0; s < 2; ++s)
                if (g[0] >= box[s][0] && g[0] <= box[s][1] && g[1] >= box[s][2] && g[1] <= box[s][3] &&
                    g[2] >= box[s][4] && g[2] <= box[s][5])
                    todo.push_back(child[s]);
        }
        *lost += !found;
    }
    lxo::free_bvh(&b);
    return grid ? 1 : 0;
}
