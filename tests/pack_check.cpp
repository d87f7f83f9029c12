// Packs random trees of finest-cell leaves and compares, for cells in and around
// the leaves, the octree descent through the packed nodes, the brick index and
// the uploaded cells.  Prints the number of differences.  Arguments: depth,
// max_depth, seed.
#include <algorithm>
#include <array>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>

#include "fpo_internal.h"

using namespace fpo;
using Cell = std::array<uint32_t, 3>;

int main(int argc, char **argv)
{
    if (argc < 4) return 2;
    const int D = std::atoi(argv[1]), M = std::atoi(argv[2]);
    std::mt19937 rng((unsigned)std::atoi(argv[3]));
    const uint32_t G = 1u << D;
    std::map<Cell, uint32_t> id;
    std::vector<Cell> cells;
    for (int b = 0; b < 40; ++b) {
        const uint32_t s = 1u << (rng() % 4), x = (uint32_t)(rng() % G), y = (uint32_t)(rng() % G), z = (uint32_t)(rng() % G);
        for (uint32_t k = 0; k < s * s * s; ++k) {
            const Cell c = {x + k % s, y + k / s % s, z + k / s / s};
            if (c[0] < G && c[1] < G && c[2] < G && rng() % 5 && id.emplace(c, 0u).second) cells.push_back(c);
        }
    }
    std::vector<uint8_t> depth(cells.size(), (uint8_t)D);
    std::vector<uint32_t> xyz;
    for (uint32_t j = 0; j < cells.size(); ++j) {  // (the order of generation, not Morton order)
        id[cells[j]] = j;
        xyz.insert(xyz.end(), cells[j].begin(), cells[j].end());
    }
    std::vector<float> coeffs(cells.size());
    fpo_tree_desc t{};
    t.n_leaves = (uint32_t)cells.size();
    t.max_depth = (uint32_t)M;
    t.leaf_depth = depth.data();
    t.leaf_xyz = xyz.data();
    t.coeffs = coeffs.data();
    t.aabb_size = 1.0;
    PackedTree p;
    std::string err;
    if (validate_and_pack(&t, 1, 1, &p, &err) != FPO_OK) return 3;
    if (p.top.empty()) return 4;
    const uint32_t T = G / 16;
    int bad = 0;
    for (int q = 0; q < 100000; ++q) {
        Cell c = cells[rng() % cells.size()];
        for (uint32_t &x : c) x = q % 3 == 0 ? (uint32_t)(rng() % G) : std::min(G - 1, x + (q % 3 == 1 ? (uint32_t)(rng() % 3) : 0u));
        uint32_t leaf = ~0u, node = 0;
        int lvl = 0;
        for (;;) {
            const int sh = D - 1 - lvl++;
            const uint32_t s = p.nodes[node * 8 + (((c[0] >> sh) & 1u) | (((c[1] >> sh) & 1u) << 1) | (((c[2] >> sh) & 1u) << 2))];
            if (s == 0) break;
            if (s & LEAF_BIT) { leaf = s & ~LEAF_BIT; break; }
            node = s;
        }
        const auto it = id.find(c);
        bad += (it != id.end()) != (leaf != ~0u) || (leaf != ~0u && p.perm[leaf] != it->second);
        // the brick index, as locate_brick reads it
        const uint32_t *k = &p.top[4 * ((size_t)((c[2] >> 4) * T + (c[1] >> 4)) * T + (c[0] >> 4))];
        const uint32_t j = ((c[0] >> 2) & 3u) | (c[1] & 12u) | ((c[2] & 12u) << 2), wj = k[j >> 5], bj = j & 31u;
        uint32_t found = ~0u;
        int csz;
        if (!((wj >> bj) & 1u)) {
            csz = (k[0] | k[1]) == 0 ? (int)k[3] : (((wj >> (bj & 10u)) & 0x330033u) ? 4 : 8);
        } else {
            const uint32_t n = k[2] + __builtin_popcount(wj & ((1u << bj) - 1u)) + (j & 32u ? __builtin_popcount(k[0]) : 0);
            const uint32_t *br = &p.bricks[4 * (size_t)n];
            const uint32_t i = (c[0] & 3u) | ((c[1] & 3u) << 2) | ((c[2] & 3u) << 4), wi = br[i >> 5], bi = i & 31u;
            if ((wi >> bi) & 1u) {
                found = br[2] + __builtin_popcount(wi & ((1u << bi) - 1u)) + (i & 32u ? __builtin_popcount(br[0]) : 0);
                csz = 1;
            } else {
                csz = ((wi >> (bi & 10u)) & 0x330033u) ? 1 : 2;
            }
        }
        bad += found != leaf || csz != 1 << (D - lvl);
    }
    std::printf("%d\n", bad);
    return 0;
}
