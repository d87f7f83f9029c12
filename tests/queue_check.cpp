// The fused mode's ray queue over camera frames of every shape: prints the
// number of random pixels that not exactly one slot stands for, and of slots
// past the last ray that claim a pixel.  Arguments: width, height.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "fpo_internal.h"

using namespace fpo;

int main(int argc, char **argv)
{
    if (argc < 3) return 2;
    const uint64_t W = std::strtoull(argv[1], nullptr, 10), H = std::strtoull(argv[2], nullptr, 10);
    TraverseParams p{};
    p.fr.mode = FPO_RAYS_CAMERA;
    p.fr.width = (uint32_t)W;
    p.fr.height = p.fr.rows = (uint32_t)H;
    p.fr.n_rays = (uint32_t)(W * H);
    p.tiles_x = (uint32_t)((W + TILE_W - 1) / TILE_W);
    const uint64_t tx = p.tiles_x;
    p.n_tiles = (uint32_t)(tx * ((H + TILE_H - 1) / TILE_H));
    fused_queue(p);
    const uint64_t slots = (uint64_t)p.n_tiles * 32;
    int bad = slots > (1ull << 31);  // (room for what the warps count past the end)
    std::mt19937_64 rng(1);
    uint32_t ray;
    int px, py;
    for (int q = 0; q < 200000; ++q) {
        const uint64_t i = q == 0 ? 0 : (q == 1 ? W * H - 1 : rng() % (W * H)), x = i % W, y = i / W;
        int found = 0;
        for (const uint64_t s : {i, (y / TILE_H * tx + x / TILE_W) * 32 + y % TILE_H * TILE_W + x % TILE_W}) {
            if (s >= slots || (found && s == i)) continue;
            if (slot_ray(p, (uint32_t)s, ray, px, py) && ray == i && (uint64_t)px == x && (uint64_t)py == y) ++found;
            if (s == i && i == (y / TILE_H * tx + x / TILE_W) * 32 + y % TILE_H * TILE_W + x % TILE_W) break;
        }
        bad += found != 1;
        const uint64_t s = slots - 1 - rng() % (slots < 4096 ? slots : 4096);  // about the end of the queue
        if (slot_ray(p, (uint32_t)s, ray, px, py)) bad += (uint64_t)px >= W || (uint64_t)py >= H || ray != (uint64_t)py * W + px;
    }
    std::printf("%d\n", bad);
    return 0;
}
