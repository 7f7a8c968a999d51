// Host side of the convolution layer's launches that needs no CUDA: how many CTAs share a tile.
#pragma once

namespace wici {

// SMs of a device, and its resident clusters of 1, 2, 4 and 8 CTAs (0: none fits).
struct ConvDevice {
    int sms = 0, clusters[4] = {};
};

// How a layer's `tiles` of 128 x 256 outputs with `nkb` reduction blocks (the longest tile's)
// run: on pairs of CTAs (0), one CTA a tile (1), or 2, 4 or 8 CTAs sharing one.  Modelled
// SM cycles: waves of tiles x (blocks of a CTA x 512 cycles of MMAs + the pipeline's fill
// and the epilogue, and the exchange of a split tile).  A single CTA takes about 640
// cycles a block (its ports serve all of B), a pair 540.
inline int pick_ctas(const ConvDevice &d, int tiles, int pair_tiles, int nkb) {
    auto cost = [](int units, int slots, double blocks, double cycles, double fixed) {
        return (double)((units + slots - 1) / slots) * (blocks * cycles + fixed);
    };
    int best = 1;
    double best_cost = 0.0;
    auto consider = [&](int ctas, double c) {
        if (best_cost == 0.0 || c < best_cost) {
            best = ctas;
            best_cost = c;
        }
    };
    // a device may have no resident cluster of some size
    if (d.clusters[1] > 0) consider(0, cost(pair_tiles, d.clusters[1], nkb, 540.0, 5000.0));
    for (int i = 0; i < 4; ++i) {
        const int split = 1 << i;
        if (d.clusters[i] > 0)
            consider(split, cost(tiles, d.clusters[i], (nkb + split - 1) / split, 640.0, i == 0 ? 4000.0 : 7000.0));
    }
    return best;
}

}  // namespace wici
