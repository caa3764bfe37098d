// Launch shapes of the lattice sweep and the grids of its launches (host
// arithmetic only).
#pragma once
#include <algorithm>

namespace dilbm {

struct SweepShape {
    int warps = 4;              // rows in flight per block: 2, 4 or 8
    int blocks_per_sm = 0;      // persistent blocks per SM; 0: as many as fit
};

constexpr int SHAPE_WARPS[3] = {2, 4, 8};

inline bool shape_valid(const SweepShape &s) {
    return (s.warps == 2 || s.warps == 4 || s.warps == 8) && s.blocks_per_sm >= 0;
}

// Persistent grid: num_sms x blocks per SM (capped by the shape and by the
// kernel's occupancy), but no more blocks than the work list needs.
inline long long persistent_grid(long long items, int warps, int per_sm, int num_sms, const SweepShape &sh) {
    const int bps = sh.blocks_per_sm > 0 && sh.blocks_per_sm < per_sm ? sh.blocks_per_sm : per_sm;
    long long blocks = (long long)num_sms * bps;
    const long long need = (items + warps - 1) / warps;
    if (blocks > need) blocks = need;
    return blocks > 0 ? blocks : 1;
}

struct FusedGrid {
    long long blocks;           // all of them
    int pblocks;                // the particle blocks among them
};

// The blocks of a fused launch: sweeping blocks, and particle blocks in front
// of them, up to a tenth of the resident ones, or up to the particles' share of
// the work if that is more (a particle's update taken as two segments).  A
// particle has a warp of its
// own where a warp sweeps few segments; with more, a warp updates up to eight
// particles while the others sweep.  (us per step by particle blocks: 2048 discs
// on 4096^2 in FP32, 31 of 760 blocks 222, 47 209, 64 211, 76 212; in FP16, 31
// of 912 226, 64 200, 91 201; 1056 discs in 64 lattices, 31 230, 38 231, 47 233,
// 76 239; 512 discs on 2048^2, 22 81, 43 65.5, 64 63.2, 76 63.6; 256 discs
// there, 22 61.5, 32 58, 64 56.5.  The rule gives 64, 64, 33, 64 and 32.  Many
// discs in FP32, 76 blocks and by the rule: 84000 on 4096^2 5701 and 1400, 20000
// there 1037 and 470, 4000 on 2048^2 142 and 96, 1296 on 512^2 102 and 38.)
inline FusedGrid fused_grid(long long items, long long parts, int warps, int per_sm, int num_sms, const SweepShape &sh) {
    const long long most = persistent_grid(1LL << 40, warps, per_sm, num_sms, sh);
    const long long each = std::min(std::max(items / (4 * most * warps), 1LL), 8LL);
    const long long share = most * 2 * parts / (2 * parts + std::max(items, 1LL));
    const long long pb = std::min((parts + warps * each - 1) / (warps * each), std::max({most / 10, share, 1LL}));
    const long long sweep = persistent_grid(items, warps, per_sm, num_sms, sh);
    return FusedGrid{std::max(std::min(sweep, most - pb), 1LL) + pb, (int)pb};
}

// Has every warp of that grid's sweeping blocks at most one item?
inline bool one_item_per_warp(long long items, long long parts, int warps, int per_sm, int num_sms, const SweepShape &sh) {
    const FusedGrid g = fused_grid(items, parts, warps, per_sm, num_sms, sh);
    return (g.blocks - g.pblocks) * warps >= items;
}

}  // namespace dilbm
