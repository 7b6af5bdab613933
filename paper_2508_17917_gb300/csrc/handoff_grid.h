// handoff_grid.h -- which build of the two-node hand-off kernel a mesh takes,
// and its grid (host only, no CUDA).
#pragma once

namespace dg {

struct HandoffGrid {
    int minb;        // the build: its __launch_bounds__ minimum of blocks per SM, 4 or 5
    int per_sm;      // its resident blocks per SM, at least minb
    int grid;
};

// The build for at least four blocks per SM has 128 registers, the one for
// five 96 and a few spills; occ4 and occ5 are their resident blocks per SM
// (occ5 = 0: not built).  As many blocks as are resident at once (a step's
// first stage and fused steps have grid barriers), capped by the tiles.  A
// wave of m blocks per SM takes about m units of time, so the build with the
// smaller m x waves is taken, the first if they are equal.  Measured, us a
// stage with five and with four, waves: p = 5, 60^2 quads 0.9 and 1.1: 20.5
// and 24.9; 76^2 1.4 and 1.7: 32.5 and 28.4; 90^2 1.9 and 2.4: 34.4 and 38.7;
// 100^2 2.4 and 3.0: 46.2 and 39.7; p = 3, 128^2 1.8 and 2.2: 29.8 and 32.3;
// 256^2 7.2 and 9.0: 98.6 and 95.2; p = 1, 256^2 2.7 and 3.4: 36.9 and 39.3.
// At p = 6 five spill more and are behind even in one wave against two (56^2:
// 25.9 and 24.5): not built.
inline HandoffGrid handoff_grid(int sms, int occ4, int occ5, long long tiles)
{
    auto cost = [&](int occ) {
        const long long wave = static_cast<long long>(sms) * occ;
        return occ * ((tiles + wave - 1) / wave);
    };
    HandoffGrid h{4, occ4, 0};
    if (occ5 > 0 && cost(occ5) < cost(occ4)) h = {5, occ5, 0};
    const long long wave = static_cast<long long>(sms) * h.per_sm;
    h.grid = static_cast<int>(tiles < wave ? tiles : wave);
    return h;
}

}  // namespace dg
