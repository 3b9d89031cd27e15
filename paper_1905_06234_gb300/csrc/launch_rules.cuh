// Host-side rules that shape a tensor-core launch (plain C++: no CUDA in here).
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace life {

// Shares the tiles out to the CTAs of a launch (at most one per SM), as units of one
// brick's consecutive tiles; each unit pays for its brick's fascicle table (gathered
// by the DSC, flushed by the WC).  Three ways:
//  - whole bricks, largest first, dealt to the CTAs in snake order: at the paper's size
//    (6 bricks a CTA) the CTAs' times are within 3 % of one another;
//  - the tiles in brick order, cut into one run per CTA of about equal cost, wherever
//    in a brick the cut falls, at the price of the cut bricks' tables twice.  Whole
//    bricks leave most SMs without any on the 16^3 workload (8 bricks of 4 tiles: a
//    DSC took 47 us, 25 with the tiles dealt out) and give the CTAs of the 64^3 one
//    three or four (512 bricks on 152 SMs: 142 -> 130 us);
//  - in a batch, whose problems stop at different times, so that a CTA's work has to be
//    of all of them: single tiles dealt out, each with its brick's table.
// The one whose most loaded CTA has less to do is taken (whole bricks unless the other
// is better by 5 %).  The costs, in units of an entry's time, are those of the BF16
// kernels' phases on the 64^3 and the paper workload: a tile 7 us, a table slot 0.8 ns,
// a unit 2 us, an entry 0.14 ns.  Single tiles in a batch take 8 % longer than these say
// in BF16, and 10 to 15 % less with FP32 storage, whose tiles cost more beside a table;
// hence the lines of 0.9 and 1.1 there.  Batches of equal problems, four iterations,
// whole bricks / single tiles on 152 SMs, with what the costs say: BF16 8 bricks 499 /
// 320 us (0.3), 64 of dense tiles 1015 / 805 (0.8), 108 554 / 572 (0.92), 125 529 / 634
// (1.2), of dense tiles 1137 / 1439 (1.4), 250 932 / 1050 (1.1), 324 1412 / 1427 (0.93);
// FP32 storage 862 / 517, 1514 / 1141, 921 / 849, 884 / 946, 1612 / 1878, 1453 / 1437,
// 2139 / 1896.
struct WorkShare {
    std::vector<int32_t> brick, t0, t1, cta_unit{0};
    double worst = 0.0;
    int grid() const { return (int)cta_unit.size() - 1; }
};

inline WorkShare share_out(const std::vector<int32_t>& order, const std::vector<int32_t>& btile,
                           const std::vector<int32_t>& base, const std::vector<int32_t>& bfasc, int num_sms,
                           bool batch, bool fp32) {
    constexpr double TILE_COST = 50000.0, UNIT_COST = 14000.0, SLOT_COST = 6.0;
    const int nb = (int)btile.size() - 1, nt = btile[nb], sms = std::max(num_sms, 1);
    auto unit_cost = [&](int b) { return UNIT_COST + SLOT_COST * (bfasc[b + 1] - bfasc[b]); };
    auto tile_cost = [&](int t) { return TILE_COST + (base[t + 1] - base[t]); };
    auto add = [](WorkShare& W, int b, int t0, int t1) {
        W.brick.push_back(b);
        W.t0.push_back(t0);
        W.t1.push_back(t1);
    };
    auto close_cta = [](WorkShare& W, double cost) {
        W.cta_unit.push_back((int32_t)W.brick.size());
        W.worst = std::max(W.worst, cost);
    };
    WorkShare deal, other;
    const int dgrid = std::min(sms, nb), grid = std::min(sms, nt);
    for (int c = 0; c < dgrid; ++c) {
        double cost = 0.0;
        for (int r = 0;; ++r) {
            const int k = r * dgrid + ((r & 1) ? (dgrid - 1 - c) : c);
            if (k >= nb) break;
            const int b = order[k];
            add(deal, b, btile[b], btile[b + 1]);
            cost += unit_cost(b);
            for (int t = btile[b]; t < btile[b + 1]; ++t) cost += tile_cost(t);
        }
        close_cta(deal, cost);
    }
    if (batch) {
        std::vector<int32_t> tbrick(nt);
        for (int b = 0; b < nb; ++b)
            for (int t = btile[b]; t < btile[b + 1]; ++t) tbrick[t] = b;
        for (int c = 0; c < grid; ++c) {
            double cost = 0.0;
            for (int t = c; t < nt; t += grid) {
                add(other, tbrick[t], t, t + 1);
                cost += unit_cost(tbrick[t]) + tile_cost(t);
            }
            close_cta(other, cost);
        }
    } else {
        double left = 0.0;
        for (int b = 0; b < nb; ++b) left += unit_cost(b);
        for (int t = 0; t < nt; ++t) left += tile_cost(t);
        for (int c = 0, b = 0, t = 0; c < grid; ++c) {
            const double want = left / (grid - c);
            double cost = 0.0;
            const int more = grid - 1 - c;  // each CTA after this one takes a tile at least
            while (t < nt - more) {
                const bool opens = cost == 0.0 || t == btile[b];
                const double x = tile_cost(t) + (opens ? unit_cost(b) : 0.0);
                if (more > 0 && cost > 0.0 && cost + 0.5 * x > want) break;
                if (opens) add(other, b, t, t);
                other.t1.back() = ++t;
                cost += x;
                if (t == btile[b + 1]) ++b;
            }
            left -= cost;
            if (t < nt && t != btile[b]) left += unit_cost(b);  // a cut brick's table is paid for again
            close_cta(other, cost);
        }
    }
    const double line = !batch ? 0.95 : fp32 && nt >= 2 * nb ? 1.1 : 0.9;  // (bricks of one tile are dealt alike)
    return other.worst < line * deal.worst ? other : deal;
}

// Form of a BF16 DSC launch.  y_tile: b and Y pass through a tile in shared memory (where
// it fits beside the brick table and two S stages, and rows are 16-byte aligned: can);
// stages: S stages.  The lines, from DSC calls timed in each form (us, one GB300; entries
// per tile and 128-atom chunk):
//  - The tile of Y spares the epilogue its reads of b, a few at a time (64^3 voxels, Nθ 96,
//    Na 360: 339 entries 128 -> 106, 3812 177 -> 146).  A tile of one chunk is over before
//    its b has arrived (Nθ 64, Na 128: 1005 81 -> 87, 7536 106 -> 109, 16351 132 -> 123,
//    22635 160 -> 140): it takes the tile of Y from 16384 entries on.  Bricks of one tile
//    gather a table for every tile, and the copies come on top of that (4^3 bricks, 48^3
//    voxels: 1270 112 -> 104, 2752 126 -> 129, 4978 147 -> 167): up to 2304 entries.
//  - A third and fourth stage let idle producers start on the next chunks: worth it where
//    a chunk's 256-entry blocks are for at most half of the 23 producer warps and a tile has
//    more than two chunks (64^3, Nθ 32, Na 512: 255 105 -> 81, 2864 137 -> 135, 7481 208 ->
//    226; Nθ 64, Na 360: 339 99 -> 97, 3812 130 -> 134, 5510 150 -> 158; Na 181: 1893 83 ->
//    89, 7422 120 -> 155).
constexpr int DSTAGE = 2;      // S stages of the general form, and the
constexpr int DSTAGE_MAX = 4;  // most the form with the tile of Y takes

struct DscForm {
    bool y_tile = false;
    int stages = DSTAGE;
};

template <class Fits>  // fits(stages): the form with the tile of Y and so many stages fits shared memory
inline DscForm dsc_form(int64_t n_nnz, int64_t n_tiles, int64_t n_bricks, int n_c, bool can, Fits fits) {
    DscForm F;
    const int64_t chunks = n_tiles * n_c;
    const bool pays = n_c == 1 ? n_nnz >= 16384 * chunks : n_tiles >= 2 * n_bricks || n_nnz <= 2304 * chunks;
    F.y_tile = can && pays && fits(DSTAGE);
    if (F.y_tile && n_c > 2 && n_nnz <= 23 * 256 / 2 * chunks)
        while (F.stages < DSTAGE_MAX && fits(F.stages + 1)) ++F.stages;
    return F;
}

}  // namespace life
