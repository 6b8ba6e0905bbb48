// lb_shape.h -- group size and pipeline depth of the stream-collide kernel
// (lb.cu): a function of the boxes and of what the caller asked for alone, so
// that the order of the option calls does not matter and nothing that a former
// shape cut short stays cut.  Plain C++.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace iblb {

constexpr int LB_THREADS = 256;                        // consumer threads per block (FP32 storage)
constexpr int LB_CONST_BYTES = 128;                    // a droplet's constants (LbConst)
// Dynamic shared memory of a block: the opt-in maximum of sm_100 and later
// (227 KB) less the kernel's barriers; what a shape may use of it; an SM's.
constexpr int64_t LB_SMEM_LAUNCH = 227 * 1024 - 128;
constexpr int64_t LB_SMEM_SHAPE = 227 * 1024 - 1024;
constexpr int64_t LB_SMEM_SM = 228 * 1024, LB_SMEM_BLOCK = 1024 + 128;   // reserved and static per block

// a droplet's box: mask_pitch bytes per row of inside bits (0: one viscosity)
struct LbBox {
    int nx, ny, nzf, mask_pitch;
};
// what the options ask for: cells per group (-1 not set, 0 the multiplier),
// the multiplier, stages (0 not set)
struct LbRequest {
    int cells = -1, mult = 1, stages = 0;
};
struct LbShape {
    int cells, mult, stages;     // cells 0: the multiplier
    int stage_bytes;
};

// elements per row: nx, rounded up so that rows are multiples of 16 bytes
inline int lb_pitch(int nx, int sb) { return (nx + 16 / sb - 1) / (16 / sb) * (16 / sb); }

// bytes of one stage: 19 population rows and 3 force rows per cell row, its
// inside bits with two viscosities, the group's header and with several
// droplets its droplet's constants (a multiple of 128 bytes; of 16, where two
// stages of such multiples do not fit a block)
inline int lb_stage_bytes(int rows, int pitch, int sb, bool several, int mask_pitch)
{
    const int64_t b = (int64_t)rows * (19 * pitch * sb + 3 * pitch * 4 + mask_pitch) + 16 + (several ? LB_CONST_BYTES : 0);
    const int64_t r = (b + 127) & ~(int64_t)127;
    return (int)(2 * r > LB_SMEM_LAUNCH ? b : r);
}

// rows per group for about `cells` cells (0: mult times 256 threads' rows), at
// most ny, in as many groups a plane, their rows as even as they go: a short
// last group would fall to the same blocks in every round
inline int lb_even_rows(int rows, int ny)
{
    const int gpp = (ny - 1) / rows + 1;
    return (ny - 1) / gpp + 1;
}
inline int lb_asked_rows(int cells, int mult, const LbBox &b)
{
    const int rows = cells > 0 ? (cells + b.nx / 2) / b.nx : mult * (LB_THREADS / b.nx);
    return std::min(b.ny, std::max(cells > 0 ? 1 : mult, rows));
}
// the same, and two stages of the group fit a block's shared memory
inline int lb_group_rows(int cells, int mult, const LbBox &b, int sb, bool several)
{
    int rows = lb_asked_rows(cells, mult, b);
    while (rows > 1 && 2 * (int64_t)lb_stage_bytes(rows, lb_pitch(b.nx, sb), sb, several, b.mask_pitch) > LB_SMEM_SHAPE)
        --rows;
    return lb_even_rows(rows, b.ny);
}
// Where two stages of one row fit without the inside bits only, the kernel
// reads them from global memory.
inline bool lb_mask_staged(int rows, const LbBox &b, int sb, bool several)
{
    return b.mask_pitch &&
           2 * (int64_t)lb_stage_bytes(rows, lb_pitch(b.nx, sb), sb, several, b.mask_pitch) <= LB_SMEM_LAUNCH;
}

// The shape for these boxes on sms SMs.  What was not asked for is chosen: the
// pair with the least estimated time over the persistent blocks.
// A group costs its cells plus a fixed part worth LB_GROUP_CELLS cells (its
// hand-over and the latency of one pass; 128^3 in FP16, one block's time per
// group at 256 .. 1024 cells), and half of an uneven last round is idle (the
// blocks that still run get the others' bandwidth).  Two blocks an SM, as
// registers allow, need their stages to fit half its shared memory; two
// stages instead of three make larger groups fit, which pays when a block
// has only a group or two.  Measured in the step (stream-collide, us, against
// 768 cells, three stages and a short last group a plane): 32^3 FP32 6.1 ->
// 4.6, 80^2 x 60 FP32 13.6 -> 9.8, 61 x 53 x 47 FP32 9.2 -> 7.3, 64 boxes of
// 48 to 96 in FP16 491 -> 416, 32 boxes with tau_in != tau_out 232 -> 171.
// The factors below are fitted, not derived.  The chosen shape against the best
// of 64 .. 1024 cells with two and three stages (a step without membranes, us):
// 32^3 FP32 3.88 / 3.88, 61 x 53 x 47 FP32 5.78 / 5.78, 80^2 x 60 FP32 7.95 /
// 7.95, 128^3 FP16 28.0 / 27.5, 256^2 x 128 BF16 101.1 / 101.0, 64 boxes FP16
// 301.7 / 301.7; but 8 boxes FP32 58.3 / 54.9, 128^3 FP32 54.8 / 50.0, 256^2 x
// 128 FP32 210 / 188: there two blocks an SM with groups of 256 cells, or one
// with twice that, are better than the larger groups that the 0.5 favours.
// One block an SM against two of the same group (us): 128^3 FP16 896 cells 32.4
// (three stages, one) / 29.5 (two stages, two), 80^2 x 60 FP32 512 cells 11.9 /
// 9.3; three stages against two, two blocks each: 128^3 FP16 640 cells 28.0 /
// 32.3, 64 boxes 640 cells 301.9 / 336.0, below two rounds no difference.
constexpr int LB_GROUP_CELLS = 160;
inline LbShape lb_shape(const std::vector<LbBox> &boxes, int sb, int sms, const LbRequest &ask)
{
    const bool several = boxes.size() > 1, any_cells = ask.cells < 0, any_stages = ask.stages == 0;
    // rows too long for two full stages: single rows, as many stages as fit
    LbShape s{any_cells ? 32 : ask.cells, ask.mult, any_stages ? 3 : ask.stages, 0};
    double best = 1e300;
    for (int ns = any_stages ? 2 : ask.stages; ns <= (any_stages ? 3 : ask.stages) && (any_cells || any_stages); ++ns)
        for (int cells = any_cells ? 32 : ask.cells; cells <= (any_cells ? 1024 : ask.cells); cells += 32) {
            int64_t stage = 0, groups = 0;
            double work = 0.0, largest = 0.0;
            for (const LbBox &b : boxes) {
                const int P = lb_pitch(b.nx, sb), rows = any_cells
                                                             ? lb_even_rows(lb_asked_rows(cells, ask.mult, b), b.ny)
                                                             : lb_group_rows(cells, ask.mult, b, sb, several);
                const int gpp = (b.ny - 1) / rows + 1;
                stage = std::max(stage, (int64_t)lb_stage_bytes(rows, P, sb, several, b.mask_pitch));
                groups += (int64_t)gpp * b.nzf;
                work += (double)b.nzf * ((double)gpp * LB_GROUP_CELLS + (double)b.ny * P);
                largest = std::max(largest, (double)rows * P + LB_GROUP_CELLS);
            }
            const int64_t fit = (LB_SMEM_SM / 2 >= ns * stage + LB_SMEM_BLOCK) ? 2 : 1;
            if (ns * stage > LB_SMEM_SHAPE)
                continue;
            const double blocks = (double)sms * fit, rounds = groups / blocks;
            double cost = work / blocks + 0.5 * (std::ceil(rounds) - rounds) * largest;
            if (groups <= blocks)
                cost = largest;
            // one block an SM has half the warps: slower, except where FP32's
            // traffic leaves them idle and there are rounds enough to fill in
            if (fit == 1)
                cost *= sb == 4 && rounds > 3.0 ? 0.5 : 0.6;
            if (ns == 2 && rounds > 2.0)
                cost *= 1.1;
            if (cost < best) {
                best = cost;
                s.cells = cells;
                s.stages = ns;
            }
        }
    for (const LbBox &b : boxes) {
        const int rows = lb_group_rows(s.cells, s.mult, b, sb, several);
        s.stage_bytes = std::max(s.stage_bytes,
                                 lb_stage_bytes(rows, lb_pitch(b.nx, sb), sb, several,
                                                lb_mask_staged(rows, b, sb, several) ? b.mask_pitch : 0));
    }
    // as many of the stages as fit
    while (s.stages > 2 && (int64_t)s.stages * s.stage_bytes > LB_SMEM_SHAPE)
        --s.stages;
    return s;
}

}  // namespace iblb
