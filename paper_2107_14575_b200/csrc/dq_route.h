// Host: whether a round is one kernel or two.
#pragma once

#include <stdint.h>

// What the choice looks at: tile positions of a worker, warps (or teams) of a launch, workers, whether the norms are
// given, and for odd buckets how many of them a tile holds (0 for the others).
struct RouteQuery {
    int64_t positions, units;
    int32_t M, given, odd_buckets;
};

// One pass for codes and average, or codes (all workers' tiles side by side) and then the average from
// the words?  In one pass a warp takes a position through all M workers, one after the other: P positions
// on U warps are `full` turns of M tiles and a last turn in which only a fraction f of the warps has work.
// Two kernels spread the M * P tiles evenly, but cost a launch and read the words back.  So the last turn decides: per
// worker, one pass pays for an almost empty turn (1.7 us; 1.2 with given norms; more where a tile's odd buckets are reduced
// one by one), gets back what the two kernels spend on its share f and on the full turns, and two kernels pay 7.3 us (8.65
// with odd buckets) for the second launch.  Fitted to 1000 pairs of times on one B200 (b = 2, 3, 4, 5, 8; buckets of 32 * 2^k, 96, 160, 224,
// 480, 992 and whole tensors; M = 2 to 32; 3k to 10M elements), on which the faster side is missed by 0.5 % on average
// (1.4 % with one line for all buckets, fitted at b = 5 and buckets of 512).  Some of them, b = 4, one pass / two kernels
// (us): bucket 512, 20k elements M = 4 10.9 / 11.9, M = 32 58 / 15; 600k M = 4 10.6 / 12.8, M = 8 17.3 / 15.1, M = 32 58 /
// 30; 1.5M M = 32 73 / 56; 3M M = 8 31.5 / 34.4, M = 32 109 / 102; 4.2M M = 32 129 / 136; 10M M = 32 263 / 308; bucket 2048,
// 600k M = 4 12.2 / 13.8, M = 8 19.9 / 16.9; 5.2M M = 32 179 / 189; bucket 480, 600k M = 8 25.7 / 18.7; 1.5M M = 4 13.7 / 19.9;
// 3M M = 8 45 / 41; 8M M = 8 85 / 94; bucket 96, 20k M = 4 19.4 / 16.1; 600k M = 8 32 / 21; 3M M = 8 62 / 49; 1.5M M = 4 21.6 / 24.8;
// whole tensors, 600k M = 32 53 / 42; 3M M = 8 42 / 49.
inline bool dq_one_pass(const RouteQuery& q)
{
    const int64_t full = q.positions / q.units;
    const double f = (double)(q.positions - full * q.units) / (double)q.units;
    if (q.M == 1 || f == 0.0) return true;                       // no worker to wait for, or no idle warp
    double empty = 1.7, share = 1.3, turn = 0.7, launch = 7.3;
    if (q.given) {
        empty = 1.2; share = 1.7; launch = 7.5;
    } else if (q.odd_buckets > 0) {
        const double r = (double)q.odd_buckets;
        empty = 1.83 + 0.17 * r; share = 1.82 + 0.06 * r; turn = 0.52 - 0.03 * r; launch = 8.65;
    }
    return (double)q.M * (empty - share * f - turn * (double)full) <= launch;
}
