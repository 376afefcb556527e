// Host: which of its kernels a round takes.
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

// Which kernels a round takes.
//   kWarpTiles   one kernel, a warp takes a tile through the workers
//   kCtaTiles    one kernel, a CTA takes a tile through the workers, four at a time (not for buckets of 4096)
//   kTwoKernels  codes, then the average from the words
enum RoundRoute { kWarpTiles, kCtaTiles, kTwoKernels };

// A CTA's four warps are through with a tile in a quarter of a warp's time, so with few tiles the round is as much shorter;
// with many, the barriers and the eight elements that a thread goes through at a time (a warp's lane: 32) cost more than the
// unused part of a last turn.  The line lies at 1.2 tiles a warp of the chip (0.6 for the teams of buckets of 2048, 0.25 with one
// worker), and beyond it wherever one pass by warps would lose to two kernels (teams: nowhere).  On 1183 triples of times on one
// B200 (buckets of 32, 96, 480, 512, 2048 and whole tensors, b = 4 to 8, M = 1 to 32, 3k to 13M elements, the rule attached) the
// fastest of the three is missed by 0.3 % on average and 15 % at worst; with a line of 0.6 by 0.7 %, of 2.2 by 0.7 %.  Some of them, by warps /
// two kernels / by CTAs (us), bucket 512, b = 4: 16k M = 4 10 / 12 / 6; 16k M = 16 27 / 13 / 11; 16k M = 32 49 / 15 /
// 17; 456k M = 4 11 / 13 / 7; 456k M = 16 28 / 20 / 14; 797k M = 4 11 / 14 / 9; 797k M = 8 18 / 18 / 13; 1.4M M = 4 13 /
// 17 / 11; 1.4M M = 16 36 / 32 / 30; 2.4M M = 16 54 / 48 / 42; 7.4M M = 8 57 / 71 / 64; bucket 2048, b = 5: 16k M = 4 11
// / 12 / 8; 16k M = 16 30 / 16 / 20; 456k M = 8 17 / 18 / 14; 1.4M M = 8 23 / 29 / 21; bucket 96, b = 4: 16k M = 4 15 /
// 15 / 7; 456k M = 8 24 / 19 / 12; 4.3M M = 8 60 / 66 / 58; whole tensors: 16k M = 4 13 / 16 / 10; 456k M = 8 20 / 21 /
// 14; 2.4M M = 8 47 / 47 / 44.
//
// Only where a few tiles have a great many workers does the CTA, which takes them in turn after all, lose to
// two kernels that spread them over the chip and slow down with the number of tiles first.
inline RoundRoute dq_round_route(const RouteQuery& q, const bool cta_tiles, const bool pairs)
{
    const bool one = dq_one_pass(q);
    const double m = (double)q.M, tiles = (double)q.positions;
    const double line = q.M == 1 ? 0.25 : (pairs ? 0.6 : 1.2);
    if (!cta_tiles) return one ? kWarpTiles : kTwoKernels;
    if (tiles > line * (double)q.units && (one || pairs)) return kWarpTiles;
    // what two kernels save per worker, and what they cost besides
    const double per_worker = pairs ? 0.5 : (q.odd_buckets > 0 ? 0.32 : 0.24), besides = pairs ? 5.5 : (q.odd_buckets > 0 ? 6.9 : 6.2);
    return per_worker * m - besides > 0.0005 * tiles * m ? kTwoKernels : kCtaTiles;
}

// What a CTA has a form for: given norms, and buckets of up to 1024 elements or of 2048, which are a pair of its warps'.
inline bool dq_cta_form(int32_t groups_per_bucket, bool given) { return given || groups_per_bucket <= 64; }

// The route of a call: tile positions of a worker, warps of a launch by warps, and the layout's bucket (32-element groups; where
// the norms are not given a power of two or less than 32).  lose_first: the test hook of the waits is set; a round by CTAs has no
// wait to lose, so the call takes the kernels that have.
inline RoundRoute dq_route_of(int64_t positions, int64_t warps, int32_t groups_per_bucket, int32_t M, bool given, bool lose_first)
{
    const bool teams = !given && groups_per_bucket > 32;
    RouteQuery q = {};
    q.positions = positions;
    q.units = teams ? warps / (groups_per_bucket / 32) : warps;
    q.M = M;
    q.given = given ? 1 : 0;
    q.odd_buckets = !given && (groups_per_bucket & (groups_per_bucket - 1)) != 0 ? 32 / groups_per_bucket : 0;
    return dq_round_route(q, dq_cta_form(groups_per_bucket, given) && !lose_first, teams);
}
