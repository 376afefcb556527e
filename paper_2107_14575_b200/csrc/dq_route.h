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

// Whether one kernel goes by warps.  A CTA's four warps are through with a tile in a quarter of a warp's time, so with few tiles
// the round is as much shorter; with many, the barriers and the eight elements that a thread goes through at a time (a warp's
// lane: 32) cost more than the unused part of a last turn.  x: tiles a warp (team) of the chip; by warps a turn is an x of 1,
// by CTAs one of 0.31 (teams 0.63).  By warps / by CTAs (us), at x:
//   one worker, three of a CTA's warps without a norm to take: above 0.25.  Bucket 512, b = 4 0.19 6.0 / 5.8, 0.33 7.1 / 7.2.
//   two workers and odd buckets, reduced one by one by half of the warps: above 0.3, but for the start of a second turn.  96, b = 4
//     0.20 10.1 / 7.8, 0.35 10.4 / 10.5, 0.64 11.6 / 13.0, 0.90 13.0 / 14.8, 1.07 18.0 / 17.1; 480 0.27 8.9 / 7.7, 0.64 10.0 /
//     11.1, 0.90 (l-infinity) 11.4 / 13.0, 1.07 14.8 / 14.1.
//   teams: above 0.6, and only the start of a second turn, 1.0 to 1.25, to the CTAs where one pass loses to two kernels.  2048,
//     b = 5, M = 16 0.60 39.3 / 35.8, 0.74 40.4 / 47.7, 1.01 59.7 / 55.6, 1.16 62.3 / 62.7, 1.26 60.3 / 69.3; M = 32 1.01 112 / 104;
//     b = 8 118 / 99; M = 3 1.01 16.8 / 17.7.
//   the others: above 1.2, and the end of the first turn, 0.85 to 1.0, except where a warp's l-infinity norms leave it the
//     slower way there (512, b = 8, M = 8 0.93 26.5 / 24.4) or its tile is one odd bucket (992, b = 8, M = 12 0.87 38.2 / 35.3).  512, b = 4, M = 8 0.74 21.4 / 20.8, 1.00 30.7 / 25.5, 1.15 31.6 /
//     29.5, 1.44 33.2 / 33.7; 1024, b = 6, M = 6 0.93 20.3 / 22.4; 128, b = 3, M = 3 0.93 13.9 / 15.0; 480, b = 6, l-infinity, M = 6
//     0.79 22.2 / 23.3, 0.90 22.8 / 25.2, 1.07 31.1 / 28.2; whole tensors, b = 4, M = 12 0.93 53.3 / 55.4, M = 8 1.00 46.5 / 43.4.
inline bool dq_by_warps(const RouteQuery& q, const bool one, const bool pairs, const bool linf)
{
    const double x = (double)q.positions / (double)q.units;
    if (q.M == 1) return x > 0.25;
    if (pairs) return x > 0.6 && (one || x <= 1.0 || x > 1.25);
    if (!one) return false;
    if (x > 1.0) return x > 1.2;
    if (q.odd_buckets > 0) return q.M == 2 ? x > 0.3 : q.odd_buckets > 1 && x > 0.85;
    return !linf && x > 0.85;
}

// Only where a few tiles have a great many workers does the CTA, which takes them in turn after all, lose to
// two kernels that spread them over the chip and slow down with the number of tiles first.  By CTAs / two kernels (us): 512, b = 4, 16k
// M = 16 11 / 13, M = 32 17 / 15; 2048, b = 5, 16k M = 16 19.6 / 15.5; 992, b = 8, 85k M = 24 15.1 / 16.8.
//
// All lines are fitted to 4760 quadruples of times on one B200 (three routes, and the kernels as they were before there was one by CTAs;
// buckets of 32, 96, 128, 160, 480, 512, 992, 1024, 2048 and whole tensors, 4096 beside them, b = 3 to 8, l2 and l-infinity,
// M = 1 to 32, 3k to 13M elements, the rule attached): the fastest of the three is missed by 0.6 % on average and 25 % at worst
// (l-infinity, one worker, 7 us); what dq_one_pass alone would take by more than 3 % at one point in a hundred, 14 % at worst (160, b = 5,
// 85k M = 24 20.2 / 17.7).
inline RoundRoute dq_round_route(const RouteQuery& q, const bool cta_tiles, const bool pairs, const bool linf = false)
{
    const bool one = dq_one_pass(q);
    if (!cta_tiles) return one ? kWarpTiles : kTwoKernels;
    if (dq_by_warps(q, one, pairs, linf)) return kWarpTiles;
    const double m = (double)q.M, tiles = (double)q.positions;
    // what two kernels save per worker, and what they cost besides
    const double per_worker = pairs ? 0.5 : (q.odd_buckets > 0 ? 0.32 : 0.24), besides = pairs ? 5.5 : (q.odd_buckets > 0 ? 6.9 : 6.2);
    return per_worker * m - besides > 0.0005 * tiles * m ? kTwoKernels : kCtaTiles;
}

// What a CTA has a form for: given norms, and buckets of up to 1024 elements or of 2048, which are a pair of its warps'.
inline bool dq_cta_form(int32_t groups_per_bucket, bool given) { return given || groups_per_bucket <= 64; }

// The route of a call: tile positions of a worker, warps of a launch by warps, and the layout's bucket (32-element groups; where
// the norms are not given a power of two or less than 32).  lose_first: the test hook of the waits is set; a round by CTAs has no
// wait to lose, so the call takes the kernels that have.
inline RoundRoute dq_route_of(int64_t positions, int64_t warps, int32_t groups_per_bucket, int32_t M, bool given, bool linf,
                              bool lose_first)
{
    const bool teams = !given && groups_per_bucket > 32;
    RouteQuery q = {};
    q.positions = positions;
    q.units = teams ? warps / (groups_per_bucket / 32) : warps;
    q.M = M;
    q.given = given ? 1 : 0;
    q.odd_buckets = !given && (groups_per_bucket & (groups_per_bucket - 1)) != 0 ? 32 / groups_per_bucket : 0;
    return dq_round_route(q, dq_cta_form(groups_per_bucket, given) && !lose_first, teams, !given && linf);
}
