// Rules that choose between forms of a kernel or lay out work for one, on
// sizes alone (plain C++: also compiled by the host tests).
#pragma once

#include <cstdint>

namespace roam {

// Tiles that a field's run is padded to: the least multiple of both the
// requested padding (0: none) and the tiles a kernel keeps in flight.
constexpr int tile_run(int pad, int slots)
{
    if (pad <= 0) return slots;
    int run = pad;
    while (run % slots != 0) run += pad;
    return run;
}

// Tiles that the tensor-core forward keeps in flight per SM, for about
// `samples` samples spread over n_fields fields of its width.  TMEM admits 2 at
// W = 128 and 4 at W = 64.  At W = 32 a layer is mostly the slot's barrier,
// commit round trip and waits, so six hide more than four, but at 80 registers
// a thread instead of 128, and a group of six takes 1.2 times as long as one of
// four: six pay once a field has several groups and every SM some.  Measured
// with four -> six (GB300, H = 2, BF16 / FP8, scattered points):
//   4 M in 1 field       292 -> 241 us / 336 -> 277
//   1 M in 128 fields     89 ->  82    /  99 ->  98    (61 tiles per field)
//   400 k in 16           46 ->  42    /  51 ->  49    (20 tiles per SM)
//   400 k in 128          49 ->  48    /  54 ->  56    (24 tiles per field)
//   1 M in 1024           98 -> 108    / 112 -> 126    (8 tiles per field)
//   150 k in 16           25 ->  28    /  28 ->  32    (8 tiles per SM)
constexpr int tc_slots(int W, int64_t samples, int n_fields, int n_sm)
{
    if (W > 32) return W > 64 ? 2 : 4;
    return samples >= 28 * 128 * (int64_t)n_fields && samples >= 16 * 128 * (int64_t)n_sm ? 6 : 4;
}

// Whether a map of S occupied voxels in `bricks` non-empty 8^3 bricks, split into
// networks of `per` voxels, is assigned from brick lists (one cluster of 8 blocks
// builds every network) or by the general form (whole-chip passes over all
// unassigned voxels, five launches per network).  Microseconds per network of
// either, fitted to both forms on the same maps (GB300; the first term of the
// one is its cluster barriers, of the other its launches).  Measured, lists and
// general:
//   1.5 M voxels in 18,944 bricks:    33,000 per network   49 /  74, 139,000 133 / 109
//   6.2 M in 86,528:                  15,500               34 / 115, 269,000 274 / 212
//   262 k in 512:                      8,200               29 /  52, 131,000  77 /  62
//   268 k in 168,116 (1.6 per brick):  2,000               35 /  50,  16,700 118 /  58
//   2.0 M in 1,289,647:                5,000              150 /  84
constexpr bool assign_from_bricks(int64_t S, int64_t bricks, int64_t per)
{
    const double lists = 10.0 + 1.2e-4 * (double)bricks + (double)per * (0.8e-3 + 8e-3 * (double)bricks / (double)S);
    const double general = 44.0 + 1.15e-5 * (double)S + 3.3e-4 * (double)per;
    return lists <= general;
}

// Samples that a round of a render marches, about: a ray of a mapped scene
// keeps up to 16 in its first round, and an eighth of the rays go on.
constexpr int64_t round_samples(int64_t n_rays, int round_size, bool first)
{
    return n_rays * (round_size < 16 ? round_size : 16) / (first ? 1 : 8);
}

}  // namespace roam
