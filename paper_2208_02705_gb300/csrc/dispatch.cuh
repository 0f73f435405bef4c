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

// Samples that a round of a render marches, about: a ray of a mapped scene
// keeps up to 16 in its first round, and an eighth of the rays go on.
constexpr int64_t round_samples(int64_t n_rays, int round_size, bool first)
{
    return n_rays * (round_size < 16 ? round_size : 16) / (first ? 1 : 8);
}

}  // namespace roam
