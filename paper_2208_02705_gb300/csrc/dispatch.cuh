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

}  // namespace roam
