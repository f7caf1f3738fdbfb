// stage_form.h -- which form of the FP32 stage kernel a solver's steps take beside other solvers (host only).
#pragma once

#include <atomic>

namespace vk {

// Small D2Q16 grids have two forms of the 8-row stage kernel, which give the same bits: 512 threads a tile (the
// fastest for a solver that has the GPU to itself) and 256.  Several solvers may step at once, on streams and
// threads of their own; together they fill the GPU, and then the form with less work per tile is the faster:
//   alone    512 threads, and of a grid of at most one tile per SM one CTA per SM (spread_smem)
//   shared   512 threads; another solver's tiles may lie beside its own on an SM
//   crowded  the 256-thread kernels
// us a step of all, 128 x 256 (128 tiles), WENO-5: 1 solver 16.7 / 16.9 / 17.7; 2 22.2 / 22.4 / 27.9; 4 41.7 / 27.1 /
// 26.9; 8 - / 53.5 / 44.3 (before the 512-thread form: 22.7, 27.6, 32.5, 45.1).  U3 + Komissarov: 1 12.1 / 12.2 /
// 17.0; 4 34.3 / 20.8 / 23.7; 8 - / 41.3 / 36.6 (before: 17.5, 25.2, 37.2).  181 x 384 (276 tiles), WENO-5: 2 - /
// 29.3 / 30.2; 3 - / 42.2 / 34.2; 4 - / 56.2 / 44.6 (before: 36.0, 38.5, 47.1).
enum StageForm { STAGE_ALONE = 0, STAGE_SHARED = 1, STAGE_CROWDED = 2, STAGE_FORMS = 3 };

// own tiles of a launch beside `others` in flight: four per SM (of 152) and more are a crowd
inline StageForm stage_form(long long own, long long others)
{
    return others <= 0 ? STAGE_ALONE : own + others <= 4 * 152 ? STAGE_SHARED : STAGE_CROWDED;
}

// Tiles of the solvers and batches of this process whose steps have been launched and not waited for.  It only
// guides the choice of a form: a program that waits by its own means leaves it too large, and loses the
// difference of two forms, no more.
inline std::atomic<long long> tiles_in_flight{0};

// One handle's share: enter before its launches (returns the others' tiles), leave once its stream has been waited for.
struct InFlight {
    long long mine = 0;
    long long enter(long long tiles)
    {
        if (!mine) tiles_in_flight += mine = tiles;
        return tiles_in_flight - mine;
    }
    void leave()
    {
        tiles_in_flight -= mine;
        mine = 0;
    }
};

}  // namespace vk
