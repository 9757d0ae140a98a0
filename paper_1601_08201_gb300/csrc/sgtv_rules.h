// sgtv_rules.h -- dispatch rules over sizes alone, plain C++ (no CUDA), so that
// they can be checked on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SGTV_RULE __host__ __device__ constexpr
#else
#define SGTV_RULE constexpr
#endif

namespace sgtv {

// The deviance's form for `rows` measurements of `mean` nonzeros on average: 0 the
// tiled one (where there is one), else the rows that a warp of the plain one takes
// in turn. The plain form has 16 warps a multiprocessor (two blocks of 8). What
// counts is how many rows lie behind one another in a warp (8 in the tiled form),
// and from some rows a multiprocessor on the FP64 terms, a division and a
// logarithm, which cost a warp the same for one row as for 8 side by side. So a warp
// each while there is one for every row, then the tiled form, and without it 8
// rows in turn unless they are long. Measured, microseconds, tiled / plain with 1 /
// 2 / 8 rows (FP32, 152 multiprocessors): 640 rows of 64 nonzeros 10.1 / 5.8 / 6.6 /
// 14.2, of 1400 40 / 12 / 18 / 60; 2000 rows of 64 10.4 / 10.2 / 8.5 / 14.4, of 1400 45 /
// 26 / 24 / 60; 6000 rows of 64 10.4 / 24 / 18 / 15, of 1400 54 / 69 / 67 / 71; 20,000 rows
// of 300 24 / 100 / 77 / 70, of 700 42 / 145 / 126 / 143, of 1400 75 / 232 / 217 / 260;
// 60,000 rows of 64 27 / 206 / 132 / 81.
SGTV_RULE int dev_rows_per_warp(int64_t rows, int64_t mean, int sms, bool tiled)
{
    if (rows <= 16 * int64_t(sms)) return 1;
    if (tiled) return 0;
    return mean <= 512 ? 8 : 1;
}

// Pieces that a plane (sample, channel) of n elements is cut into for the loss
// head: one where the planes alone fill `blocks` blocks, else enough to, of at
// least 1024 elements (four a thread). A sample of one channel, 256 x 256: 87 us with
// one block, 5.8 with 64; 16 channels 89 and 10.9; 8 samples of 320 channels, 64 x
// 64, one piece a plane either way.
SGTV_RULE int64_t mse_pieces(int64_t planes, int64_t n, int64_t blocks)
{
    const int64_t want = (blocks + planes - 1) / planes, most = (n + 1023) / 1024;
    return want < most ? want : most;
}

// Whether the shrink of `sites` sites goes out in blocks of a warp, one a site,
// instead of eight: FP64 sites of a small image, where a block of eight waits for
// one FP64 unit (13 x 7 x 37, the shrink alone 6.6 -> 4.8 us; an iteration of two
// passes 12.9 -> 11.3). Not in the single-pass form (`staged`: a row pass that stages
// tiles in shared memory runs beside the shrink): blocks on every multiprocessor
// are in the way of its start on those with room for its tiles, and replayed from
// graphs an iteration of 41 x 9 x 54 took 78 us instead of 44, 20 x 20 x 40 64 instead
// of 37, 2000 rows of 1500 nonzeros 214 instead of 137. Nor in FP32, where they stand
// in the way of the stacked row pass (41 x 9 x 54: shrink 2.6 -> 2.3 us, but the row
// pass 6.1 -> 7.9).
SGTV_RULE bool shrink_spread(int elem_size, bool staged, int64_t sites, int sms)
{
    return elem_size == 8 && !staged && sites < 8 * int64_t(sms);
}

// The autotuner's time of one launch of a form: the mean of `reps`, where
// timed(n, &ms) launches n times, gives the time of all and returns 0 or an error.
// Where a launch is long (50 us, so that one more wait for the stream counts for
// little), a form over 1.5 times the best so far is out of the running without
// them, if two launches by themselves say so: one alone may have been disturbed,
// and the choice is for the life of the handle.
template <typename Timed>
auto tuned_time(Timed &&timed, int reps, float so_far, float *ms) -> decltype(timed(1, ms))
{
    if (so_far > 0.05f) {
        float least = 0.f;
        for (int k = 0; k < 2; k++) {
            const auto e = timed(1, ms);
            if (e != decltype(e)(0)) return e;
            least = k == 0 || *ms < least ? *ms : least;
            if (least <= 1.5f * so_far) break;
        }
        *ms = least;
        if (least > 1.5f * so_far) return decltype(timed(1, ms))(0);
    }
    const auto e = timed(reps, ms);
    *ms /= float(reps);
    return e;
}

}  // namespace sgtv
