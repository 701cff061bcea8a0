// batch_plan.h -- how the problems of a batched solve are cut into CTAs, and
// how many of them a workspace has to hold: host arithmetic alone.
#pragma once
#include <algorithm>

namespace lsp {

// A problem's tile of its two fastest axes is one of kBatchShapes (chosen per
// problem dimension by two bits of lsp_solve_opts.batch_tiles).
constexpr int kBatchNumShapes = 3;
constexpr int kBatchShapes[kBatchNumShapes][2] = {{16, 16}, {32, 8}, {64, 4}};
// planes per CTA along the march when lsp_solve_opts.batch_chunk is 0
constexpr int kBatchMinPlanes = 4, kBatchMaxPlanes = 128;

// The local-coefficient / clipped kernels are compiled for 16 x 16 tiles.
inline int batch_shape(int batch_tiles, int ndim, bool local)
{
    return local ? 0 : (batch_tiles >> (2 * (ndim - 2))) & 3;
}

struct BatchTiling {
    int tb, ta, nbx, nby, ch, nchunks;
    long long blocks;
};

inline BatchTiling batch_tiling(int ndim, const int* n, int shape, int chunk)
{
    BatchTiling t;
    t.tb = kBatchShapes[shape][0];
    t.ta = kBatchShapes[shape][1];
    t.nbx = (n[ndim - 1] + t.tb - 1) / t.tb;
    t.nby = (n[ndim - 2] + t.ta - 1) / t.ta;
    t.ch = ndim >= 3 ? std::min(chunk, n[ndim - 3]) : 1;
    t.nchunks = ndim >= 3 ? (n[ndim - 3] + t.ch - 1) / t.ch : 1;
    t.blocks = (long long)t.nbx * t.nby * t.nchunks * (ndim == 4 ? n[0] : 1);
    return t;
}

// The work of a stage of the batch: planes of tiles, and the longest column of
// planes.
struct BatchWork {
    double planes = 0.0;
    int longest = 1;
    void add(int ndim, const int* n, int shape)
    {
        planes += (double)batch_tiling(ndim, n, shape, 1).blocks;
        if (ndim >= 3) longest = std::max(longest, n[ndim - 3]);
    }
};

// Planes per CTA when opts->batch_chunk is 0.  A stage of the whole batch has
// x = planes / (3 CTAs x SMs) planes for each resident CTA: with
// whole columns per CTA a small batch leaves most of them idle and waits for
// the largest problem's column, with short chunks the persistent launch pays
// its per-item overhead (counter, fences, dependency poll) and every CTA its
// start more often.  Best of 4 .. 128 planes in milliseconds, against the
// whole columns (128) used before, half 2-D fronts and half 3-D games, WENO5
// RK3 (persistent; graph form in brackets):
//   24 problems, x = 97: 32 planes 3.91, 128 5.06 (24: 4.04, 5.81)
//   8 problems, x = 33: 16 planes 1.20, 2.69 (8: 1.25, 3.28)
//   32 at half size, x = 21: 12 planes 0.92, 1.93 (8: 1.04, 2.30)
//   4 at 0.4 size, x = 1: 4 planes 0.31, 1.06 (4: 0.34, 1.09)
//   96 problems, x = 390: 128 planes 8.97 (32: 9.25, 64: 9.29, 128: 9.89)
// which 5 + 0.31 x (persistent) and 4 + 0.2 x (graph) meet within 3 %.
// Whole columns stay where no column is longer than x: they fill the device
// evenly as they are (263 problems of 9^3 on 64 x 4 tiles 29 % faster whole,
// 146 of 27 x 26 x 24 on 16 x 16 9 %); up to 24 planes, where a start weighs
// more, from 0.6 of the longest on (graph form: 368 of 12^3, 130 of 20 x 21 x
// 22 on 32 x 8, 14 %).  Over 250 random batches of 1 to 400 problems: 0.49
// (persistent) and 0.53 (graph) of the time of whole columns, none above 1.04.
inline int batch_auto_chunk(const BatchWork& w, int sms, bool persistent)
{
    const double x = w.planes / (3.0 * sms);
    if (x >= (w.longest <= 24 ? 0.6 : 1.0) * w.longest) return kBatchMaxPlanes;
    const double c = persistent ? 5.0 + 0.31 * x : 4.0 + 0.2 * x;
    return c >= kBatchMaxPlanes ? kBatchMaxPlanes : std::max(kBatchMinPlanes, (int)c / 2 * 2);
}

// The most CTAs this problem can have in a solve whose workspace was sized
// with `batch_chunk`: over every tile shape and, when the chunk is chosen by
// the work of the whole batch, at the shortest one, whatever the other
// problems, their shapes and the form of the launch turn out to be (a fraction
// of a per mille of the problem's fields).
inline long long batch_max_blocks(int ndim, const int* n, int batch_chunk)
{
    const int chunk = batch_chunk > 0 ? batch_chunk : kBatchMinPlanes;
    long long most = 0;
    for (int sh = 0; sh < kBatchNumShapes; ++sh)
        most = std::max(most, batch_tiling(ndim, n, sh, chunk).blocks);
    return most;
}

}  // namespace lsp
