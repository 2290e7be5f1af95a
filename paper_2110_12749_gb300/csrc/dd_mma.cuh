// Dedispersion on the tensor cores (dd_mma.cu): the plan's host tables.
#pragma once

#include <cstdint>
#include <vector>

namespace gsp {

constexpr int kMmaMaxBeams = 32;    // beams per launch
constexpr int kMmaMinBlock = 1024;  // smallest search block whose sums the kernel accumulates
constexpr int kMmaMaxBlock = 1 << 30;  // and the largest: a tile's block ends stay within 32 bits

// A run of channels (positions pos .. the next frame's pos, in order of
// increasing delay) whose rows keep their displacement R; e: how far each row
// of the block moves when the frame begins; rmax: its largest R.
struct MmaFrame {
    int32_t pos;
    int32_t rmax;
    uint8_t e[16];
};

struct MmaTables {
    std::vector<int32_t> base;     // [nblk][npos] window start of each position, relative to the tile
    std::vector<uint8_t> shift;    // [nblk][ceil(npos / 8)][16][8] shift of each (position, DM), 0..8
    std::vector<int32_t> crmax;    // [nblk][ceil(npos / 8)] largest R of the chunk's frames
    std::vector<int32_t> rlast;    // [nblk][16] R of the last frame
    std::vector<int32_t> foff;     // [nblk + 1] first frame of each block
    std::vector<MmaFrame> frames;
    int rmax = 0;                  // largest R of all
    double mean_cols_r = 0.0;      // mean over the channels of the frame's largest R
};

// What the launch and the choice of kernel need of the tables.
struct MmaShape {
    int npos = 0;  // channels, in order of increasing delay
    int rmax = 0;
    double mean_r = 0.0;
    double frames_per_block = 0.0;
};

// delays [ndm][C]; rev: positions run from the last channel to the first; the first
// npos of them.  false: a block's delays drift apart by more than a tile.
bool mma_plan_tables(const int32_t *delays, int ndm, int C, bool rev, int npos, MmaTables *t);
// How many positions to take where the rest is left to a kernel of other_rate additions
// per clock and SM and other_fixed clocks per sample of a trial, which takes rows in whole
// steps from the first on (the rest's first row, and its last one where more rows follow, is a
// multiple of step); 0 if that gains less than a twentieth.
int mma_split(const int32_t *delays, int ndm, int C, bool rev, int step, double other_rate,
              double other_fixed);
// Longest tile (output samples) for a largest R.
int mma_tile_len(int rmax);
// Estimated SM clocks of one work item (16 DM trials x T samples x nchan channels).
// add: to a series that is there already.
double mma_item_clocks(const MmaShape &m, int nchan, int T, bool add);

// The same of a whole launch of one beam, and the tile length it is least at.
double mma_launch_clocks(const MmaShape &m, int nchan, int ndm, int64_t n_out, int num_sms, bool add,
                         int *tile);
constexpr double kLaunchClocks = 14000.0;  // of any launch, beside its work items

}  // namespace gsp
