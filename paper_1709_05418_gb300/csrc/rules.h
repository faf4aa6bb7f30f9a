// rules.h -- index and size rules shared by host code and kernels.  Plain C++, so that a host
// compiler alone can evaluate them over ranges no device buffer of a test would reach.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define RPNN_RULE __host__ __device__ __forceinline__
#else
#define RPNN_RULE inline
#endif

namespace rpnn {

// Offset of shading point i in the lists of positions and directions (three floats a point).
// A render has up to 2^31 - 1 samples, so from i = 715,827,883 on the offset needs 64 bits.
RPNN_RULE int64_t query_at(int64_t i) { return 3 * i; }

// Waits of a warp whose lanes have no work while other warps of its block trace the paths they wait
// for.  `progress` counts what those warps get done (bounces of their paths, rounds taken into the
// label), so the bound is on polls during which nothing happened anywhere in the block, however
// long the record: the longest such stretch of a healthy block is one tracking call, at most
// `track_cap` collisions of about 4 us each, and a poll takes at least 0.2 us.
RPNN_RULE uint32_t path_poll_bound(uint32_t track_cap) {
    const uint64_t b = (1ull << 24) + 32ull * track_cap;
    return b > 0xffffffffull ? 0xffffffffu : (uint32_t)b;
}
struct PollBound {
    uint32_t polls, seen;
    // one more poll; false once `bound` polls in a row saw no progress
    RPNN_RULE bool poll(uint32_t progress, uint32_t bound) {
        if (progress != seen) { seen = progress; polls = 0; }
        return ++polls < bound;
    }
};

// FP32 GEMM: row tiles are blocks of grid.y, at most 65,535 of them.  The default tile (64 rows)
// takes every row count the entry points accept, a 32-row tile half of them.
RPNN_RULE bool gemm_rows_fit(int64_t M, int bm) { return (M + bm - 1) / bm <= 65535; }

// FP32 GEMM: inner sizes whose sum the tuner may split into runs (counted in K tiles of 16).
constexpr int kMinSplitK = 1024;
RPNN_RULE bool gemm_may_split(int64_t K) { return (K + 15) / 16 * 16 >= kMinSplitK; }
// One output column: a thread per row sums all K products in a row below that, as the tiled kernel
// would, which adds up to K roundings; longer sums keep the tiled kernel and its runs (at most
// K / 32 + 32 roundings, and more than one warp per 32 rows: 4,096 rows of 2,400 take 71 us tuned,
// 131 with a thread each; 100 rows of 16,384 take 85 and 791).
RPNN_RULE bool gemm_row_dot(int N, int64_t K) { return N == 1 && !gemm_may_split(K); }

// FP32 backward with all weight gradients in one launch: every layer's gradient is kept until then,
// 17,600 bytes a row.  A layer's own launches do beyond kGroupRows rows (where they fill the chip),
// and where the buffers that are missing would not fit beside what is allocated; asked again at each
// call, so that a step that could not have them once may later.  While a stream is being
// captured nothing is allocated: the buffers of the direct run before it are there or not.
constexpr int64_t kGroupRows = 1 << 17;
constexpr int64_t kGroupSlack = 64 << 20;         // for rounding of the allocations and the rest of the step
RPNN_RULE bool group_gradients(int64_t rows, int64_t missing, bool capturing, int64_t free_bytes) {
    return rows <= kGroupRows && (missing == 0 || (!capturing && missing + kGroupSlack <= free_bytes));
}
// Runs of its sums over K rows for a tile of K step bk (as many as one such GEMM takes at most).
RPNN_RULE int grouped_runs(int64_t K, int bk) {
    int runs = 1;
    while (gemm_may_split(K) && runs < 32 && (K + 15) / 16 * 16 / bk / (2 * runs) >= 4) runs *= 2;
    return runs;
}

// Path-traced renders list their shading points (28 bytes each) a slice of samples at a time, so that
// an image needs little more than its 4 bytes a sample: 470 MB of lists at most, halved while they do
// not fit, down to 2 MB.  A slice of 2^24 samples runs 0.1 s, its last paths about 1 ms of that.
constexpr int64_t kPathSlice = 1 << 24, kMinPathSlice = 1 << 16;
RPNN_RULE int64_t path_slice(int64_t samples) { return samples < kPathSlice ? samples : kPathSlice; }
RPNN_RULE int64_t path_slice_smaller(int64_t slice) { return slice / 2 > kMinPathSlice ? slice / 2 : kMinPathSlice; }

// x pass of the pyramid build: whether its warps stream along lines (64 slots a warp, as many lines as
// fit beside one another), for `levels` of `rows` lines of nx voxels; otherwise each output is a task.
// Streaming halves the arithmetic, and a thread's chain over a long line serves all its outputs; but a
// line that does not fit is an idle slot and a block has a warp per level.  Streamed against by task,
// all levels together, nx x lines: 256 x 65,536 123 and 180 us; 160 to 640 x 5,250 0.76-1.0 of the time, x
// 4,096 (64 blocks) 0.86-1.21; 96 and 128 x 10,000 1.08 and 1.04, x 16,384 0.89 and 0.83; 704 to 1,024 (25 to
// 17 lines fit) x 65,536 0.91-1.11, x 262,144 0.91-1.06, x 6,400 1.0-1.5; 1,100 to 8,192 x 4,096 and more
// 0.64-1.0 (1,536 x 4,096 1.19), x 256 0.88-1.1.  One level of 1,024 x 32,768, with the call around it, 612
// and 262 us.
RPNN_RULE bool mip_x_streams(int nx, int64_t rows, int levels, int sms) {
    const int least = nx < 144 ? 100 : (nx <= 680 ? 33 : (nx < 1088 ? 400 : 0));       // lines per SM
    return levels > 1 && nx >= 96 && rows >= least * (int64_t)sms;
}
RPNN_RULE int mip_x_lines(int nx, bool stream) {
    const int most = stream ? 64 : 32, fit = (stream ? 72 : 64) * 1024 / ((nx + 1) * 4);
    return fit < 1 ? 1 : (fit < most ? fit : most);
}

// Statistics and brick majorants: threads that take one row of bricks (a block of 256 takes as many
// rows as that gives): the fewest that read a whole line, with a voxel before and behind it, at
// once, where a row per block would be more than one wave of eight blocks an SM.  With all 256 on a
// row, lines of few voxels left most of the block idle: 1 x 2,048^2 407 us (81 now), 8 x 1,024^2 104 (24).
// Within one wave that costs nothing (64 x 128^2 6.6 us, 7.5 with 128 threads a row).
RPNN_RULE constexpr int brick_chunk(int threads) { return (threads - 2) / 8 * 8; }    // voxels a pass covers
RPNN_RULE int brick_row_threads(int nx, int64_t rows, int sms) {
    int w = 256;
    while (rows > 8 * (int64_t)sms && w > 16 && brick_chunk(w / 2) >= nx) w /= 2;
    return w;
}

// Training records: how many of them one warp starts (each a delta track with retries, so lanes
// of a warp wait for one another): one while the chip holds a warp for each.
RPNN_RULE int record_start_lanes(int64_t n, int sms) {
    int lanes = 1;
    while (lanes < 32 && lanes * 64 * (int64_t)sms < n) lanes *= 2;
    return lanes;
}
// Warps that share a record's paths: the fewer the records, the more, so that the chip stays full until
// the last ones end (4,096 records: 12.9 ms with one each, 12.0 with two; 1,024: 5.8 with two,
// 4.4 with four); but where the chip is full (28 warps an SM) none that would have fewer than 16
// paths (4,000 records of 32 paths: 6.0 ms with four warps each, 3.5 with one).
RPNN_RULE int record_warps(int64_t n, int n_max, int sms) {
    const int64_t want = (int64_t)sms * 64;
    int warps = n >= want ? 1 : (n * 2 >= want ? 2 : 4);
    while (4 * n > 28 * (int64_t)sms && warps > 1 && 16 * warps >= n_max) warps /= 2;
    return warps;
}
// ... and the lanes of each that take paths: the first warp to ask would leave none for the others
// where the paths are few (152 records of 32 paths: 2.1 ms on one warp, 1.4 on eight lanes of four).
RPNN_RULE int record_lanes(int n_max, int warps) {
    const int64_t l = ((int64_t)n_max + warps - 1) / warps;
    return l < 32 ? (int)l : 32;
}

// Path-traced renders: whether each sample's lane of the primary pass traces its path too, instead of
// listing it for a launch that deals the paths to lanes as they get free.  That launch wins by a
// third where paths are long or many; between the sizes at which the chip is half empty and several
// times full, short paths (little survives a collision, or few collisions lie across the cloud:
// `depth`, the majorant's optical depth of the unit box) are over before it has paid for itself.  Time
// of the second launch against the lane's own, 128^3 fBm and 64^3 blobs, 160^2 to 400^2: depth 5, any
// albedo 1.10-1.39; 10: 0.98-1.34; 20: 0.90-1.14 (160^2: 0.90-1.07); 50: 0.76-1.06 at albedo 0.9 and above,
// 0.86-1.13 at 0.7, 0.95-1.24 at 0.3.  512^2 x 2: 0.63-0.91 everywhere; 64^2: 0.55-1.1 above depth 2.
RPNN_RULE bool path_in_primary(int64_t samples, float albedo, float depth, int sms) {
    const int least = depth <= 6.0f ? 100 : (depth <= 12.0f || albedo <= 0.5f ? 160 : 240);   // samples per SM
    return (albedo <= 0.5f || depth <= 20.0f) && samples >= least * (int64_t)sms && samples <= 1300 * (int64_t)sms;
}

}  // namespace rpnn
