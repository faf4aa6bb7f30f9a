"""Index and size rules of csrc/rules.h over ranges no device buffer of a test reaches, compiled
with the host compiler (no GPU)."""
import ctypes
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1709_05418_gb300", "csrc")
SHIM = r"""
#include "rules.h"
using namespace rpnn;
extern "C" {
int64_t t_query_at(int64_t i) { return query_at(i); }
uint32_t t_poll_bound(uint32_t cap) { return path_poll_bound(cap); }
int t_rows_fit(int64_t M, int bm) { return gemm_rows_fit(M, bm); }
int t_row_dot(int N, int64_t K) { return gemm_row_dot(N, K); }
int t_group(int64_t rows, int64_t missing, int capturing, int64_t mem) { return group_gradients(rows, missing, capturing != 0, mem); }
int t_grouped_runs(int64_t K, int bk) { return grouped_runs(K, bk); }
int64_t t_slice(int64_t P) { return path_slice(P); }
int64_t t_slice_smaller(int64_t n) { return path_slice_smaller(n); }
int t_x_streams(int nx, int64_t rows, int levels) { return mip_x_streams(nx, rows, levels, 152); }
int t_x_lines(int nx, int stream) { return mip_x_lines(nx, stream != 0); }
int t_row_threads(int nx, int64_t rows) { return brick_row_threads(nx, rows, 152); }
int t_brick_chunk(int w) { return brick_chunk(w); }
int t_start_lanes(int64_t n) { return record_start_lanes(n, 152); }
int t_warps(int64_t n, int n_max) { return record_warps(n, n_max, 152); }
int t_lanes(int n_max, int warps) { return record_lanes(n_max, warps); }
int t_path_in_primary(int64_t P, float a, float depth) { return path_in_primary(P, a, depth, 152); }
// polls a wait makes until it gives up, or `total` if it does not; progress every `every` polls
int64_t t_polls(uint32_t bound, int64_t total, int64_t every) {
    PollBound w{0, 0};
    uint32_t progress = 0;
    for (int64_t i = 0; i < total; ++i) {
        if (every && i % every == 0) ++progress;
        if (!w.poll(progress, bound)) return i + 1;
    }
    return total;
}
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "rules.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I" + CSRC,
                    str(d / "shim.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.t_query_at.argtypes, L.t_query_at.restype = [ctypes.c_int64], ctypes.c_int64
    L.t_poll_bound.argtypes, L.t_poll_bound.restype = [ctypes.c_uint32], ctypes.c_uint32
    L.t_rows_fit.argtypes, L.t_rows_fit.restype = [ctypes.c_int64, ctypes.c_int], ctypes.c_int
    L.t_row_dot.argtypes, L.t_row_dot.restype = [ctypes.c_int, ctypes.c_int64], ctypes.c_int
    L.t_group.argtypes, L.t_group.restype = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int64], ctypes.c_int
    L.t_grouped_runs.argtypes, L.t_grouped_runs.restype = [ctypes.c_int64, ctypes.c_int], ctypes.c_int
    for f in (L.t_slice, L.t_slice_smaller):
        f.argtypes, f.restype = [ctypes.c_int64], ctypes.c_int64
    L.t_x_streams.argtypes, L.t_x_streams.restype = [ctypes.c_int, ctypes.c_int64, ctypes.c_int], ctypes.c_int
    L.t_x_lines.argtypes, L.t_x_lines.restype = [ctypes.c_int, ctypes.c_int], ctypes.c_int
    L.t_row_threads.argtypes, L.t_row_threads.restype = [ctypes.c_int, ctypes.c_int64], ctypes.c_int
    L.t_brick_chunk.argtypes, L.t_brick_chunk.restype = [ctypes.c_int], ctypes.c_int
    L.t_start_lanes.argtypes, L.t_start_lanes.restype = [ctypes.c_int64], ctypes.c_int
    L.t_warps.argtypes, L.t_warps.restype = [ctypes.c_int64, ctypes.c_int], ctypes.c_int
    L.t_lanes.argtypes, L.t_lanes.restype = [ctypes.c_int, ctypes.c_int], ctypes.c_int
    L.t_path_in_primary.argtypes, L.t_path_in_primary.restype = [ctypes.c_int64, ctypes.c_float, ctypes.c_float], ctypes.c_int
    L.t_polls.argtypes, L.t_polls.restype = [ctypes.c_uint32, ctypes.c_int64, ctypes.c_int64], ctypes.c_int64
    return L


def test_shading_point_offsets_need_64_bits(rules):
    """Up to 2^31 - 1 shading points: every offset is exact, and no kernel that reads the lists
    works one out by itself."""
    for i in (0, 1, 715827882, 715827883, 2 ** 31 - 2):
        assert rules.t_query_at(i) == 3 * i
    src = open(os.path.join(CSRC, "render.cu")).read()
    assert not re.findall(r"\bq[xd]\[3 \*", src)
    # a point's index runs to 2^31 - 1 and its grid stride beyond
    for kernel in ("k_nee_env", "k_scatter"):
        body = src[src.index(kernel + "("):]
        body = body[:body.index("\n}\n")]
        assert not re.search(r"\bint i = blockIdx", body), kernel


def test_waits_for_other_warps_are_bounded_from_the_last_progress(rules):
    """A record of millions of paths adds up more polls than the bound while its block gets on; only
    polls without any progress may end it, and those do."""
    assert rules.t_polls(1000, 1000000, 999) == 1000000
    assert rules.t_polls(1000, 1000000, 0) == 1000
    assert rules.t_polls(1000, 1000000, 5000) == 1000
    # no progress for as long as one tracking call may take; the sum does not wrap
    for cap in (0, 1000000, 2 ** 32 - 1):
        assert rules.t_poll_bound(cap) >= min(2 ** 24 + 32 * cap, 2 ** 32 - 1)
    src = open(os.path.join(CSRC, "paths.cuh")).read()
    assert "++polls" not in src and "src.idle(path_poll_bound(v.track_cap))" in src


def test_row_tiles_fit_the_grid(rules):
    """Every accepted row count (65,535 x 64) has its default tile; tiles of 32 rows end at half of it,
    and the tuner asks before it times one."""
    for bm in (32, 64, 128):
        for M in (1, bm * 65535):
            assert rules.t_rows_fit(M, bm)
        for M in (bm * 65535 + 1, 2 ** 31 - 1):
            assert not rules.t_rows_fit(M, bm)
    src = open(os.path.join(CSRC, "mlp_simt.cu")).read()
    body = src[src.index("rpnn_status tune("):]
    assert "gemm_rows_fit" in body[:body.index("cands.push_back")]


def test_long_one_column_sums_are_not_one_chain(rules):
    """A column whose sum may be split is not summed by one thread per row."""
    for K in (1, 200, 1008):
        assert rules.t_row_dot(1, K) and not rules.t_row_dot(2, K)
    for K in (1009, 2400, 16384, 2 ** 22):
        assert not rules.t_row_dot(1, K)


def test_grouped_gradients_only_where_everything_they_need_fits(rules):
    """The kept gradients and the grouped launch's workspace together decide, nothing is allocated
    under capture, and memory that is free again is used again."""
    rows, need, slack = 100000, 2 * 10 ** 9, 64 << 20
    assert rules.t_group(rows, need, 0, need + slack)
    assert not rules.t_group(rows, need, 0, need + slack - 1)          # the buffers alone would fit
    assert not rules.t_group(rows, need, 1, 2 ** 40)
    assert rules.t_group(rows, 0, 1, 0) and rules.t_group(2 ** 17, 0, 0, 0)
    assert not rules.t_group(2 ** 17 + 1, 0, 0, 2 ** 40)
    for K, bk, runs in ((1008, 16, 1), (1009, 16, 16), (1009, 8, 32), (2047, 16, 32), (2000, 16, 16), (4096, 16, 32), (10 ** 6, 8, 32)):
        assert rules.t_grouped_runs(K, bk) == runs, (K, bk)
    src = open(os.path.join(CSRC, "mlp_simt.cu")).read() + open(os.path.join(CSRC, "internal.h")).read()
    assert "group_rows" not in src               # no limit outlives the call that met it
    body = src[src.index("rpnn_status rpnn_backward_f32("):]
    assert "wgrads_need" in body[:body.index("group_gradients(")]


def test_path_renders_list_a_bounded_slice(rules):
    """The shading-point lists of a path-traced image do not grow with it (28 bytes a sample would be
    60 GB at 2^31 - 1), and shrink to 2 MB before a render gives up."""
    for P in (1, 2 ** 16, 2 ** 24, 2 ** 31 - 1):
        n = rules.t_slice(P)
        assert n == min(P, 2 ** 24) and 28 * n <= 470e6
        while n > 2 ** 16:
            assert rules.t_slice_smaller(n) < n
            n = rules.t_slice_smaller(n)
        assert 28 * n <= 2e6
    src = open(os.path.join(CSRC, "capi.cu")).read()
    body = src[src.index("static rpnn_status render_impl("):]
    assert "slice = path ? path_slice(P) : P;" in body and "q_x.reserve(slice * 3" in body


def test_x_pass_streams_where_that_was_measured_to_pay(rules):
    """Single levels, small grids and middling lines on few rows keep the form whose tasks fill every lane;
    staged lines fit the shared memory the launches ask for, whatever the length."""
    for nx, rows in ((96, 15200), (144, 5016), (256, 65536), (680, 5016), (681, 60800), (1024, 2 ** 20), (1088, 1),
                     (8192, 10 ** 6)):
        assert rules.t_x_streams(nx, rows, 2) and rules.t_x_streams(nx, rows, 9), (nx, rows)
        assert not rules.t_x_streams(nx, rows, 1)
    for nx, rows in ((64, 4096), (95, 10 ** 6), (143, 15199), (256, 5015), (768, 32768), (1024, 4096), (1087, 60799)):
        assert not rules.t_x_streams(nx, rows, 6), (nx, rows)
    for nx in range(1, 8193):
        for stream, most in ((0, 32), (1, 64)):
            n = rules.t_x_lines(nx, stream)
            assert 1 <= n <= most and n * (nx + 1) * 4 <= 72 * 1024


def test_brick_rows_take_no_more_threads_than_they_need(rules):
    """Whole bricks a pass, each with its two neighbours inside the row's threads; where there are many
    rows, short lines share a block (1 voxel: 16 rows of it)."""
    many = 65536
    for nx in range(1, 8193):
        w = rules.t_row_threads(nx, many)
        c = rules.t_brick_chunk(w)
        assert w in (16, 32, 64, 128, 256) and c % 8 == 0 and 8 <= c <= w - 2
        assert c >= nx or w == 256
        assert w == 16 or rules.t_brick_chunk(w // 2) < nx
        # a brick's last column, read from the row's own part of the shared buffer
        assert 8 * (c // 8 - 1) + 9 < w
        assert rules.t_row_threads(nx, 8 * 152) == 256
    assert rules.t_row_threads(1, many) == 16 and rules.t_row_threads(249, many) == 256


def test_few_paths_are_spread_over_a_records_warps(rules):
    """Every warp that a record gets has paths to trace, few records start a warp each, and all paths
    and records are reached whatever their number."""
    for n in (1, 152, 1064, 1065, 4863, 4864, 9727, 9728, 9729, 2 ** 32):
        lanes = rules.t_start_lanes(n)
        assert lanes in (1, 2, 4, 8, 16, 32) and (lanes == 1) == (n <= 9728)
        assert (n + 4 * lanes - 1) // (4 * lanes) <= 2 ** 31 - 1
        for n_max in (1, 2, 16, 31, 32, 33, 64, 65, 127, 128, 1024, 2 ** 31 - 1):
            warps = rules.t_warps(n, n_max)
            per = rules.t_lanes(n_max, warps)
            assert warps in (1, 2, 4) and 1 <= per <= 32
            assert per * warps >= min(n_max, 32 * warps)
            if n > 1064 and warps > 1:
                assert n_max > 16 * warps
            if n_max > 64:
                assert warps == (1 if n >= 9728 else 2 if n >= 4864 else 4)
            if n_max >= 128:
                assert per == 32


def test_short_paths_of_middle_sized_images_stay_in_the_primary_pass(rules):
    """Long paths, thumbnails and large images (and with them every image of several slices) are dealt
    to lanes by a launch of their own."""
    for a, depth in ((0.99, 5.0), (0.9, 12.0), (0.3, 50.0), (0.5, 400.0)):
        for side, there in ((64, 0), (160, 1), (256, 1), (400, 1), (512, 0)):
            assert rules.t_path_in_primary(side * side, a, depth) == there, (a, depth, side)
        assert not rules.t_path_in_primary(2 ** 24, a, depth)
    for a, depth in ((0.99, 50.0), (0.51, 20.5), (1.0, 1000.0)):
        assert not any(rules.t_path_in_primary(P, a, depth) for P in (1, 25600, 65536, 160000, 2 ** 31 - 1))
    assert rules.t_path_in_primary(200 * 200, 0.99, 20.0) and not rules.t_path_in_primary(160 * 160, 0.99, 20.0)
    assert rules.t_path_in_primary(128 * 128, 0.99, 5.0) and not rules.t_path_in_primary(128 * 128, 0.99, 10.0)
