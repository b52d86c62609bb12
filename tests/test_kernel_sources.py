"""Rules of the kernels' source that no run shows: breaking one costs a result only behind a predecessor that runs
for seconds, or only where a thread block starts late."""
import os
import re
import subprocess

import pytest

from paper_2602_15318_b200 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_15318_b200", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _between(text, start, end):
    i = text.index(start)
    return text[i:text.index(end, i)]


@pytest.mark.parametrize("name,start,end", [
    ("verify_tc.cuh", "if (warp == kProducerWarp) {", "else if (warp == kMmaWarp)"),
    ("verify_tc.cuh", "else if (warp == kMmaWarp) {", "else if (warp == kGateWarp)"),
    ("verify_tc.cuh", "else if (warp == kGateWarp) {", "else if (warp < 8)"),
    ("hsr_fuse.cuh", "if (warp == 4) {\n        if (lane == 0) {", "else if (warp == 5)"),
    ("hsr_fuse.cuh", "else if (warp == 5) {", "} else {"),
    ("hsr_fuse.cuh", "bool ok = n_kt == 0", None),
])
def test_no_bounded_wait_in_front_of_the_wait_for_the_predecessor(name, start, end):
    """A wait that gives up after a number of polls must not start while the predecessor may still run: a kernel
    that lets its dependents start early may take longer than those polls."""
    code = _code(name)
    if end is None:                                     # the projection's epilogue warps: the wait stands just before
        i = code.index(start)
        assert "wait_for_predecessors()" in code[i - 300:i]
        return
    part = _between(code, start, end)
    first = re.search(r"\b(mbar_wait|mbar_wait_warp|mbar_try_wait|wait_counter|ld_acquire)\(", part)
    assert first and 0 <= part.find("wait_for_predecessors()") < first.start()


@pytest.mark.parametrize("name,start", [
    ("verify_tc.cuh", "if (clustered) {\n"),
    ("split_gather.cuh", "if (clustered) {\n"),
    ("hsr_fuse.cuh", "if (args.n_slices == 1) {"),
    ("accept_sample.cuh", "accept_sample_kernel(const int32_t*"),
])
def test_a_cluster_meets_before_its_first_push(name, start):
    """Shared memory of another CTA of the cluster may only be written once that CTA is known to run."""
    code = _code(name)
    body = code[code.index(start):]
    push = re.search(r"\b(bulk_push|st_cluster_v4|cluster_sum)\(", body).start()
    assert 0 <= body.find("cluster_wait()") < push


def test_a_warp_is_through_with_its_stores_before_one_lane_hands_them_over():
    """P is stored by all lanes of a warp and handed over by one: every lane's wait and fence stand ahead of that arrival by
    a barrier of the warp, not by the warp happening to be converged."""
    softmax = _code("verify_tc.cuh")
    softmax = softmax[softmax.index("else if (warp < 8) {"):]
    arrivals = [m.start() for m in re.finditer(r"if \(lane == 0\) mbar_arrive\(", softmax)]
    assert len(arrivals) == 3
    for at in arrivals:
        assert re.search(r"tmem_wait_st\(\);\s*tc_fence_before\(\);\s*__syncwarp\(\);\s*$", softmax[:at])


HARNESS = r"""
#include <cstdio>
#include <vector>
#include <algorithm>
#include "common.cuh"
using namespace sparrow;
int main()
{
    for (int tile : {64, 128})
        for (int tiles = 1; tiles <= 300; tiles += tiles < 40 ? 1 : 37)
            for (int ns = 1; ns <= tiles; ++ns) {
                int at = 0;
                std::vector<int> mine, reported;
                for (int split = 0; split < ns; ++split) {
                    const TileRun r = piece_tiles(tiles, ns, split);
                    if (r.first != at || r.count < 1) { std::printf("gap: %d tiles, piece %d of %d\n", tiles, split, ns); return 1; }
                    if (!mine.empty() && r.count > mine.back()) { std::printf("a longer piece behind a shorter one\n"); return 1; }
                    at += r.count;
                    mine.push_back(r.count);
                    for (int rest : {1, tile / 2, tile}) {
                        int b, e;
                        const int n_keys = (tiles - 1) * tile + rest;
                        piece_range(n_keys, ns, split, tile, &b, &e);
                        if (b % tile || e <= b || (split == ns - 1) != (e == n_keys)) { std::printf("piece_range %d %d %d\n", n_keys, ns, split); return 1; }
                        if (rest == tile) reported.push_back((e - b) / tile);
                    }
                }
                if (at != tiles || mine.front() - mine.back() > 1) { std::printf("%d tiles in %d pieces end at %d\n", tiles, ns, at); return 1; }
                std::sort(reported.rbegin(), reported.rend());
                if (reported != mine) { std::printf("other sizes than reported: %d tiles, %d pieces\n", tiles, ns); return 1; }
            }
    std::puts("ok");
    return 0;
}
"""


def test_the_kernels_pieces_tile_the_key_range(tmp_path):
    """The kernels' own rule on the host: no gap, no overlap, whole tiles within one of each other, the longer ones
    first, and the sizes that sparrow_plan_piece_range() reports."""
    src, exe = tmp_path / "pieces.cu", tmp_path / "pieces"
    src.write_text(HARNESS)
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS[:2], "-std=c++17", "-I" + CSRC, "-o", str(exe), str(src)], check=True, timeout=600)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def _one_program(tmp_path, name, text, *flags):
    src, exe = tmp_path / (name + ".cu"), tmp_path / name
    src.write_text(text)
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS[:2], "-std=c++17", "-I" + CSRC, "-I" + os.path.join(build.ROOT, "include"), *flags,
                    "-o", str(exe), str(src)], check=True, timeout=600)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


STAGES = r"""
#include <cstdio>
#include "verify_tc.cuh"
using namespace sparrow::tc;
int main()
{
    for (int nb = 1; nb <= 2; ++nb)
        for (int n = 1; n <= 200; ++n) {
            const int depth = nb == 1 ? 3 : 2, stage = recv_stage(nb, n);
            int last = -1;
            for (int j = 0; j < n; ++j)
                if (j % depth == stage) last = j;
            if (stage < 0 || stage >= depth) { std::printf("no stage: %d blocks, %d tiles\n", nb, n); return 1; }
            if (n < depth ? last != -1 : last != recv_last_tile(nb, n)) { std::printf("%d blocks, %d tiles: last tile %d\n", nb, n, last); return 1; }
            if (nb == 1 && n >= depth && last > n - depth) { std::printf("%d tiles: stage busy until tile %d\n", n, last); return 1; }
        }
    std::puts("ok");
    return 0;
}
"""


def test_rows_of_a_cluster_come_to_a_stage_that_is_idle(tmp_path):
    """The stage that peers write to: unused where the piece does not fill the ring, else free once the tile that the producer
    waits for is through; with one row block that tile is never one of the last two."""
    _one_program(tmp_path, "stages", STAGES)


def test_the_stage_is_released_to_the_peers_behind_its_last_use():
    """The only arrival that makes a used stage of the ring writable for peers orders what was done to it ahead of their
    copies: it stands behind the wait for the stage's last product, and releases."""
    code = _code("verify_tc.cuh")
    kernel = code[code.index("verify_tc_kernel(const"):]
    producer = _between(kernel, "if (warp == kProducerWarp) {", "else if (warp == kMmaWarp)")
    at = producer.index("cluster_arrive();")
    assert 0 <= producer.find("mbar_wait(B.v_empty(recv_stage(NB, n_tiles))") < at
    late = [m.start() for m in re.finditer(r"n_tiles >= NS\)[^;]*cluster_arrive_relaxed\(\)", kernel)]
    assert len(late) == 1 and "!(warp == kProducerWarp && n_tiles >= NS)" in kernel[late[0] - 60:late[0] + 20]       # (everybody else's, at the start)
    assert kernel.count("cluster_arrive();") == 1


def test_no_kind_of_bounded_wait_in_front_of_the_wait_for_the_predecessor():
    """As above, for every wait that the sources define (by name: a function that returns whether it succeeded)."""
    names = sorted(set(re.findall(r"__forceinline__ bool (\w*wait\w*)\(", _code("verify_tc.cuh") + _code("common.cuh"))))
    assert {"mbar_wait", "mbar_wait_tight", "mbar_wait_warp", "mbar_try_wait", "mbar_test_wait", "wait_counter"} <= set(names)
    kernel = _code("verify_tc.cuh")
    kernel = kernel[kernel.index("verify_tc_kernel(const"):]
    for start, end in (("if (warp == kProducerWarp) {", "else if (warp == kMmaWarp)"), ("else if (warp == kMmaWarp) {", "else if (warp == kGateWarp)"),
                       ("else if (warp == kGateWarp) {", "else if (warp < 8)")):
        part = _between(kernel, start, end)
        first = re.search(r"\b(" + "|".join(names) + r"|ld_acquire)\(", part)
        assert first and 0 <= part.find("wait_for_predecessors()") < first.start()
