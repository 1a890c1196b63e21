"""The workspace's layout: the counters that must be zero when a call begins lie where no other call on the
same workspace puts data, whatever the two calls' batch bounds and class counts (host arithmetic only)."""
import importlib
import subprocess

B = importlib.import_module("paper_2607_02612_gb300.build")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "common.cuh"
int main(int argc, char **argv) {
    for (int k = 1; k + 1 < argc; k += 2) {
        const fz::WsLayout L = fz::ws_layout(atoi(argv[k]), atoi(argv[k + 1]));
        const size_t at[5] = {L.cnt, L.plan, L.partials, L.lg, L.total};
        size_t end = L.total;   // of the counters: where the next block begins
        for (size_t v : at)
            if (v > L.counters && v < end) end = v;
        printf("%zu %zu %zu\n", L.counters, end, L.total);
    }
}
"""


def test_counters_are_out_of_reach_of_other_bounds(tmp_path):
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(PROGRAM)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", f"-I{B.INCLUDE}", f"-I{B.CSRC}", "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    calls = [(b, c) for b in (0, 1, 7, 1025, 1100, 4096, 8192, 100000, 524280) for c in (1, 1000, 1100, 4000)]
    out = subprocess.run([str(exe), *[str(v) for bc in calls for v in bc]], check=True, capture_output=True, text=True)
    layouts = [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    assert len(layouts) == len(calls)
    for (b1, c1), (lo, end, _) in zip(calls, layouts):
        used = lo + 4 * (1 + -(-max(b1, 1) // 8))   # the plan's counter and one per tile of 8 samples
        assert used <= end, (b1, c1)
        for (b2, c2), (lo2, end2, total2) in zip(calls, layouts):
            # the other call's data: everything of its own layout but its counters
            for d0, d1 in ((0, lo2), (end2, total2)):
                assert used <= d0 or d1 <= lo, f"counters of {b1} x {c1} lie in the data of {b2} x {c2}"
