"""Which per-sample kernel a call takes, over batch bounds, lengths and widths (the host's choice; no GPU needed).

The forms give the same results, so a wrong choice shows only in the time: the expected routes are the ones measured
to be no slower than the general kernel (float32), or than CTAs of 256 threads (bf16), at the sizes on each side."""
import importlib
import os
import subprocess

import pytest

B = importlib.import_module("paper_2607_02612_gb300.build")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "launch.h"
// float32: F tokens key_dim batch known -> ok cluster; bf16: T tokens key_dim batch -> ok tiled threads
int main(int argc, char **argv) {
    for (int k = 1; k + 4 < argc; k += 5) {
        const int tokens = atoi(argv[k + 1]), dim = atoi(argv[k + 2]), batch = atoi(argv[k + 3]), known = atoi(argv[k + 4]);
        if (argv[k][0] == 'F') {
            fz::ImageParams p{};
            p.in.max_batch = batch;
            p.in.max_tokens = tokens;
            p.in.max_rows = (long long)batch * tokens;
            p.dim = p.kdim = dim;
            p.do_merge = 1;
            p.kc = fz::image_geometry(FUSION_F32, tokens, dim, 1).kc;
            static const unsigned char mask = 0;
            p.plan_args.exit_mask = known ? nullptr : &mask;
            const fz::F32Geometry g = fz::image_f32_geometry(p);
            printf("%d %d\n", g.ok, g.cluster);
        } else {
            const fz::TcGeometry g = fz::image_tc_geometry(FUSION_BF16, tokens, dim, dim, (long long)batch * tokens, 1, 111, batch);
            printf("%d %d %d\n", g.ok, g.tiled, g.threads);
        }
    }
}
"""


@pytest.fixture(scope="module")
def routes(tmp_path_factory):
    """A function from queries (kind, tokens, dim, batch, known) to the printed choices."""
    d = tmp_path_factory.mktemp("routes")
    (d / "routes.cu").write_text(PROGRAM)
    lib = os.path.dirname(B.build())
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", f"-I{B.INCLUDE}", f"-I{B.CSRC}", "-o", str(d / "routes"), str(d / "routes.cu"),
                    f"-L{lib}", "-lfusion", "-Xlinker", f"-rpath={lib}"], check=True, capture_output=True)

    def ask(queries):
        out = subprocess.run([str(d / "routes"), *[str(v) for q in queries for v in q]], check=True, capture_output=True, text=True)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return ask


def test_float32_merges_leave_the_general_kernel_only_where_measured_faster(routes):
    """0: the general kernel; else CTAs per sample of the streamed one."""
    expected = {
        # (tokens, key width, batch bound, everyone known to continue)
        (65, 384, 76, 0): 2, (65, 384, 77, 0): 1, (65, 1024, 152, 0): 1, (66, 384, 153, 0): 1, (65, 48, 8192, 0): 1,
        # with an exit check
        (197, 384, 15, 0): 8, (197, 384, 16, 0): 8, (197, 768, 30, 0): 8, (300, 192, 31, 0): 4, (300, 48, 19, 0): 4,
        (100, 768, 37, 0): 4, (100, 768, 72, 0): 4, (100, 768, 73, 0): 2, (150, 384, 76, 0): 2, (577, 192, 72, 0): 4,
        (577, 192, 73, 0): 2, (700, 384, 60, 0): 4, (700, 384, 76, 0): 2, (257, 48, 73, 0): 0, (700, 48, 60, 0): 0,
        (100, 384, 77, 0): 2, (100, 384, 114, 0): 2, (100, 384, 115, 0): 0, (197, 384, 152, 0): 2, (577, 384, 100, 0): 2, (300, 384, 152, 0): 2, (150, 1024, 100, 0): 2,
        (80, 1024, 77, 0): 0, (129, 768, 152, 0): 0, (257, 384, 100, 0): 0, (400, 192, 100, 0): 0, (577, 48, 100, 0): 0,
        (800, 192, 100, 0): 0, (100, 1024, 153, 0): 0, (300, 384, 200, 0): 0, (197, 384, 304, 0): 0, (80, 384, 200, 0): 1,
        (80, 768, 200, 0): 0, (80, 384, 400, 0): 1, (100, 384, 457, 0): 1, (197, 192, 2000, 0): 1, (257, 192, 608, 0): 0,
        (577, 48, 608, 0): 0, (129, 48, 64, 0): 2, (130, 48, 64, 0): 0, (80, 80, 153, 0): 0, (80, 192, 153, 0): 1,
        # without
        (197, 384, 15, 1): 8, (197, 384, 16, 1): 4, (100, 768, 36, 1): 4, (100, 768, 37, 1): 2, (197, 192, 37, 1): 4,
        (577, 192, 72, 1): 4, (700, 384, 37, 1): 2, (150, 384, 76, 1): 2, (300, 48, 76, 1): 0, (129, 48, 76, 1): 2,
        (80, 48, 77, 1): 0, (100, 384, 100, 1): 0, (197, 192, 152, 1): 0, (577, 384, 100, 1): 2, (300, 192, 77, 1): 2,
        (257, 192, 77, 1): 0, (100, 384, 200, 1): 1, (197, 384, 304, 1): 1, (197, 384, 400, 1): 0, (257, 192, 200, 1): 0,
        (700, 192, 305, 1): 0,
    }
    got = routes([("F", *q) for q in expected])
    for (q, want), (ok, cluster) in zip(expected.items(), got):
        assert (cluster if ok else 0) == want, q


def test_long_bf16_merges_stay_on_the_tensor_cores(routes):
    """Every length past one tile up to 962 tokens (two stages and the metadata fill an SM's shared memory)."""
    lengths = range(258, 963)
    for n, (ok, tiled, _) in zip(lengths, routes([("T", n, 384, 64, 0) for n in lengths])):
        assert ok and tiled, n


def test_small_bf16_ctas_only_where_measured_faster(routes):
    """Threads of a CTA over (tokens, width, batch bound): four CTAs per SM, three, or too much shared memory."""
    expected = {
        (65, 384, 304): 256, (65, 384, 305): 128, (100, 192, 305): 128, (65, 768, 323): 256, (65, 768, 324): 128,
        (33, 1024, 305): 128, (17, 1024, 8192): 128,
        (100, 384, 323): 256, (100, 384, 324): 128, (100, 384, 456): 128, (100, 384, 457): 256, (100, 384, 1024): 256,
        (100, 384, 1025): 128, (100, 768, 456): 128, (100, 768, 1025): 256, (129, 192, 500): 256, (129, 192, 2500): 128,
        (129, 64, 500): 128, (129, 384, 2500): 256, (130, 64, 2500): 256, (197, 384, 2500): 256,
    }
    for (q, want), (ok, _, threads) in zip(expected.items(), routes([("T", *q, 0) for q in expected])):
        assert ok and threads == want, q
