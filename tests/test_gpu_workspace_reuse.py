"""One workspace for calls of different batch bounds and heads, as a program has it that sizes the workspace for its
largest batch and meets a shorter one (GPU only): every call against the oracle."""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

import oracle  # noqa: E402
import parity as P  # noqa: E402
from paper_2607_02612_gb300 import runner  # noqa: E402
from test_gpu_edges import make_batch, make_head  # noqa: E402
from test_gpu_large_batch import gap_tau  # noqa: E402
from workloads import POOL_SPATIAL, StageSpec, make_mlp_head  # noqa: E402

pytestmark = pytest.mark.gpu

BOUNDS = (8192, 4096, 1100, 16000, 2000)   # falling and rising: leftovers of larger and of smaller bounds
DIM = 16


def batch_of(n, dtype):
    return make_batch(np.random.default_rng(n).integers(1, 8, n), DIM, dtype, seed=n, sizes="u1to4")


def tokens_equal(g, o, dtype, nb, label, ids=None):
    """Counts, offsets and kept rows exactly, token rows within the dtype's tolerance."""
    np.testing.assert_array_equal(g["offsets"][:nb + 1], o["offsets"][:nb + 1], err_msg=label)
    t = int(o["offsets"][nb])
    if "keep_idx" in o:
        np.testing.assert_array_equal(g["keep_idx"][:t], o["keep_idx"][:t], err_msg=label)
    np.testing.assert_array_equal(g["sizes"][:t], o["sizes"][:t], err_msg=label)
    if t:
        e = P.rel_err_rows(P.as_float(g["x"], dtype)[:t], P.as_float(o["x"], dtype)[:t])
        assert e.max() <= P.TOL[dtype], (label, float(e.max()))


def run_stage(f, b, spec, label):
    r, rho, head = P.stage_tensors(spec, b.dtype)
    mlp = runner.mlp_head_tensors(spec.mlp_head, b.dtype) if spec.mlp_head is not None else None
    g = P.to_host(f.stage(P.device_batch(b), P.flags_of(spec), r, rho, None if mlp else head, mlp_head=mlp), b.dtype)
    assert int(f.status.item()) == 0, label
    o = oracle.stage(b, spec)
    assert int(g["batch"][0]) == o["n_out"], label
    if spec.exit:
        np.testing.assert_array_equal(g["exit_mask"], o["exit_mask"], err_msg=label)
    np.testing.assert_array_equal(g["ids"][:o["n_out"]], o["ids"], err_msg=label)
    tokens_equal(g, o, b.dtype, o["n_out"], label)


def merge(f, b, rng):
    r = rng.integers(0, 4, b.batch).astype(np.int32)
    g = P.to_host(f.merge(P.device_batch(b), torch.from_numpy(r).cuda()), b.dtype)
    o = oracle.merge(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, r)
    assert int(f.status.item()) == 0
    tokens_equal(g, o, b.dtype, b.batch, f"merge {b.batch}")


def prune(f, b, rng):
    rho = rng.uniform(0.2, 1.0, b.batch).astype(np.float32)
    g = P.to_host(f.prune(P.device_batch(b), torch.from_numpy(rho).cuda()), b.dtype)
    o = oracle.prune(b.dtype, b.offsets, b.x, b.sizes, b.scores, rho)
    assert int(f.status.item()) == 0
    tokens_equal(g, o, b.dtype, b.batch, f"prune {b.batch}")


def compact(f, b, rng):
    mask = (rng.random(b.batch) < 0.3).astype(np.uint8)
    g = P.to_host(f.compact(P.device_batch(b), torch.from_numpy(mask).cuda()), b.dtype)
    o = oracle.compact(b.dtype, b.offsets, b.x, b.sizes, b.scores, mask)
    assert int(f.status.item()) == 0 and int(g["batch"][0]) == o["n_out"]
    np.testing.assert_array_equal(g["ids"][:o["n_out"]], o["ids"])
    tokens_equal(g, o, b.dtype, o["n_out"], f"compact {b.batch}")


def stage(f, b, rng, classes=0, mlp=False):
    spec = StageSpec(True, bool(classes) or mlp, True, r=rng.integers(0, 3, b.batch).astype(np.int32),
                     rho=rng.uniform(0.4, 1.0, b.batch).astype(np.float32))
    if mlp:
        spec.mlp_head = make_mlp_head(rng, POOL_SPATIAL, DIM, 16, 20, b.dtype)
        spec.mlp_head.tau = 2.0
        spec.mlp_head.tau = gap(oracle.stage(b, spec)["max_prob"])
    elif classes:
        spec.head = make_head(DIM, classes, b.dtype, 0.5, scale=0.8)
        spec.head.tau = gap_tau(b, spec.head, 0.4)
    run_stage(f, b, spec, f"stage {b.batch} classes {classes} mlp {mlp}")


def gap(c):
    """A threshold in the widest gap between neighbouring confidences around the median."""
    c = np.sort(c)
    lo = len(c) // 2 - 5
    k = lo + int(np.argmax(np.diff(c[lo:lo + 11])))
    return float(np.float32(0.5 * (float(c[k]) + float(c[k + 1]))))


CALLS = {
    "merge": merge, "prune": prune, "compact": compact, "stage": stage,
    "stage_exit": lambda f, b, rng: stage(f, b, rng, classes=20),
    "stage_wide_head": lambda f, b, rng: stage(f, b, rng, classes=1100),
    "stage_mlp": lambda f, b, rng: stage(f, b, rng, mlp=True),
}


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("call", list(CALLS))
def test_one_workspace_many_bounds(call, dtype):
    """The same call over falling and rising bounds on one workspace."""
    f = runner.Fusion(max(BOUNDS), 1100)
    for k, n in enumerate(BOUNDS):
        CALLS[call](f, batch_of(n, dtype), np.random.default_rng(k))


def test_one_workspace_all_calls():
    """Every call in turn on one workspace, each over another bound than the one before."""
    f = runner.Fusion(max(BOUNDS), 1100)
    for k, call in enumerate([c for _ in range(2) for c in CALLS]):
        CALLS[call](f, batch_of(BOUNDS[k % len(BOUNDS)], "bf16"), np.random.default_rng(k))
