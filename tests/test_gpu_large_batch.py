"""Batches beyond one wave of CTAs (GPU only): the exit check in tiles of 16, 32 and 64 samples, the
compaction plan in tiles, and the per-sample kernels that read it, against the oracle."""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

import oracle  # noqa: E402
import parity as P  # noqa: E402
import paper_2607_02612_gb300 as fz  # noqa: E402
from paper_2607_02612_gb300 import runner  # noqa: E402
from test_gpu_edges import make_batch, make_head, run_stage_and_compare  # noqa: E402
from workloads import StageSpec  # noqa: E402

pytestmark = pytest.mark.gpu


def gap_tau(b, head, share):
    """tau in the widest gap near the upper `share` of the oracle's confidences: no decision at it."""
    c = np.sort(oracle.exit_check(b.dtype, b.offsets, b.x, head)["max_prob"])[::-1]
    k = max(1, int(share * len(c)))
    at = range(max(1, k - 4), min(len(c), k + 5))
    k = max(at, key=lambda j: c[j - 1] - c[j])
    return float(np.float32(0.5 * (float(c[k - 1]) + float(c[k]))))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("batch,classes,dim", [
    (2433, 10, 16),       # 16-sample tiles, a short last K-block
    (2440, 128, 80),      # a whole class tile
    (9729, 100, 384),     # 64-sample tiles of one class tile, a ragged last tile
    (313, 1000, 384),     # 16-sample tiles, clusters of 8, a short last class tile
    (641, 257, 1024),     # the widest rows, three class tiles
])
def test_exit_check_many_samples(dtype, batch, classes, dim):
    b = make_batch(np.full(batch, 1), dim, dtype, seed=batch)
    head = make_head(dim, classes, dtype, 0.5, scale=3.0 / np.sqrt(dim))
    head.tau = gap_tau(b, head, 0.3)
    f = runner.Fusion(batch, classes)
    g = P.to_host(f.exit_check(P.device_batch(b), runner.head_tensors(head, dtype)), dtype)
    assert int(f.status.item()) == 0
    rep = P.Report()
    P.compare_exit(rep, dtype, np.arange(batch), g["exit_mask"], g["logits"], g["max_prob"],
                   oracle.exit_check(dtype, b.offsets, b.x, head))
    rep.check()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("batch,classes,merge,prune", [
    (1025, 20, True, True), (1025, 1100, True, False), (2500, 20, True, True), (4300, 0, True, True),
    (1060, 0, False, True), (2500, 20, False, False)])
def test_stage_with_tiled_plan(dtype, batch, classes, merge, prune):
    """Batches above the fused plan's bound: the plan after either exit kernel, or alone."""
    rng = np.random.default_rng(batch)
    b = make_batch(rng.integers(1, 24, batch), 64, dtype, seed=batch, sizes="u1to4")
    head = None
    if classes:
        head = make_head(64, classes, dtype, 0.5, scale=0.4)
        head.tau = gap_tau(b, head, 0.4)
    r = rng.integers(0, 12, batch).astype(np.int32) if merge else None
    rho = rng.uniform(0.2, 1.0, batch).astype(np.float32) if prune else None
    run_stage_and_compare(b, StageSpec(merge, head is not None, prune, r=r, rho=rho, head=head),
                          f"B={batch} C={classes}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("count,classes", [(0, 20), (1, 20), (37, 20), (1088, 20), (37, 0)])
def test_tiled_plan_device_count(dtype, count, classes):
    """A device batch count below the host bound, with ids: only its samples are planned."""
    batch = 1100
    rng = np.random.default_rng(count)
    b = make_batch(rng.integers(1, 20, batch), 64, dtype, seed=7)
    db = P.device_batch(b)
    db.batch = torch.tensor([count], dtype=torch.int32, device="cuda")
    ids = rng.permutation(batch).astype(np.int32)
    db.ids = torch.from_numpy(ids).cuda()
    head = make_head(64, 20, dtype, 0.5, scale=0.4)
    head.tau = gap_tau(b, head, 0.4)
    r = rng.integers(0, 9, batch).astype(np.int32)
    rho = rng.uniform(0.2, 1.0, batch).astype(np.float32)
    f = runner.Fusion(batch, 20)
    flags = 7 if classes else 5
    o = f.stage(db, flags, torch.from_numpy(r).cuda(), torch.from_numpy(rho).cuda(),
                runner.head_tensors(head, dtype) if classes else None)
    torch.cuda.synchronize()
    assert int(f.status.item()) == 0
    nb = int(o["batch"][0])
    if count == 0:
        assert nb == 0 and int(o["offsets"][0]) == 0
        return
    sub = make_batch(np.diff(b.offsets)[:count], 64, dtype)
    t = int(b.offsets[count])
    sub.x, sub.keys, sub.sizes, sub.scores = b.x[:t], b.x[:t], b.sizes[:t], b.scores[:t]
    ref = oracle.stage(sub, StageSpec(True, bool(classes), True, r=r[ids[:count]], rho=rho[ids[:count]],
                                      head=head if classes else None))
    assert nb == ref["n_out"]
    np.testing.assert_array_equal(o["offsets"][:nb + 1].cpu().numpy(), ref["offsets"])
    np.testing.assert_array_equal(o["ids"][:nb].cpu().numpy(), ids[ref["ids"]])
    rows = int(ref["offsets"][-1])
    np.testing.assert_array_equal(o["keep_idx"][:rows].cpu().numpy(), ref["keep_idx"])


def test_tiled_plan_rejects_malformed_offsets():
    """One bad sample among many: the status bit, an empty output batch, no token row written."""
    b = make_batch(np.full(1200, 8), 64, "bf16", seed=3)
    db = P.device_batch(b)
    offs = db.offsets.clone()
    offs[700] = int(offs[699]) - 1
    db.offsets = offs
    f = runner.Fusion(1200, 20)
    head = runner.head_tensors(make_head(64, 20, "bf16", 0.5), "bf16")
    for flags in (5, 7):
        f.status.zero_()
        o = f.stage_outputs(db, 7, head)
        o["x"].fill_(7)
        f.stage(db, flags, torch.full((1200,), 2, dtype=torch.int32, device="cuda"),
                torch.full((1200,), 0.5, device="cuda"), head, out=o)
        torch.cuda.synchronize()
        assert int(f.status.item()) & fz.FUSION_DEV_BAD_OFFSETS
        assert int(o["batch"][0]) == 0 and int(o["offsets"][0]) == 0 and torch.all(o["x"] == 7)


@pytest.mark.parametrize("counts,dim,keys,kdim", [
    ([65, 64, 33, 34, 17, 3, 2, 1] * 2, 384, "alias", None),     # one wave, clusters; tile edges
    ([65, 64, 33, 34, 17, 3, 2, 1] * 50, 80, "alias", None),     # 400 samples: small CTAs, a short stage
    ([66, 40, 5] * 120, 64, "separate", 48),                     # just past the small kernel
    ([197, 98, 1, 130], 384, "separate", 400),                   # clusters of 8, two norm blocks
    ([197, 196] * 60, 32, "alias", None),                        # clusters of 2
    ([129, 128, 113] * 110, 16, "alias", None),                  # one CTA per sample, several tiles per warp
    ([577, 300], 1024, "alias", None),                           # long samples, narrow stages
    ([650, 1], 64, "separate", 96)])
def test_float32_merge_tiles(counts, dim, keys, kdim):
    b = make_batch(counts, dim, "f32", seed=len(counts), keys=keys, kdim=kdim, sizes="u1to4")
    rng = np.random.default_rng(1)
    r = np.minimum(rng.integers(0, 40, len(counts)), np.asarray(counts) // 2).astype(np.int32)
    rho = rng.uniform(0.3, 1.0, len(counts)).astype(np.float32)
    run_stage_and_compare(b, StageSpec(True, False, True, r=r, rho=rho), f"{counts[:4]} x {len(counts)}")


@pytest.mark.parametrize("counts,dim,keys,kdim", [
    ([65, 64, 33, 17, 3, 2, 1] * 45, 384, "alias", None),       # 315 samples: four stages, some stay resident
    ([129, 128, 97, 9] * 77, 192, "separate", 128),             # the longest samples of the small CTAs
    ([130, 65] * 153, 64, "alias", None),                       # one token past them
    ([33, 1] * 520, 1024, "alias", None)])                      # with the tiled plan, wide rows
def test_bf16_merge_small_ctas(counts, dim, keys, kdim):
    b = make_batch(counts, dim, "bf16", seed=len(counts), keys=keys, kdim=kdim, sizes="u1to4")
    rng = np.random.default_rng(2)
    r = np.minimum(rng.integers(0, 40, len(counts)), np.asarray(counts) // 2).astype(np.int32)
    rho = rng.uniform(0.3, 1.0, len(counts)).astype(np.float32)
    run_stage_and_compare(b, StageSpec(True, False, True, r=r, rho=rho), f"{counts[:4]} x {len(counts)}")


@pytest.mark.parametrize("counts,dim", [
    ([258, 257, 259, 300, 17, 1], 128),      # one pass, two M-tiles; short samples in the same call
    ([513, 514, 512, 258], 64),              # two M-tiles of 128 rows exactly, one row over, three
    ([577, 640, 641, 130], 192),             # three M-tiles: passes of 160 columns, the last ones ragged
    ([769, 770, 771, 300], 64),              # four M-tiles: passes of 128
    ([900, 860], 128), ([1024, 3], 64),      # the longest samples, and those the general kernel takes
    ([962, 947, 3, 300], 320)])              # two stages next to the metadata, refilled in turn
def test_bf16_merge_long_samples(counts, dim):
    b = make_batch(counts, dim, "bf16", seed=len(counts), sizes="u1to4")
    rng = np.random.default_rng(3)
    r = np.minimum(rng.integers(20, 200, len(counts)), np.asarray(counts) // 2).astype(np.int32)
    rho = rng.uniform(0.3, 1.0, len(counts)).astype(np.float32)
    run_stage_and_compare(b, StageSpec(True, False, True, r=r, rho=rho), f"{counts}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("counts,dim,prune", [
    ([197, 1, 2, 130], 768, True), ([90, 17, 33] * 25, 112, True), ([1024, 5], 16, True),
    ([65, 3] * 200, 384, True), ([40, 1, 7] * 30, 1024, False),
    ([600, 5], 768, True), ([300, 225, 2] * 40, 64, True), ([260, 1, 450] * 30, 1024, True)])   # 512 threads, 512, 256
def test_prune_and_compact_column_parts(dtype, counts, dim, prune):
    """A sample's columns shared by several CTAs (few samples), and one CTA per sample (many)."""
    b = make_batch(counts, dim, dtype, seed=len(counts), sizes="u1to4")
    rng = np.random.default_rng(4)
    rho = rng.uniform(0.2, 1.0, len(counts)).astype(np.float32) if prune else None
    run_stage_and_compare(b, StageSpec(False, False, prune, rho=rho), f"{counts[:4]} x {len(counts)} d={dim}")


@pytest.mark.parametrize("batch,dim", [(3, 128), (40, 272), (2440, 128), (9729, 80), (641, 272)])
def test_layernorm_rounds_once(batch, dim):
    """The exit check's LayerNorm in every tile size: with identity weights the logits are its bf16 rows,
    each of which is the nearest bf16 value to the 64-bit one (beta cancels much of many elements).  The
    slack is the float-float evaluation's relative error, 2^-40 of the terms."""
    g = torch.Generator().manual_seed(batch)
    x = (torch.randn((batch, dim), generator=g) * 3 + torch.randn((batch, 1), generator=g)).bfloat16()
    gamma = (1 + 0.3 * torch.randn(dim, generator=g)).bfloat16()
    beta = torch.randn(dim, generator=g).bfloat16()
    eps = float(np.float32(1e-6))
    xc = x.cuda()
    b = runner.DeviceBatch("bf16", dim, batch, 1, batch, xc, xc, torch.ones(batch, device="cuda"), None,
                           torch.arange(batch + 1, dtype=torch.int32, device="cuda"))
    head = runner.HeadTensors(gamma.cuda(), beta.cuda(), eps, torch.eye(dim).bfloat16().cuda(), torch.zeros(dim).cuda(), 1e-6)
    f = runner.Fusion(batch, dim)
    o = f.exit_check(b, head)
    assert int(f.status.item()) == 0 and bool(o["exit_mask"].all())
    u = o["logits"].cpu()
    xd = x.double()
    d = xd - xd.mean(1, keepdim=True)
    v = d / torch.sqrt((d * d).mean(1, keepdim=True) + eps) * gamma.double()
    want = v + beta.double()
    assert torch.equal(u, u.bfloat16().float())
    err = (u.double() - want).abs()
    slack = 2.0 ** -40 * (v.abs() + beta.double().abs())
    bits = u.bfloat16().view(torch.int16)
    for step in (-1, 1):
        other = (bits + step).view(torch.bfloat16).double()
        ok = (err <= (other - want).abs() + slack) | ~torch.isfinite(other)
        assert bool(ok.all()), int((~ok).sum())
