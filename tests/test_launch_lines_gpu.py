"""Calls that the launch rules send to one kernel or form, timed against the one
they could have taken: on either side of a line the rule's choice must not be
the slower one by more than a margin that is above what timings on one box
differ by."""

import pytest
import torch

from paper_2609_08368_gb300 import api
from paper_2609_08368_gb300 import milesloss as ml
from paper_2609_08368_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _fastest(call, reps=5, n=12):
    best = float("inf")
    for _ in range(3):
        call()
    for _ in range(reps):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        for _ in range(n):
            call()
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1) / n)
    return best * 1e3


def _at(rows, cols, off, like):
    """A [rows, cols] tensor that starts `off` elements past a 16-byte boundary."""
    return torch.empty(off + rows * cols, dtype=like, device=DEV)[off:].view(rows, cols)


def _batch(dtype, rows, vocab, off, off_out, topk=0):
    rec = wl.shrink(wl.RECIPES["fp32" if dtype == "f32" else "glm"], n_prompts=2, group_size=8,
                    traj_len=rows // 16, vocab=vocab, topk=topk)
    w = wl.make(rec, DEV)
    z = _at(rows, vocab, off, w.logits.dtype).copy_(w.logits)
    w = wl.Workload(**{**w.__dict__, "logits": z})
    if topk:
        w.params = dict(w.params, opd_topk=topk, opd_coef=0.2)
    buf = api.alloc(rows, 16, w.n_groups, DEV, vocab=vocab, dlogits_dtype=w.logits.dtype)
    buf.dlogits = _at(rows, vocab, off_out, w.logits.dtype)
    return w, buf


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_gradient_of_rows_misaligned_against_each_other(dtype):
    """Element by element where dLogits lie differently from the logits: at most
    so much slower than the vectors of rows that lie alike (3.7 to 4.7 times)."""
    times = []
    for off, off_out in ((1, 1), (3, 0)):
        w, buf = _batch(dtype, 4096, 16632, off, off_out)
        api.fwd(w, buf)
        times.append(_fastest(lambda: api.bwd(w, buf)))
    assert times[1] <= 5.2 * times[0], times


@pytest.mark.parametrize("dtype,vocab,off,topk,mode", [
    ("bf16", 201, 1, 0, "fused"), ("bf16", 201, 1, 8, "fused"), ("bf16", 511, 1, 8, "fwd"),
    ("bf16", 1537, 1, 0, "fused"), ("bf16", 3001, 1, 8, "fused"), ("bf16", 1025, 1, 0, "fwd"),
    ("bf16", 320, 0, 0, "fused"), ("bf16", 2048, 0, 8, "fused"), ("bf16", 3072, 0, 0, "fused"),
    ("f32", 1025, 1, 0, "fused"), ("f32", 1025, 1, 0, "fwd"), ("f32", 3001, 1, 8, "fused")])
def test_short_unaligned_rows_take_the_faster_kernel(dtype, vocab, off, topk, mode):
    """Logits that start `off` elements past a boundary, dLogits that do too
    (or, where the logits are aligned, two elements past one)."""
    w, buf = _batch(dtype, 16384, vocab, off, off or 2, topk)
    call = (lambda: api.fwd_bwd(w, buf)) if mode == "fused" else (lambda: api.fwd(w, buf))
    chosen = _fastest(call)
    with ml.launch_overrides(sweep_kernel="cluster"):
        other = _fastest(call)
    assert chosen <= 1.06 * other, (chosen, other)


@pytest.mark.parametrize("dtype,vocab,topk,mode", [
    ("bf16", 8192, 64, "fused"), ("bf16", 9216, 16, "fused"), ("bf16", 9216, 64, "fused"),
    ("bf16", 9216, 32, "fwd"), ("bf16", 9216, 64, "fwd"), ("f32", 4608, 32, "fused"),
    ("f32", 4608, 64, "fused")])
def test_short_rows_with_topk_take_the_faster_kernel(dtype, vocab, topk, mode):
    w, buf = _batch(dtype, 16384, vocab, 0, 0, topk)
    call = (lambda: api.fwd_bwd(w, buf)) if mode == "fused" else (lambda: api.fwd(w, buf))
    chosen = _fastest(call)
    with ml.launch_overrides(sweep_kernel="cluster"):
        other = _fastest(call)
    assert chosen <= 1.06 * other, (chosen, other)


def test_gradient_sweep_of_fp32_rows_runs_at_the_copy_rate():
    """Of 32,768 rows x 32,768: its bytes (the training rows' logits, every
    dLogit) in little more than the time a copy of as many takes."""
    w = wl.make(wl.shrink(wl.RECIPES["fp32"], n_prompts=64, group_size=8, traj_len=64), DEV)
    buf = api.alloc(w.n_rows, 512, w.n_groups, DEV, vocab=w.vocab, dlogits_dtype=w.logits.dtype)
    api.fwd(w, buf)
    sweep = _fastest(lambda: api.bwd(w, buf), reps=8)
    trains = float((w.loss_mask != 0).float().mean())
    half = int(w.logits.numel() * (1 + trains) / 2)  # elements read, and as many written
    src, dst = w.logits.view(-1)[:half], buf.dlogits.view(-1)[:half]
    copy = _fastest(lambda: dst.copy_(src), reps=8)
    assert sweep <= 1.04 * copy, (sweep, copy)
