"""A call's kernels start beside one another where that pays (programmatic
dependents); recording events around the sweep makes the same call run them one
after the other. No call may be slower for the overlap. The margin is far above
what one box's timings differ by, and far below what a sweep loses that gets
its places on the GPU in two rounds (20 to 40 %).
The same for the group statistics, which a kernel of their own forms where the
advantage kernel would take longer."""

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
    return best


# rows of 146 KB in clusters of four (few and many advantage CTAs, one row a
# cluster and twenty), 88 KB in clusters of two, the streaming kernel with one, two
# and four CTAs per SM and in clusters, the short-row kernel
@pytest.mark.parametrize("vocab,rows,n_traj", [
    (75008, 128, 64), (75008, 1024, 8), (75008, 4096, 64), (75008, 4096, 512),
    (45056, 4096, 64), (151936, 2048, 64), (32768, 4096, 64), (16384, 8192, 64),
    (262144, 1024, 64), (4096, 8192, 64),
])
@pytest.mark.parametrize("estimator", ["grpo", "reinforcepp"])
def test_overlap_does_not_slow_a_call(vocab, rows, n_traj, estimator):
    rec = wl.shrink(wl.RECIPES["glm"], n_prompts=n_traj // 8, group_size=8,
                    traj_len=rows // n_traj, vocab=vocab)
    w = wl.make(rec, DEV)
    params = dict(w.params, estimator=estimator)
    buf = api.alloc(w.n_rows, n_traj, w.n_groups, DEV, vocab=vocab, dlogits_dtype=w.logits.dtype)

    def call():
        api.fwd_bwd(w, buf, params=params)

    overlapped = _fastest(call)
    ev = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for e in ev:  # (torch makes the events' handles when they are first recorded)
        e.record()
    ml.rl_set_sweep_events(*ev)
    try:
        apart = _fastest(call)
    finally:
        ml.rl_set_sweep_events()
    assert overlapped <= 1.08 * apart, f"{overlapped * 1e3:.1f} us against {apart * 1e3:.1f} one by one"


@pytest.mark.parametrize("estimator,n_traj,few,many", [
    ("reinforcepp_baseline", 2048, 64, 512), ("gspo", 2048, 64, 512), ("grpo", 4096, 16, 256)])
def test_many_groups_cost_little_more_than_few(estimator, n_traj, few, many):
    times = []
    for n_groups in (few, many):
        rec = wl.shrink(wl.RECIPES["glm"], n_prompts=n_groups, group_size=n_traj // n_groups,
                        traj_len=2, vocab=2048)
        w = wl.make(rec, DEV)
        params = dict(w.params, estimator=estimator)
        buf = api.alloc(w.n_rows, n_traj, n_groups, DEV, vocab=2048, dlogits_dtype=w.logits.dtype)
        times.append(_fastest(lambda: api.fwd_bwd(w, buf, params=params)))
    assert times[1] <= 1.5 * times[0], [f"{t * 1e3:.1f} us" for t in times]
