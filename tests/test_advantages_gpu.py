"""GRPO advantages at the edges of the advantage kernels' split: one
trajectory or thousands (past the shared-memory tables), one row each or
several thousand, groups whose members are scattered, with and without the
one-sample distillation term."""

import numpy as np
import pytest
import torch

import _parity as P
from paper_2609_08368_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n_prompts,group,traj_len", [
    (1, 1, 1), (1, 1, 5000), (1, 3, 2049), (2, 8, 128), (1, 17, 121), (3, 5, 137), (40, 4, 3),
    (256, 2, 5), (512, 4, 1), (700, 5, 1), (3, 1024, 2),
])
@pytest.mark.parametrize("opd", [0.0, 0.3])
def test_grpo_advantages(n_prompts, group, traj_len, opd):
    rec = wl.shrink(wl.RECIPES["tiny"], n_prompts=n_prompts, group_size=group, traj_len=traj_len,
                    vocab=16, reward="normal", mask="prefix_u0_half", teacher_noise=0.2,
                    rho_noise=0.1)
    w = wl.make(rec, DEV)
    rng = np.random.default_rng(n_prompts * 1000 + traj_len)
    w.group_id.copy_(torch.from_numpy(rng.permutation(P.np_(w.group_id))))
    w.loss_mask.copy_(torch.from_numpy((rng.random(w.n_rows) < 0.7).astype(np.uint8)))
    params = dict(w.params, opd_coef=opd)
    g, o = P.run_gpu(w, params=params), P.run_oracle(w, params=params)
    assert g["err"] == 0
    # fp32 of a double computation in both
    np.testing.assert_allclose(g["A"], o["A_traj"], rtol=1e-6, atol=1e-7)
    np.testing.assert_array_equal(g["group_sizes"], o["group_sizes"])
    assert g["stats"]["n_tokens"] == int(w.loss_mask.sum())
    P.assert_dlogits_close(g["dlogits_t"].float().cpu().numpy(), o["dlogits"])


@pytest.mark.parametrize("estimator", ["grpo", "reinforcepp_baseline", "gspo"])
@pytest.mark.parametrize("n_prompts,group", [
    (1, 3007), (1, 3008), (1, 3044), (1, 3045), (1, 3066), (1, 3067),
    (1, 3071), (1, 3072),                            # the last tables of 48 KB, the first past them
    (381, 8), (383, 8),                              # group statistics in a kernel of their own
])
def test_trajectory_tables_at_the_shared_memory_limit(n_prompts, group, estimator):
    """A launch that asks for nothing has 48 KB for the tables and the kernel's
    own shared memory together."""
    rec = wl.shrink(wl.RECIPES["tiny"], n_prompts=n_prompts, group_size=group, traj_len=1, vocab=16,
                    reward="normal", mask="none")
    w = wl.make(rec, DEV)
    params = dict(w.params, estimator=estimator)
    g, o = P.run_gpu(w, params=params), P.run_oracle(w, params=params)
    assert g["err"] == 0
    np.testing.assert_allclose(g["A"], o["A_traj"], rtol=1e-6, atol=1e-7)
    np.testing.assert_array_equal(g["group_sizes"], o["group_sizes"])
    P.assert_dlogits_close(g["dlogits_t"].float().cpu().numpy(), o["dlogits"])
