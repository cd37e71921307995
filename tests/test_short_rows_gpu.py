"""The short-row sweep against the cluster kernel it stands in for: every
output the same to the bit, at the edges of its shapes (rows of one vector, of
exactly 4, 8, 16 KB and a vector more, with and without elements past the last
whole vector), and against the oracle."""

import numpy as np
import pytest
import torch

import _parity as P
from paper_2609_08368_gb300 import milesloss as ml
from paper_2609_08368_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _same(a, b):
    for k in ("logp", "H", "A"):
        np.testing.assert_array_equal(a[k], b[k])
    assert a["stats"] == b["stats"] and a["err"] == b["err"]
    if "dlogits_t" in a:
        assert torch.equal(a["dlogits_t"].view(torch.uint8), b["dlogits_t"].view(torch.uint8))


@pytest.mark.parametrize("dtype,vocab,ld,dl", [
    ("bf16", 3, 8, "bf16"), ("bf16", 8, 8, "bf16"), ("bf16", 2048, 2048, "bf16"),
    ("bf16", 2055, 2056, "bf16"), ("bf16", 4096, 4104, "f32"), ("bf16", 4101, 4104, "bf16"),
    ("bf16", 8192, 8192, "bf16"), ("bf16", 8200, 8200, "f32"), ("bf16", 10239, 10240, "bf16"),
    ("f32", 5, 8, "f32"), ("f32", 1024, 1024, "f32"), ("f32", 1030, 1032, "f32"),
    ("f32", 2052, 2052, "bf16"), ("f32", 4097, 4100, "f32"), ("f32", 5119, 5120, "f32"),
])
def test_short_rows_match_the_cluster_kernel(dtype, vocab, ld, dl):
    rec = wl.shrink(wl.RECIPES["fp32" if dtype == "f32" else "glm"], n_prompts=2, group_size=3,
                    traj_len=7, vocab=vocab, rho_noise=0.3, mask="prefix_u0_half")
    w = wl.make(rec, DEV, ld=ld)
    if vocab > 100:
        w.logits[2, :40] = -float("inf")  # a first vector of -inf, an overflow of the reference
        w.logits[4, vocab - 1] = 300.0
        w.targets[2], w.targets[4] = 50, vocab - 1
    w.targets[0] = vocab                  # a bad target: an error and a row of zeros
    ddt = torch.float32 if dl == "f32" else torch.bfloat16
    for mode in ("fused", "split"):
        a = P.run_gpu(w, mode=mode, dl_dtype=ddt, grad_loss=0.7, ld_out=ld)
        with ml.launch_overrides(sweep_kernel="cluster"):
            b = P.run_gpu(w, mode=mode, dl_dtype=ddt, grad_loss=0.7, ld_out=ld)
        a["dlogits_t"], b["dlogits_t"] = (x["dlogits_t"][:, :vocab].contiguous() for x in (a, b))
        _same(a, b)
        assert a["err"] == 5


@pytest.mark.parametrize("vocab,K", [(1000, 1), (3001, 40), (8000, 64), (10000, 16)])
def test_short_rows_topk(vocab, K):
    rec = wl.shrink(wl.RECIPES["glm"], n_prompts=1, group_size=4, traj_len=6, vocab=vocab, topk=K,
                    rho_noise=0.3, mask="none")
    w = wl.make(rec, DEV, ld=-(-vocab // 8) * 8)
    w.topk_ids[5, K - 1] = -1
    params = dict(w.params, opd_topk=K, opd_coef=0.5)
    a = P.run_gpu(w, params=params)
    with ml.launch_overrides(sweep_kernel="cluster"):
        b = P.run_gpu(w, params=params)
    # (the compiler contracts the two kernels' sums past the last vector
    # differently here: an ulp of a log-prob or entropy)
    for k in ("logp", "H"):
        np.testing.assert_allclose(a[k], b[k], rtol=3e-7, atol=1e-6)
    P.assert_dlogits_close(a["dlogits_t"][:, :vocab].float().cpu().numpy(),
                           b["dlogits_t"][:, :vocab].float().cpu().numpy())
    assert a["err"] == b["err"] == 9


def test_short_rows_more_rows_than_the_first_wave():
    """Later CTAs take the advantages early; the oracle checks both kinds."""
    rec = wl.shrink(wl.RECIPES["glm"], n_prompts=2, group_size=4, traj_len=700, vocab=512)
    w = wl.make(rec, DEV)
    g, o = P.run_gpu(w), P.run_oracle(w)
    np.testing.assert_allclose(g["logp"], o["logp"], atol=P.logp_tol(w), rtol=0)
    P.assert_dlogits_close(g["dlogits_t"].float().cpu().numpy(), o["dlogits"])
