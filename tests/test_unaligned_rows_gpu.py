"""Rows that do not start on a 16-byte boundary, in the logits or in dLogits:
every misalignment of both, against the float64 oracle and, bit for bit in the
row statistics, against the same rows in a padded, aligned tensor."""

import numpy as np
import pytest
import torch

import _parity as P
from paper_2609_08368_gb300 import api
from paper_2609_08368_gb300 import milesloss as ml
from paper_2609_08368_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SENTINEL = 3.0


def _offset(rows, ld, off, dtype, fill):
    """A [rows, ld] tensor that starts `off` elements into its buffer, which
    holds `fill` before and after it."""
    big = torch.full((off + rows * ld + 64,), fill, dtype=dtype, device=DEV)
    return big, big[off:off + rows * ld].view(rows, ld)


# vocabularies at the edges of the launch plans (bytes of a bf16 row: one
# vector and a bit, the short rows, 24, 40 and 56 KB with four CTAs per SM, 66
# and 100 KB with two, 150 KB as halves, 200 and 250 KB with one, 500 KB on a
# cluster); (elements the logits and dLogits start past a boundary, padding of ld
# and ld_out)
@pytest.mark.parametrize("dtype,vocab,off,pad,off_out,pad_out,dl", [
    ("bf16", 11, 1, 0, 1, 0, "bf16"),
    ("bf16", 2047, 3, 0, 3, 0, "bf16"),
    ("bf16", 12001, 0, 0, 0, 0, "bf16"),
    ("bf16", 20003, 5, 2, 5, 2, "bf16"),
    ("bf16", 28671, 7, 1, 2, 0, "bf16"),    # dLogits misaligned against the logits
    ("bf16", 33001, 0, 7, 0, 7, "f32"),
    ("bf16", 50001, 2, 0, 2, 0, "bf16"),
    ("bf16", 75003, 1, 0, 0, 5, "bf16"),
    ("bf16", 100003, 6, 0, 6, 0, "bf16"),
    ("bf16", 125004, 0, 4, 4, 0, "bf16"),   # aligned logits, misaligned dLogits
    ("bf16", 250001, 1, 0, 1, 0, "bf16"),
    ("f32", 3001, 1, 0, 1, 0, "f32"),
    ("f32", 10002, 2, 0, 3, 0, "f32"),
    ("f32", 33003, 3, 0, 1, 0, "bf16"),
    ("f32", 40001, 0, 0, 0, 0, "f32"),
])
def test_unaligned_rows(dtype, vocab, off, pad, off_out, pad_out, dl):
    rec = wl.shrink(wl.RECIPES["fp32" if dtype == "f32" else "glm"], n_prompts=1, group_size=3,
                    traj_len=5, vocab=vocab, rho_noise=0.3, mask="none")
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    ddt = torch.float32 if dl == "f32" else torch.bfloat16
    al = -(-vocab // 8) * 8 + 8
    w = wl.make(rec, DEV, ld=al)
    w.logits[2, :3] = -float("inf")   # exact path, at a row's start ...
    w.logits[3, vocab - 2:vocab] = -float("inf")
    w.logits[4, 4] = 300.0            # ... and an overflow of the running reference
    w.targets[:5] = torch.tensor([0, vocab - 1, 4, 4, 4])
    want = P.run_gpu(w, mode="fwd")
    big, z = _offset(w.n_rows, vocab + pad, off, tdt, float("nan"))
    z[:, :vocab] = w.logits[:, :vocab]
    wu = wl.Workload(**{**w.__dict__, "logits": z})
    o = P.run_oracle(w)
    for mode in ("fused", "split"):
        buf = api.alloc(w.n_rows, 3, 1, DEV, vocab=vocab, dlogits_dtype=ddt)
        bigd, buf.dlogits = _offset(w.n_rows, vocab + pad_out, off_out, ddt, SENTINEL)
        if mode == "fused":
            api.fwd_bwd(wu, buf)
        else:
            api.fwd(wu, buf)
            api.bwd(wu, buf)
        torch.cuda.synchronize()
        assert ml.rl_loss_check_device_error(buf.workspace) == 0
        got = dict(logp=P.np_(buf.token_logprobs), H=P.np_(buf.entropy))
        tol = P.logp_tol(w)
        np.testing.assert_allclose(got["logp"], o["logp"], atol=tol, rtol=1e-6)
        np.testing.assert_allclose(got["H"], o["H"], atol=tol, rtol=1e-6)
        if mode == "split" and dtype == "bf16" and vocab * 2 >= 20 * 1024:
            # (streamed either way: summed in the same order)
            np.testing.assert_array_equal(got["logp"], want["logp"])
            np.testing.assert_array_equal(got["H"], want["H"])
        P.assert_dlogits_close(buf.dlogits[:, :vocab].float().cpu().numpy(), o["dlogits"])
        # nothing outside the rows' columns is written
        assert (buf.dlogits[:, vocab:] == SENTINEL).all()
        assert (bigd[:off_out] == SENTINEL).all() and (bigd[-64:] == SENTINEL).all()


def test_unaligned_topk_and_vocab_shards():
    """Top-K candidates are gathered through the shift; a column shard whose
    columns start at an odd id is unaligned too."""
    rec = wl.shrink(wl.RECIPES["glm"], n_prompts=1, group_size=2, traj_len=8, vocab=30001, topk=16,
                    rho_noise=0.3, mask="none")
    w = wl.make(rec, DEV)
    params = dict(w.params, opd_topk=16, opd_coef=0.5)
    g = P.run_gpu(w, params=params)
    assert g["err"] == 0
    al = wl.Workload(**{**w.__dict__, "logits": torch.nn.functional.pad(w.logits, (0, 7))})
    a = P.run_gpu(al, params=params)
    tol = P.logp_tol(w)
    np.testing.assert_allclose(g["logp"], a["logp"], atol=tol, rtol=0)
    P.assert_dlogits_close(g["dlogits_t"].float().cpu().numpy(),
                           a["dlogits_t"][:, :30001].float().cpu().numpy())
    cols, shards = [0, 14999, 30001], []
    for k in range(2):
        wk = wl.Workload(**{**w.__dict__, "logits": w.logits[:, cols[k]:cols[k + 1]]})
        buf = api.alloc(w.n_rows, 2, 1, DEV, vocab=cols[k + 1] - cols[k],
                        dlogits_dtype=torch.bfloat16)
        shards.append(api.VocabShard(wk, k, cols, buf, params=params))
    api.vocab_sharded_fwd_bwd_local([shards])
    torch.cuda.synchronize()
    for s in shards:
        assert ml.rl_loss_check_device_error(s.buf.workspace) == 0
    np.testing.assert_allclose(P.np_(shards[0].buf.token_logprobs), g["logp"], atol=tol, rtol=0)
    both = torch.cat([s.buf.dlogits for s in shards], 1).float().cpu().numpy()
    P.assert_dlogits_close(both, g["dlogits_t"].float().cpu().numpy())


@pytest.mark.parametrize("vocab,off,topk", [
    (1025, 0, 0), (3001, 1, 0), (10002, 2, 0), (18435, 3, 0), (20001, 0, 8), (20482, 1, 0),
    (40001, 0, 0), (65539, 1, 0), (70001, 0, 0), (130003, 2, 0),
])
@pytest.mark.parametrize("mode", ["fused", "split"])
def test_unaligned_fp32_keeps_the_cluster_kernels_sums(vocab, off, topk, mode):
    """One, two, four and eight virtual slices, slices that end inside a
    chunk, a row's last elements in a slice of their own: every output as the
    cluster kernel has it."""
    rec = wl.shrink(wl.RECIPES["fp32"], n_prompts=1, group_size=3, traj_len=37 if vocab < 9000 else 5,
                    vocab=vocab, topk=topk)
    w = wl.make(rec, DEV)
    w.logits[1, :300] = -float("inf")
    w.targets[1] = vocab - 1
    w.logits[3, vocab // 2] = 120.0
    w.targets[3] = vocab // 2
    _, z = _offset(w.n_rows, vocab, off, torch.float32, float("nan"))
    z.copy_(w.logits)
    w = wl.Workload(**{**w.__dict__, "logits": z})
    params = dict(w.params, **(dict(opd_topk=topk, opd_coef=0.4) if topk else {}))
    got = P.run_gpu(w, mode=mode, params=params)
    with ml.launch_overrides(sweep_kernel="cluster"):
        want = P.run_gpu(w, mode=mode, params=params)
    assert got["err"] == want["err"] == 0
    if topk:  # (the candidates' parts merge in another order)
        np.testing.assert_allclose(got["logp"], want["logp"], rtol=3e-7, atol=1e-6)
        P.assert_dlogits_close(P.np_(got["dlogits_t"]), P.np_(want["dlogits_t"]))
        return
    np.testing.assert_array_equal(got["logp"], want["logp"])
    np.testing.assert_array_equal(got["H"], want["H"])
    assert torch.equal(got["dlogits_t"], want["dlogits_t"])


@pytest.mark.parametrize("dtype,vocab", [("f32", 10001), ("bf16", 20001)])
def test_unaligned_nan_stays_in_its_row(dtype, vocab):
    """A NaN logit reaches its own dLogit (as in an aligned row) and no other
    row's outputs."""
    rec = wl.shrink(wl.RECIPES["fp32" if dtype == "f32" else "glm"], n_prompts=1, group_size=2,
                    traj_len=6, vocab=vocab, mask="none")
    w = wl.make(rec, DEV)
    clean = P.run_gpu(w)
    w.logits[5, 777] = float("nan")
    got = P.run_gpu(w)
    rest = [r for r in range(w.n_rows) if r != 5]
    np.testing.assert_array_equal(got["logp"][rest], clean["logp"][rest])
    assert torch.isnan(got["dlogits_t"][5, 777])
    assert torch.equal(got["dlogits_t"][rest], clean["dlogits_t"][rest])
