"""Calls behind other work, eagerly and in a captured graph: the first kernel
of a small call and the sweep of a chunk of rows are launched as programmatic
dependents of whatever is in front of them (a copy, a memset, another kernel,
the join of two streams, an earlier call), and may read nothing that this has
still to write. What is in front is slowed down, so that a kernel that does not
wait for it reads the old inputs; outputs must be those of a call made alone, to
the bit."""

import pytest
import torch

import _parity as P
from paper_2609_08368_gb300 import api
from paper_2609_08368_gb300 import milesloss as ml
from paper_2609_08368_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SLOW = 400_000  # clocks (0.2 ms) before the work in front of a call


def _workload(vocab, traj_len, seed=7):
    return wl.make(wl.shrink(wl.RECIPES["glm"], n_prompts=2, group_size=4, traj_len=traj_len,
                             vocab=vocab, rho_noise=0.3, seed=seed), DEV)


def _buf(w):
    return api.alloc(w.n_rows, int(w.rewards.shape[0]), w.n_groups, DEV, vocab=w.vocab,
                     dlogits_dtype=w.logits.dtype, fill_nan=True)


def _out(buf):
    torch.cuda.synchronize()
    assert ml.rl_loss_check_device_error(buf.workspace) == 0
    return [t.clone().view(torch.uint8) for t in
            (buf.token_logprobs, buf.entropy, buf.advantages, buf.dlogits, buf.stats)]


def _in_front(order, w, src, buf, side, other):
    """Fills w.logits with src on the current stream, in one of the orders."""
    main = torch.cuda.current_stream()
    half = w.n_rows // 2
    if order == "copy":
        torch.cuda._sleep(SLOW)
        w.logits.copy_(src)
    elif order == "kernel":
        torch.cuda._sleep(SLOW)
        torch.mul(src, 1.0, out=w.logits)
    elif order == "memset":
        w.logits.copy_(src)
        torch.cuda._sleep(SLOW)
        buf.workspace.zero_()
    elif order == "join":
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.cuda._sleep(SLOW)
            w.logits[:half].copy_(src[:half])
        w.logits[half:].copy_(src[half:])
        main.wait_stream(side)
    elif order == "event":
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.cuda._sleep(SLOW)
            w.logits.copy_(src)
            done = torch.cuda.Event()
            done.record(side)
        main.wait_event(done)
    elif order == "call":
        w.logits.copy_(src)
        torch.cuda._sleep(SLOW)
        api.fwd_bwd(other, buf)   # the same workspace and outputs, other inputs


def _run(captured, body, again):
    """body() eagerly, or captured and replayed twice (again() in between)."""
    if not captured:
        body()
        return
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        body()
    g.replay()
    again()
    g.replay()


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("order", ["copy", "kernel", "memset", "join", "event", "call"])
@pytest.mark.parametrize("vocab,traj_len", [(4096, 64), (12288, 256), (100000, 16), (12001, 64)])
def test_call_behind(vocab, traj_len, order, captured):
    w, other = _workload(vocab, traj_len), _workload(vocab, traj_len, seed=8)
    src, buf, side = w.logits.clone(), _buf(w), torch.cuda.Stream()
    api.fwd_bwd(w, buf)
    want = _out(buf)

    def stale():
        torch.cuda.synchronize()
        w.logits.copy_(other.logits)
        torch.cuda.synchronize()

    def body():
        _in_front(order, w, src, buf, side, other)
        api.fwd_bwd(w, buf)

    stale()
    _run(captured, body, stale)
    for a, b in zip(_out(buf), want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("order", ["copy", "kernel", "event"])
@pytest.mark.parametrize("vocab", [100000, 28672, 12001])
def test_blocks_of_rows_behind(vocab, order, captured):
    """A chunked call whose blocks of logits are made one at a time, in one
    buffer, in front of their sweeps."""
    w = _workload(vocab, 40)
    src, buf, side, step = w.logits, _buf(w), torch.cuda.Stream(), 96
    api.fwd_bwd_chunked(w, buf, step)
    want = _out(buf)
    block = torch.empty((step, vocab), dtype=src.dtype, device=DEV)

    def body():
        main = torch.cuda.current_stream()
        api._rows_call(w, buf, ml.RL_PHASE_BEGIN, 0, w.n_rows, None, None)
        for r0 in range(0, w.n_rows, step):
            r1 = min(w.n_rows, r0 + step)
            z = block[:r1 - r0]
            if order == "event":
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    torch.cuda._sleep(SLOW)
                    z.copy_(src[r0:r1])
                    done = torch.cuda.Event()
                    done.record(side)
                main.wait_event(done)
            else:
                torch.cuda._sleep(SLOW)
                if order == "copy":
                    z.copy_(src[r0:r1])
                else:
                    torch.mul(src[r0:r1], 1.0, out=z)
            api._rows_call(w, buf, ml.RL_PHASE_ROWS, r0, r1, z, buf.dlogits[r0:r1])
        api._rows_call(w, buf, ml.RL_PHASE_END, 0, w.n_rows, None, None)

    def stale():
        torch.cuda.synchronize()
        block.fill_(1.0)
        buf.dlogits.fill_(float("nan"))
        torch.cuda.synchronize()

    stale()
    _run(captured, body, stale)
    for a, b in zip(_out(buf), want):
        assert torch.equal(a, b)
