"""Failure detection and context hygiene, without faulting or hanging anything.

* A bounded device-side wait that runs out: the failure-injection build of the attention kernel
  (its producer stops early, its waits give up after 4096 polls) must return, report
  RAPID3_ERR_TIMEOUT through the status word, and leave the context usable.
* The tensor-map cache of a context: one context fed more distinct buffers than it has cache
  slots must keep computing with the right tensors.
* A call whose launch is refused reports it once: the next call starts without it."""
import ctypes
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2509_22323_b200 import binding, inputs
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda"
POISON = 0x7FC1
ERR_CUDA, ERR_TIMEOUT = -4, -5


def poison_like(t):
    return torch.full(t.shape, POISON, dtype=torch.int16, device=t.device).view(torch.bfloat16)


@pytest.mark.parametrize("D,stop_group", [(128, 0), (128, 2), (128, 5), (64, 1), (64, 3)])
def test_wait_that_runs_out_sets_the_status_and_returns(D, stop_group):
    wl = inputs.Workload("timeout", 2, 2, D, 64, 16, 2.0, (0.5, 1.0), rope=(D == 128), seed=91)   # nb = 5
    Q, K, V = inputs.make_qkv(wl, 0, device=DEV)
    ctx = binding.Context(wl.batch, wl.heads, wl.head_dim, wl.n_text, wl.n_image)
    acts, ratios = [2, 2], [0.5, 1.0]
    want = poison_like(Q)
    ctx.rapid3_gated_step(Q, K, V, want, acts, ratios, wl.softmax_scale)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0

    scratch = poison_like(Q)
    ctx.rapid3_debug_inject_timeout(Q, K, V, scratch, stop_group, wl.softmax_scale)
    torch.cuda.synchronize()                       # the kernel returned: nothing waits for ever
    assert ctx.last_status() == ERR_TIMEOUT
    assert ctx.last_status() == 0                  # reading the status cleared it
    assert (scratch[1].view(torch.int16) == np.int16(POISON)).all()     # only image 0 was launched

    # the context still computes: bit-identical to before the failure, and right against the oracle
    out = poison_like(Q)
    ctx.rapid3_gated_step(Q, K, V, out, acts, ratios, wl.softmax_scale)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert torch.equal(out.view(torch.int16), want.view(torch.int16))
    ref = oracle.gated_step(Q.cpu(), K.cpu(), V.cpu(), acts, ratios, wl.n_text, wl.softmax_scale)
    for b in range(2):
        parity.compare_outputs(out[b], ref[b]["out"], f"after a timeout, img {b}")


@pytest.mark.parametrize("D,n_blocks,stop_group", [(64, 40, 0), (64, 40, 2), (64, 40, 40), (128, 36, 0), (128, 36, 1), (128, 36, 3)])
def test_a_wait_that_runs_out_leaves_rows_in_parts_unwritten(D, n_blocks, stop_group):
    """A context whose attention works on lists in parts: a launch that has given up adds up neither the parts of the call before
    nor memory that nothing has written.  The launch after it does."""
    gen = torch.Generator(device=DEV).manual_seed(n_blocks)
    q, k, v = (torch.randn((1, 2, 64 * n_blocks, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    ctx = binding.Context(1, 2, D, 64, 64 * (n_blocks - 1))
    want = None
    for _ in range(2):                             # on a new context, and after a call that has left its parts
        n0, scratch = ctx.launch_count(), poison_like(q)
        ctx.rapid3_debug_inject_timeout(q, k, v, scratch, stop_group)
        torch.cuda.synchronize()
        assert ctx.launch_count() - n0 == 2        # attention, sum of the parts
        assert ctx.last_status() == ERR_TIMEOUT
        assert (scratch.view(torch.int16) == np.int16(POISON)).all()
        out = poison_like(q)
        ctx.rapid3_sparse_joint_attn(q, k, v, out)
        torch.cuda.synchronize()
        assert ctx.last_status() == 0
        want = out if want is None else want
        assert torch.equal(out.view(torch.int16), want.view(torch.int16))
    ref = (q[0].double() @ k[0].double().transpose(1, 2) * D ** -0.5).softmax(-1) @ v[0].double()
    assert float((want[0].double() - ref).abs().max()) <= 2 ** -7 * float(v.abs().max())    # P and the result rounded to bf16


@pytest.mark.parametrize("D,n_blocks,H,stop_group", [(64, 6, 3, 0), (64, 6, 3, 5), (64, 21, 2, 1), (64, 21, 2, 20), (64, 21, 2, 21),
                                                     (128, 8, 3, 0), (128, 19, 2, 2), (128, 19, 2, 18), (128, 19, 2, 19)])
def test_a_wait_that_runs_out_by_turns(D, n_blocks, H, stop_group):
    """A context whose tiles take the key blocks by turns: the copies stop before the first block, or so late that one of the two tiles has
    all of its own.  Neither waits for good for what the other would hand it, nothing is written, and the steps after it are whole."""
    gen = torch.Generator(device=DEV).manual_seed(n_blocks)
    q, k, v = (torch.randn((1, H, 64 * n_blocks, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    ctx = binding.Context(1, H, D, 64, 64 * (n_blocks - 1))
    want = {}
    for ratio in (1.0, 0.5):
        want[ratio] = poison_like(q)
        ctx.rapid3_gated_step(q, k, v, want[ratio], [2], [ratio])
    for _ in range(2):
        n0, scratch = ctx.launch_count(), poison_like(q)
        ctx.rapid3_debug_inject_timeout(q, k, v, scratch, stop_group)
        torch.cuda.synchronize()
        assert ctx.launch_count() - n0 == 1
        assert ctx.last_status() == ERR_TIMEOUT
        assert ctx.last_status() == 0
        assert (scratch.view(torch.int16) == np.int16(POISON)).all()
        for ratio in (1.0, 0.5):
            out = poison_like(q)
            ctx.rapid3_gated_step(q, k, v, out, [2], [ratio])
            torch.cuda.synchronize()
            assert ctx.last_status() == 0
            assert torch.equal(out.view(torch.int16), want[ratio].view(torch.int16))
    ref = (q[0].double() @ k[0].double().transpose(1, 2) * D ** -0.5).softmax(-1) @ v[0].double()
    assert float((want[1.0][0].double() - ref).abs().max()) <= 2 ** -7 * float(v.abs().max())    # P and the result rounded to bf16


@pytest.mark.parametrize("D", [64, 128])
def test_a_wait_that_ran_out_does_not_delay_the_end_by_the_sequence(D):
    """512 key blocks: 256 thread blocks, two rounds of them, each over after 4096 polls and 16 more for each of the next 32
    key blocks at most, under 10 us a poll: 92 ms.  (256 polls at every key block that was left took 0.5 s.)"""
    q = torch.randn((1, 2, 512 * 64, D), device=DEV).to(torch.bfloat16)
    out = torch.zeros_like(q)
    ctx = binding.Context(1, 2, D, 0, 512 * 64)
    took = []
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx.rapid3_debug_inject_timeout(q, q, q, out, 1)
        torch.cuda.synchronize()
        took.append(time.perf_counter() - t0)
        assert ctx.last_status() == ERR_TIMEOUT
    assert min(took) < 0.2, took


def test_injection_entry_refuses_bad_arguments():
    ctx = binding.Context(1, 1, 64, 64, 256)
    Q = torch.zeros((1, 1, 320, 64), dtype=torch.bfloat16, device=DEV)
    for bad in (-1, 6):
        with pytest.raises(binding.Rapid3Error):
            ctx.rapid3_debug_inject_timeout(Q, Q, Q, Q, bad)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0


def test_one_context_many_distinct_buffers():
    """Fixed Q, K, V and a new output tensor per call -- more distinct base pointers than the context
    caches tensor maps for -- then fresh Q/K/V as well: every call must equal a fresh context's result."""
    wl = inputs.Workload("maps", 2, 2, 128, 64, 16, 2.0, (0.5, 1.0), rope=True, seed=93)
    acts, ratios = [2, 2], [0.5, 1.0]
    Q, K, V = inputs.make_qkv(wl, 0, device=DEV)
    fresh = binding.Context(wl.batch, wl.heads, wl.head_dim, wl.n_text, wl.n_image)
    want = poison_like(Q)
    fresh.rapid3_gated_step(Q, K, V, want, acts, ratios, wl.softmax_scale)
    torch.cuda.synchronize()
    ctx = binding.Context(wl.batch, wl.heads, wl.head_dim, wl.n_text, wl.n_image)
    outs = [poison_like(Q) for _ in range(12)]
    assert len({o.data_ptr() for o in outs}) == 12
    for o in outs:
        ctx.rapid3_gated_step(Q, K, V, o, acts, ratios, wl.softmax_scale)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    for n, o in enumerate(outs):
        assert torch.equal(o.view(torch.int16), want.view(torch.int16)), f"call {n}"
    # rotate all four tensors
    for step in range(1, 6):
        Q2, K2, V2 = inputs.make_qkv(wl, step, device=DEV)
        a, b = poison_like(Q2), poison_like(Q2)
        ctx.rapid3_gated_step(Q2, K2, V2, a, acts, ratios, wl.softmax_scale)
        other = binding.Context(wl.batch, wl.heads, wl.head_dim, wl.n_text, wl.n_image)
        other.rapid3_gated_step(Q2, K2, V2, b, acts, ratios, wl.softmax_scale)
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"step {step}"
    ref = oracle.gated_step(Q.cpu(), K.cpu(), V.cpu(), acts, ratios, wl.n_text, wl.softmax_scale)
    for b in range(2):
        parity.compare_outputs(outs[-1][b], ref[b]["out"], f"many buffers img {b}")


def test_a_refused_launch_is_reported_once():
    """A call on a stream whose capture has been invalidated is refused by the runtime; the call after it, on a sound
    stream, is not."""
    wl = inputs.Workload("refused", 1, 2, 64, 64, 8, 2.0, (0.5,), seed=95)
    Q, K, V = inputs.make_qkv(wl, 0, device=DEV)
    out = torch.zeros_like(Q)
    ctx = binding.Context(wl.batch, wl.heads, wl.head_dim, wl.n_text, wl.n_image)
    ctx.rapid3_gated_step(Q, K, V, out, [2], [0.5], wl.softmax_scale)
    torch.cuda.synchronize()
    want = out.clone()
    delta = V.clone()
    cudart = ctypes.CDLL("libcudart.so.12")                  # torch's own, already loaded
    stream = torch.cuda.Stream()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    for ratio in (0.5, 1.0):                                 # the pooling kernel is the first to be refused, then the attention
        assert cudart.cudaStreamBeginCapture(handle, 1) == 0     # thread-local mode
        assert cudart.cudaStreamSynchronize(handle) != 0         # not permitted: the capture is invalid from here on
        with torch.cuda.stream(stream), pytest.raises(binding.Rapid3Error) as e:
            ctx.rapid3_gated_step(Q, K, V, out, [2], [ratio], wl.softmax_scale)
        assert e.value.code == ERR_CUDA
        assert cudart.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0
        cudart.cudaGetLastError()
        binding.rapid3_cache_step(Q, out, delta, [2])        # judged by the last error of the library's own runtime
    out.zero_()
    ctx.rapid3_gated_step(Q, K, V, out, [2], [0.5], wl.softmax_scale)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert torch.equal(out.view(torch.int16), want.view(torch.int16))
