"""Launches that may start before the kernel ahead of them has finished: chains of calls in
which each one consumes what the one before it wrote, queued without a pause, give the bits of
the same calls made one at a time."""
import numpy as np
import pytest

import rqc_inputs as ri

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def chain(qfx, S, B, dims, precision, variant, pause):
    """Steps of K = N through S[i], each on the output of the one before; all outputs."""
    P, K, Sd = dims
    outs, b = [], B
    for s in S:
        b = qfx.contract_step(s, b, P, K, K, K, Sd, precision=precision, variant=variant)
        if pause:
            qfx.sync()
        outs.append(b)
    qfx.sync()
    return outs


@pytest.mark.parametrize("precision,variant,dims", [
    ("bf16x3", 13, (3, 64, 1030)), ("bf16x3", -1, (3, 64, 1030)), ("tf32x3", 13, (129, 32, 130)),
    ("bf16x2", 13, (1, 128, 20003)), ("bf16x3", -1, (16, 64, 2048)), ("bf16x3", 12, (3, 64, 1030)),
    ("fp32", -1, (3, 64, 1031)), ("fp32", -1, (5, 24, 130))])
def test_steps_on_the_output_of_the_step_before(qfx, precision, variant, dims):
    """Rows that no tensor map describes are read by per-thread loads, and Sd that is no
    multiple of 16 makes row tiles share 128-byte lines."""
    P, K, Sd = dims
    S = [torch.from_numpy(ri.random_complex(K * K, seed=30 + i) / np.float32(np.sqrt(2 * K))).cuda() for i in range(6)]
    B = torch.from_numpy(ri.random_complex(P * K * Sd, seed=29)).cuda()
    want = chain(qfx, S, B, dims, precision, variant, True)
    for _ in range(4):
        for a, b in zip(chain(qfx, S, B, dims, precision, variant, False), want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("precision,bound", [("bf16x3", 1e-5), ("tf32x3", 3e-5)])
def test_chunks_added_into_the_result(qfx, precision, bound):
    """A contraction of K = 4096 takes four launches, each of which adds into what the one
    before wrote: the same bits every time, and the FP32 plan's amplitudes within the mode's
    bound."""
    c = ri.rqc(5, 5, 32, seed=2)
    x1 = torch.tensor(ri.random_bitstrings(25, 2, seed=3).view(np.int64), device="cuda")
    plan = qfx.Plan(qfx.Circuit(c), n_open=2, family="tree", precision=precision)
    assert any(s["K"] == 4096 and s["variant"] >= 10 for s in plan.steps)
    ws = torch.empty(plan.workspace_bytes(2), dtype=torch.uint8, device="cuda")
    first = qfx.amplitudes(plan, x1, workspace=ws)
    for _ in range(4):
        assert torch.equal(qfx.amplitudes(plan, x1, workspace=ws), first)
    ref = qfx.amplitudes(qfx.Plan(qfx.Circuit(c), n_open=2, family="tree"), x1)
    qfx.sync()
    err = (first - ref).abs()
    assert bool((err <= bound * torch.clamp(ref.abs(), min=2.0 ** -12.5)).all()), float(err.max())


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_inputs_from_two_streams(qfx, precision):
    """A step whose operands come from two streams that join before it, called directly and
    from a captured graph replayed with other values."""
    P, K, N, Sd = 3, 64, 64, 4096
    s0, b0 = (torch.from_numpy(ri.random_complex(n, seed=7)).cuda() for n in (K * N, P * K * Sd))
    scratch = torch.empty(max(256, qfx.qfx.step_scratch_bytes(K, N, precision)), dtype=torch.uint8, device="cuda")
    S, B, out = torch.empty_like(s0), torch.empty_like(b0), torch.empty(P * N * Sd, dtype=torch.complex64, device="cuda")
    main, side = torch.cuda.Stream(), torch.cuda.Stream()

    def work():
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.mul(b0, 2.0, out=B)
            torch.add(B, b0, out=B)
        with torch.cuda.stream(main):
            torch.mul(s0, 0.5, out=S)
            main.wait_stream(side)
            qfx.contract_step(S, B, P, K, N, N, Sd, precision=precision, out=out, scratch=scratch)

    def want():
        ref = qfx.contract_step(0.5 * s0, 2.0 * b0 + b0, P, K, N, N, Sd, precision=precision)
        qfx.sync()
        return ref

    def check():
        torch.cuda.synchronize()
        assert torch.equal(out, want())

    torch.cuda.synchronize()
    for _ in range(3):
        work()
        check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        work()
    for i in range(3):
        s0.copy_(torch.from_numpy(ri.random_complex(K * N, seed=40 + i)))
        b0.copy_(torch.from_numpy(ri.random_complex(P * K * Sd, seed=50 + i)))
        torch.cuda.synchronize()
        graph.replay()
        check()
