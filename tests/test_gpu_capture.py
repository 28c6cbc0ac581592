"""Calls captured into a CUDA graph: every entry point that only enqueues work, replayed on other inputs in the same buffers,
gives the bits of the call itself."""
import numpy as np
import pytest
import torch

from paper_2601_04342_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2601_04342_b200 import build
    build.build()


def _dev(wl, seed):
    x = synth.make_inputs(wl.with_(seed=wl.seed + seed), phi_scale=1.5, v_frame_offsets=True)
    d = {n: x[n].cuda() for n in ("q", "k", "v")}
    d["phi_q"], d["phi_k"] = ({n: t.cuda() for n, t in x[m].items()} for m in ("phi_q", "phi_k"))
    return d


def _fill(to, of):
    for n in ("q", "k", "v"):
        to[n].copy_(of[n])


def _captured(call):
    call()                                                     # attributes, static scratch: before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


BF16 = synth.Workload("capture", 2, 3, 128, 7, 9, 17, 2, 1, "bf16", True, seed=synth.BASE_SEED + 500)
FP32 = synth.Workload("capture32", 1, 24, 128, 7, 15, 20, 1, 1, "fp32", False, seed=synth.BASE_SEED + 510)


@pytest.mark.parametrize("which", ["forward", "qk", "bidirectional", "stream", "stream_qk", "static", "fp32"])
def test_replays_give_the_bits_of_the_call(which):
    from paper_2601_04342_b200 import binding
    wl = FP32 if which == "fp32" else BF16.with_(n_heads=1, B=1) if which == "static" else BF16
    sets = [_dev(wl, s) for s in range(3)]
    d, out = sets[0], torch.empty_like(sets[0]["q"])
    args = (wl.T, wl.H, wl.W, wl.Tc, wl.To)
    qk = which.endswith("qk")
    op = None if which == "static" else binding.for_workload(wl, bidirectional=which == "bidirectional", qk_transform=qk)
    if qk:
        ang = torch.arange(wl.N, dtype=torch.float64)[:, None] * 10000.0 ** (-torch.arange(64, dtype=torch.float64) / 64)[None, :]
        op.set_qk_transform(cos=ang.cos().float().cuda(), sin=ang.sin().float().cuda())

    def call():
        if which == "static":
            binding.forward_static(d["q"], d["k"], d["v"], d["phi_q"], d["phi_k"], *args, dtype=wl.dtype, out=out)
        elif which.startswith("stream"):
            op.stream_begin(wl.B, wl.H, wl.W, wl.Tc, wl.To)
            for f0 in range(0, wl.T, wl.Tc):
                f1 = min(f0 + wl.Tc, wl.T)
                sl = slice(f0 * wl.HW, f1 * wl.HW)
                op.stream_step(d["q"][:, :, sl], d["k"][:, :, sl], d["v"][:, :, sl], d["phi_q"], d["phi_k"], f1 - f0, out=out[:, :, sl])
        else:
            op.forward(d["q"], d["k"], d["v"], d["phi_q"], d["phi_k"], *args, out=out)

    graph = _captured(call)
    for s in (1, 2, 1):
        _fill(d, sets[s])
        out.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        replayed = out.clone()
        out.fill_(float("nan"))
        call()
        torch.cuda.synchronize()
        assert torch.isfinite(out.float()).all() and torch.equal(replayed, out)
    if op is not None:
        assert op.status() == 0
        op.close()
    del graph


def test_a_replay_on_values_that_cannot_be_split_leaves_nothing_behind():
    """Replays carry the epochs of the capture.  One on values of 2^39 and more gives what the call gives, and the replays
    after it are right and run without the CUDA-core kernels again (they take about five times as long here)."""
    from paper_2601_04342_b200 import binding
    wl = FP32.with_(n_heads=60, T=9)
    sets = [_dev(wl, s) for s in range(2)]
    d, out = sets[0], torch.empty_like(sets[0]["q"])
    plain = {n: d[n].clone() for n in ("q", "k", "v")}
    op = binding.for_workload(wl)
    call = lambda: op.forward(d["q"], d["k"], d["v"], d["phi_q"], d["phi_k"], wl.T, wl.H, wl.W, wl.Tc, wl.To, out=out)   # noqa: E731
    graph = _captured(call)
    assert op.last_launches == 7                               # state, read-out and window each on the tensor cores, with their stand-ins

    def timed():
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(); graph.replay(); b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return float(np.median(times))

    def expected():                                            # before any replay: the call carries an epoch of its own
        call()
        return out.clone()

    unsafe = {}
    for name in ("k", "v", "q"):
        _fill(d, plain)
        d[name][0, :, 700, 3] = 2.0 ** 45
        unsafe[name] = (d[name].clone(), expected())
    _fill(d, sets[1])
    other = expected()
    _fill(d, plain)
    before = timed()
    for name in ("k", "v", "q"):
        _fill(d, plain)
        d[name].copy_(unsafe[name][0])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, unsafe[name][1])
    _fill(d, sets[1])
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, other)
    after = timed()
    assert after < 1.5 * before, f"{before:.3f} ms a replay before, {after:.3f} ms after"
    assert op.status() == 0
    op.close()
    del graph
