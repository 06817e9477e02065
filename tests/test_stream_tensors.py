"""Tensors that a call allocates for itself (outputs, workspaces, the zeroed
gradient) belong to the stream that the call runs on: on the CPU with stand-ins
for the library and the streams, on the GPU beside a busy current stream."""
import contextlib

import pytest

from tests.gpu_util import rel_l2, to_dev, torch_cuda


class _Stream:
    def __init__(self, handle):
        self.cuda_stream = handle


class _Library:
    def __getattr__(self, name):
        return lambda *args: 0


# call, tensors it allocates, tensors that the caller gets
CALLS = {
    "step": (lambda p, b, x, s: p.step(x, 0.1, stream=s), 2, 1),
    "step_adjoint": (lambda p, b, x, s: p.step_adjoint(x, 0.1, stream=s), 2, 1),
    "step_host": (lambda p, b, x, s: p.step_host(x, x, 0.1, stream=s, blocking=False), 1, 0),
    "grad_depth": (lambda p, b, x, s: p.grad_depth(x, x, 0.1, stream=s), 2, 1),
    "step_backward": (lambda p, b, x, s: p.step_backward(x, x, 0.1, stream=s), 3, 2),
    "batch": (lambda p, b, x, s: b.step(x, stream=s), 2, 1),
}


@pytest.mark.parametrize("call", sorted(CALLS))
def test_call_owned_tensors_are_made_on_the_calls_stream(monkeypatch, call):
    torch = pytest.importorskip("torch")
    from paper_2008_11607_gb300 import rexi

    plan, batch = object.__new__(rexi.Plan), object.__new__(rexi.Batch)
    for obj in (plan, batch):
        obj._lib, obj._h = _Library(), None
    plan.nx = plan.ny = 4
    batch.workspace_bytes = 256
    x = torch.zeros(3, 4, 4, dtype=torch.complex128)
    current, side = _Stream(1), _Stream(2)
    active, made, kept = [current], [], []

    @contextlib.contextmanager
    def on(stream):
        active.append(stream)
        yield
        active.pop()

    def record(fn):
        def wrapped(*args, **kw):
            made.append(active[-1])
            if kw.get("device") == "cuda":
                kw["device"] = "cpu"
            return fn(*args, **kw)
        return wrapped

    monkeypatch.setattr(torch.cuda, "Stream", _Stream)
    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: active[-1])
    for name in ("empty", "empty_like", "zeros"):
        monkeypatch.setattr(torch, name, record(getattr(torch, name)))
    monkeypatch.setattr(torch.Tensor, "new_empty", record(torch.Tensor.new_empty))
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda t, s: kept.append(s))
    fn, count, returned = CALLS[call]
    fn(plan, batch, x, side)
    assert made == [side] * count
    assert kept == [current] * returned  # what the caller keeps, it uses on its own stream
    del made[:], kept[:]
    fn(plan, batch, x, None)
    assert made == [current] * count and kept == []


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["grad_depth", "step_backward"])
def test_gradient_on_a_side_stream_beside_a_busy_current_stream(call):
    """The current stream has work queued when the call on the side stream runs."""
    torch = torch_cuda()
    from paper_2008_11607_gb300 import inputs, rexi

    nx, ny = 40, 21
    H = torch.from_numpy(inputs.variable_depth(nx, ny, seed=3)).cuda()
    plan = rexi.Plan(nx, ny, depth=H)
    plan.set_krylov(rtol=1e-12)
    plan.set_krylov_method("shared")
    dt = 10.0 / plan.rho
    x = to_dev(torch, inputs.white_real_state(nx, ny, seed=2))
    g = to_dev(torch, inputs.white_real_state(nx, ny, seed=4))
    ref = plan.step_backward(x, g, dt)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)  # some 50 ms
    got = getattr(plan, call)(x, g, dt, stream=side)
    side.synchronize()
    torch.cuda.synchronize()
    got = got if call == "step_backward" else (ref[0], got)
    for a, b in zip(got, ref):
        assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) < 1e-13
