"""The output tensor that Subgraph.run makes: the same tensor whatever is active on the calling thread."""
import contextlib

import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode

from paper_2212_01005_b200 import workloads as WL

pytestmark = pytest.mark.gpu


class Factories(TorchDispatchMode):
    def __init__(self):
        super().__init__()
        self.seen = []

    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        self.seen.append(str(func))
        return func(*args, **(kwargs or {}))


@contextlib.contextmanager
def deterministic():
    torch.use_deterministic_algorithms(True)
    try:
        yield
    finally:
        torch.use_deterministic_algorithms(False)


CONTEXTS = {"plain": contextlib.nullcontext, "inference": torch.inference_mode, "no_grad": torch.no_grad, "dispatch": Factories,
            "autocast": lambda: torch.autocast("cuda"), "deterministic": deterministic, "stream": lambda: torch.cuda.stream(torch.cuda.Stream()),
            "profiler": lambda: torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU])}


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("name", list(CONTEXTS))
def test_output_tensor(ago, name, fp32):
    if fp32:
        ops = [("conv2d", dict(O=16, R=3, S=3, stride=1, pad=1, groups=16)), ("bias_add", {}), ("relu6", {})]
        wl = WL.Workload("d", [0], [(1, 5, 7, 16)], ops, samples=1)
    else:
        wl = WL.dw_dw("d", [0], 1, 9, 16)
    dtype = torch.float32 if fp32 else torch.bfloat16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    draw = lambda shape, t: torch.randn(shape, generator=gen, device="cuda").to(t)  # noqa: E731
    inputs = [draw(s, dtype) for s in wl.input_shapes]
    weights = [draw(s, torch.float32 if k == "bias" else dtype) for s, k in zip(wl.weight_shapes, wl.weight_kinds)]
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused", dtype=ago.AGO_FP32 if fp32 else ago.AGO_BF16)
    given = torch.full_like(inputs[0], float("nan"))
    sg.run(inputs, weights, out=given)
    torch.cuda.synchronize()
    with CONTEXTS[name]() as active:
        out = sg.run(inputs, weights)
        assert out.is_inference() == (name == "inference")
        if name == "dispatch":
            assert any("empty" in f for f in active.seen)
        torch.cuda.current_stream().synchronize()
    if name == "profiler":
        assert any(e.key == "aten::empty" for e in active.key_averages())
    assert out.shape == given.shape and out.dtype == dtype and out.device == given.device and out.is_contiguous() and not out.requires_grad
    assert out.data_ptr() != given.data_ptr() and torch.equal(out, given)
    sg.close()
