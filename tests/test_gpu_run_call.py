"""The native call behind `Subgraph.run`: what it returns, which stream it uses, when it attaches a workspace, how it fails."""
import os
import subprocess
import sys
import threading

import pytest

from paper_2212_01005_b200 import workloads as WL
from helpers import to_device

pytestmark = pytest.mark.gpu


def handle(ago, wl, mode="fused"):
    return ago.Subgraph(wl.ops, wl.input_shapes, mode=mode), to_device(wl, WL.generate(wl))


def test_run_returns_the_given_output_and_allocates_its_own(ago):
    import torch
    sg, (ins, ws) = handle(ago, WL.pw_pw("call", [301], 2, 9, 64, 32, 64))
    own = sg.run(ins, ws)
    given = torch.empty_like(own)
    assert sg.run(ins, ws, out=given) is given
    assert sg.run(tuple(ins), tuple(ws)).shape == sg.output_shape
    torch.cuda.synchronize()
    assert torch.equal(own, given) and own.dtype == torch.bfloat16
    sg.close()


def test_run_attaches_a_workspace_and_uses_the_stream_it_is_given(ago):
    import torch
    sg, (ins, ws) = handle(ago, WL.ffn("call_ffn", [302], 512, 768, 3072, 1))
    assert sg.workspace_bytes > 0
    ref = sg.run(ins, ws)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    a = sg.run(ins, ws, stream=side.cuda_stream)
    with torch.cuda.stream(side):
        b = sg.run(ins, ws)
    torch.cuda.synchronize()
    scale = float(ref.float().abs().max())
    for o in (a, b):          # the additions arrive in any order: one bf16 step
        assert float((o.float() - ref.float()).abs().max()) <= 2.0 ** -7 * scale
    assert sg.status() == ago.AGO_OK
    sg.close()


def test_run_rejects_what_it_cannot_launch(ago):
    sg, (ins, ws) = handle(ago, WL.pw_pw("call_bad", [303], 1, 8, 64, 32, 64))
    with pytest.raises(ago.AgoError):
        sg.run(ins, ws[:-1])                      # a weight short
    with pytest.raises(ago.AgoError):
        sg.run([t.cpu() for t in ins], ws)        # no CPU path
    with pytest.raises((TypeError, IndexError)):
        sg.run([], ws)
    sg.close()


def test_run_from_two_threads_on_streams_of_their_own(ago):
    import torch
    sg0, (ins0, ws0) = handle(ago, WL.pw_pw("call_t0", [304], 4, 20, 96, 24, 96))
    sg1, (ins1, ws1) = handle(ago, WL.mbv2_block("call_t1", [305], 2, 14, 32, 192, 32, 1, True))
    refs = [sg0.run(ins0, ws0), sg1.run(ins1, ws1)]
    torch.cuda.synchronize()
    outs = [[], []]

    def work(k, sg, ins, ws):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(50):
                outs[k].append(sg.run(ins, ws))
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=work, args=a) for a in ((0, sg0, ins0, ws0), (1, sg1, ins1, ws1))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert all(torch.equal(o, refs[0]) for o in outs[0])
    scale = float(refs[1].float().abs().max())    # chunks are added in the order the groups finish: one bf16 step
    assert all(float((o.float() - refs[1].float()).abs().max()) <= 2.0 ** -7 * scale for o in outs[1])
    sg0.close(); sg1.close()


@pytest.mark.parametrize("wl", [
    WL.pw_pw("call_many", [309], 1, 6, 64, 32, 64), WL.mbv2_block("call_many", [310], 1, 12, 64, 96, 64, 1, True), WL.attention("call_many", [311], 1, 32, 1, 64),
    WL.Workload("call_many", [312], [(1, 5, 6, 16)], WL.resnet_block("x", [0], 1, 8, 16).ops, samples=1), WL.unfold_chain("call_many", [313], 1, 4, 9, 32, 64),
], ids=["pw_pw", "block", "attention", "residual", "unfold"])
def test_one_handle_from_two_threads_on_new_addresses(ago, wl):
    # every run meets addresses that the handle has not seen: the two threads' runs change what it remembers about them at once
    import torch
    runs = 300
    sg, (ins, ws) = handle(ago, wl)
    ref = sg.run(ins, ws)

    def copies(t):      # the tensor at `runs` places, 256 bytes apart or more
        step = -(-t.numel() * t.element_size() // 256) * 256 // t.element_size()
        flat = torch.zeros(runs * step, dtype=t.dtype, device=t.device).view(runs, step)
        flat[:, :t.numel()] = t.flatten()
        return [flat[i, :t.numel()].view(t.shape) for i in range(runs)]

    places = [[copies(t) for t in ins + ws] for _ in range(2)]
    torch.cuda.synchronize()
    outs, start = [[], []], threading.Barrier(2)

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            for i in range(runs):
                args = [p[i] for p in places[k]]
                outs[k].append(sg.run(args[:len(ins)], args[len(ins):]))
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert sg.status() == ago.AGO_OK and [len(o) for o in outs] == [runs, runs]
    scale = float(ref.float().abs().max())
    for o in outs[0] + outs[1]:
        assert float((o.float() - ref.float()).abs().max()) <= 2.0 ** -7 * scale      # the block's chunks: one bf16 step
    sg.close()


def test_run_takes_whatever_has_a_device_and_an_address(ago):
    # arrays of another library, more weights than the handle reads, a stream as a ctypes pointer
    import ctypes
    import torch

    class Array:
        def __init__(self, t, device):
            self.t, self.device = t, device

        def data_ptr(self):
            return self.t.data_ptr()

    stream = torch.cuda.current_stream().cuda_stream
    for wl in (WL.pw_pw("call_duck", [306], 1, 8, 64, 32, 64), WL.ffn("call_duck_ffn", [307], 64, 128, 256, 1)):
        sg, (ins, ws) = handle(ago, wl)
        ref = sg.run(ins, ws)
        outs = [sg.run([Array(t, t.device) for t in ins], [Array(w, w.device) for w in ws]), sg.run([Array(t, torch.device("cuda")) for t in ins], ws),
                sg.run(ins, ws + [ws[0]] * 100), sg.run(ins, ws, stream=ctypes.c_void_p(stream or None))]
        torch.cuda.synchronize()
        assert sg.status() == ago.AGO_OK
        scale = float(ref.float().abs().max())
        for o in outs:
            assert float((o.float() - ref.float()).abs().max()) <= 2.0 ** -7 * scale      # split sums arrive in any order: one bf16 step
        sg.close()
    with pytest.raises(ago.AgoError):
        sg2, (ins, ws) = handle(ago, wl)
        sg2.run([Array(t.cpu(), torch.device("cpu")) for t in ins], ws)


FOREIGN = """
import ctypes
import numpy as np
import torch
from oracle import oracle as O
from paper_2212_01005_b200 import binding as B, workloads as WL

rt = ctypes.CDLL("libcudart.so.12")      # the one torch has loaded

class Array:
    device = "cuda:0"
    def __init__(self, a):
        a = np.ascontiguousarray(a)
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)) == 0
        assert rt.cudaMemcpy(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes), 1) == 0
        self.address = p.value
    def data_ptr(self):
        return self.address

wl = WL.pw_pw("call_foreign", [308], 1, 8, 64, 32, 64)
data = WL.generate(wl)
bf16 = lambda a: (np.ascontiguousarray(a, np.float32).view(np.uint32) >> 16).astype(np.uint16)      # the values are bf16 numbers
ins = [Array(bf16(a)) for a in data["inputs"]]
ws = [Array(a.astype(np.float32) if k == "bias" else bf16(a)) for a, k in zip(data["weights"], wl.weight_kinds)]
sg = B.Subgraph(wl.ops, wl.input_shapes, mode="fused")
out = sg.run(ins, ws)
ref = O.run_chain(wl.ops, data["inputs"], data["weights"])
got = out.double().cpu().numpy()
assert sg.status() == B.AGO_OK and tuple(out.shape) == sg.output_shape
assert abs(got - ref).max() <= 1e-2 * abs(ref).max() + 1e-3
"""


def test_run_is_the_first_that_asks_torch_for_the_device():
    # a process whose arrays are all another library's: nothing has initialised torch's CUDA state when the output is made
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FOREIGN], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
