"""Calls of one context on several streams: compress calls of different workers side by side, and whole steps on streams that the
caller orders by events.  Every run is compared bit for bit with the same calls one after the other."""
import os
import subprocess
import sys

import pytest
import torch

import paper_2411_19870_b200 as demo

pytestmark = pytest.mark.gpu

W = 3
# name, shapes, chunk size or chunk shapes, k, caller-supplied basis: more chunks than a grid has CTAs or slots (chunks on demand)
SETS = {
    "s64_and_vectors": ([(4096, 2048), (2048,), (128, 64)], 64, 32, False),
    "s32": ([(2048, 4096)], 32, 8, False),
    "s128": ([(4096, 4096), (512,)], 128, 32, False),
    "s64_basis": ([(4096, 4096)], 64, 32, True),
    "nd_classes": ([(1024, 512, 3, 3), (9000, 512), (640,)], [(16, 16, 3, 3), (15, 64), (20,)], 12, False),
}


class Run:
    def __init__(self, name):
        shapes, chunk, k, basis = SETS[name]
        kw = dict(chunk=chunk) if isinstance(chunk, int) else dict(chunk_shapes=chunk)
        self.tr = demo.DemoTransform(shapes, topk=k, beta=0.9, lr=1e-3, weight_decay=0.1, num_workers=W, **kw)
        if basis:
            gen = torch.Generator().manual_seed(1)
            self.tr.set_basis(torch.linalg.qr(torch.randn(64, 64, generator=gen, dtype=torch.float64))[0].float())
        gen = torch.Generator("cuda").manual_seed(2)
        self.g = [[torch.randn(s, device="cuda", generator=gen).bfloat16() for s in shapes] for _ in range(W)]
        self.m = [[torch.randn(s, device="cuda", generator=gen) for s in shapes] for _ in range(W)]
        self.x = [torch.randn(s, device="cuda", generator=gen) for s in shapes]
        self.p = [torch.zeros(self.tr.payload_bytes, dtype=torch.uint8, device="cuda") for _ in range(W)]

    def compress(self, w):
        self.tr.compress(w, self.g[w], self.m[w], self.p[w])

    def results(self):
        torch.cuda.synchronize()
        assert self.tr.device_status() == 0
        return [v for m in self.m for v in m] + self.x + self.p


def same(a, b):
    return all(torch.equal(u, v) for u, v in zip(a.results(), b.results()))


@pytest.mark.parametrize("name", SETS)
def test_compress_of_different_workers_side_by_side(name):
    ref, run = Run(name), Run(name)
    streams = [torch.cuda.Stream() for _ in range(W)]
    for r in (ref, run):
        for w in range(W):
            r.compress(w)  # (the pointer tables of this worker are on the device from here on)
    torch.cuda.synchronize()
    for _ in range(6):
        for w in range(W):
            ref.compress(w)
    for _ in range(6):
        for w, st in enumerate(streams):
            with torch.cuda.stream(st):
                run.compress(w)
    for r in (ref, run):
        torch.cuda.synchronize()
        r.tr.decode_apply(r.p, r.x)
    assert same(ref, run)


@pytest.mark.parametrize("name", SETS)
def test_steps_on_streams_ordered_by_events(name):
    ref, run = Run(name), Run(name)
    torch.cuda.synchronize()
    for _ in range(4):
        for w in range(W):
            ref.compress(w)
        ref.tr.decode_apply(ref.p, ref.x)
    streams, last = [torch.cuda.Stream() for _ in range(2)], None
    for step in range(4):
        for call in range(W + 1):
            st = streams[(step + call) % 2]
            if last is not None:
                st.wait_event(last)
            with torch.cuda.stream(st):
                run.compress(call) if call < W else run.tr.decode_apply(run.p, run.x)
                last = torch.cuda.Event()
                last.record()
    assert same(ref, run)


@pytest.mark.parametrize("name", SETS)
def test_queued_steps_equal_steps_waited_for(name):
    """Kernels may be resident before the work queued before them has finished, and the second kernel of a call runs beside the first:
    many calls with nothing waited for in between against the same calls each waited for."""
    ref, run = Run(name), Run(name)
    torch.cuda.synchronize()
    for r, wait in ((ref, True), (run, False)):
        for _ in range(12):
            for w in range(W):
                r.compress(w)
                if wait:
                    torch.cuda.synchronize()
            r.tr.decode_apply(r.p, r.x)
            if wait:
                torch.cuda.synchronize()
    assert same(ref, run)


RESET = """
import ctypes, glob, sys
from paper_2411_19870_b200 import binding

rt = ctypes.CDLL(glob.glob(sys.prefix + "/lib/python3*/site-packages/nvidia/cuda_runtime/lib/libcudart.so*")[0])
lib = binding.load_library()


def compress():
    ctx, bufs = ctypes.c_void_p(), []
    desc = (binding.DemoTensorDesc * 1)()
    desc[0].ndim, desc[0].shape[0], desc[0].shape[1] = 2, 256, 256
    assert lib.demo_init(ctypes.byref(ctx), ctypes.byref(binding.DemoConfig(0.9, 128, 32, 1e-3, 0.1, 1, 0)), desc, 1, 0) == 0
    for n in (4 * 256 * 256, 4 * 256 * 256, lib.demo_payload_bytes(ctx)):
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(n)) == 0 and rt.cudaMemset(p, 0, ctypes.c_size_t(n)) == 0
        bufs.append(p)
    one = lambda p: (ctypes.c_void_p * 1)(p.value)
    status = lib.demo_compress(ctx, 0, one(bufs[0]), one(bufs[1]), bufs[2], None), lib.demo_device_status(ctx, None)
    lib.demo_free(ctx)
    for p in bufs:
        rt.cudaFree(p)
    return status


assert compress() == (0, 0)
assert rt.cudaDeviceReset() == 0
assert compress() == (0, 0)
print("both")
"""


def test_a_context_made_after_the_process_reset_its_cuda_context():
    """The limit on a kernel's shared memory goes with the CUDA context of the process: it is set again after cudaDeviceReset (in a process
    of its own: torch's memory would go too)."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.stdout.split() == ["both"], r.stdout + r.stderr


def test_contexts_of_different_sizes_do_not_lower_each_other_s_limits():
    """The same N-D kernels with much and with little shared memory, by turns."""
    made = []
    for chunk in ((128, 64), (16, 32), (64, 127), (8, 128)):
        shape = tuple(2 * c for c in chunk)
        tr = demo.DemoTransform([shape], chunk_shapes=[chunk], topk=32, beta=0.9, lr=1e-3, weight_decay=0.1, num_workers=1)
        m, x = torch.zeros(shape, device="cuda"), torch.zeros(shape, device="cuda")
        made.append((tr, [torch.ones(shape, device="cuda").bfloat16()], [m], [x], torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda")))
    for _ in range(2):
        for tr, g, m, x, p in made:
            tr.compress(0, g, m, p)
            tr.decode_apply([p], x)
            assert tr.device_status() == 0
    for tr, *_ in made:
        tr.close()
