"""Edges of the size ranges the kernel variants are chosen by, against the fp64 oracle (rules and tolerances of
tests/parity.py, every chunk)."""
import contextlib
import ctypes
import math
import types

import numpy as np
import pytest
import torch

from paper_2411_19870_b200 import inputs
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["tensor_scaled", "student_t_ties"])
@pytest.mark.parametrize("k", [48, 49, 64, 65, 128, 192, 193])
def test_s64_list_and_dense_row_stage(k, kind):
    """s = 64: k = 48 is the last with a listed row stage, k = 192 the last bounded by quarter rows; an all-zero tile and a
    single non-zero element among ordinary ones."""
    wl = inputs.Workload("s64k", [(3 * 64, 4 * 64), (64, 64)], chunk=64, topk=k, num_workers=2, grad_kind=kind,
                         grad_dtype=torch.float32 if k % 2 else torch.bfloat16)
    r = parity.Runner(wl, max_chunks=10**9, seed=k)
    for step in range(2):
        grads = [st.next() for st in r.streams]
        for g in grads:
            g[0][:64, :64] = 0
            g[0][64:128, :64] = 0
            g[0][70, 5] = 0.5
        r.step(grads=grads)
    r.close()


@pytest.mark.parametrize("kind", ["tensor_scaled", "student_t_ties"])
@pytest.mark.parametrize("k", [1, 12, 13, 32, 33, 128, 129, 1024])
def test_s32_bounds_list_and_search(k, kind):
    """s = 32: bound from row and half-row maxima, listed and dense row stage, bounded and unbounded search; more chunks than
    the grid has warps, all-zero tiles and tiles of one element."""
    wl = inputs.Workload("s32k", [(55 * 32, 56 * 32), (32, 96)], chunk=32, topk=k, num_workers=2, grad_kind=kind,
                         grad_dtype=torch.float32 if k % 2 else torch.bfloat16)
    r = parity.Runner(wl, max_chunks=200, seed=k)
    for step in range(2):
        grads = [st.next() for st in r.streams]
        for g in grads:
            g[0][:32, :32] = 0
            g[0][32:64, :32] = 0
            g[0][40, 5] = 0.5
            g[1][:, :32] = 0
            g[1][:, 32:64] = 0
            g[1][3, 40] = -0.25
        r.step(grads=grads)
    r.close()


@pytest.mark.parametrize("k", [1, 2, 9, 31, 128, 129])
def test_s128_halves_of_the_row_stage(k):
    """s = 128: the list of records cut between the halves of a CTA where a row ends; more chunks than CTAs, chunks with all
    their coefficients in one row or in one column."""
    wl = inputs.Workload("s128k", [(18 * 128, 17 * 128)], chunk=128, topk=k, num_workers=2, grad_kind="tensor_scaled",
                         grad_dtype=torch.float32 if k % 2 else torch.bfloat16)
    r = parity.Runner(wl, max_chunks=60, seed=k)
    for step in range(2):
        grads = [st.next() for st in r.streams]
        for g in grads:
            g[0][:128, :128] = g[0][:1, :128].clone()
            g[0][128:256, :128] = g[0][128:256, :1].clone()
        r.step(grads=grads)
    r.close()


@pytest.mark.parametrize("s", [32, 64, 128])
@pytest.mark.parametrize("k,workers,agg", [(64, 17, 0), (65, 5, 2), (128, 5, 0), (129, 3, 1), (256, 3, 2), (512, 2, 0), (513, 2, 0)])
def test_decode_large_k(s, k, workers, agg):
    """Records in parts of 64 (short last part), several workers per batch, one, and none staged; colliding coordinates."""
    wl = inputs.Workload("dk", [(2 * s, 3 * s)], chunk=s, topk=k, num_workers=workers, grad_kind="normal", grad_std=0.01)
    r = parity.Runner(wl, max_chunks=10**9, seed=k, agg=agg)
    base = [g.clone() for g in r.streams[0].next()]
    grads = [[(b.float() + 0.3 * o.float()).to(b.dtype) for b, o in zip(base, st.next())] for st in r.streams]
    r.step(grads=grads)
    r.close()


@pytest.mark.parametrize("k,agg", [(48, 0), (49, 2), (64, 2), (65, 0), (192, 0), (193, 2)])
def test_tensor_core_pairs(k, agg):
    """s = 64 under a random basis: listed and dense row stage, decode by warp order and by barriers, four and three groups per CTA;
    2406 chunks, more pairs than the grid has groups, the second tensor's one chunk alone in the last pair's second half."""
    wl = inputs.Workload("tc", [(37 * 64, 65 * 64), (64, 64)], chunk=64, topk=k, num_workers=2, grad_kind="normal", grad_std=0.01,
                         grad_dtype=torch.float32 if k % 2 else torch.bfloat16)
    r = parity.Runner(wl, max_chunks=300, gauss=inputs.basis_gaussian(k, 64).numpy(), agg=agg)
    for _ in range(2):
        r.step()
    assert r.tr.device_status() == 0
    r.close()


@pytest.mark.parametrize("shapes,chunks,k", [
    ([(64, 32, 7, 7), (32,)], [(32, 4, 7, 7), (32,)], 40),         # kernel windows of 7 x 7; a lossless vector
    ([(32, 16, 2, 2), (24, 4, 6, 6)], [(16, 16, 2, 2), (8, 4, 6, 6)], 17),
    ([(32, 48, 3)], [(32, 48, 1)], 33),                            # 1536 rows of one element: no row table
    ([(128, 64), (64, 384)], [(64, 32), (32, 128)], 64),           # two threads per line; ten chunks in one class with extents of 128
    ([(58, 128), (62, 93)], [(29, 64), (31, 31)], 32),             # odd dense extents, one and two lines per thread
    ([(127, 127)], [(127, 127)], 300),                             # the largest dense chunk: both tiles and B fill the SM
    ([(64, 96)], [(16, 32)], 400),                                 # k close to the chunk: the list overflows
])
def test_nd_extents(shapes, chunks, k):
    r = parity.NdRunner(shapes, chunks, topk=k, num_workers=2, grad_std=0.02)
    for _ in range(2):
        r.step()
    r.close()


def test_nd_ties_and_untouched_chunks():
    """Equal magnitudes straddling the k-th place inside the candidate list (a few equal coefficients) and beyond it
    (+-a everywhere), a constant chunk, an all-zero chunk."""
    r = parity.NdRunner([(64, 48)], [(32, 24)], topk=20, num_workers=1, grad_dtype=torch.float32)
    g = torch.zeros(64, 48, device="cuda")
    g[:32, 24:] = 0.25
    sign = torch.where(torch.rand(32, 24, device="cuda", generator=torch.Generator("cuda").manual_seed(3)) < 0.5, -1.0, 1.0)
    g[32:, :24] = 0.125 * sign
    g[32, 24] = 1.0
    r.inputs = types.SimpleNamespace(random_tensor=lambda *a: g)  # the gradient of every step
    for _ in range(2):
        r.step()
    r.close()


@pytest.mark.parametrize("k", [1, 4, 8, 9, 63, 64])
def test_small_tiles_8(k):
    """s = 8: four tiles per warp, an odd number of them, records beyond one round of lanes, lossless."""
    wl = inputs.Workload("s8", [(3 * 8, 7 * 8), (8, 8), (5 * 8,)], chunk=8, topk=k, num_workers=9, grad_kind="student_t_ties")
    r = parity.Runner(wl, max_chunks=10**9, seed=k)
    for _ in range(2):
        r.step()
    r.close()


@pytest.mark.parametrize("k,agg", [(2, 0), (16, 2), (17, 1), (130, 2), (256, 0)])
def test_small_tiles_16(k, agg):
    wl = inputs.Workload("s16", [(3 * 16, 3 * 16), (16, 32)], chunk=16, topk=k, num_workers=3, grad_kind="student_t_ties",
                         grad_dtype=torch.float32)
    r = parity.Runner(wl, max_chunks=10**9, seed=k, agg=agg)
    for _ in range(2):
        r.step()
    r.close()


@pytest.mark.parametrize("s,k,workers", [(8, 3, 2), (16, 16, 9), (32, 5, 17), (64, 33, 5), (128, 1, 3), (128, 97, 2)])
def test_segments(s, k, workers):
    """1-D tensors alone, more than one tensor per warp's search (33 and up), tied and zero segments among them."""
    shapes = [(s * (1 + t % 3),) for t in range(37)]
    wl = inputs.Workload("seg", shapes, chunk=s, topk=k, num_workers=workers, grad_kind="student_t_ties")
    r = parity.Runner(wl, max_chunks=10**9, seed=s + k)
    for _ in range(2):
        r.step()
    r.close()


@pytest.mark.parametrize("shapes", [[(64, 64)], [(64,), (64, 64 * 3), (64 * 65,), (128, 64)], [(64 * 64,)] * 40])
def test_apply_signs_pieces(shapes):
    """Tensors of a piece of 1024 elements and less, several, and with a remainder; many tensors per block."""
    import paper_2411_19870_b200 as demo

    tr = demo.DemoTransform(shapes, chunk=64, topk=4, beta=0.9, lr=0.125, weight_decay=0.5, num_workers=1)
    gen = torch.Generator("cuda").manual_seed(7)
    x = [torch.randn(s, device="cuda", generator=gen) for s in shapes]
    signs = [torch.randint(-1, 2, s, device="cuda", generator=gen, dtype=torch.int8) for s in shapes]
    want = [v.double() - 0.125 * (s.double() + 0.5 * v.double()) for v, s in zip(x, signs)]
    tr.apply_signs(signs, x)
    for got, ref in zip(x, want):  # two fused multiply-adds: at most one rounding each of values below 4
        assert (got.double() - ref).abs().max().item() <= 2 ** -22
    tr.close()


class Flat:
    """A set of equal tensors laid one behind the other in flat buffers, and the calls on it through the C ABI with pointer
    arrays made once (the binding would look at every tensor in every call)."""

    def __init__(self, count, shape, chunk, topk, basis=None):
        import paper_2411_19870_b200 as demo

        self.tr = demo.DemoTransform([shape] * count, chunk=chunk, topk=topk, beta=0.9, lr=1e-3, weight_decay=0.1, num_workers=1)
        if basis is not None:
            self.tr.set_basis(basis)
        n, gen = count * math.prod(shape), torch.Generator("cuda").manual_seed(11)
        self.m = torch.randn(n, device="cuda", generator=gen)
        self.g = torch.randn(n, device="cuda", generator=gen).bfloat16()
        self.x = torch.randn(n, device="cuda", generator=gen)
        each = math.prod(shape)
        rows = torch.zeros(count, -(-each // 16) * 16, dtype=torch.int8, device="cuda")  # tensors start on 16-byte boundaries
        self.signs = rows[:, :each]
        self.payload = torch.zeros(self.tr.payload_bytes, dtype=torch.uint8, device="cuda")

        def pointers(t):
            step = (rows.shape[1] if t is self.signs else each) * t.element_size()
            return (ctypes.c_void_p * count)(*range(t.data_ptr(), t.data_ptr() + count * step, step))

        self.ptr = {k: pointers(getattr(self, k)) for k in ("m", "g", "x", "signs")}
        self.payloads = (ctypes.c_void_p * 1)(self.payload.data_ptr())

    def call(self, what):
        lib, ctx, p = self.tr.lib, self.tr._ctx, self.ptr
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        if what == "compress":
            st = lib.demo_compress(ctx, 0, p["g"], p["m"], ctypes.c_void_p(self.payload.data_ptr()), stream)
        elif what == "decode":
            st = lib.demo_decode_apply(ctx, self.payloads, 1, p["x"], stream)
        elif what == "signs":
            st = lib.demo_decode_signs(ctx, self.payloads, 1, p["signs"], stream)
        else:
            st = lib.demo_apply_signs(ctx, p["signs"], p["x"], stream)
        assert st == 0, what

    def device_us(self, what):
        """Time of one call on the device (calls of a captured graph), the best of several."""
        self.call(what)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(4):
                self.call(what)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = math.inf
        for _ in range(8):
            t0.record()
            graph.replay()
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1) / 4 * 1e3)
        return best


def check_many_tensors(count, shape, chunk, calls, slower, topk=4, basis=None):
    """`count` tensors against one tensor of the same chunks: the same bits, and a call at most `slower` times as long (a call
    looks its tensors up in a table; a search one entry after the other makes it tens of times as long)."""
    many = Flat(count, shape, chunk, topk, basis)
    one = Flat(1, (count * shape[0],) + shape[1:], chunk, topk, basis)
    for what in ("compress", "decode", "signs", "apply"):
        many.call(what)
        one.call(what)
    for k in ("m", "payload", "x", "signs"):
        assert torch.equal(getattr(many, k).reshape(-1), getattr(one, k).reshape(-1)), k
    for what in calls:
        a, b = many.device_us(what), one.device_us(what)
        assert a <= slower * b + 5.0, "%s: %.1f us, one tensor %.1f us" % (what, a, b)
    many.tr.close()
    one.tr.close()


@pytest.mark.parametrize("count", [2, 32, 33, 1024, 1025, 20000])
@pytest.mark.parametrize("s", [8, 64, 128])
def test_many_vectors(s, count):
    check_many_tensors(count, (s,), s, ["compress", "decode"] if count == 20000 else [], 5.0)


@pytest.mark.parametrize("count,shape", [(33, (64,)), (20000, (8,)), (20000, (64,)), (3000, (128,)), (5000, (32, 32)), (20000, (64, 64))])
def test_apply_signs_many_tensors(count, shape):
    """Pieces of a thread (less than half a block's piece on average) and of a block, each with more than 32 tensors to skip."""
    check_many_tensors(count, shape, shape[0], ["apply"] if count > 1000 else [], 5.0)


@pytest.mark.parametrize("count,s,basis", [(3, 64, False), (1000, 64, False), (20000, 64, False), (5000, 32, False), (2000, 128, False),
                                           (32, 64, True), (33, 64, True), (1000, 64, True), (20000, 64, True)])
def test_many_matrices(count, s, basis):
    """One chunk per tensor: the walks over the tensor table skip a grid's worth of entries between two chunks of a CTA."""
    b = torch.linalg.qr(torch.randn(s, s, dtype=torch.float64, generator=torch.Generator().manual_seed(5)))[0].float() if basis else None
    # (s = 64 and 128 acquire two tensor maps for every chunk, about a microsecond each; a few tensors per chunk slot only)
    check_many_tensors(count, (s, s), s, ["compress", "decode"] if count >= 1000 else [], 5.0, basis=b)


@pytest.mark.parametrize("chunk,k,workers,agg", [
    ((16, 32), 32, 17, 0), ((16, 32), 33, 17, 2), ((16, 32), 256, 3, 2), ((16, 32), 257, 3, 0), ((16, 32), 511, 2, 1),  # a warp, one list per batch
    ((32, 64), 32, 19, 2), ((32, 64), 100, 11, 0), ((32, 64), 512, 3, 2), ((32, 64), 513, 3, 2), ((32, 64), 1500, 2, 0),  # more threads, no batches
    ((4, 8, 6, 5), 40, 5, 2), ((13, 64), 90, 6, 2),                                  # an odd number of dense axes: the tiles change places
])
def test_nd_decode_batches(chunk, k, workers, agg):
    """Records of several workers per batch, two and more batches, a short last one, lists longer than a batch; colliding coordinates."""
    r = parity.NdRunner([tuple(3 * c for c in chunk)], [chunk], topk=k, num_workers=workers, grad_std=0.02, agg=agg)
    for _ in range(2):
        r.step()
    r.close()


def nd_device_us(shape, chunk, k, workers, what):
    """Time of one call on an N-D context, the best of several."""
    import paper_2411_19870_b200 as demo

    shapes = [shape, (48, 48)]  # (the second keeps square chunks on the N-D kernels)
    tr = demo.DemoTransform(shapes, chunk_shapes=[chunk, (3, 16)], topk=k, beta=0.9, lr=1e-3, weight_decay=0.1, num_workers=workers)
    gen = torch.Generator("cuda").manual_seed(3)
    g = [torch.randn(s, device="cuda", generator=gen).bfloat16() for s in shapes]
    m, x = ([torch.zeros(s, device="cuda") for s in shapes] for _ in range(2))
    pay = [torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda") for _ in range(workers)]
    for w in range(workers):
        tr.compress(w, g, m, pay[w])
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = math.inf
    for _ in range(8):
        t0.record()
        for _ in range(10):
            tr.compress(0, g, m, pay[0]) if what == "compress" else tr.decode_apply(pay, x)
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1) / 10 * 1e3)
    tr.close()
    return best


@pytest.mark.parametrize("shape,chunk", [((2048, 2048), (32, 128)), ((512, 512, 3, 3), (32, 32, 3, 3))])
def test_nd_decode_time_of_long_lists(shape, chunk):
    """512 records per chunk and 64 workers are 64 times the records of k = 8: added by one warp they took 7 and 11 times as long, by all threads 3 and 5."""
    short, long_ = nd_device_us(shape, chunk, 8, 64, "decode"), nd_device_us(shape, chunk, 512, 64, "decode")
    assert long_ <= 6 * short, "k = 8 %.1f us, k = 512 %.1f us" % (short, long_)


@pytest.mark.parametrize("shape,chunk,k", [((512, 512, 1, 1), (32, 32, 1, 1), 128), ((512, 512, 1, 1), (32, 32, 1, 1), 1000), ((1024, 1024), (16, 32), 256),
                                           ((1024, 1024), (16, 32), 512), ((7475, 512), (13, 32), 300)])
def test_nd_compress_time_of_large_k(shape, chunk, k):
    """Much of a small chunk kept: ordering the records by counting pairs, and the radix select with 32 threads, took 2.7 to 7 times as
    long as k = 32."""
    short, long_ = nd_device_us(shape, chunk, 32, 1, "compress"), nd_device_us(shape, chunk, k, 1, "compress")
    assert long_ <= 2.2 * short, "k = 32 %.1f us, k = %d %.1f us" % (short, k, long_)


@pytest.mark.parametrize("k", [108, 111, 135, 136, 150, 400, 767, 768])
def test_nd_numbered_records(k):
    """Chunks of 768 elements around k^2 = 24 M and up to all of them, padded tiles, equal magnitudes at the k-th place, a tile with few
    non-zero coefficients, an all-zero one."""
    r = parity.NdRunner([(96, 48)], [(32, 24)], topk=k, num_workers=1, grad_dtype=torch.float32)
    gen = torch.Generator("cuda").manual_seed(k)
    sign = torch.where(torch.rand(96, 48, device="cuda", generator=gen) < 0.5, -1.0, 1.0)
    g = torch.randn(96, 48, device="cuda", generator=gen)
    g[:32, 24:] = 0.0
    g[32:64, :24] = 0.125 * sign[32:64, :24]
    g[32:64, 24:] = 0.25
    # With most of a chunk kept the residual is the rounding of both transforms: some 5 * 2^-23 of the largest |B|, here about 4 * 2^-6, which
    # stays below the absolute tolerance of 1e-7.
    g *= 2.0 ** -6 if k > 300 else 1.0
    r.inputs = types.SimpleNamespace(random_tensor=lambda *a: g)
    for _ in range(2):
        r.step()
    r.close()


@pytest.mark.parametrize("shapes,chunks,classes,agg", [
    # one class, 4900 chunks, a CTA takes several and changes between one dense axis (the tiles change places) and two
    ([(60 * 13, 40 * 32), (50 * 9, 50 * 40)], [(13, 32), (9, 40)], 1, 0),
    ([(60 * 13, 40 * 32), (50 * 9, 50 * 40)], [(13, 32), (9, 40)], 1, 2),
    # a class of 2400 chunks and one of 400 beside it
    ([(60 * 13, 40 * 32), (160, 640, 3, 3)], [(13, 32), (16, 16, 3, 3)], 2, 2),
])
def test_nd_many_chunks_and_classes(shapes, chunks, classes, agg):
    """Chunks on demand, changes of layout inside a CTA and classes side by side, every chunk against the oracle; the signs handed out and
    applied leave the parameters of decode_apply."""
    r = parity.NdRunner(shapes, chunks, topk=12, num_workers=2, grad_std=0.02, agg=agg)
    for _ in range(2):
        n = r.tr.launch_count
        x = [p.clone() for p in r.params]
        r.step()
        assert r.tr.launch_count - n == classes * (r.W + 1)
        signs = [torch.zeros(s, dtype=torch.int8, device="cuda") for s in r.shapes]
        r.tr.decode_signs(r.payloads, signs)
        r.tr.apply_signs(signs, x)
        assert all(torch.equal(a, b) for a, b in zip(x, r.params))
    r.close()


@pytest.mark.parametrize("shapes,s,k", [([(20001 * 8,), (19321 * 8,)], 8, 3), ([(2501 * 64,)], 64, 9), ([(1301 * 128,)], 128, 17),
                                        ([(139 * 8, 139 * 8)], 8, 5), ([(99 * 16, 97 * 16), (5000 * 16,)], 16, 7)])
def test_small_chunks_beyond_one_round(shapes, s, k):
    """More segments and tiles than the grid takes in one round, the last round and the last warp partly filled."""
    wl = inputs.Workload("small", shapes, chunk=s, topk=k, num_workers=2, grad_kind="student_t_ties")
    r = parity.Runner(wl, max_chunks=400, seed=s)
    for _ in range(2):
        r.step()
    # (the sample holds the last chunk; the energy identity covers all of them)
    r.step(invariants=True)
    r.close()


def steps_with(shapes, chunk, k, f32, basis, domain, bad):
    import paper_2411_19870_b200 as demo

    kw = dict(chunk=chunk) if isinstance(chunk, int) else dict(chunk_shapes=chunk)
    tr = demo.DemoTransform(shapes, topk=k, beta=0.9, lr=1e-3, weight_decay=0.1, num_workers=2,
                            grad_dtype=demo.DEMO_F32 if f32 else demo.DEMO_BF16, **kw)
    if basis:
        tr.set_basis(torch.linalg.qr(torch.randn(64, 64, dtype=torch.float64, generator=torch.Generator().manual_seed(2)))[0].float())
    if domain:
        tr.set_momentum_domain(demo.DEMO_MOMENTUM_DCT)
    gen = torch.Generator("cuda").manual_seed(9)
    m = [[torch.zeros(s, device="cuda") for s in shapes] for _ in range(2)]
    x = [torch.randn(s, device="cuda", generator=gen) for s in shapes]
    p = [torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda") for _ in range(2)]
    for step in range(2):
        for w in range(2):
            g = [torch.randn(s, device="cuda", generator=gen) for s in shapes]
            if bad and step == 0:
                flat = g[0].view(-1)
                flat[3], flat[flat.numel() // 2], flat[-2] = float("nan"), float("inf"), float("-inf")
            tr.compress(w, [v if f32 else v.bfloat16() for v in g], m[w], p[w])
        tr.decode_apply(p, x)
    assert tr.device_status() == 0
    layout = [tr.payload_layout(t) for t in range(len(shapes))]
    tr.close()
    return m, x, p, layout


@pytest.mark.parametrize("chunk,k,f32,basis,domain", [
    (8, 20, True, False, False), (16, 5, False, False, False), (16, 100, True, False, False), (32, 20, True, False, False),
    (32, 40, False, False, False), (64, 64, False, False, False), (64, 200, True, False, False), (64, 64, True, False, True), (128, 130, True, False, False),
    (128, 300, False, False, False), (64, 32, False, True, False), (64, 60, True, True, False),
    ([(12, 29), (7, 3, 3)], 20, True, False, False), ([(12, 29), (7, 3, 3)], 100, False, False, False), ([(32, 64), (16, 4, 4)], 600, True, False, False),
])
def test_non_finite_gradients_per_variant(chunk, k, f32, basis, domain):
    """NaN and infinities in the first tensor, in every variant of the selection: records still distinct, ascending and in range, the
    second tensor the same bits as without them."""
    square = isinstance(chunk, int)
    shapes = [(4 * chunk, 3 * chunk), (2 * chunk, 2 * chunk)] if square else [tuple(3 * c for c in ch) for ch in chunk]
    per = [chunk * chunk] * 2 if square else [math.prod(c) for c in chunk]
    clean = steps_with(shapes, chunk, k, f32, basis, domain, False)
    dirty = steps_with(shapes, chunk, k, f32, basis, domain, True)
    assert torch.equal(clean[1][1], dirty[1][1])
    for w in range(2):
        assert torch.equal(clean[0][w][1], dirty[0][w][1])
        rec = dirty[2][w].view(torch.int32).view(-1, 2)[:, 0].cpu().numpy()
        for (first, n, k_eff), elems in zip(dirty[3], per):
            idx = rec[first:first + n * k_eff].reshape(n, k_eff)
            assert idx.min() >= 0 and idx.max() < elems
            assert k_eff == 1 or np.all(np.diff(idx, axis=1) > 0)


@pytest.mark.parametrize("s", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("k", [1, 40, 64, 65, 128, 129, 200, 256, 257, 512, 513])
def test_decode_adds_in_the_order_of_the_workers(s, k):
    """2^25 + 1 - 2^25 is 0 in fp32 in this order and 1 or 0 in others: three workers send these values for one coordinate that stands
    first in the lists of workers 0 and 2 and last in worker 1's, all other values are zero.  The signs and the update agree."""
    import paper_2411_19870_b200 as demo

    M = s * s
    if k > M // 4:
        pytest.skip("the lists need room on both sides of the coordinate")
    lr = 2.0 ** -3
    tr = demo.DemoTransform([(2 * s, s)], chunk=s, topk=k, beta=0.9, lr=lr, weight_decay=0.0, num_workers=3)
    at = M // 2
    pay = [torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda") for _ in range(3)]
    for w, (value, first) in enumerate(((2.0 ** 25, True), (1.0, False), (-2.0 ** 25, True))):
        idx = torch.arange(k) + (at if first else at - k + 1)
        rec = pay[w].view(torch.int32).view(2, k, 2)
        rec[:, :, 0] = idx.int().cuda()
        pay[w].view(torch.float32).view(2, k, 2)[:, 0 if first else k - 1, 1] = value
    signs = [torch.ones(2 * s, s, dtype=torch.int8, device="cuda")]
    tr.decode_signs(pay, signs)
    assert int(signs[0].abs().sum()) == 0
    x = [torch.randn(2 * s, s, device="cuda")]
    before = x[0].clone()
    tr.decode_apply(pay, x)
    assert torch.equal(x[0], before)
    tr.set_decode_mode(demo.DEMO_AGG_SUM, demo.DEMO_PHI_IDENTITY)
    tr.decode_apply(pay, x)
    assert torch.equal(x[0], before)
    tr.close()


@pytest.mark.parametrize("kind", ["normal", "ties", "zero", "one", "full"])
@pytest.mark.parametrize("k", [193, 255, 1000, 4095, 4096])
def test_s64_search_of_the_threshold(k, kind):
    """s = 64 above the bound of the lists: all keys equal, all zero, a single non-zero coefficient, fewer than k of them, everything kept;
    on DCT and caller-supplied basis, every chunk against the oracle."""
    for gauss in (None, inputs.basis_gaussian(3, 64).numpy()):
        wl = inputs.Workload("s64s", [(2 * 64, 3 * 64)], chunk=64, topk=k, num_workers=1, grad_kind="normal", grad_dtype=torch.float32)
        r = parity.Runner(wl, max_chunks=10**9, seed=k, gauss=gauss)
        g = r.streams[0].next()
        # (most of a chunk kept leaves the rounding of both transforms, some 5 * 2^-23 of the largest |B|, as the residual: inputs below
        # 2^-4 keep it under the absolute tolerance of 1e-7)
        g[0].mul_(2.0 ** -6 / max(1e-30, float(g[0].abs().max())))
        if kind == "ties":
            g[0].copy_(torch.where(g[0] < 0, -(2.0 ** -8), 2.0 ** -8))
        if kind in ("zero", "one"):
            g[0].zero_()
        if kind == "one":
            g[0][::64, ::64] = 2.0 ** -6
        if kind == "full":
            g[0][64:] = 2.0 ** -6
        r.step(grads=[g])
        r.close()


@pytest.mark.parametrize("basis", [False, True])
def test_s64_compress_time_above_the_lists(basis):
    """k = 193 is searched among all coefficients, k = 192 among a list: by a radix select it took 2.7 times as long, on all-zero tiles nine
    times."""
    times = {}
    for k in (192, 193):
        f = Flat(1, (4096, 4096), 64, k, torch.linalg.qr(torch.randn(64, 64, dtype=torch.float64))[0].float() if basis else None)
        times[k] = f.device_us("compress")
        f.g.zero_()
        f.m.zero_()
        times[-k] = f.device_us("compress")
        f.tr.close()
    assert times[193] <= 2.0 * times[192] and times[-193] <= 2.2 * times[-192], times


@pytest.mark.parametrize("shapes,s,k,workers,agg", [([(8 * 8, 37 * 8), (40,)], 8, 9, 8, 0), ([(8 * 8, 38 * 8), (40,)], 8, 20, 9, 2),
                                                    ([(4 * 16, 5 * 16)], 16, 17, 8, 2), ([(18 * 16, 17 * 16)], 16, 40, 8, 0)])
def test_small_tiles_many_workers(shapes, s, k, workers, agg):
    """Eight workers and lists longer than a tile's lanes: up to 296 tiles on the dense kernels, more on the small-chunk ones."""
    wl = inputs.Workload("st", shapes, chunk=s, topk=k, num_workers=workers, grad_kind="student_t_ties")
    r = parity.Runner(wl, max_chunks=10**9, seed=k, agg=agg)
    for _ in range(2):
        r.step()
    r.close()


def test_decode_time_of_long_lists_on_few_small_tiles():
    """64 workers' lists of half a tile, 256 tiles of 16 x 16: with 16 threads per tile 2.4 times as long as with 256."""
    import paper_2411_19870_b200 as demo

    wl = inputs.Workload("st", [(256, 256)], chunk=16, topk=128, num_workers=64, grad_kind="normal")
    r = parity.Runner(wl, max_chunks=4)
    r.step(check=False)
    times = {}
    for path in (demo.DEMO_PATH_AUTO, demo.DEMO_PATH_GENERIC):
        r.tr.set_path(path)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times[path] = math.inf
        for _ in range(8):
            t0.record()
            for _ in range(8):
                r.tr.decode_apply(r.payloads, r.params)
            t1.record()
            torch.cuda.synchronize()
            times[path] = min(times[path], t0.elapsed_time(t1))
    assert times[demo.DEMO_PATH_AUTO] <= 1.4 * times[demo.DEMO_PATH_GENERIC], times
    r.close()


@pytest.mark.parametrize("s,per_sm", [(32, 16), (64, 6), (64, 8), (128, 2)])
@pytest.mark.parametrize("rounds,extra", [(1, 0), (1, 1), (2, -1), (2, 0), (2, 1), (3, -1), (3, 0), (3, 1), (4, 3)])
def test_chunks_of_the_first_rounds(s, per_sm, rounds, extra):
    """Every chunk is processed once whether a CTA's second chunk is fixed or drawn (up to three rounds of the decode kernels' grid, or more): one
    row of chunks in one call against the same chunks in contexts of at most one chunk per SM, whose grids hold them all at once and draw
    nothing, bit for bit, over two calls.  ``per_sm``: chunks of a round per SM (s = 32: eight CTAs of two; s = 64: eight, six where the senders
    are counted)."""
    import paper_2411_19870_b200 as demo

    sms, k = torch.cuda.get_device_properties(0).multi_processor_count, 3
    n = rounds * per_sm * sms + extra
    g = torch.randn(s, n * s, device="cuda", generator=torch.Generator("cuda").manual_seed(n))

    def run(first, count):
        tr = demo.DemoTransform([(s, count * s)], chunk=s, topk=k, beta=0.9, lr=0.125, weight_decay=0.1, num_workers=1, grad_dtype=demo.DEMO_F32)
        if per_sm == 6:
            tr.set_decode_mode(demo.DEMO_AGG_COUNT_MEAN, demo.DEMO_PHI_SIGN)
        part = g[:, first * s:(first + count) * s].contiguous()
        gs, ms, xs = [part], [0.5 * part], [0.25 * part]
        pay = torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda")
        for _ in range(2):
            tr.compress(0, gs, ms, pay)
            tr.decode_apply([pay], xs)
        assert tr.device_status() == 0
        tr.close()
        return pay, ms[0], xs[0]

    whole = run(0, n)
    parts = [run(first, min(sms, n - first)) for first in range(0, n, sms)]
    assert torch.equal(whole[0], torch.cat([p[0] for p in parts]))
    assert torch.equal(whole[1], torch.cat([p[1] for p in parts], 1))
    assert torch.equal(whole[2], torch.cat([p[2] for p in parts], 1))


@pytest.mark.parametrize("s,k,workers", [(32, 1, 2), (32, 40, 9), (64, 1, 3), (64, 33, 17), (64, 70, 5), (64, 600, 3)])
def test_senders_of_every_place_of_a_row(s, k, workers):
    """Count-normalised mean: coordinates of every column sent by none, one and several workers."""
    wl = inputs.Workload("cm", [(2 * s, 3 * s)], chunk=s, topk=k, num_workers=workers, grad_kind="normal", grad_std=0.01)
    r = parity.Runner(wl, max_chunks=10**9, seed=k, agg=2)
    base = [g.clone() for g in r.streams[0].next()]
    r.step(grads=[[(b.float() + 0.2 * o.float()).to(b.dtype) for b, o in zip(base, st.next())] for st in r.streams])
    r.close()


@pytest.mark.parametrize("s", [8, 16, 32, 64, 128])
def test_vectors_under_a_callers_basis(s):
    """1-D tensors read the basis by columns on the way there and by rows on the way back: a matrix that is not symmetric, set twice."""
    wl = inputs.Workload("vb", [(3 * s,), (s, 2 * s), (s,)], chunk=s, topk=max(1, s // 4), num_workers=2, grad_kind="normal", grad_std=0.01)
    r = parity.Runner(wl, max_chunks=10**9)
    for seed in (1, 2):
        q = np.linalg.qr(np.random.default_rng(seed).standard_normal((s, s)))[0]
        r.set_basis(basis=np.ascontiguousarray(q, dtype=np.float32))
        r.step()
    r.set_basis()
    r.step()
    r.close()


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("shape,chunk,k", [
    ((32, 128), (16, 32), 5),            # rows of whole quads in the tensor and in the tile, the last axis read by quads
    ((24, 80), (8, 16), 128),            # the same, everything kept: no list of lines
    ((64, 24), (32, 8), 12), ((48, 12), (3, 4), 3),
    ((48, 64, 3, 3), (16, 32, 3, 3), 31),  # rows of 288 elements across two axes, the tile's rows not quads
    ((4, 48, 3, 3), (4, 16, 3, 3), 9),   # one chunk deep: the rows are the chunk
    ((32, 36, 5, 5), (8, 12, 5, 5), 20), ((14, 21, 6, 6), (7, 7, 6, 6), 17),
    ((30, 33), (6, 11), 7),              # rows of 11: element by element
    ((30, 36), (5, 12), 7), ((29 * 3, 128), (29, 64), 32), ((64, 62), (32, 31), 40),
    ((128, 8), (128, 4), 30),
])
def test_nd_rows_and_lines(shape, chunk, k, f32):
    """Chunks whose rows are whole 16-byte pieces of the tensor, of the tile, of both, or not; odd and even extents multiplied out;
    first axes whose kept lines are listed (several records per line among them) and others."""
    r = parity.NdRunner([shape, (shape[-1] * 4,)], [chunk, (chunk[-1],)], topk=k, num_workers=2, grad_std=0.02,
                        grad_dtype=torch.float32 if f32 else torch.bfloat16)
    for _ in range(2):
        r.step()
    r.close()


def test_compress_time_of_several_tensors_below_four_chunks_per_sm():
    """s = 64, sets of 16-chunk tensors: 576 chunks are compressed in 0.91 of the time of 640, as their number says.  (1.01 where their first
    chunks, below four per SM, were all looked up and requested in the same moment.)"""
    import paper_2411_19870_b200 as demo

    times = {}
    for n in (36, 40):
        tr = demo.DemoTransform([(256, 256)] * n, chunk=64, topk=32, beta=0.9, lr=0.1, weight_decay=0.1, num_workers=4)
        sets = [[[torch.randn((256, 256), device="cuda").to(d) for _ in range(n)] for d in (torch.bfloat16, torch.float32)] for _ in range(4)]
        pay = [torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda") for _ in range(4)]
        graph = torch.cuda.CUDAGraph()
        for captured in (False, True):
            with torch.cuda.graph(graph) if captured else contextlib.nullcontext():
                for w, (g, m) in enumerate(sets):
                    tr.compress(w, g, m, pay[w])
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times[n] = math.inf
        for _ in range(10):
            t0.record()
            for _ in range(20):
                graph.replay()
            t1.record()
            torch.cuda.synchronize()
            times[n] = min(times[n], t0.elapsed_time(t1))
        del graph
        tr.close()
    assert times[36] <= 0.96 * times[40], times


def _graph_time(calls, repeats=20):
    """Device time of the captured calls, the shortest of ten loops."""
    graph = torch.cuda.CUDAGraph()
    calls()
    with torch.cuda.graph(graph):
        calls()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = math.inf
    for _ in range(10):
        t0.record()
        for _ in range(repeats):
            graph.replay()
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1))
    return best


def test_time_of_a_few_segments_of_128():
    """Compress of one segment of 128 elements takes 1.4 times as long as of one of 64, whose table is a quarter as large (2.3 times where its
    elements of the basis were fetched in four turns behind one another)."""
    import paper_2411_19870_b200 as demo

    times = {}
    for s in (64, 128):
        tr = demo.DemoTransform([(s,)], chunk=s, topk=8, beta=0.9, lr=0.1, weight_decay=0.1, num_workers=1)
        g, m = [torch.randn(s, device="cuda").bfloat16()], [torch.randn(s, device="cuda")]
        pay = torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda")
        times[s] = _graph_time(lambda: [tr.compress(0, g, m, pay) for _ in range(4)])
        tr.close()
    assert times[128] <= 1.9 * times[64], times


@pytest.mark.parametrize("counted", [False, True])
def test_segments_of_128_in_two_rounds_and_more(counted):
    """Decode of vectors at s = 128 has a form for up to two rounds of blocks and one for more: one vector of both kinds of length, and in halves
    that take the first form, bit for bit."""
    import paper_2411_19870_b200 as demo

    sms, s, W = torch.cuda.get_device_properties(0).multi_processor_count, 128, 3
    n = 16 * sms + 7
    gen = torch.Generator("cuda").manual_seed(n)
    g = [torch.randn(n * s, device="cuda", generator=gen) for _ in range(W)]

    def run(first, count):
        tr = demo.DemoTransform([(count * s,)], chunk=s, topk=9, beta=0.9, lr=0.125, weight_decay=0.1, num_workers=W, grad_dtype=demo.DEMO_F32)
        tr.set_decode_mode(demo.DEMO_AGG_COUNT_MEAN if counted else demo.DEMO_AGG_SUM, demo.DEMO_PHI_IDENTITY)
        gs = [v[first * s:(first + count) * s].contiguous() for v in g]
        ms, x = [0.5 * v for v in gs], 0.25 * gs[0]
        pay = [torch.zeros(tr.payload_bytes, dtype=torch.uint8, device="cuda") for _ in range(W)]
        for _ in range(2):
            for w in range(W):
                tr.compress(w, [gs[w]], [ms[w]], pay[w])
            tr.decode_apply(pay, [x])
        tr.close()
        return torch.cat(ms), x

    whole, parts = run(0, n), [run(0, n // 2), run(n // 2, n - n // 2)]
    assert torch.equal(whole[1], torch.cat([p[1] for p in parts]))
    assert torch.equal(whole[0].view(W, -1), torch.cat([p[0].view(W, -1) for p in parts], 1))
