"""The native per-step calls (csrc/calls.cpp) without a device: which calls they take, and what reaches the library."""
import ctypes
import types

import pytest
import torch

from paper_2411_19870_b200 import binding, build

COMPRESS = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
DECODE = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_void_p)
APPLY = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)


class Sub(torch.Tensor):
    """A subclass answers for itself."""
    shift = 0

    def data_ptr(self):
        return super().data_ptr() + self.shift


def array(tensors):
    ptrs = [t.data_ptr() for t in tensors]
    return ptrs, (ctypes.c_void_p * len(ptrs))(*ptrs)


def pointers(address, n):
    return list((ctypes.c_void_p * n).from_address(address))


@pytest.mark.parametrize("n", [0, 1, 5])
def test_calls_pass_the_pointers_of_tensors_that_did_not_move(n):
    calls, seen = binding.load_calls(), []
    g, m, x = ([torch.zeros(8) for _ in range(n)] for _ in range(3))
    p = [torch.zeros(16, dtype=torch.uint8) for _ in range(n + 1)]
    cache = {("g", 3): array(g), ("m", 3): array(m), "x": array(x), "s": array(m), "p": array(p)}
    known = {(t.data_ptr(), t.numel()) for t in p}
    compress = COMPRESS(lambda *a: seen.append((a[0], a[1], pointers(a[2], n), pointers(a[3], n), a[4], a[5])) or 5)
    decode = DECODE(lambda *a: seen.append((a[0], pointers(a[1], n + 1), a[2], pointers(a[3], n), a[4])) or 6)
    apply = APPLY(lambda *a: seen.append((a[0], pointers(a[1], n), pointers(a[2], n), a[3])) or 7)
    address = lambda f: ctypes.cast(f, ctypes.c_void_p).value  # noqa: E731
    go = lambda **k: calls.compress(address(compress), 64, cache, known, 3, ("g", 3), k.get("g", g), ("m", 3), k.get("m", tuple(m)),  # noqa: E731
                                    k.get("p", p[0]), 77)
    assert go() == 5 and seen.pop() == (64, 3, cache[("g", 3)][0], cache[("m", 3)][0], p[0].data_ptr(), 77)
    assert calls.decode(address(decode), 0, cache, known, p, "x", x, 9) == 6
    assert seen.pop() == (None, cache["p"][0], n + 1, cache["x"][0], 9)
    assert calls.apply_signs(address(apply), 64, cache, m, x, 9) == 7 and seen.pop() == (64, cache["s"][0], cache["x"][0], 9)
    # everything else is left to the checked way: other places, another number, unknown payloads, no entry, an iterator
    assert go(g=g + [torch.zeros(8)]) is None and go(p=torch.zeros(16, dtype=torch.uint8)) is None and go(p=p[0][:8]) is None
    assert calls.compress(address(compress), 64, {}, known, 3, ("g", 3), g, ("m", 3), m, p[0], 77) is None
    assert calls.decode(address(decode), 0, cache, set(), p, "x", x, 9) is None
    assert go(m=iter(m)) is None
    if n:
        moved = [torch.zeros(8)] + g[1:]
        assert go(g=moved) is None
        same = [g[0].as_subclass(Sub)] + g[1:]
        assert go(g=same) == 5 and seen.pop()[2] == cache[("g", 3)][0]
        same[0].shift = 16
        assert go(g=same) is None
    assert not seen


def test_errors_of_the_arguments_are_raised():
    calls = binding.load_calls()
    with pytest.raises(TypeError):
        calls.compress(1, 2)
    with pytest.raises(TypeError):
        calls.decode("no address", 0, {}, set(), [], "x", [], 0)
    with pytest.raises(AttributeError):
        calls.apply_signs(1, 0, {"s": ([1], (ctypes.c_void_p * 1)(1))}, [object()], [], 0)


def views(t):
    """Tensors at t's address that are not t: another shape, order, type, or part of it."""
    return {"transposed": t.t(), "columns": t[:, :4], "rows": t[:1], "reshaped": t.view(8, 4), "flat": t.view(-1), "type": t.view(torch.int32),
            "half": t.view(torch.float16)[:, :8]}


@pytest.mark.parametrize("view", sorted(views(torch.zeros(4, 8))))
def test_a_known_address_with_another_layout_is_not_taken(view):
    calls, seen = binding.load_calls(), []
    g, m, x = (torch.zeros(4, 8) for _ in range(3))
    p = torch.zeros(16, dtype=torch.uint8)
    f32 = calls.layouts(torch.float32, -1, [(4, 8)])
    cache = {k: array([t]) + (f32,) for k, t in ((("g", 0), g), (("m", 0), m), ("x", x), ("s", m))}
    cache["p"] = array([p])
    known = {(p.data_ptr(), p.numel())}
    fn = [f(lambda *a: seen.append(a) or 0) for f in (COMPRESS, DECODE, APPLY)]
    at = [ctypes.cast(f, ctypes.c_void_p).value for f in fn]
    go = lambda g, m, x, p: (calls.compress(at[0], 0, cache, known, 0, ("g", 0), [g], ("m", 0), [m], p, 0),  # noqa: E731
                             calls.decode(at[1], 0, cache, known, [p], "x", [x], 0), calls.apply_signs(at[2], 0, cache, [m], [x], 0))
    assert go(g, m, x, p) == (0, 0, 0) and len(seen) == 3
    assert go(views(g)[view], m, x, p) == (None, 0, 0)
    assert go(g, views(m)[view], x, p) == (None, 0, None)
    assert go(g, m, views(x)[view], p) == (0, None, None)
    assert go(g, m, x, p.view(torch.int8)) == (None, None, 0)
    assert go(g, m, x, torch.zeros(32, dtype=torch.uint8).set_(p.untyped_storage(), 0, (4, 4), (1, 4))) == (None, None, 0)
    assert go(g.as_subclass(Sub), m, x, p) == (0, 0, 0) and go(views(g)[view].as_subclass(Sub), m, x, p) == (None, 0, 0)
    # the payload is held to the tensors' device as well
    cache["x"] = cache["x"][:2] + (calls.layouts(torch.float32, 0, [(4, 8)]),)
    assert go(g, m, x, p)[1:] == (None, None)


def test_layouts_refuses_what_it_cannot_read():
    calls = binding.load_calls()
    for bad in ((1, -1, []), (torch.float32, "0", []), (torch.float32, -1, 3), (torch.float32, -1, [("a",)]), (torch.float32, -1, [(1 << 70,)])):
        with pytest.raises((TypeError, OverflowError)):
            calls.layouts(*bad)
    with pytest.raises(ValueError):
        calls.apply_signs(1, 0, {"s": ([], (ctypes.c_void_p * 0)(), "not layouts")}, [], [], 0)


def test_a_module_of_another_python_or_torch_is_not_loaded(monkeypatch):
    """Their internals are compiled into it: only the one whose name says the running versions counts as built, and is loaded."""
    binding.load_calls()
    own = build.calls_path()
    ran = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **k: ran.append(cmd) or types.SimpleNamespace(returncode=1, stdout="", stderr=""))
    assert build.build_calls() == own and not ran
    for target, name, value in ((torch, "__version__", "9.9.0+cu999"), (build.sysconfig, "get_config_var", lambda n: "cpython-399-x86_64-linux-gnu")):
        with monkeypatch.context() as m:
            m.setattr(target, name, value)
            assert build.calls_path() != own
            with pytest.raises(RuntimeError):
                build.build_calls()
            assert len(ran) == 1 and ran.pop()[0].endswith("g++")
            m.setattr(binding, "_calls", None)
            with pytest.raises(RuntimeError, match="missing"):
                binding.load_calls()
    assert build.calls_path() == own


@pytest.fixture
def host_only(monkeypatch):
    """A DemoTransform of one 4 x 8 tensor around functions that write down what reaches the library."""
    seen = []
    apply = APPLY(lambda *a: seen.append("native") or 0)
    note = lambda name: lambda *a: seen.append(name) or 0  # noqa: E731
    lib = types.SimpleNamespace(demo_init=lambda *a: 0, demo_payload_bytes=lambda c: 16, demo_apply_signs=note("python"), demo_step_host=note("host"),
                                demo_free=lambda c: None, entry_points={"demo_apply_signs": ctypes.cast(apply, ctypes.c_void_p).value})
    monkeypatch.setattr(binding, "load_library", lambda: lib)
    tr = binding.DemoTransform([(4, 8)], chunk=4, topk=1, beta=0.9, lr=0.1, weight_decay=0.0, num_workers=1, device=-1)
    tr.device, tr.keep, tr.seen = None, apply, seen
    return tr


@pytest.mark.parametrize("view", sorted(views(torch.zeros(4, 8))))
def test_every_call_checks_the_layout(host_only, view):
    x, s = torch.zeros(4, 8), torch.zeros(4, 8, dtype=torch.int8)
    for _ in range(3):
        host_only.apply_signs([s], [x], stream=1)
    assert host_only.seen == ["native"] * 3
    for args in (([s], [views(x)[view]]), ([s.t()], [x]), ([views(x)[view].as_subclass(Sub)], [x]), ([s], iter([views(x)[view]]))):
        with pytest.raises(ValueError):
            host_only.apply_signs(*args, stream=1)
    assert len(host_only.seen) == 3


def test_tensors_of_step_host_are_not_taken_as_checked(host_only):
    x, s = torch.zeros(4, 8, dtype=torch.int32), torch.zeros(4, 8, dtype=torch.int8)
    p = torch.zeros(16, dtype=torch.uint8)
    host_only.apply_signs([s], [torch.zeros(4, 8)], stream=1)
    host_only.step_host([[x]], [[x]], [[x]], [p], [x], stream=1)
    with pytest.raises(ValueError):
        host_only.apply_signs([s], [x], stream=1)
    assert host_only.seen == ["native", "host"]


@pytest.mark.parametrize("n", [1, 5, 70])
def test_tensors_at_new_addresses_take_the_native_way(n):
    calls, seen = binding.load_calls(), []
    f32 = calls.layouts(torch.float32, -1, [(4, 8 + i) for i in range(n)])
    cache = {k: ([], (ctypes.c_void_p * 0)(), f32) for k in (("g", 0), ("m", 0), "x", "s")}
    fn = (COMPRESS(lambda *a: seen.append([a[1], pointers(a[2], n), pointers(a[3], n), a[4]]) or 0),
          DECODE(lambda *a: seen.append([pointers(a[1], a[2]), pointers(a[3], n)]) or 0), APPLY(lambda *a: seen.append([pointers(a[1], n), pointers(a[2], n)]) or 0))
    at = [ctypes.cast(f, ctypes.c_void_p).value for f in fn]
    keep = []
    for _ in range(3):
        g, m, x = ([torch.zeros(4, 8 + i) for i in range(n)] for _ in range(3))
        p = [torch.zeros(16, dtype=torch.uint8) for _ in range(n)]
        known = {(t.data_ptr(), t.numel()) for t in p}
        keep += [g, m, x, p]  # (so that the next ones lie elsewhere)
        G, M, X, P = ([t.data_ptr() for t in v] for v in (g, m, x, p))
        assert calls.compress(at[0], 0, cache, known, 0, ("g", 0), g, ("m", 0), tuple(m), p[-1], 0) == 0 and seen.pop() == [0, G, M, P[-1]]
        assert calls.decode(at[1], 0, cache, known, tuple(p), "x", x, 0) == 0 and seen.pop() == [P, X]
        assert calls.apply_signs(at[2], 0, cache, m, x, 0) == 0 and seen.pop() == [M, X]
        # a payload not seen before, a subclass that was never asked, a list that is too short or too long
        assert calls.decode(at[1], 0, cache, known, p + [torch.zeros(16, dtype=torch.uint8)], "x", x, 0) is None
        assert calls.apply_signs(at[2], 0, cache, m[:-1] + [m[-1].as_subclass(Sub)], x, 0) is None
        assert calls.apply_signs(at[2], 0, cache, m[:-1], x, 0) is None and calls.apply_signs(at[2], 0, cache, m, x + x[:1], 0) is None
    assert not seen


def test_a_subclass_takes_the_native_way_where_it_was_asked(host_only):
    s, x = torch.zeros(4, 8, dtype=torch.int8), torch.zeros(4, 8).as_subclass(Sub)
    for _ in range(3):
        host_only.apply_signs([s], [x], stream=1)
    x.shift = 16
    host_only.apply_signs([s], [x], stream=1)
    host_only.apply_signs([s], [torch.zeros(4, 8)], stream=1)
    assert host_only.seen == ["python", "native", "native", "python", "native"]
