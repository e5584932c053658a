"""The native per-step calls (csrc/calls.cpp) without a device: which calls they take, and what reaches the library."""
import ctypes

import pytest
import torch

from paper_2411_19870_b200 import binding

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
