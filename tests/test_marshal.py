"""The binding's extension for plain arguments: what is not plain is left to the Python marshalling, and both do the same."""
import os
import subprocess
import sys
import warnings

import numpy as np
import pytest
import torch
from torch.overrides import TorchFunctionMode
from torch.utils._python_dispatch import TorchDispatchMode

from paper_2509_16989_b200 import binding, build


class Sub(torch.Tensor):
    pass


def functions():
    # an extension that was built and is not in use is a failure; none only where it cannot be built
    if not os.path.exists(build.marshal_path()):
        try:
            build.build_marshal()
        except (OSError, RuntimeError) as e:
            pytest.skip("the extension cannot be built here: %s" % e)
        binding._bind_plain(binding.lib())
    binding.lib()
    assert binding._gemv_plain is not None
    return sys.modules["paper_2509_16989_b200._marshal"]


@pytest.mark.parametrize("kind", ["missing", "broken", "another torch"])
def test_an_extension_that_cannot_serve_is_reported(kind, tmp_path, monkeypatch):
    functions()
    for name in ("_gemv_plain", "_gemv_host_plain", "_gemm_skinny_plain", "_gemm_skinny_ws_plain"):
        monkeypatch.setattr(binding, name, None)
    path = tmp_path / "_marshal.so"
    if kind == "broken":
        path.write_bytes(b"no library")
    if kind == "another torch":
        real = build.marshal_path()
        monkeypatch.setattr(torch, "__version__", "0.0.0+none")
        assert not os.path.exists(build.marshal_path())  # it looks for a file of its own name
        path = real
    monkeypatch.setattr(build, "marshal_path", lambda: str(path))
    with pytest.warns(RuntimeWarning, match={"missing": "not there", "broken": "does not load", "another torch": "built for torch"}[kind]):
        binding._bind_plain(binding.lib())
    assert binding._gemv_plain is None


def test_a_usable_extension_is_not_reported():
    functions()
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        binding._bind_plain(binding.lib())


def test_left_alone_on_the_cpu():
    # nothing here is on a device: every function returns None and has done nothing
    m = functions()
    b, h = torch.zeros(4096, dtype=torch.uint8), torch.zeros(256, dtype=torch.float16)
    for args in ((b, h, h, 16, 256, 3), (None, h, h, 16, 256, 3), (b, h, h, 16.0, 256, 3), (b, h, h, np.int64(16), 256, 3), (b, h, h, -16, 256, 3),
                 (b, h, h, 1 << 40, 256, 3), (b, h, h, True, 256, 3), (b, h, h, 16, 256, None), (b, h), (b.as_subclass(Sub), h, h, 16, 256, 3)):
        assert m.gemv(*args) is None and m.gemm_skinny(*args) is None
    assert m.gemm_skinny_ws(b, h, h, b, 16, 256, 2) is None and m.gemv_host(b, h, h, h, h, 16, 256, 3) is None


def test_what_was_refused_stays_refused_on_the_cpu():
    b, h = torch.zeros(4096, dtype=torch.uint8), torch.zeros(256, dtype=torch.float16)
    with pytest.raises(TypeError):
        binding.ptqtp_gemv(b, 16, 256, h, y=h, fmt=3)
    with pytest.raises(TypeError):
        binding.ptqtp_gemm_skinny(b, 16, 256, h.reshape(1, 256), Y=h, fmt=3)


def test_addresses_are_four_and_not_null():
    m = functions()
    for args, error in (((1, 2, 3), TypeError), ((0, 0, 0, 0), ValueError), ((None, 1, 2, 3), TypeError)):
        with pytest.raises(error):
            m.bind(*args)


@pytest.mark.gpu
def test_nothing_is_called_before_there_are_addresses():
    # in a process of its own, where nothing has given them
    functions()
    code = """
import importlib.util, torch
spec = importlib.util.spec_from_file_location("_marshal", %r)
m = importlib.util.module_from_spec(spec)
spec.loader.exec_module(m)
b, h = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda"), torch.zeros(1152, dtype=torch.float16, device="cuda")
p = h.cpu()
assert m.gemv(b, h, h, 40, 1152, 3) is None and m.gemm_skinny(b, h, h, 40, 1152, 3) is None
assert m.gemm_skinny_ws(b, h, h, b, 40, 1152, 2) is None and m.gemv_host(b, p, p, h, h, 40, 1152, 3) is None
""" % build.marshal_path()
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300)


@pytest.mark.gpu
@pytest.mark.parametrize("fmt", [1, 2, 3])
def test_both_ways_do_the_same(fmt):
    functions()
    assert binding._gemv_plain is not None
    n, k, M = 40, 1152, 3
    g = torch.Generator(device="cuda").manual_seed(7)
    t = lambda: torch.randint(-1, 2, (n, k), generator=g, device="cuda", dtype=torch.int8)  # noqa: E731
    s = lambda: torch.rand((n, k // 128), generator=g, device="cuda").half()  # noqa: E731
    blob = binding.ptqtp_pack(t(), t(), s(), s(), fmt=fmt)[0]
    X = torch.randn((M, k), generator=g, device="cuda").half()
    names = [v for v in vars(binding) if v.endswith("_plain") and v.startswith("_gem")]
    kept = {v: getattr(binding, v) for v in names}

    def outcome(call):
        try:
            out = call()
            torch.cuda.synchronize()
            return out.cpu()
        except (TypeError, RuntimeError) as e:
            return type(e).__name__ + str(getattr(e, "status", ""))

    class Functions(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    class Dispatch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    def under(mode, call):
        def f():
            with mode():
                return call()
        return f

    y = lambda *shape: torch.zeros(shape or (n,), dtype=torch.float16, device="cuda")  # noqa: E731
    x, host = X[0], lambda v: v.cpu().pin_memory()  # noqa: E731
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    G, S, W, H = binding.ptqtp_gemv, binding.ptqtp_gemm_skinny, binding.ptqtp_gemm_skinny_ws, binding.ptqtp_gemv_host
    calls = {
        "plain": lambda: G(blob, n, k, x, y=y(), fmt=fmt),
        "numpy sizes": lambda: G(blob, np.int64(n), np.int32(k), x, y=y(), fmt=fmt),
        "a stream": lambda: G(blob, n, k, x, y=y(), stream=torch.cuda.current_stream(), fmt=fmt),
        "no output": lambda: G(blob, n, k, x, fmt=fmt),
        "subclass": lambda: G(blob, n, k, x.as_subclass(Sub), y=y(), fmt=fmt),
        "parameter": lambda: G(blob, n, k, torch.nn.Parameter(x), y=y(), fmt=fmt),
        "wrong type": lambda: G(blob, n, k, x.float(), y=y(), fmt=fmt),
        "strided": lambda: G(blob, n, k, torch.zeros(2 * k, device="cuda").half()[::2], y=y(), fmt=fmt),
        "misaligned": lambda: G(blob, n, k, torch.zeros(k + 8, device="cuda").half()[1:k + 1], y=y(), fmt=fmt),
        "host": lambda: G(blob, n, k, x.cpu(), y=y(), fmt=fmt),
        "short blob": lambda: G(blob[:256], n, k, x, y=y(), fmt=fmt),
        "unknown format": lambda: G(blob, n, k, x, y=y(), fmt=9),
        "bad shape": lambda: G(blob, n, k + 1, x, y=y(), fmt=fmt),
        "function mode": under(Functions, lambda: G(blob, n, k, x, y=y(), fmt=fmt)),
        "dispatch mode": under(Dispatch, lambda: G(blob, n, k, x, y=y(), fmt=fmt)),
        "vmap": lambda: torch.func.vmap(lambda v: G(blob, n, k, v, y=v.new_zeros(n), fmt=fmt))(X),
        "rows": lambda: S(blob, n, k, X, Y=y(M, n), fmt=fmt),
        "rows, numpy sizes": lambda: S(blob, np.int64(n), k, X, Y=y(M, n), fmt=fmt),
        "too many rows": lambda: S(blob, n, k, X.repeat(30, 1), Y=y(3 * 30, n), fmt=fmt),
        "workspace": lambda: W(blob, n, k, X, Y=y(M, n), workspace=ws, fmt=fmt),
        "short workspace": lambda: W(blob, n, k, X, Y=y(M, n), workspace=ws[:16], fmt=fmt),
        "host buffers": lambda: H(blob, n, k, host(x), host(y()), y(k), y(), fmt=fmt),
        "host buffers on the device": lambda: H(blob, n, k, x, host(y()), y(k), y(), fmt=fmt),
    }
    got = {name: outcome(call) for name, call in calls.items()}
    try:
        for v in names:
            setattr(binding, v, None)
        want = {name: outcome(call) for name, call in calls.items()}
    finally:
        for v, f in kept.items():
            setattr(binding, v, f)
    for name in calls:
        if isinstance(want[name], str):
            assert got[name] == want[name], name
        else:
            assert torch.equal(got[name], want[name]), name
    assert not isinstance(want["plain"], str) and torch.equal(got["plain"], got["numpy sizes"])
