"""The native argument marshalling against the general path: it leaves every
argument that is not of the ordinary kind to the Python code (which raises or
handles it), and for ordinary arguments both give the same bytes and errors.
"""
import ctypes
import importlib
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2608_27370_gb300 as P
from paper_2608_27370_gb300 import workloads as W
import _native_harness as H

DEV = "cuda"
u8, i32, bf16, f32 = torch.uint8, torch.int32, torch.bfloat16, torch.float32


def _buffers(dev, M=256, N=384, K=128):
    e = lambda dt, *s: torch.zeros(s, dtype=dt, device=dev)  # noqa: E731
    op = lambda r, c, role=P.ROLE_ACT: P.FP8Operand(e(u8, r, c), e(u8, *P.scale_vec_shape(r, c)), role=role)  # noqa: E731
    b = dict(x=e(bf16, M, K), st=e(i32, 1), ws=e(u8, 64), amax=e(i32, 1), xo=op(M, K), xt=op(K, M), wo=op(N, K),
             wt=op(K, N), dyo=op(M, N), dyt=op(N, M), y=e(bf16, M, N), dx=e(bf16, M, K), dw=e(bf16, N, K),
             main=e(f32, N, K), rstd=e(f32, M), gu=e(bf16, M, 2 * K), a=e(bf16, M, K), w=e(bf16, N, K), sf=e(f32, 1))
    b["dxo"], b["dxt"] = op(M, K), op(K, M)
    b["table"] = (P.puro_fp8_weight_t * 1)()
    return b


def _native_args(b, M=256, N=384, K=128):
    """Every native function with a whole set of ordinary arguments."""
    q = lambda o, t: (o.data, o.scale, t.data, t.scale)  # noqa: E731
    st = (b["st"], None)
    return {
        "puro_fp8_amax": (b["x"], b["amax"], None),
        "puro_fp8_quantize": (b["x"], 0, 1, 0, None, *q(b["xo"], b["xt"]), *st),
        "puro_fp8_quantize_rmsnorm": (b["x"], None, 1e-6, 0, b["rstd"], b["a"], *q(b["xo"], b["xt"]), *st),
        "puro_fp8_quantize_swiglu": (b["gu"][:, :K], b["gu"][:, K:], 0, b["a"], *q(b["xo"], b["xt"]), *st),
        "puro_fp8_quantize_weights": (ctypes.addressof(b["table"]), 1, 0, *st),
        "puro_fp8_linear_fprop": (b["xo"], b["wo"], b["y"], b["ws"], *st),
        "puro_fp8_linear_dgrad": (b["dyo"], b["wt"], b["dx"], b["ws"], *st),
        "puro_fp8_linear_wgrad": (b["dyt"], b["xt"], b["dw"], b["ws"], *st),
        "puro_fp8_linear_wgrad_main_grad": (b["dyt"], b["xt"], b["main"], b["ws"], *st),
        "puro_fp8_linear_backward": (b["dyo"], b["wt"], b["dx"], b["dyt"], b["xt"], b["dw"], b["ws"], *st),
        "puro_fp8_linear_dgrad_quantize": (b["dyo"], b["wt"], 0, b["dx"], *q(b["dxo"], b["dxt"]), *st),
        "puro_bf16_linear_fprop": (b["x"], b["w"], b["y"], M, N, K, *st),
        "puro_bf16_linear_dgrad": (b["y"], b["dw"], b["dx"], M, N, K, *st),
        "puro_bf16_linear_wgrad": (b["y"], b["x"], b["dw"], M, N, K, *st),
    }


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    """Path of the native module built to run without a GPU."""
    return H.build(tmp_path_factory.mktemp("harness"))


def _odd_arguments(m):
    """What an argument may be instead, ordinary for some of them; m shows tensors as CUDA ones."""
    whole = torch.zeros(64, 64)
    yield from (None, object(), "x", 1.5, float("inf"), 3, True, 2 ** 31, 2 ** 70, np.zeros(4), whole, torch.zeros(0),
                torch.zeros(4, device="meta"), torch.nested.nested_tensor([torch.zeros(2)]))
    for dt in (bf16, f32, u8, i32, torch.uint32, torch.float64, torch.int64):
        yield m.as_cuda(torch.zeros((2, 3), dtype=dt))
        yield m.as_cuda(torch.zeros((256, 128), dtype=dt))
    yield from (m.as_cuda(t) for t in (whole.t(), whole[:, :8], torch.zeros(0), torch.zeros(2, 3, 4, dtype=bf16),
                                       torch.zeros(6, dtype=bf16), torch.zeros(128, 512, dtype=bf16).t(),
                                       torch.zeros(256, 512, dtype=bf16)[:, :128]))
    yield torch.nn.Parameter(m.as_cuda(torch.zeros((256, 128), dtype=bf16)))
    codes, scale = m.as_cuda(torch.zeros((8, 16), dtype=u8)), m.as_cuda(torch.zeros(4))
    yield from (P.FP8Operand(codes, scale, 1, 0, 1), P.FP8Operand(codes, m.as_cuda(whole.t())),
                P.FP8Operand(m.as_cuda(torch.zeros(8, dtype=u8)), scale), P.FP8Operand(codes.view(torch.int8), scale),
                P.FP8Operand(codes, torch.zeros(4)), P.FP8Operand(codes, None), P.FP8Operand(codes, scale, True),
                P.FP8Operand(codes, scale, 2 ** 40))
    yield type("Other", (P.FP8Operand,), {})(codes, scale)


@pytest.mark.parametrize("name", sorted(_native_args(_buffers("cpu"))))
def test_native_calls_the_library_as_ctypes_does(name, harness, monkeypatch):
    """Ordinary arguments are accepted; whatever is accepted reaches the library with the arguments
    of the general path; nothing else reaches it.  Every argument in turn is replaced."""
    lib = H.Recorder()
    m = H.load(harness, lib.addresses)
    monkeypatch.setattr(P, "_lib", lib)
    monkeypatch.setattr(P, "_native", P._CtypesOnly())
    monkeypatch.setattr(P, "_stream", lambda stream: H.STREAM if stream is None else int(stream))
    fn, table = getattr(m, name), (P.puro_fp8_weight_t * 1)()
    table.count = 1
    ordinary = [H.shown_as_cuda(m, a) for a in _native_args(_buffers("cpu"))[name]]
    if name == "puro_fp8_quantize_weights":
        ordinary[0] = ctypes.addressof(table)

    def same(args):
        """Whether the native function accepted; if so, compared."""
        lib.calls.clear()
        got = fn(*args)
        if got is None:
            assert not lib.calls
            return False
        assert got == lib.STATUS
        if name == "puro_fp8_quantize_weights":
            args = [table, *args[2:]] if args[:2] == ordinary[:2] else None
        if args is not None:
            with pytest.raises(P.PuroError):
                getattr(P, name)(*args)
            native, general = lib.calls
            assert native == general
        return True

    assert same(ordinary)
    assert fn() is None and fn(*ordinary, None) is None  # another number of arguments
    for k, a in enumerate(ordinary):
        for odd in _odd_arguments(m):
            if name == "puro_fp8_quantize_weights" and k < 2:
                continue  # made by the binding
            accepted = same([*ordinary[:k], odd, *ordinary[k + 1:]])
            if type(odd) in (object, str, bool, np.ndarray) or (torch.is_tensor(odd) and not odd.is_cuda):
                assert not accepted


def test_native_refuses_an_incomplete_library(harness):
    lib = H.Recorder()
    m = H.load(harness, lib.addresses)
    with pytest.raises(ValueError, match="no address of puro_bf16_linear_wgrad"):
        m.set_library({k: v for k, v in lib.addresses.items() if k != "puro_bf16_linear_wgrad"})


def test_native_declines_tensors_whose_memory_cannot_be_accessed(harness):
    """In a process of its own: a function that throws without the interpreter's lock ends it."""
    env = dict(os.environ, PYTHONPATH=os.pathsep.join(p for p in sys.path if p))
    r = subprocess.run([sys.executable, H.__file__, harness], capture_output=True, text=True, env=env)
    assert r.returncode == 0 and r.stdout.split("\n")[-2] == "declined all", (r.returncode, r.stdout, r.stderr)


@pytest.mark.parametrize("kind", ["another torch", "missing", "not a module"])
def test_without_a_usable_native_module_calls_go_through_ctypes(kind, monkeypatch, tmp_path):
    monkeypatch.setattr(P, "_native", None)
    if kind == "another torch":
        monkeypatch.setattr(torch, "__version__", "2.0.0")
        assert P._build._stale()  # and it is rebuilt
    else:
        monkeypatch.setattr(P._build, "NATIVE", str(tmp_path / "_native.so"))
        if kind == "not a module":
            (tmp_path / "_native.so").write_text("x")
    with pytest.warns(UserWarning, match="marshalled by ctypes"):
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            P.puro_fp8_amax(torch.zeros((4, 4), dtype=bf16), torch.zeros(1, dtype=i32))
    with pytest.raises(ValueError, match="must be a CUDA tensor"):  # and says so once
        P.puro_bf16_linear_fprop(*(torch.zeros((4, 4), dtype=bf16) for _ in range(3)), 4, 4, 4)


@pytest.fixture
def copy_of_the_package(tmp_path):
    """The package a second time in this process, from other files."""
    shutil.copytree(os.path.dirname(P.__file__), tmp_path / "puro_copy",
                    ignore=shutil.ignore_patterns("_build", "__pycache__"))
    sys.path.insert(0, str(tmp_path))
    try:
        yield importlib.import_module("puro_copy")
    finally:
        sys.path.remove(str(tmp_path))
        for name in [n for n in sys.modules if n.split(".")[0] == "puro_copy"]:
            del sys.modules[name]


def test_a_copy_of_the_package_brings_no_second_binding_to_the_library(copy_of_the_package):
    C = copy_of_the_package
    P._load_native(), C._load_native()
    address = lambda lib: ctypes.cast(lib.puro_fp8_amax, ctypes.c_void_p).value  # noqa: E731
    assert address(P.load_library()) != address(C.load_library())
    # linked by name, the copy's module would find the library loaded first
    with pytest.raises(AttributeError):
        ctypes.CDLL(C._build.NATIVE).puro_fp8_amax


@pytest.mark.gpu
def test_a_copy_of_the_package_calls_its_own_library(copy_of_the_package):
    """The wait bound set through one copy (by ctypes) holds for that copy's hot calls alone."""
    C = copy_of_the_package
    x = W.normal_bf16((4096, 4096), 1.0, DEV, 60)
    got = {}
    for bounded in (P, C):
        bounded.puro_set_wait_timeout_ns(0)
        try:
            for p in (P, C):
                status = torch.zeros(1, dtype=torch.int32, device=DEV)
                q = p.quantize(x, p.E4M3)
                p.puro_fp8_quantize(x, p.E4M3, p.SCALE_BLOCK, p.ROLE_ACT, None, q.rowwise.data, q.rowwise.scale,
                                    q.colwise.data, q.colwise.scale, status)
                got[bounded, p] = p.puro_fp8_get_status(status)
        finally:
            bounded.puro_set_wait_timeout_ns(2_000_000_000)
    assert got == {(b, p): P.PURO_ERR_TIMEOUT if b is p else P.PURO_OK for b in (P, C) for p in (P, C)}


def _random(b):
    for k, t in enumerate(("x", "w", "gu")):
        b[t].copy_(W.normal_bf16(tuple(b[t].shape), 1.0, DEV, 40 + k))
    for k, t in enumerate(("xo", "xt", "wo", "wt", "dyo", "dyt")):
        r = W.normal_bf16((b[t].rows, b[t].red), 1.0, DEV, 50 + k)
        P.puro_fp8_quantize(r, 0, 1, 0, None, b[t].data, b[t].scale)


def _calls(b, M=256, N=384, K=128):
    for name, args in _native_args(b, M, N, K).items():
        if name == "puro_fp8_quantize_weights":
            q = P.Quantized(b["wo"], P.FP8Operand(b["wt"].data, b["wt"].scale))
            yield name, lambda q=q: P.puro_fp8_quantize_weights([(b["w"], q)], 0, b["st"])
        else:
            yield name, lambda name=name, args=args: getattr(P, name)(*args)
    yield "stream object", lambda: P.puro_fp8_linear_fprop(b["xo"], b["wo"], b["y"], b["ws"], b["st"],
                                                           torch.cuda.current_stream())
    yield "per-tensor", lambda: P.puro_fp8_quantize(b["x"], 1, 0, 0, b["amax"], b["xo"].data, b["sf"], b["xt"].data,
                                                    None)
    yield "keywords", lambda: P.puro_fp8_linear_dgrad(b["dyo"], b["wt"], dx=b["dx"], dev_status=b["st"])


@pytest.mark.gpu
def test_both_paths_give_the_same_bytes():
    P._load_native()
    got = []
    native = P._native
    try:
        for route in (native, P._CtypesOnly()):
            P._native = route
            b = _buffers(DEV)
            _random(b)
            if route is native:  # they are taken, not handed back
                for name, args in _native_args(b).items():
                    assert getattr(native, name)(*args) == P.PURO_OK, name
                b["main"].zero_()
            for name, call in _calls(b):
                call()
            torch.cuda.synchronize()
            flat = []
            for k in sorted(b):
                v = b[k]
                flat += [v.data, v.scale] if isinstance(v, P.FP8Operand) else [v] if torch.is_tensor(v) else []
            got.append([t.contiguous().view(u8) for t in flat])
    finally:
        P._native = native
    assert all(torch.equal(a, c) for a, c in zip(*got))
    assert any(int(t.count_nonzero()) for t in got[0])


@pytest.mark.gpu
@pytest.mark.parametrize("route", ["native", "general"])
def test_errors_are_the_same(route):
    native = P._load_native()
    b = _buffers(DEV)
    q = (b["xo"].data, b["xo"].scale, b["xt"].data, b["xt"].scale)
    try:
        P._native = native if route == "native" else P._CtypesOnly()
        with pytest.raises(ValueError, match="x has dtype"):
            P.puro_fp8_quantize(b["x"].float(), 0, 1, 0, None, *q)
        with pytest.raises(ValueError, match="x must be contiguous"):
            P.puro_fp8_quantize(b["gu"][:, :128], 0, 1, 0, None, *q)
        with pytest.raises(ValueError, match="scale has dtype"):
            P.puro_fp8_quantize(b["x"], 0, 1, 0, None, q[0], b["sf"], q[2], q[3])
        with pytest.raises(ValueError, match="out must be a CUDA tensor"):
            P.puro_fp8_linear_fprop(b["xo"], b["wo"], b["y"].cpu())
        with pytest.raises(ValueError, match="unit column stride"):
            P.puro_fp8_quantize_swiglu(b["gu"].t(), b["gu"].t(), 0, None, *q)
        with pytest.raises(AttributeError):
            P.puro_fp8_linear_fprop(None, b["wo"], b["y"])
        for call in (lambda: P.puro_fp8_quantize(b["x"], 7, 1, 0, None, *q),
                     lambda: P.puro_fp8_linear_fprop(b["xo"], b["dyo"], b["y"]),
                     lambda: P.puro_fp8_linear_fprop(b["xo"], b["wo"], None),
                     lambda: P.puro_fp8_linear_fprop(P.FP8Operand(b["xo"].data[:0], b["xo"].scale), b["wo"], b["y"]),
                     lambda: P.puro_fp8_quantize_rmsnorm(b["x"], None, -1.0, 0, b["rstd"], None, *q)):
            with pytest.raises(P.PuroError) as e:
                call()
            assert e.value.status == P.PURO_ERR_INVALID_ARG
    finally:
        P._native = native
