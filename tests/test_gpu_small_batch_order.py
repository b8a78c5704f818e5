"""Stream order of the small-batch kernels, which are launched as dependents of one another at every overlap level: chains in
which every call reads what the call before it wrote, blobs written directly ahead of a call, the workspace and the output
shared by consecutive calls.  All results are compared bit for bit with synchronised calls."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2509_16989_b200 import binding, build
from paper_2509_16989_b200.inputs import make_case
from gpu_util import assert_parity, dev, oracle_y, pack_case

pytestmark = pytest.mark.gpu
V2, V3 = binding.FORMAT_V2, binding.FORMAT_V3
N = 2048
SMALL = 896                                              # columns and rows of a matrix whose batches the workspace kernel takes
SIZES = [(N, 2), (N, 5), (N, 6), (N, 24), (SMALL, 24)]

# name -> (format, call); what it runs on 2048 x 2048 by the number of rows, and on 896 x 896 at 24:
#   gemv5/gemm7  two rows: batch-1 tiles kernel; more: warp MMAs on int8 activations
#   gemm7 fp16   warp MMAs on fp16 activations; 24 rows of 2048 x 2048: tcgen05 kernel
#   gemm8        tcgen05 kernel, two CTAs per row block
#   format 2     up to three rows: register-stationary kernel; five and six: warp MMAs (and a batch-1 launch for a row left alone); 24:
#                tcgen05 kernel
#   workspace    format 2: up to six rows warp MMAs, 24 tcgen05 kernel; 24 rows of 896 x 896: conversion kernel and workspace kernel
FORMS = {
    "gemv5/gemm7": (V3, lambda p, X, Y, ws, n: binding.ptqtp_gemm_skinny_cfg(p, n, n, X, Y=Y, path=5)),
    "gemm7 fp16": (V3, lambda p, X, Y, ws, n: binding.ptqtp_gemm_skinny_cfg(p, n, n, X, Y=Y, path=6)),
    "gemm8": (V3, lambda p, X, Y, ws, n: binding.ptqtp_gemm_skinny_cfg(p, n, n, X, Y=Y, path=6, k_split=2)),
    "format 2": (V2, lambda p, X, Y, ws, n: binding.ptqtp_gemm_skinny(p, n, n, X, Y=Y, fmt=V2)),
    "workspace": (V2, lambda p, X, Y, ws, n: binding.ptqtp_gemm_skinny_ws(p, n, n, X, Y=Y, workspace=ws, fmt=V2)),
}


@pytest.fixture(scope="module")
def layers():
    # two layers of either size with a gain of about one, so that long chains stay in the range of fp16
    out = {}
    for n in (N, SMALL):
        for seed in (50, 51):
            c = make_case(n, n, seed=seed)
            for a in ("alpha1", "alpha2"):
                c[a] = (c[a].astype(np.float32) * 1.28 * (2048 / n) ** 0.5).astype(np.float16)
            out.setdefault(n, []).append({V2: pack_case(c, V2), V3: pack_case(c, V3)})
    return out


def workspace(n, M):
    return torch.empty(binding.gemm_skinny_workspace_size(n, n, M, fmt=V2), dtype=torch.uint8, device="cuda")


@pytest.fixture(scope="module")
def neighbours(tmp_path_factory):
    """The kernels of dependent_launch.cu."""
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "dependent_launch.cu")
    out = str(tmp_path_factory.mktemp("native") / "dependent_launch.so")
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + [src, "-o", out], check=True)
    lib = ctypes.CDLL(out)
    vp = ctypes.c_void_p
    lib.run_late_writer.argtypes = [vp, ctypes.c_int, ctypes.c_longlong, vp]
    lib.run_early_reader.argtypes = [vp, vp, vp]
    return lib


@pytest.fixture(autouse=True)
def default_level():
    old = binding.ptqtp_set_overlap(0)
    yield
    binding.ptqtp_set_overlap(old)


def bits(t):
    return t.cpu().numpy().view(np.uint16)


def every_pair():
    """Names in an order in which every one follows every one, itself included."""
    names, out = list(FORMS), []
    for i, a in enumerate(names):
        out.append(a)
        for b in names[i + 1:]:
            out += [a, b]
        out.append(a)
    return out + [names[0]] + names[::-1]


@pytest.mark.parametrize("n,M", SIZES)
def test_the_workspace_kernel_is_reached(layers, n, M):
    # it alone writes the workspace
    ws = workspace(n, M).fill_(0xA5)
    fmt, call = FORMS["workspace"]
    call(layers[n][0][fmt], dev(make_case(n, n, seed=57, M=M)["x"]), torch.empty((M, n), dtype=torch.float16, device="cuda"), ws, n)
    assert bool((ws != 0xA5).any()) == (n == SMALL)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("n,M", SIZES)
def test_chain_of_every_kernel_behind_every_kernel(layers, n, M, level, graph):
    order = every_pair()
    assert len({(a, b) for a, b in zip(order, order[1:])}) == len(FORMS) ** 2
    X = dev(make_case(n, n, seed=52, M=M)["x"])
    ws = workspace(n, M)
    Y = [torch.empty((M, n), dtype=torch.float16, device="cuda") for _ in order]
    Z = [torch.empty((M, n), dtype=torch.float16, device="cuda") for _ in range(2)]

    def chain(ys, sync=False):
        for i, name in enumerate(order):
            fmt, call = FORMS[name]
            call(layers[n][i % 2][fmt], X if i == 0 else ys[(i - 1) % len(ys)], ys[i % len(ys)], ws, n)
            if sync:
                torch.cuda.synchronize()

    chain(Y, sync=True)
    want = [bits(y) for y in Y]
    assert np.isfinite(want[-1].view(np.float16)).all() and np.abs(want[-1].view(np.float16).astype(np.float64)).max() > 1e-2
    binding.ptqtp_set_overlap(level)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for ys in (Y, Z):                                # every result kept, then two buffers that take turns
            for y in ys:
                y.fill_(float("nan"))
            if graph:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=stream):
                    chain(ys)
                for _ in range(3):
                    g.replay()
            else:
                chain(ys)
                chain(ys)
            stream.synchronize()
    for i, y in enumerate(Y):
        assert np.array_equal(bits(y), want[i]), (i, order[i])
    assert np.array_equal(bits(Z[(len(order) - 1) % 2]), want[-1])
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("n,M", SIZES)
def test_blob_written_by_a_kernel_directly_ahead_at_level_0(layers, n, M):
    # the blob of every call is rewritten by an elementwise kernel, and the call before that is one that releases its dependents early
    X = dev(make_case(n, n, seed=53, M=M)["x"])
    ws = workspace(n, M)
    for name, (fmt, call) in FORMS.items():
        want = []
        for lay in layers[n]:
            y = torch.empty((M, n), dtype=torch.float16, device="cuda")
            call(lay[fmt], X, y, ws, n)
            want.append(bits(y))
        blob = torch.empty_like(layers[n][0][fmt])
        ys = [torch.empty((M, n), dtype=torch.float16, device="cuda") for _ in range(6)]
        torch.cuda.synchronize()
        for i, y in enumerate(ys):
            torch.add(layers[n][i % 2][fmt], 0, out=blob)
            call(blob, X, y, ws, n)
        torch.cuda.synchronize()
        for i, y in enumerate(ys):
            assert np.array_equal(bits(y), want[i % 2]), (name, i)


@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("n,M", SIZES)
def test_pack_directly_before_a_call(n, M, level):
    # the same blob is packed anew and used by the next call without any synchronisation
    cs = [make_case(n, n, seed=54 + i, M=M) for i in range(2)]
    X = dev(cs[0]["x"])
    planes = [tuple(dev(c[k]) for k in ("T1", "T2", "alpha1", "alpha2")) for c in cs]
    ws = workspace(n, M)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    refs = [oracle_y(dict(c, x=cs[0]["x"])) for c in cs]
    binding.ptqtp_set_overlap(level)
    for name, (fmt, call) in FORMS.items():
        blob = torch.empty(binding.packed_size(n, n, fmt=fmt), dtype=torch.uint8, device="cuda")
        ys = [torch.empty((M, n), dtype=torch.float16, device="cuda") for _ in range(6)]
        torch.cuda.synchronize()
        for i, y in enumerate(ys):
            binding.ptqtp_pack(*planes[i % 2], packed=blob, dev_status=status, fmt=fmt)
            call(blob, X, y, ws, n)
        torch.cuda.synchronize()
        for i, y in enumerate(ys):
            assert_parity(y.cpu().numpy(), refs[i % 2], cs[0]["x"], "%s call %d" % (name, i))
            assert np.array_equal(bits(y), bits(ys[i % 2])), (name, i)
    assert int(status.item()) == 0


@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("n,M", [(N, 6), (SMALL, 24)])
def test_small_batch_behind_batch_1_and_back(layers, n, M, level):
    # activations of a batch written row by row by batch-1 calls, and a row of a small-batch result read by a batch-1 call
    x = dev(make_case(n, n, seed=56, M=M)["x"])
    ws = workspace(n, M)

    def run(sync):
        out = []
        for name, (fmt, call) in FORMS.items():
            X = torch.full((M, n), float("nan"), dtype=torch.float16, device="cuda")
            Y, z = torch.empty((M, n), dtype=torch.float16, device="cuda"), torch.empty(n, dtype=torch.float16, device="cuda")
            torch.cuda.synchronize()
            for m in range(M):
                binding.ptqtp_gemv(layers[n][0][fmt], n, n, x[m], y=X[m], fmt=fmt)
                if sync:
                    torch.cuda.synchronize()
            call(layers[n][1][fmt], X, Y, ws, n)
            if sync:
                torch.cuda.synchronize()
            binding.ptqtp_gemv(layers[n][0][fmt], n, n, Y[M - 1], y=z, fmt=fmt)
            torch.cuda.synchronize()
            out.append((name, bits(Y), bits(z)))
        return out

    want = run(True)
    binding.ptqtp_set_overlap(level)
    for (name, Y, z), (_, Yw, zw) in zip(run(False), want):
        assert np.array_equal(Y, Yw) and np.array_equal(z, zw), name


@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("n,M", SIZES)
def test_a_call_in_stream_order_releases_the_next_kernel_after_all_that_came_before(layers, neighbours, n, M, level):
    # level 0, and the call after a pack at levels 1 and 2: a kernel behind the call that reads without waiting sees what a kernel ahead
    # of the call writes late, although that one released its dependents at once
    X = dev(make_case(n, n, seed=58, M=M)["x"])
    Y = torch.empty((M, n), dtype=torch.float16, device="cuda")
    ws = workspace(n, M)
    c = make_case(16, 128, seed=59)
    planes = tuple(dev(c[k]) for k in ("T1", "T2", "alpha1", "alpha2"))
    small = torch.empty(binding.packed_size(16, 128, fmt=V3), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    word, seen = (torch.zeros(64, dtype=torch.int32, device="cuda") for _ in range(2))
    stream = torch.cuda.Stream()
    for name, (fmt, call) in FORMS.items():
        with torch.cuda.stream(stream):
            call(layers[n][0][fmt], X, Y, ws, n)               # loads the kernels
            binding.ptqtp_set_overlap(level)
            for i in range(4):
                stream.synchronize()
                if level:
                    binding.ptqtp_pack(*planes, packed=small, dev_status=status, fmt=V3)
                assert neighbours.run_late_writer(word.data_ptr(), i + 1, 200_000, stream.cuda_stream) == 0
                call(layers[n][0][fmt], X, Y, ws, n)
                assert neighbours.run_early_reader(word.data_ptr(), seen.data_ptr() + 4 * i, stream.cuda_stream) == 0
            stream.synchronize()
            binding.ptqtp_set_overlap(0)
        assert seen[:4].tolist() == [1, 2, 3, 4], name
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("n,M", [(N, 5), (N, 24), (SMALL, 24)])
def test_two_blobs_packed_directly_before_two_calls(n, M, level):
    # the second call reads a blob whose pack is two kernels ahead of it
    cs = [make_case(n, n, seed=60 + i, M=M) for i in range(2)]
    X = dev(cs[0]["x"])
    planes = [tuple(dev(c[k]) for k in ("T1", "T2", "alpha1", "alpha2")) for c in cs]
    ws = workspace(n, M)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = {}
    for name, (fmt, call) in FORMS.items():
        for i in range(2):
            y = torch.empty((M, n), dtype=torch.float16, device="cuda")
            call(binding.ptqtp_pack(*planes[i], fmt=fmt)[0], X, y, ws, n)
            want[name, i] = bits(y)
    binding.ptqtp_set_overlap(level)
    for a, (fmt_a, call_a) in FORMS.items():
        for b, (fmt_b, call_b) in FORMS.items():
            blobs = [torch.empty(binding.packed_size(n, n, fmt=f), dtype=torch.uint8, device="cuda") for f in (fmt_a, fmt_b)]
            ys = [torch.empty((M, n), dtype=torch.float16, device="cuda") for _ in range(8)]
            torch.cuda.synchronize()
            for i in range(4):
                binding.ptqtp_pack(*planes[i % 2], packed=blobs[0], dev_status=status, fmt=fmt_a)
                binding.ptqtp_pack(*planes[(i + 1) % 2], packed=blobs[1], dev_status=status, fmt=fmt_b)
                call_a(blobs[0], X, ys[2 * i], ws, n)
                call_b(blobs[1], X, ys[2 * i + 1], ws, n)
            torch.cuda.synchronize()
            for i in range(4):
                assert np.array_equal(bits(ys[2 * i]), want[a, i % 2]), (a, b, i)
                assert np.array_equal(bits(ys[2 * i + 1]), want[b, (i + 1) % 2]), (a, b, i)
    assert int(status.item()) == 0


@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("form", ["format 3", "format 2"])
def test_polls_of_the_tcgen05_kernel_do_not_count_the_time_of_the_kernel_ahead(neighbours, form, level):
    # a kernel ahead that releases its dependents at once and works for longer than the polls of a wait last (a launch alone is healthy
    # with 16; 256 run out within these 30 ms); more superblocks per CTA than the ring of codes has stages
    n, k, M = (300, 8192, 24) if form == "format 3" else (2048, 16384, 24)
    c = make_case(n, k, seed=61, M=M)
    packed, X = pack_case(c, V3 if form == "format 3" else V2), dev(c["x"])
    Y = torch.empty((M, n), dtype=torch.float16, device="cuda")
    word = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()

    def call():
        if form == "format 3":
            binding.ptqtp_gemm_skinny_cfg(packed, n, k, X, Y=Y, path=6, k_split=1)
        else:
            binding.ptqtp_gemm_skinny(packed, n, k, X, Y=Y, fmt=V2)

    binding.ptqtp_kernel_status_clear()
    with torch.cuda.stream(stream):
        call()
        stream.synchronize()
        want = bits(Y)
        Y.zero_()
        binding.ptqtp_set_overlap(level)
        old = binding.ptqtp_set_wait_limit(256)
        try:
            stream.synchronize()
            assert neighbours.run_late_writer(word.data_ptr(), 1, 30_000_000, stream.cuda_stream) == 0
            call()
            stream.synchronize()
        finally:
            binding.ptqtp_set_wait_limit(old)
    assert word.item() == 1
    status = binding.ptqtp_kernel_status()
    binding.ptqtp_kernel_status_clear()
    assert status == 0 and np.array_equal(bits(Y), want)
    assert_parity(Y.cpu().numpy(), oracle_y(c), c["x"], form)


@pytest.mark.parametrize("fmt", [V2, V3])
@pytest.mark.parametrize("late", ["pack T1", "pack T2", "pack alpha1", "pack alpha2", "unpack codes", "unpack scales", "unpack header", "decompose W"])
def test_conversions_follow_stream_order_between_dependent_launches(neighbours, late, fmt):
    # a kernel ahead that releases its dependents at once and writes late what the call reads, each operand in turn; a kernel behind that reads
    # without waiting sees what that kernel wrote
    n, k = 48, 1152
    c = make_case(n, k, seed=62)
    form, what = late.split()
    planes = dict((v, dev(c[v])) for v in ("T1", "T2", "alpha1", "alpha2"))
    blob = binding.ptqtp_pack(*planes.values(), fmt=fmt)[0]
    W, status = torch.randn((n, k), generator=torch.Generator().manual_seed(5)).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")

    def call():
        if form == "pack":
            return binding.ptqtp_pack(*planes.values(), packed=torch.empty_like(blob), dev_status=status, fmt=fmt)
        return binding.ptqtp_unpack(blob, n, k, dev_status=status, fmt=fmt) if form == "unpack" else binding.ptqtp_decompose(W)

    # the late word: four trits, two scales, the bytes of four columns, the scales of a row pair, the version of the format, or a weight
    word = 0
    if form == "unpack":
        other = planes["alpha1"].clone()
        other[0, 0] += 1
        scales = int((binding.ptqtp_pack(planes["T1"], planes["T2"], other, planes["alpha2"], fmt=fmt)[0] != blob).nonzero()[0])
        word = {"codes": 64, "scales": scales // 4, "header": 2}[what]
    source = blob if form == "unpack" else W if form == "decompose" else planes[what]
    words = source.flatten().view(torch.int32)[word:]
    old = int(words[0].item())
    new = {"T1": 0x0100ff01, "T2": 0x0100ff01, "alpha1": 0x3c003800, "alpha2": 0x3c003800, "codes": 0x55555555, "scales": 0x3c003800, "header": 99,
           "W": 0x3f800000}[what]
    assert old != new
    stream, seen = torch.cuda.Stream(), torch.zeros(8, dtype=torch.int32, device="cuda")
    kept = []
    with torch.cuda.stream(stream):
        for i in range(4):
            value = new if i % 2 == 0 else old
            status.zero_()
            words[0] = value
            want = [t.clone() for t in call()]
            words[0] = old if i % 2 == 0 else new
            status.zero_()
            stream.synchronize()
            assert neighbours.run_late_writer(words.data_ptr(), value, 200_000, stream.cuda_stream) == 0
            got = call()
            assert neighbours.run_early_reader(words.data_ptr(), seen.data_ptr() + 4 * i, stream.cuda_stream) == 0
            stream.synchronize()
            assert all(torch.equal(g, w) for g, w in zip(got, want)), i
            assert int(seen[i].item()) == value
            kept.append(want)
    # the word matters
    assert any(not torch.equal(a, b) for a, b in zip(kept[0], kept[1]))
