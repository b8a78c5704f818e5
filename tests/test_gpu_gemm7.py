"""GPU parity of the warp-MMA small-batch kernel (fp16 activations on format 3, 15-bit block fixed point on formats 3 and 2)
against the fp64 oracle, at the edges of its tiles: row pairs, superblocks and slices, column tiles, one launch or several,
columns in chunks, matrices taller than a launch; exact integer cases, the give-up path of its bounded waits.  (The library gives
some of the larger cases to other kernels: fp16 with more than 32 rows and 16 rows of 4100 x 6144, on either format, to the tcgen05
kernel, more than 16 rows of format 2 to the workspace kernel.)"""
import numpy as np
import pytest
import torch

from paper_2509_16989_b200 import binding
from paper_2509_16989_b200.inputs import make_case
from gpu_util import assert_parity, dev, oracle_y, pack_case

pytestmark = pytest.mark.gpu
V2, V3 = binding.FORMAT_V2, binding.FORMAT_V3
KINDS = ("fp16", "int8", "format2")


def run(kind, packed, N, K, X):
    if kind == "format2":
        Y = binding.ptqtp_gemm_skinny_ws(packed, N, K, X, fmt=V2)
    else:
        Y = binding.ptqtp_gemm_skinny_cfg(packed, N, K, X, path=6 if kind == "fp16" else 5)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


def pack_for(kind, c):
    return pack_case(c, V2 if kind == "format2" else V3)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("N,K,M", [(1, 128, 5), (15, 384, 8), (17, 512, 9), (33, 640, 16), (47, 2048, 7), (64, 2176, 6), (31, 4224, 13),
                                   (2375, 1920, 5), (4100, 6144, 16), (1500, 9728, 5), (200, 14336, 4), (97, 28672, 11)])
def test_edges(kind, N, K, M):
    c = make_case(N, K, seed=N + K + M, M=M)
    Y = run(kind, pack_for(kind, c), N, K, dev(c["x"]))
    assert_parity(Y, oracle_y(c), c["x"], "%s %d x %d, %d rows" % (kind, N, K, M))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("M", [2, 3, 4, 5, 8, 9, 12, 15, 16, 17, 24, 25, 32, 33, 63, 64])
def test_every_number_of_column_tiles(kind, M):
    N, K = 330, 10240                                        # long enough for the warp-MMA kernel from two rows on
    c = make_case(N, K, seed=100 + M, M=M)
    Y = run(kind, pack_for(kind, c), N, K, dev(c["x"]))
    assert_parity(Y, oracle_y(c), c["x"], "%s %d rows" % (kind, M))


@pytest.mark.parametrize("kind", ["int8", "format2"])
@pytest.mark.parametrize("level", [0, 1, 2])
def test_overlap_levels_give_the_same_bits(kind, level):
    # every x but the first is written by a copy kernel directly ahead of the call
    N, K, M = 1040, 9216, 4
    c = make_case(N, K, seed=7, M=M)
    packed = pack_for(kind, c)
    X0 = dev(c["x"])
    want = run(kind, packed, N, K, X0)
    old = binding.ptqtp_set_overlap(level)
    try:
        for rep in range(4):
            X = torch.zeros_like(X0)
            X.add_(X0)
            assert np.array_equal(run(kind, packed, N, K, X).view(np.uint16), want.view(np.uint16)), (level, rep)
    finally:
        binding.ptqtp_set_overlap(old)


@pytest.mark.parametrize("kind", KINDS)
def test_columns_in_chunks(kind):
    # no CTA has room for its columns: activations come in chunks, sums wait in shared memory
    N, K, M = 40, 147456, 6
    c = make_case(N, K, seed=3, M=M)
    Y = run(kind, pack_for(kind, c), N, K, dev(c["x"]))
    assert_parity(Y, oracle_y(c), c["x"], kind)
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("kind", KINDS)
def test_matrix_taller_than_a_launch(kind):
    N, K, M = 600_011, 128, 6
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    trits = lambda: torch.randint(-1, 2, (N, K), generator=g, device="cuda", dtype=torch.int8)  # noqa: E731
    scale = lambda: (torch.randn((N, 1), generator=g, device="cuda") * 0.02).abs().half()  # noqa: E731
    T1, T2, a1, a2 = trits(), trits(), scale(), scale()
    X = torch.randn((M, K), generator=g, device="cuda").half()
    packed, _ = binding.ptqtp_pack(T1, T2, a1, a2, fmt=V2 if kind == "format2" else V3)
    Y = run(kind, packed, N, K, X)
    W = a1.double() * T1.double() + a2.double() * T2.double()
    assert_parity(Y, (X.double() @ W.T).cpu().numpy(), X.cpu().numpy(), kind)


@pytest.mark.parametrize("N,K,M,writes", [(8192, 28672, 8, True), (8192, 32768, 8, False), (4096, 28672, 8, False), (8192, 28672, 3, True)])
def test_workspace_call_leaves_uneven_clusters_to_the_workspace_kernel(N, K, M, writes):
    # 14 slices over clusters of eight: the kernel that converts X into the workspace is faster; 16 slices, or clusters of four: not
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    trits = lambda: torch.randint(-1, 2, (N, K), generator=g, device="cuda", dtype=torch.int8)  # noqa: E731
    scale = lambda: (torch.randn((N, K // 128), generator=g, device="cuda") * 0.02).abs().half()  # noqa: E731
    T1, T2, a1, a2 = trits(), trits(), scale(), scale()
    X = torch.randn((M, K), generator=g, device="cuda").half()
    packed, _ = binding.ptqtp_pack(T1, T2, a1, a2, fmt=V2)
    ws = torch.full((binding.gemm_skinny_workspace_size(N, K, M, fmt=V2),), 0xA5, dtype=torch.uint8, device="cuda")
    Y = binding.ptqtp_gemm_skinny_ws(packed, N, K, X, workspace=ws, fmt=V2)
    assert bool((ws != 0xA5).any()) == writes
    rows = torch.cat([torch.arange(64, device="cuda"), torch.arange(N - 64, N, device="cuda")])
    W = a1[rows].double().repeat_interleave(128, 1) * T1[rows].double() + a2[rows].double().repeat_interleave(128, 1) * T2[rows].double()
    assert_parity(Y[:, rows].cpu().numpy(), (X.double() @ W.T).cpu().numpy(), X.cpu().numpy(), "%d x %d" % (N, K))


@pytest.mark.parametrize("kind", KINDS)
def test_exact_on_integers(kind):
    N, K, M = 200, 10240, 7
    c = make_case(N, K, seed=13, M=M)
    rng = np.random.default_rng(4)
    c["x"] = rng.integers(-2, 3, (M, K)).astype(np.float16)
    c["alpha1"] = np.ones_like(c["alpha1"])
    c["alpha2"] = np.full_like(c["alpha2"], 2.0)
    exact = c["x"].astype(np.int64) @ (c["T1"].astype(np.int64) + 2 * c["T2"].astype(np.int64)).T
    assert np.all(np.abs(exact) < 2048)
    assert np.array_equal(run(kind, pack_for(kind, c), N, K, dev(c["x"])).astype(np.int64), exact)


def test_small_and_large_activations():
    # fp16 operands: the whole range of a half, subnormal ones included, next to large ones in one group
    N, K, M = 64, 1024, 5
    c = make_case(N, K, seed=17, M=M)
    rng = np.random.default_rng(8)
    c["x"] = (rng.standard_normal((M, K)) * np.exp2(rng.integers(-22, 8, (M, K)))).astype(np.float16)
    Y = run("fp16", pack_for("fp16", c), N, K, dev(c["x"]))
    ref = oracle_y(c)
    # A group's sum of (trit + 1) x is eight MMA steps, each cut off at 2^-23 of the largest number in it, at most twice the sum
    # of magnitudes: 2^-19 of that sum, scaled (2^-19.4 seen); then one rounding to fp16.
    bound = 2.0 ** -19 * np.abs(c["x"].astype(np.float64)).sum(1, keepdims=True) * float(c["alpha1"].max() + c["alpha2"].max()) \
        + 2.0 ** -11 * np.abs(ref) + 2.0 ** -24
    assert np.all(np.abs(Y.astype(np.float64) - ref) <= bound)


@pytest.mark.parametrize("k_split", [0, 1])
@pytest.mark.parametrize("N,K,M", [(47, 640, 8), (64, 4096, 5), (330, 10240, 16), (33, 2048, 32)])
def test_columns_whose_trits_are_zero_add_nothing(N, K, M, k_split):
    # fp16 operands: one column per scale group holds 20000 and more, with trit 0 in both planes, next to multiples of 2^-10 below
    # 2^-7.  Every sum without those columns is a multiple of 2^-10 below 2^14, exact in fp32, and every result one below 2,
    # exact in fp16; 20000 added and taken off again leaves multiples of 2^-8 at best.
    c = make_case(N, K, seed=19 + M, M=M)
    rng = np.random.default_rng(9)
    c["x"] = (rng.integers(-7, 8, (M, K)) * 2.0 ** -10 * (rng.random((M, K)) < 0.2)).astype(np.float16)
    cols = np.arange(37, K, 128)
    c["x"][:, cols] = (20000 + 16 * rng.integers(0, 1000, (M, cols.size))).astype(np.float16)
    c["T1"][:, cols] = c["T2"][:, cols] = 0
    c["alpha1"] = np.ones_like(c["alpha1"])
    c["alpha2"] = np.full_like(c["alpha2"], 2.0)
    exact = c["x"].astype(np.float64) @ (c["T1"].astype(np.float64) + 2 * c["T2"].astype(np.float64)).T
    assert np.all(np.abs(exact) < 2)
    Y = binding.ptqtp_gemm_skinny_cfg(pack_for("fp16", c), N, K, dev(c["x"]), path=6, k_split=k_split)
    assert np.array_equal(Y.cpu().numpy().astype(np.float64), exact)


def test_infinite_activations_reach_the_same_rows_on_both_kernels():
    # an infinity times a trit of 0 is NaN, times other trits an infinity, whichever kernel takes fp16 operands
    N, K, M = 90, 1024, 6
    c = make_case(N, K, seed=23, M=M)
    c["x"][1, 5], c["x"][2, 700], c["x"][4, 1000] = np.inf, -np.inf, np.nan
    packed = pack_for("fp16", c)
    want, got = (binding.ptqtp_gemm_skinny_cfg(packed, N, K, dev(c["x"]), path=6, k_split=k).cpu().numpy() for k in (1, 0))
    assert np.isinf(want[1]).any() and np.isnan(want[1]).any()
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    assert np.all(np.isfinite(got[[0, 3, 5]]))


@pytest.mark.parametrize("kind", KINDS)
def test_bounded_wait_gives_up_reports_and_recovers(kind):
    N, K, M = 700, 9216, 12
    c = make_case(N, K, seed=66, M=M)
    packed = pack_for(kind, c)
    binding.ptqtp_kernel_status_clear()
    try:
        binding.ptqtp_test_fail_next_wait(1)
        Y = run(kind, packed, N, K, dev(c["x"]))
    finally:
        binding.ptqtp_test_fail_next_wait(0)
    assert np.isnan(Y.astype(np.float64)).all()
    assert binding.ptqtp_kernel_status() == binding.ERR_CUDA
    binding.ptqtp_kernel_status_clear()
    assert_parity(run(kind, packed, N, K, dev(c["x"])), oracle_y(c), c["x"], "after the failure")
    assert binding.ptqtp_kernel_status() == 0
