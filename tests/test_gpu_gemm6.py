"""GPU parity of the tcgen05 small-batch kernel on formats 3 and 2 (fp16 trits from tensor memory against fp16
activations, fp32 accumulators in tensor memory) against the fp64 oracle: ragged shapes, every batch size class,
every K split of a cluster, exact integer cases, the library's dispatch and the give-up path of its bounded waits."""
import numpy as np
import pytest
import torch

from paper_2509_16989_b200 import binding
from paper_2509_16989_b200.inputs import make_case
from gpu_util import assert_parity, dev, oracle_y, pack_case

pytestmark = pytest.mark.gpu
V3 = binding.FORMAT_V3


def _run(c, packed, N, K, **kw):
    Y = binding.ptqtp_gemm_skinny_cfg(packed, N, K, dev(c["x"]), path=6, **kw)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


@pytest.mark.parametrize("N,K,M", [(1, 128, 2), (5, 256, 5), (7, 1152, 16), (33, 2048, 17), (130, 3200, 31),
                                   (257, 5120, 32), (64, 14336, 33), (1000, 6144, 48), (37, 36864, 49),
                                   (192, 3072, 64), (2400, 4096, 9), (129, 640, 2), (255, 512, 64), (256, 384, 20)])
@pytest.mark.parametrize("k_split", [0, -1])             # 0: the warp-MMA kernel where the library takes it, up to 32 rows
def test_ragged_shapes_and_batch_sizes(N, K, M, k_split):
    c = make_case(N, K, seed=900 + N + M, M=M)
    Y = _run(c, pack_case(c, V3), N, K, k_split=k_split)
    assert_parity(Y, np.atleast_2d(oracle_y(c)), np.atleast_2d(c["x"]), "N=%d K=%d M=%d" % (N, K, M))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("K", [128, 384, 512, 640, 2176, 4608])
def test_every_number_of_tiles_and_groups_left_over(K):
    # blocks of one to eight tiles (quarters of a block empty or half full), rows that no 16-byte store takes, superblocks of one to four
    # groups at the end, more and fewer superblocks than stages, both sides of every class of batch sizes
    for i, N in enumerate((1, 15, 17, 40, 63, 79, 96, 113, 128, 136, 241)):
        for M in ((16, 33), (17, 48), (32, 64), (9, 49))[i % 4]:
            c = make_case(N, K, seed=600 + N + M, M=M)
            packed = pack_case(c, V3)
            for k_split in (-1, 1, 0):
                Y = _run(c, packed, N, K, k_split=k_split)
                assert_parity(Y, np.atleast_2d(oracle_y(c)), np.atleast_2d(c["x"]), "N=%d K=%d M=%d split %d" % (N, K, M, k_split))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("K,k_split", [(128, 1), (256, 1), (640, 2), (1664, 1), (1792, -1), (3200, 1), (3840, 2), (6272, 1), (7808, 4)])
def test_partial_sums_over_a_last_superblock_of_one_or_two_groups(K, k_split):
    # the partial sums are written where the codes and scales of superblocks 0, 3, 6, ... of a CTA were: a CTA whose last superblock is one
    # of these and has one or two groups; many row blocks, the same bits every time, rows and scales so different that one taken for
    # another shows
    N = 4100
    for M in (5, 16, 33, 64):
        c = make_case(N, K, seed=700 + K + M, M=M)
        c["alpha1"] = (c["alpha1"].astype(np.float32) * np.exp2(np.arange(N) % 5)[:, None]).astype(np.float16)
        packed, x = pack_case(c, V3), dev(c["x"])
        Y = [binding.ptqtp_gemm_skinny_cfg(packed, N, K, x, path=6, k_split=k_split) for _ in range(40)]
        assert all(torch.equal(Y[0].view(torch.int16), y.view(torch.int16)) for y in Y[1:])
        assert_parity(Y[0].cpu().numpy(), oracle_y(c), c["x"], "K=%d M=%d split %d" % (K, M, k_split))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("K", [1024, 2048, 2176, 4608, 6272])
def test_format_2_with_and_without_a_workspace(K):
    # full slices and a last one of one to many groups, blocks with quarters empty, both sides of every class of batch sizes; the calls
    # with and without a workspace give the same bits (no row is left alone by passes of four; up to 16 rows of K = 1024 both run the warp MMAs)
    V2 = binding.FORMAT_V2
    for i, N in enumerate((1602, 1777, 2049, 2400)):
        for M in ((10, 36), (16, 64), (18, 48), (32, 50))[i]:
            c = make_case(N, K, seed=800 + N + M, M=M)
            packed, x = pack_case(c, V2), dev(c["x"])
            ws = torch.empty(binding.gemm_skinny_workspace_size(N, K, M, fmt=V2), dtype=torch.uint8, device="cuda")
            Y = binding.ptqtp_gemm_skinny_ws(packed, N, K, x, workspace=ws, fmt=V2).cpu().numpy()
            ref = np.atleast_2d(oracle_y(c))
            assert_parity(Y, ref, c["x"], "N=%d K=%d M=%d" % (N, K, M))
            assert np.linalg.norm(Y - ref) / np.linalg.norm(ref) < 2.5e-4          # one rounding to fp16: 2.1e-4 (and block fixed point: 2.3e-4)
            assert np.array_equal(Y.view(np.uint16), binding.ptqtp_gemm_skinny(packed, N, K, x, fmt=V2).cpu().numpy().view(np.uint16))
        # a batch whose last row a batch-1 launch takes when there is no workspace, and this kernel when there is
        M = (17, 33, 21, 61)[i]
        c = make_case(N, K, seed=850 + N, M=M)
        packed, x, ref = pack_case(c, V2), dev(c["x"]), oracle_y(c)
        assert_parity(binding.ptqtp_gemm_skinny(packed, N, K, x, fmt=V2).cpu().numpy(), ref, c["x"], "N=%d K=%d M=%d" % (N, K, M))
        assert_parity(binding.ptqtp_gemm_skinny_ws(packed, N, K, x, fmt=V2).cpu().numpy(), ref, c["x"], "N=%d K=%d M=%d workspace" % (N, K, M))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("fmt,N,K,M,fp16", [(2, 1024, 1536, 10, False), (2, 2048, 1536, 12, False), (2, 1536, 1024, 16, False), (2, 20480, 2048, 10, False),
                                            (2, 128, 28672, 10, False), (2, 128, 28672, 6, False), (2, 1280, 2048, 12, True), (2, 4096, 1024, 16, True),
                                            (2, 2048, 3072, 10, True), (2, 1024, 1536, 18, True), (3, 2048, 1536, 18, True), (3, 4096, 1024, 20, True),
                                            (3, 5003, 512, 32, True), (3, 20480, 512, 24, True), (3, 2560, 1536, 25, True)])
def test_either_side_of_the_lines_between_the_kernels(fmt, N, K, M, fp16):
    # one column of 20000 per scale group, with trit 0 in both planes, next to others below 2^-7: with fp16 operands it adds nothing, block
    # fixed point (the warp MMAs on format 2) has no bits left for the others
    g = torch.Generator(device="cuda")
    g.manual_seed(N + M)
    trits = lambda: torch.randint(-1, 2, (N, K), generator=g, device="cuda", dtype=torch.int8)  # noqa: E731
    scale = lambda: (torch.randn((N, K // 128), generator=g, device="cuda") * 0.02).abs().half()  # noqa: E731
    T1, T2, a1, a2 = trits(), trits(), scale(), scale()
    T1[:, 37::128] = T2[:, 37::128] = 0
    X = (torch.randn((M, K), generator=g, device="cuda") * 2.0 ** -9).half()
    X[:, 37::128] = 20000.0
    W = a1.double().repeat_interleave(128, 1) * T1.double() + a2.double().repeat_interleave(128, 1) * T2.double()
    ref = X.double() @ W.T
    packed, _ = binding.ptqtp_pack(T1, T2, a1, a2, fmt=fmt)
    Y = binding.ptqtp_gemm_skinny(packed, N, K, X, fmt=fmt).double()
    error = float((Y - ref).norm() / ref.norm())
    assert error < 1e-3 if fp16 else error > 0.1, error
    X = torch.randn((M, K), generator=g, device="cuda").half()
    Y = binding.ptqtp_gemm_skinny(packed, N, K, X, fmt=fmt).cpu().numpy()
    assert_parity(Y, (X.double() @ W.T).cpu().numpy(), X.cpu().numpy(), "%d x %d, %d rows" % (N, K, M))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("k_split", [1, 2, 4, 8])
@pytest.mark.parametrize("N,K,M", [(300, 4096, 24), (130, 1536, 64), (2050, 512, 7), (48, 7168, 40)])
def test_every_k_split(N, K, M, k_split):
    # a cluster of k_split CTAs shares the columns of a block of 128 rows (some CTAs get no superblock when K is short)
    c = make_case(N, K, seed=77 + k_split, M=M)
    Y = _run(c, pack_case(c, V3), N, K, k_split=k_split)
    assert_parity(Y, oracle_y(c), c["x"], "N=%d K=%d M=%d split %d" % (N, K, M, k_split))
    assert binding.ptqtp_kernel_status() == 0


@pytest.mark.parametrize("N,K,M", [(14336, 4096, 64), (4096, 14336, 16), (1024, 4096, 37), (4096, 4096, 8),
                                   (28672, 4096, 33)])
@pytest.mark.parametrize("k_split", [0, -1])
def test_full_size_shapes(N, K, M, k_split):
    c = make_case(N, K, seed=5 + M, M=M)
    Y = _run(c, pack_case(c, V3), N, K, k_split=k_split)
    assert_parity(Y, oracle_y(c), c["x"], "N=%d K=%d M=%d" % (N, K, M))
    assert binding.ptqtp_kernel_status() == 0


def test_exact_on_integers():
    # integer activations, scales 1 and 2: every product and every fp32 sum is exact, so the result is the integer
    # matrix product for every batch size class and K split
    N, K, M = 200, 4096, 64
    c = make_case(N, K, seed=13, M=M)
    rng = np.random.default_rng(4)
    c["x"] = rng.integers(-3, 4, (M, K)).astype(np.float16)
    c["alpha1"] = np.ones_like(c["alpha1"])
    c["alpha2"] = np.full_like(c["alpha2"], 2.0)
    exact = (c["x"].astype(np.int64) @ c["T1"].astype(np.int64).T) + 2 * (c["x"].astype(np.int64) @ c["T2"].astype(np.int64).T)
    assert np.all(np.abs(exact) < 2048)
    packed = pack_case(c, V3)
    for m in (1, 15, 16, 17, 33, 64):
        for k_split in (1, 4):
            cm = dict(c, x=c["x"][:m].copy())
            Y = _run(cm, packed, N, K, k_split=k_split)
            assert np.array_equal(Y.astype(np.int64), exact[:m]), (m, k_split)


@pytest.mark.parametrize("N,K,M", [(300, 4096, 40), (14336, 4096, 16), (4096, 4096, 64)])
def test_the_tcgen05_kernel_can_be_asked_for_with_a_split_of_its_own(N, K, M):
    # k_split = -1 is one of the explicit splits, bit for bit; 0 is the library's choice, which for up to 32 rows is another kernel or the
    # one that sums the groups of a superblock by themselves first (the last bits of fp32: some of 229376 results round to another fp16 number)
    c = make_case(N, K, seed=88, M=M)
    packed = pack_case(c, V3)
    own, chosen = (_run(c, packed, N, K, k_split=k).view(np.uint16) for k in (-1, 0))
    assert any(np.array_equal(own, _run(c, packed, N, K, k_split=k).view(np.uint16)) for k in (1, 2, 4, 8))
    assert np.array_equal(own, chosen) == (M > 32)


def test_rows_do_not_depend_on_their_neighbours():
    # row m of the result is a function of row m of X alone: the same row inside batches of different size and at a
    # different position gives the same bits
    N, K = 300, 2048
    c = make_case(N, K, seed=31, M=40)
    packed = pack_case(c, V3)
    full = _run(c, packed, N, K, k_split=2)
    part = _run(dict(c, x=c["x"][8:24].copy()), packed, N, K, k_split=2)
    assert np.array_equal(full[8:24].view(np.uint16), part.view(np.uint16))


def test_library_dispatch():
    # the library takes fp16 operands where the fixed cost of the tcgen05 kernel would pay: many rows, or a matrix of some size
    def same(a, b):
        torch.cuda.synchronize()
        return np.array_equal(a.cpu().numpy().view(np.uint16), b.cpu().numpy().view(np.uint16))
    N, K = 4096, 4096
    c = make_case(N, K, seed=40, M=64)
    packed = pack_case(c, V3)
    for M, path in ((64, 6), (16, 6), (4, 5)):
        X = dev(c["x"][:M].copy())
        assert same(binding.ptqtp_gemm_skinny(packed, N, K, X, fmt=V3), binding.ptqtp_gemm_skinny_cfg(packed, N, K, X, path=path)), M
    N, K = 520, 3072
    c = make_case(N, K, seed=41, M=64)
    packed = pack_case(c, V3)
    for M, path in ((64, 6), (8, 5), (7, 5)):
        X = dev(c["x"][:M].copy())
        assert same(binding.ptqtp_gemm_skinny(packed, N, K, X, fmt=V3), binding.ptqtp_gemm_skinny_cfg(packed, N, K, X, path=path)), M


def test_argument_checks():
    N, K = 64, 512
    c = make_case(N, K, seed=1, M=8)
    x = dev(c["x"])
    p3 = pack_case(c, V3)
    for kw in (dict(path=4), dict(path=6, k_split=3), dict(path=6, k_split=16), dict(path=6, k_split=-2)):
        with pytest.raises(binding.PtqtpError) as e:
            binding.ptqtp_gemm_skinny_cfg(p3, N, K, x, **kw)
        assert e.value.status == binding.ERR_CONFIG


@pytest.mark.parametrize("k_split", [1, 4])
def test_bounded_wait_gives_up_reports_and_recovers(k_split):
    # the first wait of every CTA is made to give up: all rows come out as NaN, the status word reports it, the
    # CTAs still meet at their cluster barriers and free their tensor memory, and the next call is healthy
    N, K, M = 700, 2048, 12
    c = make_case(N, K, seed=66, M=M)
    packed = pack_case(c, V3)
    ref = oracle_y(c)
    binding.ptqtp_kernel_status_clear()
    assert binding.ptqtp_kernel_status() == 0
    try:
        binding.ptqtp_test_fail_next_wait(1)
        Y = _run(c, packed, N, K, k_split=k_split)
    finally:
        binding.ptqtp_test_fail_next_wait(0)
    assert np.isnan(Y.astype(np.float64)).all()
    assert binding.ptqtp_kernel_status() == binding.ERR_CUDA
    binding.ptqtp_kernel_status_clear()
    for _ in range(3):                                       # tensor memory was freed: later launches allocate again
        Y = _run(c, packed, N, K, k_split=k_split)
    assert_parity(Y, ref, c["x"], "after the failure")
    assert binding.ptqtp_kernel_status() == 0


def test_many_launches_on_two_streams_give_the_same_bits():
    # tensor memory is allocated and freed by every CTA: launches that share the SMs (two streams, back to back) must
    # neither starve one another nor change a result
    N, K = 2400, 2048
    cs = [make_case(N, K, seed=300 + i, M=M) for i, M in enumerate((9, 24, 40, 64))]
    packed = [pack_case(c, V3) for c in cs]
    xs = [dev(c["x"]) for c in cs]
    want = []
    for c, p, x in zip(cs, packed, xs):
        want.append(binding.ptqtp_gemm_skinny_cfg(p, N, K, x, path=6, k_split=-1).cpu().numpy().view(np.uint16))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [[torch.empty((x.shape[0], N), dtype=torch.float16, device="cuda") for x in xs] for _ in range(2)]
    torch.cuda.synchronize()
    for rep in range(25):
        for si, st in enumerate(streams):
            with torch.cuda.stream(st):
                for i in range(4):
                    j = (i + si + rep) % 4
                    binding.ptqtp_gemm_skinny_cfg(packed[j], N, K, xs[j], Y=outs[si][j], path=6, k_split=(1, 2, 4)[rep % 3],
                                                  stream=st)
    torch.cuda.synchronize()
    assert binding.ptqtp_kernel_status() == 0
    # the sum over a cluster is in rank order, but the split changes which partial sums exist: compare like with like
    for si in range(2):
        for j in range(4):
            got = outs[si][j].cpu().numpy()
            assert_parity(got, oracle_y(cs[j]), cs[j]["x"], "stream %d case %d" % (si, j))
    for j in range(4):
        a = binding.ptqtp_gemm_skinny_cfg(packed[j], N, K, xs[j], path=6, k_split=-1).cpu().numpy().view(np.uint16)
        assert np.array_equal(a, want[j])
