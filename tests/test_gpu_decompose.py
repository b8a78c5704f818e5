"""GPU trit-plane decomposition (ptqtp_decompose) against the CPU oracle: identical planes, scales to 1e-12, the
same number of sweeps and the same error and change histories; the hand-worked 2 x 4 example; degenerate groups."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest
import torch

from golden_io import load_worked_2x4
from oracle.c_oracle import decompose_c
from oracle.decompose import decompose, reconstruction_error
from paper_2509_16989_b200 import binding, build
from paper_2509_16989_b200.inputs import make_activations, make_weights
from gpu_util import assert_parity, dev, oracle_y

pytestmark = pytest.mark.gpu


def run(W, **kw):
    T1, T2, a1, a2, info = binding.ptqtp_decompose(dev(np.ascontiguousarray(W, dtype=np.float32)), details=True, **kw)
    return dict(T1=T1.cpu().numpy(), T2=T2.cpu().numpy(), alpha1_fp16=a1.cpu().numpy(), alpha2_fp16=a2.cpu().numpy(), **info)


def assert_same(got, ref, what=""):
    assert got["sweeps"] == ref["sweeps"], what
    assert np.array_equal(got["T1"], ref["T1"]) and np.array_equal(got["T2"], ref["T2"]), what
    for k in ("alpha1", "alpha2"):
        assert np.all(np.abs(got[k] - ref[k]) <= 1e-12 * np.maximum(1.0, np.abs(ref[k]))), what
        assert np.array_equal(got[k + "_fp16"].view(np.uint16), ref[k + "_fp16"].view(np.uint16)), what
    assert np.allclose(got["delta_history"], ref["delta_history"], rtol=1e-12, atol=1e-300), what
    assert np.allclose(got["err_history"], ref["err_history"], rtol=1e-10, atol=1e-300), what


def test_worked_2x4_example():
    g = load_worked_2x4()
    W = np.array([[float(v) for v in row] for row in g["W"]], dtype=np.float32)
    out = run(W, group=4)
    assert out["sweeps"] == g["n_sweeps"]
    for row in (0, 1):
        want = g["canon"][row]
        assert list(out["T1"][row]) == want["T1"] and list(out["T2"][row]) == want["T2"]
        assert abs(out["alpha1"][row, 0] - float(want["alpha"][0])) < 5e-6
        assert abs(out["alpha2"][row, 0] - float(want["alpha"][1])) < 5e-6
    # the squared error after every sweep (both rows together), and the final total of 2
    for t in range(1, g["n_sweeps"] + 1):
        want = float(g["sweeps"][(t, 0)]["E"] + g["sweeps"][(t, 1)]["E"])
        assert abs(out["err_history"][t - 1] - want) < 1e-4
    assert abs(out["err_history"][-1] - float(g["Etotal"])) < 1e-5
    # without the normal form the planes of the last sweep come back as they are
    raw = run(W, group=4, canonicalize=False)
    for row in (0, 1):
        last = g["sweeps"][(g["n_sweeps"], row)]
        assert list(raw["T1"][row]) == last["T1"] and list(raw["T2"][row]) == last["T2"]
        assert abs(raw["alpha1"][row, 0] - float(last["alpha"][0])) < 5e-6


@pytest.mark.parametrize("N,K,seed", [(512, 4096, 40), (37, 1152, 41), (1, 128, 42), (130, 256, 43)])
def test_matches_the_cpu_oracle(N, K, seed):
    W = make_weights(N, K, seed=seed)
    assert_same(run(W), decompose_c(W), "N=%d K=%d" % (N, K))
    assert_same(run(W, canonicalize=False), decompose_c(W, canonicalize=False), "raw iterate")


@pytest.mark.parametrize("G", [4, 32, 64, 256])
def test_other_group_sizes_and_sweep_limits(G):
    W = make_weights(48, 1024, seed=50 + G)
    assert_same(run(W, group=G), decompose_c(W, G=G), "G=%d" % G)
    assert_same(run(W, group=G, t_max=3), decompose_c(W, G=G, T_max=3), "three sweeps")
    assert_same(run(W, group=G, eps=1e-2), decompose_c(W, G=G, eps=1e-2), "loose eps")


def test_degenerate_groups():
    rng = np.random.default_rng(7)
    W = (rng.standard_normal((64, 512)) * 0.02).astype(np.float32)
    W[3, 128:256] = 0.0                 # an all-zero group: alpha = 0, planes 0, no NaN
    W[5, :128] = 0.25                   # a constant group
    W[7, 256:384] = np.where(rng.random(128) < 0.5, 0.5, -0.5).astype(np.float32)     # exactly one level
    W[9, :] = 0.0
    W[11, 384:] = np.repeat(np.array([1.0, -2.0, 3.0, 0.0], np.float32), 32)
    W[13, 0] = 1e4                      # a huge outlier
    W[15, :128] = -0.0
    got, ref = run(W), decompose_c(W)
    assert_same(got, ref, "degenerate")
    assert np.all(np.isfinite(got["alpha1"])) and np.all(np.isfinite(got["alpha2"]))
    assert not got["T1"][3, 128:256].any() and not got["T2"][3, 128:256].any()
    assert got["alpha1"][3, 1] == 0.0 and got["alpha2"][3, 1] == 0.0
    # and the numpy oracle agrees on a slice (the C oracle is bit-identical to it)
    sub = decompose(W[:16])
    assert np.array_equal(run(W[:16])["T1"], sub["T1"])


def _special(kind, rng):
    """Weights at which the sorted sums, the runs of the quantiser or the second pass can go wrong."""
    W = (rng.standard_normal((70, 640)) * 0.02).astype(np.float32)
    if kind == "inexact sums":          # magnitudes too far apart for exact sums, in every group of half of the rows
        W[::2] *= np.exp2(rng.integers(-40, 3, W[::2].shape)).astype(np.float32)
    elif kind == "few values":          # ties everywhere: multiples of 1/8, zeros of both signs among them
        W = (rng.integers(-4, 5, W.shape) / 8).astype(np.float32)
        W[3:9] *= -1.0
    elif kind == "short mantissas":     # as from a 16-bit checkpoint
        W = torch.from_numpy(W).bfloat16().float().numpy()
    elif kind == "one plane":           # W = c * sign: the second scale is nothing but rounding
        W = (np.where(rng.random(W.shape) < 0.5, 1.0, -1.0) * 0.3).astype(np.float32)
    elif kind == "planes":              # what two planes represent: the error falls to the rounding of its own sums
        t = rng.integers(-1, 2, (2,) + W.shape)
        W = (0.02 * t[0] + 0.0075 * t[1]).astype(np.float32)
    elif kind == "extremes":
        W[:20] *= np.float32(1e-41)     # subnormal
        W[20:40] *= np.float32(1e36)
    return W


@pytest.mark.parametrize("kind", ["inexact sums", "few values", "short mantissas", "one plane", "planes", "extremes"])
@pytest.mark.parametrize("G,kw,okw", [(128, {}, {}), (20, {}, {}), (160, {"eps": 1e-2}, {"eps": 1e-2}),
                                      (5, {"t_max": 2}, {"T_max": 2}), (64, {"eps": 0.0, "t_max": 30}, {"eps": 0.0, "T_max": 30})])
def test_sorted_sweeps_match_the_oracle(kind, G, kw, okw):
    W = _special(kind, np.random.default_rng(70 + G))
    assert_same(run(W, group=G, **kw), decompose_c(W, G=G, **okw), "%s G=%d" % (kind, G))


@pytest.mark.parametrize("G", [1, 3, 16, 31, 32, 33, 63, 64, 65, 128, 129, 132, 255, 256])
def test_every_sort_width_and_ragged_batches_of_group_rows(G):
    # sorts of 32, 64, 128 and 256 values with and without padding, vector loads and single ones, the last batch of 32 group-rows and
    # of eight cut short; magnitudes repeated with both signs, zeros of both signs among them
    rng = np.random.default_rng(400 + G)
    for rows in (1, 7, 9, 33):
        W = (rng.standard_normal((rows, G)) * 0.02).astype(np.float32)
        W[:, ::3] = np.copysign(W[:, :1], W[:, ::3])
        W[::2, 1::5] = np.copysign(np.float32(0.0), W[::2, 1::5])
        for canonicalize in (True, False):
            assert_same(run(W, group=G, canonicalize=canonicalize), decompose_c(W, G=G, canonicalize=canonicalize), "%d x %d" % (rows, G))


@pytest.mark.parametrize("rows,K,G,kw,okw", [(2048, 4096, 128, {}, {}), (1000, 1536, 24, {"t_max": 12}, {"T_max": 12}),
                                             (1024, 2048, 32, {"eps": 0.05}, {"eps": 0.05})])
def test_lanes_that_take_one_group_row_after_the_other(rows, K, G, kw, okw):
    # more group-rows than the lanes of the device: group-rows of every length of run beside each other in a warp, zeros, constants,
    # inexact sums, subnormal and huge weights, and errors that are next to nothing among them
    rng = np.random.default_rng(500 + G)
    W = (rng.standard_normal((rows, K)) * 0.02).astype(np.float32)
    W[rng.random(W.shape) < 1e-3] *= 20
    g = W.reshape(-1, G)
    n = g.shape[0]
    pick = lambda share: rng.random(n) < share  # noqa: E731
    g[pick(0.02)] = 0.0
    g[pick(0.02)] = np.float32(0.25)
    m = pick(0.02)
    g[m] *= np.exp2(rng.integers(-40, 3, g[m].shape)).astype(np.float32)
    g[pick(0.01)] *= np.float32(1e-41)
    g[pick(0.01)] *= np.float32(1e30)
    m = pick(0.02)
    g[m] = (0.02 * rng.integers(-1, 2, g[m].shape) + 0.0075 * rng.integers(-1, 2, g[m].shape)).astype(np.float32)
    assert_same(run(W, group=G, **kw), decompose_c(W, G=G, **okw), "%d x %d G=%d" % (rows, K, G))


@pytest.mark.parametrize("t_max", [1, 2, 999, 1000])
def test_histories_with_and_without_room_for_the_records(t_max):
    # few weights and many sweeps: the records of errors find no room beside the planes
    for rows, G in ((1, 128), (3, 16), (40, 128)):
        W = (np.random.default_rng(600 + rows).standard_normal((rows, 2 * G)) * 0.02).astype(np.float32)
        assert_same(run(W, group=G, t_max=t_max, eps=0.0), decompose_c(W, G=G, T_max=t_max, eps=0.0), "%d %d" % (rows, t_max))


@pytest.mark.parametrize("kind", ["normal", "few values", "short mantissas", "one plane", "planes", "extremes", "inexact sums"])
@pytest.mark.parametrize("G", [128, 64, 20, 256])
def test_scales_bit_for_bit(kind, G):
    # every operation of the solve is rounded on its own, so the unrounded scales are the oracle's to the last bit, sweep by sweep
    W = _special(kind, np.random.default_rng(900 + G))[:, :2 * G]
    for t_max in (1, 2, 3, 9, 50):
        got, ref = run(W, group=G, t_max=t_max, canonicalize=False), decompose_c(W, G=G, T_max=t_max, canonicalize=False)
        for k in ("alpha1", "alpha2"):
            assert np.array_equal(got[k].view(np.uint64), ref[k].view(np.uint64)), (t_max, k)


def test_one_reciprocal_serves_both_divisions(tmp_path):
    # the shared reciprocal with two corrections per quotient against IEEE divisions, and both against numpy: sums as they occur, counts of
    # 0 to 256 weights, determinants from that of lambda alone (1e-16) on, weights from subnormal to huge, sums of zero
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "alpha_step.cu")
    out = str(tmp_path / "alpha_step.so")
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-I", build.CSRC, src, "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.run_compare.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    rng = np.random.default_rng(11)
    n = 4_000_000
    n11, n22 = rng.integers(0, 257, n), rng.integers(0, 257, n)
    n11[::50], n22[::70] = 0, 0
    n12 = np.rint((2 * rng.random(n) - 1) * np.minimum(n11, n22)).astype(np.int64)
    n12[::9] = np.minimum(n11, n22)[::9]
    same = rng.random(n) < 0.05                          # both planes alike: singular but for lambda
    n22, n12 = np.where(same, n11, n22), np.where(same, n11, n12)
    unit = np.exp2(rng.integers(-149, 105, n).astype(np.float64))
    b1, b2 = (np.rint((2 * rng.random(n) - 1) * 2.0 ** rng.integers(0, 30, n)) * unit for _ in range(2))
    b2 = np.where(same, b1, b2)
    lam = np.where(rng.random(n) < 0.7, 1e-8, 10.0 ** (-8 * rng.random(n)))
    v = np.stack([n11, n22, n12, b1 + 0.0, b2 + 0.0, lam], axis=1).astype(np.float64)
    d_in, d_out, differ = dev(v), torch.empty((n, 3), dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    assert lib.run_compare(d_in.data_ptr(), n, d_out.data_ptr(), differ.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    got = d_out.cpu().numpy()
    assert int(differ.item()) == 0
    n11, n22, n12, b1, b2, lam = v.T
    with np.errstate(all="ignore"):
        A11, A22 = n11 + lam, n22 + lam
        det = A11 * A22 - n12 * n12
        kappa = ((A11 * A11 + A22 * A22) + (2.0 * n12) * n12) / np.abs(det)
        grown = np.maximum(np.where(kappa >= 1e6, np.minimum(lam * np.sqrt(kappa / 1e6), 1.0), lam), 1e-8)
        A11, A22 = n11 + grown, n22 + grown
        det = A11 * A22 - n12 * n12
        want = np.stack([(A22 * b1 - n12 * b2) / det, (A11 * b2 - n12 * b1) / det, grown], axis=1)
    assert np.isfinite(want).all() and np.array_equal(got.view(np.uint64), want.view(np.uint64))


def _total_error(W, T1, T2, a1, a2, G):
    # the levels rounded once, as the T-step forms them; an fp32 weight minus such a level fits into the 64 bits of an extended double
    level = a1.reshape(-1, 1) * T1.reshape(-1, G) + a2.reshape(-1, 1) * T2.reshape(-1, G)
    d = W.reshape(-1, G).astype(np.longdouble) - level.astype(np.longdouble)
    return (d * d).sum()


@pytest.mark.parametrize("G", [128, 256, 100, 64, 20, 16])
def test_error_of_a_group_row_in_full_precision(G):
    # one group-row at a time, from weights that two planes hardly describe to ones that they describe to 2^-30 of the sum of the squares:
    # the error after a sweep is that sum minus what the planes explain, and what is left is good to its own last bit.  Bound: the parts are
    # held to twice the precision, so one rounding, 2^-53; twice that, because the parts below it were rounded as well.
    rng = np.random.default_rng(800 + G)
    left = []
    for noise in (1.0, 0.3, 0.1, 0.05, 0.03, 0.02, 0.01, 1e-3, 1e-4):
        for most in (1, 2) * 3:                          # around 0 and one or two levels of either sign
            W = (np.copysign(0.01, rng.standard_normal((1, G))) * rng.integers(0, most + 1, (1, G)) +
                 rng.standard_normal((1, G)) * 0.01 * noise).astype(np.float32)
            for t_max in (1, 2, 7, 20):
                got = run(W, group=G, t_max=t_max, eps=0.0, canonicalize=False)
                want = _total_error(W, got["T1"], got["T2"], got["alpha1"], got["alpha2"], G)
                assert abs(np.longdouble(got["err_history"][-1]) - want) <= 2.0 ** -52 * want, (noise, t_max)
                left.append(float(want) / float((W.astype(np.float64) ** 2).sum()))
    assert min(left) < 2.0 ** -20 and max(left) > 2.0 ** -6 and sum(2.0 ** -11 < v < 2.0 ** -9 for v in left) > 3


@pytest.mark.parametrize("t_max", [2, 30, 31, 32, 33, 62, 63, 64, 65, 100])
def test_histories_past_the_sweep_at_which_the_last_group_row_repeats(t_max):
    # eps = 0 goes on to t_max; a warp per sweep, 32 at a time, sweep 0 among them
    rng = np.random.default_rng(700 + t_max)
    W = (rng.standard_normal((256, 1024)) * 0.02).astype(np.float32)
    for w in (W, np.sign(W) * np.float32(0.25), np.zeros_like(W)):
        assert_same(run(w, t_max=t_max, eps=0.0), decompose_c(w, T_max=t_max, eps=0.0))


@pytest.mark.parametrize("G", [128, 20, 7])
def test_non_finite_weights_stay_in_their_group_rows(G):
    # a NaN or an infinity makes the scales of its group-row NaN in the first sweep and its planes 0 (no candidate is nearer than
    # another); the rule is then never met, and the other group-rows are those of t_max sweeps
    W = (np.random.default_rng(90 + G).standard_normal((40, 8 * G)) * 0.02).astype(np.float32)
    hurt = np.zeros((40, 8), bool)
    for row, col, v in ((0, 3, np.nan), (5, 2 * G, np.inf), (5, 7 * G + 1, -np.inf), (39, 8 * G - 1, np.nan), (17, G, np.inf),
                        (17, G + 2, -np.inf)):
        W[row, col] = v
        hurt[row, col // G] = True
    ref = decompose_c(np.where(np.isfinite(W), W, np.float32(0.01)), G=G, T_max=9, eps=0.0)
    for canonicalize in (True, False):
        got = run(W, group=G, t_max=9, canonicalize=canonicalize)
        if not canonicalize:
            ref = decompose_c(np.where(np.isfinite(W), W, np.float32(0.01)), G=G, T_max=9, eps=0.0, canonicalize=False)
        assert got["sweeps"] == 9
        cols = np.repeat(hurt, G, axis=1)
        for k in ("T1", "T2"):
            assert np.array_equal(got[k][~cols], ref[k][~cols]) and not got[k][cols].any()
        for k in ("alpha1", "alpha2"):
            assert np.all(np.abs(got[k][~hurt] - ref[k][~hurt]) <= 1e-12) and np.isnan(got[k][hurt]).all()
            assert np.array_equal(got[k + "_fp16"][~hurt].view(np.uint16), ref[k + "_fp16"][~hurt].view(np.uint16))
            assert np.isnan(got[k + "_fp16"][hurt]).all()
        assert np.isnan(got["delta_history"]).all() and np.isnan(got["err_history"]).all()


def test_decompose_pack_gemv_pipeline_on_the_gpu():
    # W -> planes on the GPU -> pack -> GEMV, never leaving the device; checked against the oracle's layer product
    # on the same planes and against the dense product at the level of the reconstruction error
    N, K = 1024, 4096
    W = make_weights(N, K, seed=60)
    T1, T2, a1, a2 = binding.ptqtp_decompose(dev(W))
    x = make_activations(K, seed=61)
    for fmt in (binding.FORMAT_V2, binding.FORMAT_V3):
        packed, st = binding.ptqtp_pack(T1, T2, a1, a2, fmt=fmt)
        y = binding.ptqtp_gemv(packed, N, K, dev(x), fmt=fmt)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        c = dict(T1=T1.cpu().numpy(), T2=T2.cpu().numpy(), alpha1=a1.cpu().numpy(), alpha2=a2.cpu().numpy(), x=x)
        assert_parity(y.cpu().numpy(), oracle_y(c), x, "fmt %d" % fmt)
    err = reconstruction_error(W, c["T1"], c["T2"], c["alpha1"], c["alpha2"])
    assert 0.10 < err < 0.25
    dense = W.astype(np.float64) @ x.astype(np.float64)
    assert np.linalg.norm(y.cpu().numpy().astype(np.float64) - dense) / np.linalg.norm(dense) < 2.5 * err


def test_argument_checks():
    L = binding.lib()
    assert L.ptqtp_decompose_workspace_size(8, 256, 128, 50) > 0
    for bad in ((0, 256, 128, 50), (8, 200, 128, 50), (8, 256, 0, 50), (8, 256, 512, 50), (8, 256, 128, 0), (8, 256, 128, 1001)):
        assert L.ptqtp_decompose_workspace_size(*bad) == 0
    W = dev(make_weights(8, 256, seed=1))
    with pytest.raises(binding.PtqtpError) as e:
        binding.ptqtp_decompose(W, group=100)
    assert e.value.status == binding.ERR_SHAPE
