"""Parity of mpq_output_error (Eq. 11) with the oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from paper_2002_09049_gb300 import binding, workloads as wlm
from _parity import compare_err

pytestmark = pytest.mark.gpu


def gpu_err(X, W, codes, scales, k_max, groups=1, dev="cuda:0"):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    err = binding.mpq_output_error(t(X), t(W), t(codes), t(scales), k_max, groups=groups)
    torch.cuda.synchronize()
    return err.cpu().numpy()


@pytest.mark.parametrize("C,d,N,K", [(1, 1, 1, 1), (3, 5, 7, 2), (5, 33, 70, 4), (7, 64, 64, 3),
                                     (11, 147, 129, 4), (4, 1000, 65, 2), (64, 576, 512, 4),
                                     (2, 17, 300, 16),
                                     # d % 16 == 0 (CTA-pair kernel): several pair tiles with a
                                     # part-filled last pair, an empty odd CTA, ragged row tiles
                                     # split over a cluster, k_max + 1 from 2 to 17
                                     (130, 256, 600, 4), (30, 128, 1000, 1), (9, 32, 300, 16),
                                     (50, 512, 1100, 6), (3, 48, 20, 8),
                                     # k_max + 1 = 8 and 16: no channel pairing separates the
                                     # stores' bank halves there (layout unchanged, results too)
                                     (40, 96, 300, 7), (17, 64, 260, 15),
                                     (3, 8192, 300, 4)])          # the longest rows taken
def test_shared_input(gpu, oracle, C, d, N, K):
    W = wlm.random_weights(C, d, C + d + N, "normal")
    q = oracle.quantize_layer(W, 4, 32, K)
    X = wlm.random_calibration(N, d, 7 + d)
    e_or = oracle.output_error(X, 1, W, q["codes"], q["scales"], K)
    e_gpu = gpu_err(X, W, q["codes"], q["scales"], K)
    compare_err(e_gpu, e_or)


@pytest.mark.parametrize("C,d,N,K", [(1, 9, 1, 1), (6, 9, 100, 8), (40, 9, 1024, 8), (3, 25, 77, 4),
                                     (5, 300, 33, 16),
                                     # two rows a thread: chunks of 256 rows, 32 elements at most
                                     (3, 32, 257, 8), (3, 33, 257, 8), (7, 9, 255, 3), (2, 31, 513, 16),
                                     (4, 1, 1025, 1), (5, 16, 129, 9)])
def test_per_channel_input(gpu, oracle, C, d, N, K):
    W = wlm.random_weights(C, d, 3 * C + d, "laplace")
    q = oracle.quantize_layer(W, 4, 64, K)
    X = wlm.random_calibration(N, d, 11, groups=C)
    e_or = oracle.output_error(X, C, W, q["codes"], q["scales"], K)
    e_gpu = gpu_err(X, W, q["codes"], q["scales"], K, groups=C)
    compare_err(e_gpu, e_or)


def test_config1_layer(gpu, oracle):
    wl = wlm.WORKLOADS["c1"]
    W = wlm.make_weights(wl, 0)
    X = wlm.make_calibration(wl, 0)
    q = oracle.quantize_layer(W, 4, wl.G, wl.k_max)
    worst = compare_err(gpu_err(X, W, q["codes"], q["scales"], wl.k_max),
                        oracle.output_error(X, 1, W, q["codes"], q["scales"], wl.k_max))
    assert worst < 1e-5


def test_hot_columns_input(gpu, oracle):
    """Inputs with a few large columns (the large-linear-layer workload's calibration recipe)."""
    rng = np.random.default_rng(4)
    X = rng.standard_normal((256, 512)).astype(np.float32)
    X[:, rng.choice(512, 8, replace=False)] *= 10
    W = (rng.standard_normal((24, 512)) * 0.02).astype(np.float32)
    q = oracle.quantize_layer(W, 4, 256, 8)
    compare_err(gpu_err(X, W, q["codes"], q["scales"], 8),
                oracle.output_error(X, 1, W, q["codes"], q["scales"], 8))


def test_nonfinite_weight_propagates(gpu, oracle):
    W = wlm.random_weights(3, 20, 1, "normal")
    W[1, 2] = np.nan
    q = oracle.quantize_layer(W, 4, 16, 2)
    X = wlm.random_calibration(10, 20, 2)
    e = gpu_err(X, W, q["codes"], q["scales"], 2)
    assert np.all(np.isnan(e[1])) and np.all(np.isfinite(e[[0, 2]]))


@pytest.mark.parametrize("x_exp,w_exp", [(40, -60), (-50, 30), (0, -40)])
def test_operand_scaling_extremes(gpu, oracle, x_exp, w_exp):
    """fp16 operands are scaled per residual vector and per layer of X: inputs scaled by powers of
    two far from 1 (the oracle's double result scales exactly), residuals that reach 0 after one
    point, and calibration rows many binades below the others."""
    C, d, N, K = 40, 256, 300, 6
    W = wlm.random_weights(C, d, 3, "normal")
    W[5] = np.ldexp(np.round(W[5] * 64), -8).astype(np.float32)    # few distinct values
    W[6] = 0.0
    X = wlm.random_calibration(N, d, 4)
    X[::7] *= np.float32(2.0 ** -30)
    W = np.ldexp(W, w_exp).astype(np.float32)
    X = np.ldexp(X, x_exp).astype(np.float32)
    q = oracle.quantize_layer(W, 4, 32, K)
    compare_err(gpu_err(X, W, q["codes"], q["scales"], K),
                oracle.output_error(X, 1, W, q["codes"], q["scales"], K))


def test_nonfinite_on_the_pair_path(gpu, oracle):
    """Rows a multiple of 16 (scaled fp16 operands): the range pass skips NaN in its maxima, and
    the NaN still propagates -- a NaN weight into its channel's errors only, a NaN calibration
    input into every error."""
    W = wlm.random_weights(40, 64, 5, "normal")
    W[7, 3] = np.nan
    q = oracle.quantize_layer(W, 4, 16, 3)
    X = wlm.random_calibration(300, 64, 6)
    e = gpu_err(X, W, q["codes"], q["scales"], 3)
    assert np.all(np.isnan(e[7])) and np.all(np.isfinite(np.delete(e, 7, axis=0)))
    compare_err(e, oracle.output_error(X, 1, W, q["codes"], q["scales"], 3))
    X[100, 10] = np.nan
    assert np.all(np.isnan(gpu_err(X, W, q["codes"], q["scales"], 3)))


@pytest.mark.parametrize("C,d,N,K,bits", [(130, 256, 600, 4, 4), (64, 576, 1024, 8, 4),
                                          (9, 32, 300, 16, 3), (3, 147, 100, 4, 4)])
def test_ranges_from_the_greedy_search(gpu, oracle, C, d, N, K, bits):
    """mpq_quantize_layer's rmax output is max |r| of every residual vector (w, then each step's
    residual, exactly as the oracle's recursion gives them), and mpq_output_error with it gives
    bit for bit the errors it gives measuring the ranges itself (also for rows the tensor-core
    path cannot take, which ignore it), within 1e-5 of the oracle."""
    W = wlm.random_weights(C, d, 3 * C + d, "normal")
    W[1, 3] = np.nan                                   # a non-finite channel: NaN ranges
    X = wlm.random_calibration(N, d, 11 + d)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(gpu)
    rmax = torch.empty((C, K + 1), dtype=torch.float32, device=gpu)
    codes, scales, _, _ = binding.mpq_quantize_layer(t(W), bits, 64, K, rmax=rmax)
    e1 = binding.mpq_output_error(t(X), t(W), codes, scales, K, rmax=rmax)
    e0 = binding.mpq_output_error(t(X), t(W), codes, scales, K)
    torch.cuda.synchronize()
    o = oracle.quantize_layer(W, bits, 64, K)
    want = np.concatenate([np.abs(W).max(axis=1, keepdims=True),
                           np.abs(o["residuals"]).max(axis=2).T], axis=1)
    want[1, :] = np.nan
    np.testing.assert_array_equal(rmax.cpu().numpy(), want.astype(np.float32))
    assert torch.equal(torch.nan_to_num(e1, nan=-1.0), torch.nan_to_num(e0, nan=-1.0))
    keep = np.arange(C) != 1
    e_or = oracle.output_error(X, 1, W[keep], o["codes"][:, keep], o["scales"][keep], K)
    compare_err(e1.cpu().numpy()[keep], e_or)


# channel tiles are 2 floor(128 / (k_max + 2)) channels (24 at k_max = 8), row tiles 256 calibration
# rows, steps 64 elements: one less, exactly and one more of each; every row tile in one CTA pair
# or shared by several; the largest k_max
@pytest.mark.parametrize("C,d,N,K", [(24, 64, 256, 8), (23, 48, 255, 8), (25, 80, 257, 8),
                                     (84, 16, 70, 1), (85, 272, 513, 1), (7, 320, 2049, 16),
                                     (33, 1040, 1500, 6), (2000, 64, 700, 4)])
def test_point_chain_tiles(gpu, oracle, C, d, N, K):
    """The contraction over the points (codes and the last residual): tile edges, through the
    pooled and the fixed-scratch entry point (bit for bit the same), against the oracle."""
    W = wlm.random_weights(C, d, C + d + K, "t")
    X = wlm.random_calibration(N, d, 9 + d)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(gpu)
    codes, scales, _, _ = binding.mpq_quantize_layer(t(W), 4, 32, K)
    e = binding.mpq_output_error(t(X), t(W), codes, scales, K)
    e_fixed = binding.mpq_output_error_noalloc(t(X), t(W), codes, scales, K)
    torch.cuda.synchronize()
    assert torch.equal(e, e_fixed)
    some = np.unique(np.concatenate([np.arange(min(C, 30)), np.arange(max(0, C - 30), C)]))
    q, s = codes.cpu().numpy()[:, some], scales.cpu().numpy()[some]
    compare_err(e.cpu().numpy()[some], oracle.output_error(X, 1, W[some], q, s, K))


@pytest.mark.parametrize("K", [1, 5, 16])
def test_codes_that_are_not_nearest_values(gpu, oracle, K):
    """Codes and scales of the caller's own, under which residuals grow: those channels take plain
    fp32 sums, the others (nearest codes) the chain."""
    C, d, N = 60, 144, 300
    rng = np.random.default_rng(K)
    W = wlm.random_weights(C, d, 21, "normal")
    q = oracle.quantize_layer(W, 4, 32, K)
    codes, scales = q["codes"].copy(), q["scales"].copy()
    for k in (0, 3, 41, 59):
        codes[:, k] = rng.integers(-7, 8, size=(K, d)).astype(np.int8)
        scales[k] = (10.0 ** rng.uniform(0, 3, size=K)).astype(np.float32)
    codes[:, 7] = 0
    scales[7] = 1e30                                   # a scale far above its residual, codes 0
    X = wlm.random_calibration(N, d, 5)
    compare_err(gpu_err(X, W, codes, scales, K), oracle.output_error(X, 1, W, codes, scales, K))


@pytest.mark.parametrize("grow", [1.15, 1.35, 1.9])
def test_residuals_that_grow_step_by_step(gpu, oracle, grow):
    """Codes that add to the residual, a little at each of 16 points (9, 122 and 29,000 times in all):
    no single step doubles it, and the first errors are as exact as the last."""
    C, d, N, K = 20, 160, 300, 16
    W = wlm.random_weights(C, d, 3, "normal")
    codes, scales = np.zeros((K, C, d), np.int8), np.zeros((C, K), np.float32)
    r = W.copy()
    for n in range(K):
        scales[:, n] = np.abs(r).max(1) * np.float32(grow - 1) / 7
        codes[n] = np.rint(-r * np.float32(grow - 1) / scales[:, n:n + 1]).clip(-7, 7)
        r = r - scales[:, n:n + 1] * codes[n]
    X = wlm.random_calibration(N, d, 5)
    compare_err(gpu_err(X, W, codes, scales, K), oracle.output_error(X, 1, W, codes, scales, K))


@pytest.mark.parametrize("C,d,N,K", [(60, 144, 300, 5), (400, 64, 70, 1), (25, 257, 257, 9),
                                     (30, 1040, 33, 16), (15, 601, 100, 16), (9, 8192, 40, 8)])
def test_every_channel_grows(gpu, oracle, C, d, N, K):
    """Layers of channels that the chain cannot take, more of them than blocks that look for them, rows
    longer than shared memory holds residuals of: the pooled and the fixed-scratch entry points (which
    regenerate different lengths at a time) give the same errors bit for bit."""
    rng = np.random.default_rng(C + d)
    W = wlm.random_weights(C, d, 21, "normal")
    codes = rng.integers(-7, 8, size=(K, C, d)).astype(np.int8)
    scales = rng.uniform(1, 3, size=(C, K)).astype(np.float32)
    X = wlm.random_calibration(N, d, 5)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(gpu)
    args = (t(X), t(W), t(codes), t(scales), K)
    e = binding.mpq_output_error(*args)
    assert torch.equal(e, binding.mpq_output_error_noalloc(*args))
    compare_err(e.cpu().numpy(), oracle.output_error(X, 1, W, codes, scales, K))


# rows that tile copies cannot address: around 16 elements and a 64-element step, channel and row
# tile edges as above, where the chain takes them and just below; off: elements that X, W and
# (x 4) the codes start past a 16-byte boundary
@pytest.mark.parametrize("C,d,N,K,off", [(24, 255, 256, 9, 0), (25, 257, 257, 9, 0), (52, 193, 129, 3, 0),
                                         (51, 193, 300, 3, 0), (52, 191, 300, 3, 0),
                                         (86, 321, 513, 1, 0), (33, 1039, 1500, 6, 0),
                                         (15, 601, 300, 16, 0), (700, 207, 700, 4, 0),
                                         (2000, 300, 128, 8, 0), (43, 256, 300, 4, 1),
                                         (61, 275, 300, 3, 3)])
def test_rows_of_any_length(gpu, oracle, C, d, N, K, off):
    """Padded copies (pooled scratch, with and without the search's ranges) and the gather (fixed
    scratch) give bit for bit the same errors, within 1e-5 of the oracle."""
    W = wlm.random_weights(C, d, C + d + K, "t")
    X = wlm.random_calibration(N, d, 9 + d)

    def t(a, pad):
        a = torch.from_numpy(np.ascontiguousarray(a)).to(gpu)
        store = torch.empty(a.numel() + 64, dtype=a.dtype, device=gpu)
        out = store[pad:pad + a.numel()].view(a.shape)
        return out.copy_(a)

    o = oracle.quantize_layer(W, 4, 32, K)
    rmax = np.concatenate([np.abs(W).max(axis=1, keepdims=True),
                           np.abs(o["residuals"]).max(axis=2).T], axis=1).astype(np.float32)
    args = (t(X, off), t(W, off), t(o["codes"], 4 * off), t(o["scales"], 0), K)
    e = binding.mpq_output_error(*args)
    e_rmax = binding.mpq_output_error(*args, rmax=t(rmax, 0))
    e_fixed = binding.mpq_output_error_noalloc(*args)
    torch.cuda.synchronize()
    assert torch.equal(e, e_fixed) and torch.equal(e, e_rmax)
    compare_err(e.cpu().numpy(), oracle.output_error(X, 1, W, o["codes"], o["scales"], K))


@pytest.mark.parametrize("C,d,N,K", [(60, 144, 300, 5), (25, 257, 257, 9), (30, 1040, 600, 16), (90, 64, 70, 1)])
def test_scales_that_end_in_nan(gpu, oracle, C, d, N, K):
    """A channel whose points end at a NaN scale (a refused step of the adaptive grid: this and every
    later scale NaN, codes 0) keeps its errors before that point."""
    W = wlm.random_weights(C, d, 7 * C + d, "normal")
    q = oracle.quantize_layer(W, 4, 32, K)
    codes, scales = q["codes"].copy(), q["scales"].copy()
    for k, n in ((0, 0), (1, K - 1), (C // 2, K // 2), (C - 1, 0)):
        scales[k, n:] = np.nan
        codes[n:, k] = 0
    X = wlm.random_calibration(N, d, 5)
    e = gpu_err(X, W, codes, scales, K)
    o = oracle.output_error(X, 1, W, codes, scales, K)
    assert np.array_equal(np.isnan(e), np.isnan(o)) and np.isnan(o).any()
    compare_err(np.where(np.isnan(o), 0, e), np.where(np.isnan(o), 0, o))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(gpu)
    e_fixed = binding.mpq_output_error_noalloc(t(X), t(W), t(codes), t(scales), K).cpu().numpy()
    assert np.array_equal(e, e_fixed, equal_nan=True)


def test_refused_steps_of_the_adaptive_grid(gpu, oracle):
    """The adaptive grid's refusals through the output error: errors up to the refused step."""
    W = wlm.random_weights(64, 144, 11, "normal")
    X = wlm.random_calibration(300, 144, 12)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(gpu)
    _, _, _, ncand = binding.mpq_quantize_layer_adaptive(t(W), 4, 4, max_cand=10 ** 15)
    cap = int(ncand.float().median())   # (about half of the steps refused)
    codes, scales, _, _ = binding.mpq_quantize_layer_adaptive(t(W), 4, 4, max_cand=cap)
    e = binding.mpq_output_error(t(X), t(W), codes, scales, 4).cpu().numpy()
    o = oracle.output_error(X, 1, W, codes.cpu().numpy(), scales.cpu().numpy(), 4)
    assert np.array_equal(np.isnan(e), np.isnan(o)) and np.isnan(o).any() and np.isfinite(o[:, 0]).all()
    compare_err(np.where(np.isnan(o), 0, e), np.where(np.isnan(o), 0, o))


@pytest.mark.parametrize("C,d,N,K,pad", [(134, 1378, 128, 6, 0), (134, 1376, 128, 6, 0), (64, 576, 512, 4, 0),
                                         (300, 200, 200, 4, 1), (40, 2064, 300, 16, 0)])
def test_ranges_of_this_call(gpu, C, d, N, K, pad):
    """The kernels of a call are launched before the ones ahead of them have finished: each uses this
    call's max |X| and residual ranges, whole.  Inputs whose ranges change from call to call give
    the same errors every time (rows that are copied, split in place, and measured)."""
    W = torch.randn(C, d, device=gpu)
    codes, scales, _, _ = binding.mpq_quantize_layer(W, 8, 16, K)
    rmax = torch.empty((C, K + 1), device=gpu)
    binding.mpq_quantize_layer(W, 8, 16, K, codes=codes, scales=scales, rmax=rmax)
    inputs = []
    for i in range(4):
        x = torch.empty(N * d + pad, device=gpu)[pad:].view(N, d)
        inputs.append(x.copy_(torch.randn(N, d, device=gpu) * 10.0 ** (2 * i - 3)))
    first = []
    for i in range(80):
        e = binding.mpq_output_error(inputs[i % 4], W, codes, scales, K, rmax=rmax if i % 8 < 4 else None)
        if i < 4:
            first.append(e)
            torch.cuda.synchronize()
            y = inputs[i].double() @ W.double().T
            assert torch.allclose(e[:, 0].double(), y.square().mean(0), rtol=1e-5, atol=0)
        else:
            assert torch.equal(e, first[i % 4])
