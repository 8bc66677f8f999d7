"""FP32 detection in the FP16 x3 form (detect_h3.cuh) with queries outside the factor range: rows far from
every entry (the unfactored exponent), rows whose norms cancel (direct differences, any number of them in a
tile of 256 queries), and both beside rows inside the range, against the FP64 oracle.

Tolerance: an unmarked term is off by less than 2e-6 of its coefficient (H3Guard), one by direct differences
by 2^-23 of an exponent of at most 20 where it matters; sums of some hundred such terms and the FP32 linear
part stay below 1e-5 of the output scale."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import assert_hard_match, assert_soft_close, gpu_params, load_state, oracle_state_fp32, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5


def run(M, K, ent, gam, clin, rx, sigma=0.5):
    D = ent.shape[0]
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=sigma, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    soft, hard = apsm.detect(gp, st, to_dev(rx))
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), rx)
    assert apsm.read_status(st) == 0
    again, _ = apsm.detect(gp, st, to_dev(rx))
    assert torch.equal(torch.view_as_real(soft), torch.view_as_real(again))
    return soft.cpu().numpy(), hard.cpu().numpy(), ref


def data(M, K, D, N):
    ent, gam, clin = synth.random_state(M, K, D, instance=D + M)
    return ent.copy(), gam, clin, synth.make_instance(M, K, 4, N, 10.0, instance=N + K).rx_data.copy()


SHAPES = [(16, 2, 290, 700), (16, 9, 1025, 257), (32, 2, 97, 300), (32, 11, 700, 513), (64, 2, 97, 300),
          (64, 6, 513, 257), (64, 16, 300, 600)]


@pytest.mark.parametrize("M,K,D,N", SHAPES)
def test_large_common_offset(M, K, D, N):
    """||r||^2 >> ||r - r_t||^2 for every pair: every row by direct differences."""
    ent, gam, clin, rx = data(M, K, D, N)
    rng = np.random.default_rng(M)
    base = (rng.standard_normal(M) + 1j * rng.standard_normal(M)) * (1.6 if M > 16 else 3.2)
    soft, hard, ref = run(M, K, (ent + base).astype(np.complex64), gam, clin, (rx * 0.5 + base).astype(np.complex64), 0.8)
    assert_soft_close(soft, ref, tol=TOL)
    assert_hard_match(hard, ref, tol=TOL)


@pytest.mark.parametrize("M,K,D,N", SHAPES)
def test_rows_far_outside(M, K, D, N):
    """Some rows, then all, far larger than any entry: no kernel term is left of them."""
    ent, gam, clin, rx = data(M, K, D, N)
    rx[::37] *= 40.0
    soft, hard, ref = run(M, K, ent, gam, clin, rx)
    assert_soft_close(soft, ref, tol=TOL)
    assert_hard_match(hard, ref, tol=TOL)
    soft, _, ref = run(M, K, ent, gam, clin, rx * np.float32(30))
    assert_soft_close(soft, ref, tol=TOL)


@pytest.mark.parametrize("scale", [10.0, 1e2, 1e4])
@pytest.mark.parametrize("n_near", [1, 8, 9, 33, 130, 256])
@pytest.mark.parametrize("M,K,D", [(16, 4, 600), (32, 3, 200), (64, 6, 130), (64, 16, 129)])
def test_marked_rows_among_others(M, K, D, n_near, scale):
    """n_near rows of a tile lie on or beside large entries (the terms there are of order one), also turned by a
    quarter (the other half of the real split).  No linear part, so that the kernel sum is all there is."""
    N = 300
    ent, gam, clin, rx = data(M, K, D, N)
    ent[::3] *= np.float32(scale)
    rows = np.random.default_rng(n_near).permutation(256)[:n_near]
    for i in rows:
        e = ent[3 * (i % ((D + 2) // 3))]
        near = e + (0.1 / np.sqrt(M) * (i % 2)) * rx[i] if scale < 1e3 else e
        rx[i] = (near * (1, 1j, -1j)[i % 3]).astype(np.complex64)
    soft, hard, ref = run(M, K, ent, gam, np.zeros_like(clin), rx)
    # the scale of the outputs is that of single terms: of all rows' sums, not of the small ones alone
    err = np.abs(soft - ref)
    assert err.max() <= TOL * np.abs(gam).max() * np.sqrt(D)


@pytest.mark.parametrize("M", [16, 32, 64])
def test_nan_and_overflowing_rows_beside_marked_ones(M):
    K, D, N = 4, 300, 300
    ent, gam, clin, rx = data(M, K, D, N)
    ent[::5] *= np.float32(30)
    for i in range(0, N, 4):
        rx[i] = ent[5 * (i % 60)]
    clin = np.zeros_like(clin)
    clean = rx.copy()
    rx[3, 1], rx[40, 0], rx[77] = np.nan, np.nan, 1e25   # (||rx[77]||^2 overflows FP32: no term is left)
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    y = apsm.detect(gp, st, to_dev(rx))[0].cpu().numpy()
    assert np.isnan(y[[3, 40]]).all() and (y[77] == 0).all()
    ok = np.setdiff1d(np.arange(N), [3, 40, 77])
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), clean)
    assert np.abs(y[ok] - ref[ok]).max() <= TOL * np.abs(gam).max() * np.sqrt(D)


@pytest.mark.parametrize("M", [16, 32, 64])
def test_rows_of_very_different_scales(M):
    """Entries and queries from 1e-12 to 1e3 of unit norm in one tile, a zero row and a row with one dominant
    antenna: the power of two per row keeps every distance (sigma spans the large ones)."""
    K, D, N = 4, 300, 300
    ent, gam, clin, rx = data(M, K, D, N)
    scale = np.array([1.0, 1e-12, 1e-4, 30.0, 1e3], np.float32)
    ent *= scale[np.arange(D) % 5][:, None]
    rx *= scale[np.arange(N) % 4][:, None]
    ent[7], rx[11] = 0, 0
    ent[8, 1:] *= 1e-6
    rx[12, :-1] *= 1e-6
    soft, _, ref = run(M, K, ent, gam, clin, rx, sigma=4.0)
    assert_soft_close(soft, ref, tol=TOL)
