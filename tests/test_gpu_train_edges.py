"""Edges of the training kernels: the blocked window warp (window and block lengths that fill and
just miss a warp, chunks of one block or one live-range warp, ragged last blocks) against the oracle, and
the adjoint's team form (windows at its limits, user counts that leave a team part empty, samples
beyond one staging ring) against the FP64 numpy model of the same recurrence."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import to_dev
from test_adjoint_pull_form import forward_direct, reverse_push
from test_gpu_parity import _compare_training, _train_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,P,W", [(4, 2, 8, 3), (8, 3, 16, 15), (4, 1, 17, 16), (8, 2, 64, 17), (16, 5, 65, 23),
                                     (4, 2, 72, 24), (8, 3, 129, 2), (16, 7, 200, 13)])
def test_blocked_training_matches_oracle(M, K, P, W):
    inst = synth.make_instance(M, K, P, 100, 10.0, instance=P + W)
    op = oracle.Params(M=M, K=K, W=W, D=P, sigma=0.5, mu=0.5, eps=0.01, w_L=0.5)
    gp, st, cl, ref = _train_both(op, inst)
    _compare_training(op, inst, gp, st, cl, ref, tol_coef=1e-4)  # the tolerance of the other training checks


@pytest.mark.parametrize("M,K,P,W", [(8, 1, 30, 1), (8, 3, 40, 14), (8, 4, 45, 15), (4, 2, 60, 30), (4, 2, 60, 31),
                                     (4, 5, 50, 32), (16, 7, 70, 8), (4, 2, 300, 9), (2, 2, 5, 12)])
def test_adjoint_matches_fp64_model(M, K, P, W):
    """FP32 sums of up to 2P W terms with FP64 taps: about 2P W 2^-24 of the largest term, 3e-4 at the
    longest case; a factor of ten above that, as in the finite-difference check."""
    sig, mu, eps, wL = 0.6, 0.6, 0.05, 0.4
    inst = synth.make_instance(M, K, P, 16, 10.0, instance=P + W)
    rng = np.random.default_rng(W)
    c0 = (0.1 * (rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K)))).astype(np.complex64)
    D = max(P, (W + 2) // 2)  # (a capacity holds the window)
    p = apsm.Params(M=M, K=K, window=W, dict_cap=D, sigma=sig, mu=mu, eps=eps, w_L=wL)
    dg = np.zeros((apsm.dict_alloc(p), 2, K), np.float32)
    dg[:P] = 0.1 * rng.standard_normal((P, 2, K))
    dc = (0.1 * (rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K)))).astype(np.complex64)
    ds, dc0 = apsm.train_backward(p, to_dev(inst.rx_pilot), to_dev(inst.sym_pilot), to_dev(dg), to_dev(dc), clin0=to_dev(c0))

    rx = np.asarray(inst.rx_pilot).astype(np.complex64).astype(np.complex128)
    X = np.empty((2 * P, 2 * M))
    X[0::2] = np.concatenate([rx.real, rx.imag], axis=1)
    X[1::2] = np.concatenate([rx.imag, -rx.real], axis=1)
    sc, wb = np.zeros(4), np.zeros((M, K), complex)
    for k in range(K):
        b = np.empty(2 * P)
        b[0::2], b[1::2] = inst.sym_pilot[:, k].real, inst.sym_pilot[:, k].imag
        w0 = np.concatenate([c0[:, k].real, c0[:, k].imag]).astype(np.float64)
        _, _, tape = forward_direct(X, b, W, D, sig, mu, eps, wL, w0)
        gfin = dg[:P, :, k].astype(np.float64).reshape(-1)
        wfin = np.concatenate([dc[:, k].real, dc[:, k].imag]).astype(np.float64)
        s, w = reverse_push(X, W, D, sig, mu, wL, tape, gfin, wfin)
        sc += s
        wb[:, k] = w[:M] + 1j * w[M:]
    assert np.abs(dc0.cpu().numpy() - wb).max() <= 3e-3 * np.abs(wb).max()
    assert np.abs(ds.cpu().numpy() - sc).max() <= 3e-3 * np.abs(sc).max()
    assert torch.isfinite(ds).all()


@pytest.mark.parametrize("W", [7, 16, 30])
def test_single_warp_and_team_forms_give_the_same_bits(W):
    """Past two team CTAs per SM an instance runs one warp per user: the same bits as its own call."""
    M, K, P, n = 4, 2, 24, 320
    p = apsm.Params(M=M, K=K, window=W, dict_cap=P, sigma=0.6, mu=0.7, eps=0.02, w_L=0.4)
    xs = [synth.make_instance(M, K, P, 4, 10.0, instance=i) for i in range(3)]
    rp = torch.stack([to_dev(xs[i % 3].rx_pilot) for i in range(n)])
    sp = torch.stack([to_dev(xs[i % 3].sym_pilot) for i in range(n)])
    g = torch.Generator(device="cpu").manual_seed(W)
    dg = (0.1 * torch.randn((n, apsm.dict_alloc(p), 2, K), generator=g)).cuda()
    dc = (0.1 * torch.randn((n, M, K), dtype=torch.complex64, generator=g)).cuda()
    ds, dc0 = apsm.train_backward_batched(p, rp, sp, dg, dc)
    for i in (0, 1, 151, n - 1):
        ds1, dc1 = apsm.train_backward(p, rp[i], sp[i], dg[i], dc[i])
        assert torch.equal(ds[i], ds1) and torch.equal(dc0[i], dc1)
