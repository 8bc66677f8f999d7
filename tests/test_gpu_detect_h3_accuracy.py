"""FP32 detection in the FP16 x3 form: no further from the FP64 oracle than the form without it (the FMA engine at
64 antennas, TF32 x3 below), over entries and vectors of few users, whose Gram sums grow the most in one
direction, and of as many users as antennas, whose filter terms are large and cancel.  Root mean square over
some thousand outputs; 5 % for the sample.  And the edges of whole waves of query tiles (152 CTAs of 256
queries unsplit, the rest split), within 1e-5: the exponents here are below 6, off by 2^-21 of that."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import assert_soft_close, gpu_params, load_state, oracle_state_fp32, rms, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,D", [(64, 1, 500), (64, 2, 300), (64, 2, 700), (64, 3, 500), (64, 4, 500), (64, 6, 500),
                                   (64, 8, 500), (64, 12, 500), (64, 16, 500), (32, 2, 500), (32, 11, 500),
                                   (16, 2, 500), (16, 8, 500), (16, 16, 300), (16, 16, 1500)])
def test_error_is_not_above_the_form_without_it(M, K, D):
    rng, e_new, e_old = np.random.default_rng(1000 * M + K), [], []
    for i in range(4):
        inst = synth.make_instance(M, K, D, 500, 15.0, instance=100 * i + K)
        gam = (0.05 * rng.standard_normal((D, 2, K))).astype(np.float32)
        # the filter of least squares on the pilots, as strong as the linear part has it (w_L = 0.5)
        clin = np.linalg.lstsq(inst.rx_pilot.conj(), inst.sym_pilot.conj(), rcond=None)[0].astype(np.complex64) * 2
        op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
        gp = gpu_params(op)
        st = load_state(gp, inst.rx_pilot, gam, clin)
        ref = oracle.detect(op, oracle_state_fp32(M, inst.rx_pilot, gam, clin), inst.rx_data)
        try:
            for opt, out in ((1, e_new), (0, e_old)):
                apsm.set_option("detect_tma", opt)
                out.append(np.abs(apsm.detect(gp, st, to_dev(inst.rx_data))[0].cpu().numpy() - ref))
        finally:
            apsm.set_option("detect_tma", 1)
    assert rms(e_new) <= 1.05 * rms(e_old)


@pytest.mark.parametrize("M,K,D", [(16, 2, 300), (16, 6, 290), (32, 5, 100), (32, 16, 1), (32, 7, 31), (32, 2, 33),
                                   (64, 2, 70), (64, 6, 33), (64, 9, 32), (64, 16, 31)])
@pytest.mark.parametrize("extra", [-1, 0, 1, 300])
def test_edges_of_whole_waves(M, K, D, extra):
    wave = 256 * torch.cuda.get_device_properties(0).multi_processor_count
    N = wave + extra
    ent, gam, clin = synth.random_state(M, K, D, instance=M + K)
    rx = synth.random_state(M, 1, N, instance=7)[0]
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    soft = torch.full((N, K), float("nan"), dtype=torch.complex64, device="cuda")
    apsm.detect(gp, st, to_dev(rx), soft=soft)
    assert bool(torch.isfinite(torch.view_as_real(soft)).all())
    rows = np.unique(np.clip(np.concatenate([np.arange(0, N, 199), np.arange(wave - 260, wave + 300),
                                             np.arange(N - 40, N)]), 0, N - 1))
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), np.ascontiguousarray(rx[rows]))
    assert_soft_close(soft.cpu().numpy()[rows], ref, tol=1e-5)
    assert apsm.read_status(st) == 0


@pytest.mark.parametrize("M,K,D,N", [(64, 6, 96, 700), (64, 6, 97, 700), (64, 16, 128, 300), (64, 16, 129, 300),
                                     (64, 2, 32, 12500), (64, 2, 32, 12501), (64, 11, 20, 15000), (64, 11, 20, 15001),
                                     (32, 4, 64, 500), (32, 4, 65, 500), (32, 5, 32, 500), (32, 5, 33, 500),
                                     (32, 5, 32, 16384), (32, 5, 32, 16385)])
def test_either_side_of_the_line_to_the_former_form(M, K, D, N):
    ent, gam, clin = synth.random_state(M, K, D, instance=M + K)
    rx = synth.random_state(M, 1, N, instance=9)[0]
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    soft = apsm.detect(gp, st, to_dev(rx))[0].cpu().numpy()
    rows = np.unique(np.concatenate([np.arange(0, N, 37), np.arange(max(N - 300, 0), N)]))
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), np.ascontiguousarray(rx[rows]))
    assert_soft_close(soft[rows], ref, tol=1e-5)
    try:   # the same call in the form without FP16 products, of which the outputs are an FP32 rounding away
        apsm.set_option("detect_tma", 0)
        plain = apsm.detect(gp, st, to_dev(rx))[0].cpu().numpy()
    finally:
        apsm.set_option("detect_tma", 1)
    former = not (D > (64 if K <= 4 else 32) or N > 16384) if M == 32 else \
        not (D > (128 if K > 12 else 96) or N * D > (400000 if K <= 8 else 300000))
    assert np.array_equal(soft, plain) == former
