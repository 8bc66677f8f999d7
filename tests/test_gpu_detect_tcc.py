"""BF16/FP16 detection with the coefficient sums on the tensor cores (detect_tcc.cuh): the edges of its
tiles (128 queries, 64 entries in four chunks, one per epilogue group) and of its rings (two Gram
operands, three accumulators, three coefficient stages), and pairs close enough for direct
differences in every group, against the FP64 oracle;
the last five cases: dictionaries of one to ten tiles with more query tiles than SMs (half CTAs)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import assert_hard_match, assert_soft_close, gpu_params, load_state, oracle_state_fp32, to_dev

pytestmark = pytest.mark.gpu
TOL = 2e-2  # the bound of every reduced-precision detection test here: BF16 Gram, FP32 sums


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("M,K,D,N", [
    (16, 1, 1, 1), (16, 3, 16, 127), (16, 5, 17, 128), (16, 6, 64, 129), (32, 2, 65, 300), (32, 12, 193, 40),
    (64, 16, 256, 260), (64, 7, 257, 129), (64, 4, 385, 5), (32, 8, 449, 128), (16, 16, 1025, 500),
    (16, 6, 128, 19457), (16, 2, 64, 19700), (32, 5, 100, 20000), (16, 12, 129, 19600),
    (16, 2, 577, 19457)])
def test_edges_and_direct_differences(M, K, D, N, dtype):
    ent, gam, clin = synth.random_state(M, K, D, instance=D + M)
    inst = synth.make_instance(M, K, 4, N, 10.0, instance=N + K)
    rx = inst.rx_data.copy()
    # every third query sits on an entry, some turned by a quarter (the other half of the real split)
    for i in range(0, N, 3):
        rx[i] = ent[(5 * i) % D] * (1, 1j, -1j)[i % 3 if i % 2 else 0] * np.float32(1 + 1e-4)
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op, dtype=dtype)
    st = load_state(gp, ent, gam, clin)
    ws = apsm.detect_workspace(gp, N)
    soft, hard = apsm.detect(gp, st, to_dev(rx), workspace=ws)
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), rx)
    assert_soft_close(soft.cpu().numpy(), ref, tol=TOL, what=dtype)
    assert_hard_match(hard.cpu().numpy(), ref, tol=TOL)
    for _ in range(3):
        again, _ = apsm.detect(gp, st, to_dev(rx), workspace=ws)
        assert torch.equal(soft, again)                 # fixed order of every sum
    assert apsm.read_status(st) == 0
