"""FP32 detection at 32 and 64 antennas, and at 16 above 256 entries, with the Gram as three FP16 products (detect_h3.cuh): the
edges of its tiles (256 queries, 32 entries), of the split of the dictionary over a cluster, of the
user buckets, and rows that the FP16 scaling has to carry, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import assert_hard_match, assert_soft_close, gpu_params, load_state, oracle_state_fp32, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,D,N", [
    (64, 16, 1, 1), (64, 1, 31, 255), (64, 3, 32, 256), (64, 6, 33, 257), (64, 12, 257, 513), (64, 5, 700, 40),
    (32, 16, 1, 300), (32, 2, 64, 256), (32, 7, 95, 1000), (32, 11, 1025, 700), (32, 4, 2048, 3),
    (16, 6, 257, 1), (16, 1, 288, 255), (16, 16, 700, 257), (16, 5, 1025, 513), (16, 2, 2048, 40), (16, 12, 289, 300),
    (16, 8, 300, 1000)])
def test_tile_edges_match_oracle(M, K, D, N):
    ent, gam, clin = synth.random_state(M, K, D, instance=D + M)
    inst = synth.make_instance(M, K, 4, N, 10.0, instance=N + K)
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    soft, hard = apsm.detect(gp, st, to_dev(inst.rx_data))
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), inst.rx_data)
    assert_soft_close(soft.cpu().numpy(), ref)
    assert_hard_match(hard.cpu().numpy(), ref)
    again, _ = apsm.detect(gp, st, to_dev(inst.rx_data))
    assert torch.equal(soft, again)                     # fixed order of every sum
    assert apsm.read_status(st) == 0


@pytest.mark.parametrize("M", [16, 32, 64])
def test_rows_of_very_different_scales(M):
    """Entries and queries from 1e-12 to 1e3 of unit norm in one tile, a zero row and a row with one
    dominant antenna: the power of two per row keeps every distance (sigma spans the large ones)."""
    K, D, N = 4, 70 if M > 16 else 300, 300
    ent, gam, clin = synth.random_state(M, K, D, instance=3)
    inst = synth.make_instance(M, K, 4, N, 10.0, instance=9)
    rx = inst.rx_data.copy()
    ent, scale = ent.copy(), np.array([1.0, 1e-12, 1e-4, 30.0, 1e3], np.float32)
    ent *= scale[np.arange(D) % 5][:, None]
    rx *= scale[np.arange(N) % 4][:, None]
    ent[7], rx[11] = 0, 0
    ent[8, 1:] *= 1e-6
    rx[12, :-1] *= 1e-6
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=4.0, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    soft, _ = apsm.detect(gp, st, to_dev(rx))
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), rx)
    assert_soft_close(soft.cpu().numpy(), ref)


@pytest.mark.parametrize("M", [16, 32, 64])
def test_infinite_and_nan_rows_stay_where_they_are(M):
    """An entry of infinite norm contributes nothing; a query with a NaN gives NaN for itself only."""
    K, D, N = 2, 40 if M > 16 else 300, 20
    ent, gam, clin = synth.random_state(M, K, D, instance=4)
    inst = synth.make_instance(M, K, 4, N, 10.0, instance=8)
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    ent[5] = 1e25                                        # squared norm overflows FP32
    rx = inst.rx_data.copy()
    gp = gpu_params(op)
    keep = np.delete(np.arange(D), 5)
    st = load_state(gp, ent, gam, clin)
    soft, _ = apsm.detect(gp, st, to_dev(rx))
    ref = oracle.detect(op, oracle_state_fp32(M, ent[keep], gam[keep], clin), rx)
    assert_soft_close(soft.cpu().numpy(), ref)
    rx[3, 1] = np.nan
    soft, _ = apsm.detect(gp, st, to_dev(rx))
    y = soft.cpu().numpy()
    assert np.isnan(y[3]).all()
    others = np.delete(np.arange(N), 3)
    assert_soft_close(y[others], ref[others])
