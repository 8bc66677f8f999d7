"""FP32 detection with 16 antennas and dictionaries of up to 256 entries: the TMA-staged form, plain and balanced
over the SMs (above 256 entries, where the FP16 x3 form takes over, the same calls no longer reach it)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import assert_hard_match, assert_soft_close, gpu_params, load_state, oracle_state_fp32, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,D,N", [(6, 256, 8192), (6, 200, 3001), (12, 255, 5000), (2, 193, 40000), (16, 256, 777),
                                   (4, 130, 65), (8, 129, 19456)])
def test_balanced_and_plain(K, D, N):
    M = 16
    ent, gam, clin = synth.random_state(M, K, D, instance=3 * D + K)
    inst = synth.make_instance(M, K, 4, N, 10.0, instance=N + K)
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op)
    st = load_state(gp, ent, gam, clin)
    ws = apsm.detect_workspace(gp, N)
    assert ws is not None and ws.numel() > 0
    used = 4 * ((N + 127) // 128)            # arrival counters, then the parts of split query tiles
    rx = to_dev(inst.rx_data)
    soft, hard = apsm.detect(gp, st, rx, workspace=ws)
    if N >= 700:
        assert torch.count_nonzero(ws[used:]) > 0   # the balanced kernel ran: it left parts behind its counters
    assert torch.count_nonzero(ws[:used]) == 0
    plain, hard_plain = apsm.detect(gp, st, rx)
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), inst.rx_data)
    for y, h in ((soft, hard), (plain, hard_plain)):
        assert_soft_close(y.cpu().numpy(), ref)
        assert_hard_match(h.cpu().numpy(), ref)
    again, _ = apsm.detect(gp, st, rx, workspace=ws)
    assert torch.equal(soft, again)
    assert apsm.read_status(st) == 0


@pytest.mark.parametrize("balanced", [True, False])
def test_slots_past_the_held_entries(balanced):
    M, K, D, n, N = 16, 6, 250, 133, 4000
    ent, gam, clin = synth.random_state(M, K, n, instance=77)
    inst = synth.make_instance(M, K, 4, N, 10.0, instance=78)
    op = oracle.Params(M=M, K=K, W=1, D=D, sigma=0.5, w_L=0.5)
    gp = gpu_params(op)
    st = apsm.State(gp)
    st.dict.fill_(complex(float("nan"), float("nan")))
    st.dict_norm.fill_(float("nan"))
    st.gamma.fill_(float("nan"))
    apsm.state_set(gp, st, to_dev(np.asarray(ent, np.complex64)), to_dev(np.asarray(gam, np.float32)),
                   to_dev(np.asarray(clin, np.complex64)))
    ws = apsm.detect_workspace(gp, N) if balanced else None
    soft, hard = apsm.detect(gp, st, to_dev(inst.rx_data), workspace=ws)
    ref = oracle.detect(op, oracle_state_fp32(M, ent, gam, clin), inst.rx_data)
    assert_soft_close(soft.cpu().numpy(), ref)
    assert_hard_match(hard.cpu().numpy(), ref)


@pytest.mark.parametrize("M,K,D", [(16, 6, 257), (16, 2, 1000), (32, 5, 100), (64, 6, 70)])
def test_a_workspace_that_is_not_used_changes_nothing(M, K, D):
    """The FP16 x3 form leaves a workspace untouched and gives the bits of the call without one."""
    N = 3000
    ent, gam, clin = synth.random_state(M, K, D, instance=D)
    gp = apsm.Params(M=M, K=K, window=1, dict_cap=D, sigma=0.5, w_L=0.5)
    st = load_state(gp, ent, gam, clin)
    rx = to_dev(synth.random_state(M, 1, N, instance=2)[0])
    nb = apsm.detect_workspace_bytes(gp, N)
    assert (nb > 0) == (M == 16)
    ws = torch.zeros(max(nb, 4096), dtype=torch.uint8, device="cuda")
    soft, hard = apsm.detect(gp, st, rx, workspace=ws)
    plain, hard_plain = apsm.detect(gp, st, rx)
    assert torch.equal(soft, plain) and torch.equal(hard, hard_plain)
    assert torch.count_nonzero(ws) == 0
