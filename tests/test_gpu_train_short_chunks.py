"""Training at 64 antennas with entries that leave: chunks that shared memory cuts short, ended on a whole block or
kept to one round of tracked samples, against the oracle, and in two calls against one."""
import numpy as np
import pytest

import oracle
from paper_2201_05024_gb300 import apsm, synth

from parity import rms, to_dev
from test_gpu_parity import _compare_training, _train_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,D,W", [(240, 130, 13), (240, 130, 17), (250, 120, 20), (215, 120, 20), (216, 120, 20),
                                   (230, 90, 10), (120, 100, 24)])
def test_matches_oracle(P, D, W):
    inst = synth.make_instance(64, 2, P, 50, 10.0, instance=P + W)
    op = oracle.Params(M=64, K=2, W=W, D=D, sigma=0.5, mu=0.5, eps=0.01, w_L=0.5)
    gp, st, cl, ref = _train_both(op, inst)
    _compare_training(op, inst, gp, st, cl, ref, tol_coef=1e-4)


@pytest.mark.parametrize("W", [13, 20])
def test_two_calls_equal_one(W):
    P, D, first = 330, 120, 75
    inst = synth.make_instance(64, 2, P, 1, 10.0, instance=W)
    gp = apsm.Params(M=64, K=2, window=W, dict_cap=D, sigma=0.5, mu=0.5, eps=0.01, w_L=0.5)
    rx, sym = to_dev(inst.rx_pilot), to_dev(inst.sym_pilot)
    one = apsm.train(gp, rx, sym, apsm.State(gp))
    two = apsm.train(gp, rx[:first].contiguous(), sym[:first].contiguous(), apsm.State(gp))
    apsm.train_continue(gp, rx[first:].contiguous(), two, sym[first:].contiguous())
    a, b = one.gamma[:D].cpu().numpy(), two.gamma[:D].cpu().numpy()
    assert np.abs(a - b).max() <= 1e-4 * rms(a)     # the tolerance of trained coefficients
    assert np.array_equal(one.dict[:D].cpu().numpy(), two.dict[:D].cpu().numpy())
