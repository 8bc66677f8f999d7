"""The training adjoint's forms give the same bits: single calls (a team of four warps per user) against one batched
call of more instances than the GPU holds teams of (one warp per user), at row lengths around those from
which a row's later entries are loaded together (768 entries, 1280 with windows above 16), with remainders
of sixteen and of four times 32 entries, and with entries that leave."""
import pytest
import torch

from paper_2201_05024_gb300 import apsm

pytestmark = pytest.mark.gpu


def cn(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda"))


@pytest.mark.parametrize("M,K,W,P,D", [(4, 4, 8, 384, 384), (4, 4, 8, 385, 385), (8, 5, 16, 520, 520), (4, 4, 3, 601, 601),
                                       (4, 4, 8, 530, 450), (4, 4, 11, 700, 390), (4, 4, 20, 640, 640),
                                       (4, 4, 20, 641, 641), (4, 5, 30, 700, 660)])
def test_single_calls_equal_a_large_batch(M, K, W, P, D):
    n = torch.cuda.get_device_properties(0).multi_processor_count // 2 + 4   # two team CTAs per instance
    g = torch.Generator(device="cuda").manual_seed(P + W)
    rx = cn(g, n, P, M) * (0.5 / M) ** 0.5
    sym = torch.sign(torch.view_as_real(cn(g, n, P, K)))
    sym = torch.view_as_complex((sym * 0.5 ** 0.5).contiguous())
    p = apsm.Params(M=M, K=K, window=W, dict_cap=D, sigma=0.6, mu=0.6, eps=0.05, w_L=0.4)
    dg = 0.1 * torch.randn(n, apsm.dict_alloc(p), 2, K, generator=g, device="cuda")
    dc = 0.1 * cn(g, n, M, K)
    ds, dc0 = apsm.train_backward_batched(p, rx, sym, dg, dc)
    assert bool(torch.isfinite(ds).all())
    for i in (0, n // 2, n - 1):
        s, c = apsm.train_backward(p, rx[i].contiguous(), sym[i].contiguous(), dg[i].contiguous(), dc[i].contiguous())
        assert torch.equal(s, ds[i]) and torch.equal(torch.view_as_real(c), torch.view_as_real(dc0[i]))
