"""GPU parity at the sizes where a kernel or a dispatch rule can go wrong: tile edges, remainders, the smallest and the
largest of its range, against the oracle (fp64) on the same seeded inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2608_00938_b200 import api as _api
    return _api


from gpu_util import DEV  # noqa: E402


@pytest.mark.parametrize("B,M,H,T", [(16, 1000, 16, 200), (20, 300, 8, 640)])
def test_cross_attn_waits_never_give_up_back_to_back(api, B, M, H, T):
    """Head size 128, launches queued without a gap: no bounded wait runs out (the issuing
    thread may come arbitrarily late to its wait for a block's probabilities), and the last output is the first's."""
    d = 128
    g = torch.Generator(device=DEV)
    g.manual_seed(5)
    q, k, v = (torch.randn(*s, device=DEV, generator=g).to(torch.bfloat16) for s in ((B * M, H, d), (B, H, T, d), (B, H, T, d)))
    first, last = torch.empty_like(q), torch.empty_like(q)
    api.grace_wait_timeouts()
    api.grace_cross_attn(q, k, v, first, d ** -0.5)
    for _ in range(4000):
        api.grace_cross_attn(q, k, v, last, d ** -0.5)
    torch.cuda.synchronize()
    assert api.grace_wait_timeouts() == 0
    assert torch.equal(first, last)
