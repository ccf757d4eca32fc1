"""Surrogate inference over tile counts that leave an SM one tile, two, a full
group of three, and full groups with one or two tiles after them: a sample's
result does not depend on the tiles around it, and the input may be the output."""
import pytest
import torch

import paper_2108_11775_gb300 as pdmp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm,rest", [(0, 5), (1, 0), (1, 77), (2, 1), (3, 0), (4, 3), (5, 0), (6, 129)])
def test_results_do_not_depend_on_the_grouping(per_sm, rest):
    assert torch.cuda.is_available()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 128 * sms * per_sm + rest
    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.rand(N, 3, generator=g, device="cuda") * 5.0
    if N > 2:
        x[N // 2] = torch.tensor([3.0e7, -1.0e30, float("nan")], device="cuda")   # far outside the box
    net = pdmp.Surrogate([0.0] * 3, [5.0] * 3, [0.05, 0.07, 0.03], seed=3)
    y = net.forward(x)
    some = torch.unique(torch.cat([torch.randint(0, N, (90,), generator=g, device="cuda"),
                                   torch.tensor([0, N // 2, N - 1], device="cuda")]))
    alone = net.forward(x[some].contiguous())
    assert torch.equal(torch.nan_to_num(y[some], nan=7.0), torch.nan_to_num(alone, nan=7.0))
    assert torch.isfinite(torch.cat([y[:N // 2], y[N // 2 + 1:]])).all()
    z = x.clone()
    net.forward(z, out=z)
    assert torch.equal(torch.nan_to_num(z, nan=7.0), torch.nan_to_num(y, nan=7.0))
    assert pdmp.stream_status()[0] == 0
