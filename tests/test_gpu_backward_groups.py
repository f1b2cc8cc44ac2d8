"""How vla_backward's chunked form lays its units out over launches (-m gpu): the bits of the first and
last units of a large call against calls of their own."""
import pytest
import torch

import paper_2605_11196_b200 as vla

pytestmark = pytest.mark.gpu


def _same(got, part, own, names=("dq", "dk", "dv", "dS0", "dz0")):
    for n in names:
        assert torch.equal(getattr(got, n)[part], getattr(own, n)), n


@pytest.mark.parametrize("B,H,T,d", [(16501, 4, 8, 16), (66001, 1, 3, 32)])
def test_more_units_than_a_grids_second_dimension(B, H, T, d):
    g = torch.Generator(device="cuda").manual_seed(1)
    x = [torch.randn((B, H, T, d), generator=g, device="cuda") for _ in range(4)]
    dS_T = torch.randn((B, H, d, d), generator=g, device="cuda")
    dA_T = torch.randn((B, H, d, d), generator=g, device="cuda")
    a = vla.vla_backward(*x[:3], 1.0, x[3], dS_T=dS_T, dA_T=dA_T, want_dA0=False)
    for s in (slice(0, 2), slice(B - 2, B)):
        q, k, v, do, dS, dA = [y[s].contiguous() for y in x + [dS_T, dA_T]]
        _same(a, s, vla.vla_backward(q, k, v, 1.0, do, dS_T=dS, dA_T=dA, want_dA0=False))
    assert int(a.status.item()) == 0
