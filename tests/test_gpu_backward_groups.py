"""How vla_backward's chunked form lays its units out over launches (-m gpu): the bits of the first and
last units of a large call against calls of their own."""
import pytest
import torch

import oracle
import paper_2605_11196_b200 as vla
from paper_2605_11196_b200 import workloads as W
from parity_util import NTHREADS, rel_err, to_oracle_array

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


@pytest.mark.parametrize("tm,B,H", [(False, 1, 61), (True, 12, 5), (True, 1, 61), (True, 2, 61)])
def test_groups_of_either_layout(tm, B, H):
    """T = 8192, d = 128: 94 MB a unit, so 60 units pass 4 GiB and take turns: whole batch entries, and parts of one
    where a single entry is too large.  Explicit u, carried states and state gradients, the last units of every group."""
    T, d = 8192, 128
    g = torch.Generator(device="cuda").manual_seed(2)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    seq = (B, T, H, d) if tm else (B, H, T, d)
    q, k, v, u = [rnd(*seq).bfloat16() for _ in range(4)]
    u = torch.nn.functional.normalize(u.float(), dim=-1).bfloat16()
    do, S0, dS_T, dA_T, z0, dz_T = rnd(*seq), rnd(B, H, d, d), rnd(B, H, d, d), rnd(B, H, d, d), 5 + rnd(B, H, d).abs(), rnd(B, H, d)
    h = 0.05 * rnd(B, H, d, d)
    A0 = (h @ h.transpose(-1, -2) + 0.5 * torch.eye(d, device="cuda")).contiguous()
    flags = vla.VLA_FLAG_TOKEN_MAJOR if tm else 0
    a = vla.vla_backward(q, k, v, 1.0, do, u=u, S0=S0, A0=A0, z0=z0, dS_T=dS_T, dA_T=dA_T, dz_T=dz_T, flags=flags, want_dA0=False)
    assert int(a.status.item()) == 0
    for b, hh in [(0, 0), (B - 1, H - 1), (B // 2, H // 2), (0, H - 1), (B - 1, 0)]:
        c = lambda x: x[b:b + 1, :, hh:hh + 1].contiguous() if tm and x.dim() == 4 and x.shape[1] == T else x[b:b + 1, hh:hh + 1].contiguous()
        own = vla.vla_backward(c(q), c(k), c(v), 1.0, c(do), u=c(u), S0=c(S0), A0=c(A0), z0=c(z0), dS_T=c(dS_T), dA_T=c(dA_T),
                               dz_T=c(dz_T), flags=flags, want_dA0=False)
        for n in ("dq", "dk", "dv", "du", "dS0", "dz0"):
            assert torch.equal(c(getattr(a, n)), getattr(own, n)), (n, b, hh)


@pytest.mark.parametrize("d,T,flags", [(64, 65536, 0), (64, 65536, vla.VLA_FLAG_IDENTITY_MAP), (128, 8192, 0)])
def test_long_sequences_of_the_chunked_form(d, T, flags):
    """Whole units of the long and the throughput shape, every gradient within 1e-4 of the oracle (T 65536 of the largest entry;
    the token-level form is held to 1e-3 there)."""
    w = W.Workload("long", 1, 1, d, T, "bf16", 3)
    q, k, v = W.make_inputs(w)
    do = torch.randn((1, 1, T, d), generator=torch.Generator().manual_seed(6))
    (qa, dt), ka, va = to_oracle_array(q), to_oracle_array(k)[0], to_oracle_array(v)[0]
    ref = oracle.backward(qa, ka, va, 1.0, do.double().numpy(), in_dtype=dt, flags=flags, n_threads=NTHREADS)
    got = vla.vla_backward(q.cuda(), k.cuda(), v.cuda(), 1.0, do.cuda(), want_dA0=False, flags=flags)
    for n in ("dq", "dk", "dv", "dS0"):
        assert rel_err(getattr(got, n), getattr(ref, n)) <= 1e-4, n
