"""Chunked backward pass (vla_backward without the gradient of A0) against the fp64 backward oracle
(-m gpu): edges of chunks and blocks, every d, carried states, state gradients, explicit u, layouts, and
more units than one pass over its workspace takes."""
import pytest
import torch

import oracle
import paper_2605_11196_b200 as vla
from paper_2605_11196_b200 import workloads as W
from parity_util import NTHREADS, to_oracle_array
from test_gpu_backward import _err

pytestmark = pytest.mark.gpu
IDENT, TM = vla.VLA_FLAG_IDENTITY_MAP, vla.VLA_FLAG_TOKEN_MAJOR


def _compare(w, flags, lam, tol, u=None, carried=False, states=False, tm=False):
    g = torch.Generator().manual_seed(w.seed)
    q, k, v = W.make_inputs(w)
    n, d = (w.B, w.H), w.d
    rnd = lambda *s: torch.randn(n + s, generator=g)
    d_out, kw = rnd(w.T, d), {}
    if u is not None:
        kw["u"] = W.make_u(w, u)
    if carried:
        h = 0.1 * rnd(d, d)
        kw.update(S0=0.2 * rnd(d, d), A0=h @ h.transpose(-1, -2) + 0.5 * torch.eye(d), z0=torch.rand(n + (d,), generator=g))
    if states:
        kw.update(dS_T=rnd(d, d), dA_T=rnd(d, d), dz_T=rnd(d))
    lay = (lambda x: x.transpose(1, 2).contiguous()) if tm else (lambda x: x)
    seq = ("u",)
    dev = {a: (lay(x) if a in seq else x).cuda() for a, x in kw.items()}
    got = vla.vla_backward(lay(q).cuda(), lay(k).cuda(), lay(v).cuda(), lam, lay(d_out).cuda(), want_dA0=False,
                           flags=flags | (TM if tm else 0), **dev)
    torch.cuda.synchronize()
    assert int(got.status.item()) == 0 and got.dA0 is None
    f64 = {a: x.double().numpy() for a, x in kw.items() if a != "u"}
    ua = to_oracle_array(kw["u"])[0] if u is not None else None
    (qa, dt), ka, va = to_oracle_array(q), to_oracle_array(k)[0], to_oracle_array(v)[0]
    ref = oracle.backward(qa, ka, va, lam, d_out.double().numpy(), u=ua, in_dtype=dt, flags=flags, n_threads=NTHREADS, **f64)
    for name in ("dq", "dk", "dv", "dS0", "dz0") + (("du",) if u is not None else ()):
        x = getattr(got, name)
        e = _err(lay(x) if tm and name in ("dq", "dk", "dv", "du") else x, getattr(ref, name))
        assert e <= tol, "%s: rel err %.3e > %.1e" % (name, e, tol)


@pytest.mark.parametrize("d", [16, 32, 64, 128])
@pytest.mark.parametrize("T", [1, 15, 16, 17, 32, 33, 100])
@pytest.mark.parametrize("flags", [0, IDENT])
def test_chunked_gradients_agree_with_the_oracle(d, T, flags):
    w = W.Workload("bc", 2, 3, d, T, "bf16" if T % 2 else "f32", 40 * d + T)
    _compare(w, flags, 1.0, 2e-5 if T > 1 else 2e-4)   # (T = 1: dq cancels to rounding noise)
    _compare(w, flags, 0.1, 1e-4 if T > 1 else 2e-4)
    _compare(w, flags, 0.5, 5e-5, carried=True, states=True)
    if d >= 32:
        _compare(w, flags, 1.0, 5e-5, u=d ** -0.5, states=True, tm=True)
        _compare(w, flags, 1.0, 5e-5, u=1.0, carried=True)


def test_units_in_groups_and_long_sequences():
    """T = 4096; and a call whose workspace would pass 4 GiB, which takes its units in two groups (checked through
    the bits of the first and last units against calls of their own)."""
    w = W.Workload("bc", 1, 2, 64, 4096, "f32", 9)
    _compare(w, 0, 1.0, 5e-5)
    T, units = 2048, 200
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v, do = [torch.randn((units, 1, T, 128), generator=g, device="cuda") for _ in range(4)]
    a = vla.vla_backward(q, k, v, 1.0, do, want_dA0=False)
    for s in (slice(0, 1), slice(units - 2, units)):
        b = vla.vla_backward(q[s].contiguous(), k[s].contiguous(), v[s].contiguous(), 1.0, do[s].contiguous(), want_dA0=False)
        assert all(torch.equal(getattr(a, n)[s], getattr(b, n)) for n in ("dq", "dk", "dv", "dS0"))


@pytest.mark.parametrize("d", [16, 32, 64, 128])
@pytest.mark.parametrize("units,T", [(5, 37), (5, 16), (40, 1000)])
@pytest.mark.parametrize("explicit_u", [False, True])
def test_gradients_do_not_depend_on_what_the_workspace_held(d, units, T, explicit_u):
    """A value read before it is written, or a missing wait, shows as a difference: four calls, the workspace full of zeros, NaN,
    large numbers and what the call before left in it, give the same bits."""
    if explicit_u and d == 16:
        return
    w = W.Workload("ws", 1, units, d, T, "bf16", 3 * d + T)
    q, k, v = [x.cuda() for x in W.make_inputs(w)]
    u = W.make_u(w, d ** -0.5).cuda() if explicit_u else None
    g = torch.randn(q.shape, device="cuda")
    ws = torch.empty((vla.backward_workspace_bytes(1, units, T, d),), dtype=torch.uint8, device="cuda")
    first = None
    for fill in (0, 255, 0x6f, None):
        if fill is not None:
            ws.fill_(fill)
        r = vla.vla_backward(q, k, v, 1.0, g, u=u, workspace=ws, want_dA0=False)
        assert int(r.status.item()) == 0
        got = [r.dq, r.dk, r.dv, r.dS0, r.dz0] + ([r.du] if explicit_u else [])
        assert all(torch.isfinite(x).all() for x in got)
        first = first or got
        assert all(torch.equal(a, b) for a, b in zip(first, got))
