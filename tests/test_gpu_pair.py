"""Pair kernel (VLA_KERNEL_PAIR: the chunk algebra on warp-level tensor-core products, two CTAs per
unit) vs the fp64 CPU oracle through the C ABI (-m gpu): chunk edges, every d, both input types
and readings, explicit u, carried states, layouts, scales far from one."""
import pytest
import torch

import paper_2605_11196_b200 as vla
from paper_2605_11196_b200 import workloads as W
from parity_util import check_parity, run_gpu

pytestmark = pytest.mark.gpu

PAIR, IDENT = vla.VLA_KERNEL_PAIR, vla.VLA_FLAG_IDENTITY_MAP


def _carried(w):
    g = torch.Generator().manual_seed(3)
    M = torch.randn((w.B, w.H, w.d, w.d), generator=g) * 0.05
    return {"S0": torch.randn((w.B, w.H, w.d, w.d), generator=g) * 0.3,
            "A0": torch.eye(w.d) * 0.5 + M @ M.transpose(-1, -2), "z0": torch.rand((w.B, w.H, w.d), generator=g) * 3}


@pytest.mark.parametrize("d", [16, 32, 64, 128])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T", [1, 15, 16, 17, 33, 83, 144])
def test_pair_matches_the_oracle(d, dtype, T):
    w = W.Workload("pair", 2, 2, d, T, dtype, 7 * d + T)
    q, k, v = W.make_inputs(w)
    for flags in (0, IDENT):
        _, h, _ = check_parity(q, k, v, 1.0, 1e-5, flags=flags, kernel=PAIR, label="plain")
        check_parity(q, k, v, 0.1, 1e-4, flags=flags, kernel=PAIR, label="lambda 0.1")
        check_parity(q, k, v, 1.0, 1e-5, u=W.make_u(w, d ** -0.5), flags=flags, kernel=PAIR, label="u", **_carried(w))
        tm = lambda x: x.transpose(1, 2).contiguous()
        r = run_gpu(tm(q), tm(k), tm(v), 1.0, flags=flags | vla.VLA_FLAG_TOKEN_MAJOR, kernel=PAIR)
        assert torch.equal(r.out.transpose(1, 2), h.out) and torch.equal(r.S_T, h.S_T)


@pytest.mark.parametrize("scale", [1e-9, 1e7])
def test_pair_operand_scales_follow_the_data(scale):
    """The fp16 operands are scaled by powers of two that follow S, E and q: results keep their relative
    accuracy whatever the size of v and q; u far from unit length; A far below its start."""
    w = W.Workload("pair", 1, 3, 64, 700, "f32", 5)
    q, k, v = W.make_inputs(w)
    check_parity(q * scale, k, v * scale, 1.0, 1e-5, flags=IDENT, kernel=PAIR, label="q, v")
    check_parity(q, k, v, 1.0, 1e-5, u=W.make_u(w, 1e-3), kernel=PAIR, label="small u")
    check_parity(q, k, v, 1.0, 1e-4, u=W.make_u(w, 8.0), kernel=PAIR, label="large u")   # (as lambda = 1/64)
