"""Against the fp64 oracle (-m gpu), where they can go wrong: the Gram matrices of a cut sequence from tensor-core products
(blocks of 32 tokens with a remainder, fewer blocks than the CTAs that share a segment, several per CTA), and the pair
kernel's diag(delta)^-1/2 L^-1 operand on both sides of delta = 1e9, from where its rows carry scales of their own."""
import numpy as np
import pytest
import torch

import paper_2605_11196_b200 as vla
from paper_2605_11196_b200 import workloads as W
from parity_util import rel_err, run_gpu, run_oracle

pytestmark = pytest.mark.gpu
IDENT = vla.VLA_FLAG_IDENTITY_MAP


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("chunks", [1, 5, 9, 27])   # 16-token chunks a segment: half a block, 2.5, 4.5, 13.5 blocks
@pytest.mark.parametrize("flags", [0, IDENT])
def test_gram_blocks(d, dtype, chunks, flags):
    w = W.Workload("gram", 1, 2, d, 3 * 16 * chunks, dtype, 40 + d + chunks)
    q, k, v = W.make_inputs(w)
    ref = run_oracle(q, k, v, 0.5, flags=flags)
    r = vla.vla_forward_seqpar(q.cuda(), k.cuda(), v.cuda(), 0.5, segments=3, flags=flags)
    torch.cuda.synchronize()
    assert int(r.status.item()) == 0
    for name in ("out", "S_T", "A_T", "z_T"):   # at most 7.2e-7 was seen; without one cross term of the products A_T is off by 2.6e-5
        assert rel_err(getattr(r, name), getattr(ref, name)) <= 3e-6, name


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("flags", [0, IDENT])
def test_gram_matrix_of_a_long_segment(d, dtype, flags):
    """256 blocks of 32 tokens a CTA, where an error to one side does not average out: the matrix itself (it comes first in the
    workspace, from its first 256-byte boundary on) against 64 bits.  What is left is the rounding of k_hat to fp32, 2^-25 an
    entry, partly averaged: at most 1.7e-8 was seen, 0.6e-8 to 2.2e-8 with fp32 products, 4e-8 to 9e-8 with two-term ones."""
    seg = 4 * 256 * 32
    k = torch.randn((1, 1, 2 * seg, d), device="cuda", generator=torch.Generator("cuda").manual_seed(d)).to(dtype)
    ws = torch.zeros((vla.seqpar_workspace_bytes(1, 1, 2 * seg, d, 2),), dtype=torch.uint8, device="cuda")
    r = vla.vla_forward_seqpar(k, k, k, 1.0, segments=2, workspace=ws, flags=flags)
    torch.cuda.synchronize()
    assert int(r.status.item()) == 0
    first = -ws.data_ptr() % 256
    G = ws[first:first + d * d * 8].view(torch.float64).view(d, d)
    x = k[0, 0, :seg].double()
    x = x if flags else torch.where(x > 0, x + 1, torch.exp(x))
    x = x / x.norm(dim=-1, keepdim=True).clamp_min(1e-4)
    ref = x.T @ x
    assert float((G - ref).norm() / ref.norm()) <= 2 ** -25
    assert float((G - ref).trace().abs() / ref.trace()) <= 2 ** -25


@pytest.mark.parametrize("d", [16, 64, 128])
@pytest.mark.parametrize("lam", [2e-8, 2e-9, 9e-10, 5e-10, 1e-11])
def test_rows_of_the_back_substitution(d, lam):
    """delta starts at 1 + 1 / lambda and falls to order one within d tokens, and A loses 1 / lambda of its size meanwhile.  With
    fp32 sums in place of these products A_T was off by up to 5e-6, 2e-5, 1.8e-4 (2-norm, three seeds); three times that."""
    w = W.Workload("rows", 1, 2, d, d - 3, "f32", 15)
    q, k, v = W.make_inputs(w)
    ref = run_oracle(q, k, v, lam, flags=IDENT)
    r = run_gpu(q, k, v, lam, flags=IDENT, kernel=vla.VLA_KERNEL_PAIR)
    e = r.A_T.cpu().double().numpy() - ref.A_T
    assert np.linalg.norm(e) <= {16: 1.5e-5, 64: 6e-5, 128: 5.4e-4}[d] * np.linalg.norm(ref.A_T)
