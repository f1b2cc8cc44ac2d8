"""Against the fp64 oracle (-m gpu), where they can go wrong: the Gram matrices of a cut sequence from tensor-core products
(blocks of 32 tokens with a remainder, fewer blocks than the CTAs that share a segment, several per CTA), and the pair
kernel's diag(delta)^-1/2 (L^-1 - I) operand on both sides of delta = 1e6, from where its rows carry scales of their own."""
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


def _norm_err(x, ref):
    return np.linalg.norm(x.cpu().double().numpy() - ref) / np.linalg.norm(ref)


# largest of the kernel's own errors over seeds 15 to 18 and the lambda below, times three
@pytest.mark.parametrize("d,tol", [(16, 1.4e-5), (32, 4.2e-5), (64, 7.2e-5), (128, 1.6e-3)])
@pytest.mark.parametrize("seed", [15, 16, 17])
def test_rows_with_scales_of_their_own(d, tol, seed):
    """Past delta = 1e6 a row of the operand has a power of two of its own.  Without it A_T is off by 1.1e-4, 1.7e-3 and 8.3e-3 at
    lambda 1e-14 (d = 16, 64, 128).  (The readout there takes differences of numbers 1 / lambda apart, in every kernel; it is
    compared where it is well conditioned.)"""
    w = W.Workload("rows", 1, 2, d, d - 3, "f32", seed)
    q, k, v = W.make_inputs(w)
    for lam in (2e-6, 5e-7, 2e-8, 5e-10, 1e-13, 1e-14):
        ref = run_oracle(q, k, v, lam, flags=IDENT)
        r = run_gpu(q, k, v, lam, flags=IDENT, kernel=vla.VLA_KERNEL_PAIR)
        assert _norm_err(r.A_T, ref.A_T) <= tol, lam
        if lam > 1e-10:
            assert _norm_err(r.out, ref.out) <= 7.2e-6 and _norm_err(r.S_T, ref.S_T) <= max(tol / 10, 7.2e-6), lam


@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("lam", [0.01, 1e-3])
@pytest.mark.parametrize("flags", [0, IDENT])
def test_small_lambda_over_several_times_d_tokens(d, lam, flags):
    """After A has lost its large directions: the states no further from fp64 than the fp32 token-level kernel leaves them
    (seen: 0.02 to 0.84 of its errors), the readout within six times (seen: 0.1 to 4.3)."""
    for T in (200, 500):
        w = W.Workload("many", 4, 8, d, T, "f32", 31 + d)
        q, k, v = W.make_inputs(w)
        ref = run_oracle(q, k, v, lam, flags=flags)
        a, b = [run_gpu(q, k, v, lam, flags=flags, kernel=x) for x in (vla.VLA_KERNEL_PAIR, vla.VLA_KERNEL_TOKEN)]
        for name, times in (("S_T", 1.0), ("A_T", 1.0), ("out", 6.0)):
            assert _norm_err(getattr(a, name), getattr(ref, name)) <= times * _norm_err(getattr(b, name), getattr(ref, name)), (name, T)


@pytest.mark.parametrize("d,tol", [(64, 1.8e-5), (128, 7e-5)])
@pytest.mark.parametrize("lam", [1e-6, 1e-9])
def test_back_substitution_keeps_the_unit_diagonal(d, tol, lam):
    """A_T's 2-norm error, the geometric mean over 32 units: 1.3e-5 to 1.5e-5 and 4.9e-5 to 5.3e-5 were seen, as much as with tf32 pairs in four
    products (1.4e-5 to 1.5e-5, 5.1e-5 to 5.6e-5); 2.2e-5 and 9.4e-5 where L^-1's unit diagonal went through the truncating sum."""
    w = W.Workload("diag", 4, 8, d, d - 3, "f32", 100 + d)
    q, k, v = W.make_inputs(w)
    ref = run_oracle(q, k, v, lam, flags=IDENT).A_T.reshape(32, -1)
    x = run_gpu(q, k, v, lam, flags=IDENT, kernel=vla.VLA_KERNEL_PAIR).A_T.cpu().double().numpy().reshape(32, -1)
    e = np.linalg.norm(x - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.exp(np.log(e).mean()) <= tol
