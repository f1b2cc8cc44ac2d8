"""The three-CTA clusters of a cut sequence (one A, the segment's S and its transfer scan) against the fp64
oracle where they can go wrong: one chunk a segment, chunk counts around the input and alpha slots, and more
segments than the device holds at a time."""
import pytest
import torch

import paper_2605_11196_b200 as vla
from paper_2605_11196_b200 import workloads as W
from parity_util import rel_err, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("units,chunks,segments", [(1, 16, 16), (2, 15, 3), (3, 18, 2), (24, 18, 9)])
@pytest.mark.parametrize("with_u", [False, True])
def test_segment_clusters(d, dtype, units, chunks, segments, with_u):
    w = W.Workload("t", 1, units, d, 16 * chunks, dtype, 300 + d + chunks)
    q, k, v = W.make_inputs(w)
    u = W.make_u(w, d ** -0.5) if with_u else None
    ref = run_oracle(q, k, v, 0.5, u=u)
    dev = torch.device("cuda:0")
    mv = lambda x: None if x is None else x.to(dev).contiguous()
    r = vla.vla_forward_seqpar(mv(q), mv(k), mv(v), 0.5, segments=segments, u=mv(u))
    torch.cuda.synchronize()
    assert int(r.status.item()) == 0
    for name in ("out", "S_T", "A_T", "z_T"):
        assert rel_err(getattr(r, name), getattr(ref, name)) <= 1e-4, name
