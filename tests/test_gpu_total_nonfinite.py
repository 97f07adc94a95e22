"""The probability check of steps written in bands, beyond FP32's finite range:
an infinite bin gives an infinite sum (both signs, or NaN: NaN), and bins whose
sum over a few rows passes FP32's largest value a finite one."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _total(a, b, batched):
    """FP64 sum of the bins a[x] b[y] of two unconnected subcircuits."""
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    n = [len(a).bit_length() - 1, len(b).bit_length() - 1]
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(sum(n), [], [], n, list(range(sum(n))),
                                          [torch.from_numpy(v.reshape(1, -1)).cuda() for v in (a, b)])
        qid, na = ctx.set_qubit_roles(cid, np.zeros(sum(n), dtype=np.int8))
        out = torch.empty(1 << na, dtype=torch.float32, device="cuda")
        tot = torch.zeros(1, dtype=torch.float64, device="cuda")
        if batched:
            bid = ctx.batch_create([qid], [out], tot)
            ctx.batch_run(bid)
            ctx.batch_status(bid)
        else:
            ctx.reconstruct(qid, out, "fp32", tot)
        torch.cuda.synchronize()
        assert torch.equal(out, (torch.from_numpy(b)[:, None] * torch.from_numpy(a)[None, :]).reshape(-1).cuda()) or \
            bool(torch.isnan(out).any())
        return tot.item()


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("n", [(9, 10), (12, 9), (11, 12)])
def test_total(n, batched):
    a, b = (np.full(1 << v, 2.0 ** -v, dtype=np.float32) for v in n)
    assert _total(a, b, batched) == 1.0
    a[5] = b[7] = 1e30
    assert _total(a, b, batched) == math.inf
    a[5] = -1e30
    assert _total(a, b, batched) == -math.inf
    a[6] = 1e30
    assert math.isnan(_total(a, b, batched))
    # 32 bins of 2^122 are the most that a group of any tile adds in FP32
    a, b = np.full(1 << n[0], 2.0 ** 60, dtype=np.float32), np.full(1 << n[1], 2.0 ** 62, dtype=np.float32)
    assert _total(a, b, batched) == 2.0 ** (122 + sum(n))
