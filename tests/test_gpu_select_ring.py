"""GPU parity of the resident selection's load (vectors through a ring of three
rounds in shared memory) at its edges: slices of one round (no ring), of the
ring's length and around it, that end inside a vector, the most values the form
takes, misaligned input (no ring), with NaN, an infinity and a threshold.
Compared exactly with a full sort of the same values."""
import math

import pytest

from synthetic import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_ring_rounds(dtype):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    w = W.full_state_12q()
    c = w.circuit
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in w.probs])
        qid, _ = ctx.set_qubit_roles(cid, w.roles)
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        word = 1024 * (4 if dtype == "float32" else 2)     # values of one round of a CTA
        for n in [sms * p - 1 for p in (word, word + 4, 3 * word, 3 * word + 4, 4 * word + 8)] + [5 << 20]:
            g = torch.Generator(device="cuda").manual_seed(n)
            x = torch.empty(n + 1, dtype=getattr(torch, dtype), device="cuda").exponential_(1.0, generator=g)
            x[n // 2] = math.inf
            x[n // 3] = math.nan
            x[-2:] = 50.0                                  # the last value of the last slice is selected
            for y in (x[:n], x[1:]):                       # 16-byte aligned, and not
                for k, thr in ((1, -math.inf), (1000, -math.inf), (4096, 9.0)):
                    b, v, nf = ctx.top_bins(qid, y, k, thr)
                    idx = torch.nonzero(y >= thr).flatten()            # false for NaN
                    val, order = torch.sort(y[idx], descending=True, stable=True)
                    m = min(k, idx.numel())
                    assert int(nf.item()) == m
                    assert torch.equal(b[:m], idx[order[:m]])
                    assert torch.equal(v[:m], val[:m].double())
