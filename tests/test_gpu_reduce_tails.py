"""GPU parity of the REDUCE section's ragged tail (up to 127 records by one warp: 32 memberships and
eight records at a time), with members out of range and features beyond the fixed-point range, infinite
and NaN, bit for bit against the oracle; and of the sums added up per CTA when only the tail has records."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu
F32, I32 = synth.workloads.F32, synth.workloads.I32


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("d,K", [(1, 8), (13, 1), (32, 5)])
@pytest.mark.parametrize("n", [1, 8, 31, 33, 127, 128 + 65, 5 * 128 + 127])
def test_reduce_tail(layout, d, K, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    rng = np.random.default_rng(100 * d + n)
    fields = [rng.uniform(-300, 300, n).astype(np.float32) for _ in range(d)]   # some beyond +-256
    for f in fields:
        f[rng.random(n) < 0.05] = np.nan
        f[rng.random(n) < 0.05] = -np.inf
    fields.append(rng.integers(-2, K + 2, n).astype(np.int32))
    sec = synth.Section("reduce", (d, K), frozenset(range(d + 1)), frozenset())
    groups = [list(range(d + 1))] if layout == "aos" else [[f] for f in range(d + 1)]
    dtypes = [F32] * d + [I32]
    want = oracle.core.kmeans_reduce(sec, dtypes, [f.copy() for f in fields])
    bufs = to_device(n, dtypes, groups, fields)
    for R in (0, 32, 64, 128):
        sections = P.Sections([sec])
        try:
            P.adha_tune_override(R)
            P.adha_run_section(P.Schema(dtypes), n, P.Layout(groups), bufs, sections.arr[0])
        finally:
            P.adha_tune_override(0)
        torch.cuda.synchronize()
        assert np.array_equal(sections.outputs[0].cpu().numpy().reshape(want.shape), want), "chunk %d" % R
