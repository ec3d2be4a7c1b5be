"""GPU parity of REDUCE where the features lie in one-field groups and structs (the sums go through the tables
in shared memory, the CTA's total through the table behind them), alone and fused with an ASSIGN whose centroids
lie behind that, at the largest numbers of features and clusters; bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_fields_equal, from_device, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K", [(32, 8), (32, 1), (5, 8)])
@pytest.mark.parametrize("n", [127, 70001])
def test_reduce_of_mixed_groups(d, K, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    wl = synth.kmeans(n=n, n_features=d, k=K)
    fields = oracle.initial_fields(wl)
    fields[d] = fields[d].view(np.int32)
    want = [f.copy() for f in fields]
    oracle.section(wl.sections[0], wl.dtypes, want)
    sums = oracle.section(wl.sections[1], wl.dtypes, want)
    groups = [[d, 0], [1], list(range(2, d))]
    S, lay = P.Schema(wl.dtypes), P.Layout(groups)
    for R in (0, 32, 64):
        for fused in (False, True):
            bufs = to_device(n, wl.dtypes, groups, fields)
            sections = P.Sections(wl.sections)
            try:
                P.adha_tune_override(R)
                if fused:
                    P.adha_run_sections_fused(S, n, lay, bufs, sections)
                else:
                    for k in range(2):
                        P.adha_run_section(S, n, lay, bufs, sections.arr[k])
            finally:
                P.adha_tune_override(0)
            torch.cuda.synchronize()
            assert_fields_equal(from_device(n, wl.dtypes, groups, bufs), want, "assign, fused %s" % fused)
            assert np.array_equal(sections.outputs[1].cpu().numpy(), sums), "reduce, chunk %d, fused %s" % (R, fused)
