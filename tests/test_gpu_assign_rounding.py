"""GPU parity of ASSIGN on records whose membership is decided by the rounding of the squared distances
(one rounding for the square and the sum): the same whether a record lies in a whole chunk or in the ragged
tail, for every chunk size, and in the first or the second assign of a fused run."""
import numpy as np
import pytest
import torch

import near_ties
import synth
from gpu_util import from_device, to_device

pytestmark = pytest.mark.gpu
F32, I32 = synth.workloads.F32, synth.workloads.I32


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("d,K,pair", [(2, 2, (0, 1)), (7, 3, (0, 2)), (32, 5, (3, 4)), (9, 8, (2, 7))])
def test_assign_of_near_ties(layout, d, K, pair):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    x, cent, member = near_ties.records(d, K, pair, 12, seed=d)
    n = 16 * 128 + 127                               # a tail for chunks of 32, 64 and 128 records
    which = np.arange(n) % len(x)                    # every record in chunks and in the tail
    table = tuple(float(v) for v in cent.reshape(-1))
    secs = [synth.Section("assign", (m, K), frozenset(range(d)), frozenset([m]), table=table) for m in (d, d + 1)]
    fields = [np.ascontiguousarray(x[which, j]) for j in range(d)] + [np.full(n, -1, np.int32) for _ in range(2)]
    dtypes = [F32] * d + [I32] * 2
    groups = [list(range(d + 2))] if layout == "aos" else [[f] for f in range(d + 2)]
    S, lay = P.Schema(dtypes), P.Layout(groups)
    for R in (0, 32, 64, 128):
        for fused in (False, True):
            bufs = to_device(n, dtypes, groups, fields)
            sections = P.Sections(secs)
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
            got = from_device(n, dtypes, groups, bufs)
            for f in (d, d + 1):
                bad = np.nonzero(got[f] != member[which])[0]
                assert bad.size == 0, "field %d, chunk %d, fused %s: records %s" % (f, R, fused, bad[:5])
