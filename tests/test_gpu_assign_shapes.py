"""GPU parity of ASSIGN at the record counts and widths where its launch shape changes: narrow records long
enough for chunks of 128 in two buffers, wide ones around the limit of the 32-record chunks; against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_fields_equal, from_device, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,layout", [(1, 2, "aos"), (2, 3, "soa"), (6, 8, "aos"), (7, 5, "soa"), (7, 5, "aos"), (17, 4, "aos")])
@pytest.mark.parametrize("n", [389119, 389121, 622591, 622593, 2490369])
def test_assign_shapes(d, K, layout, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    wl = synth.kmeans(n=n, n_features=d, k=K)
    fields = oracle.initial_fields(wl)
    fields[d] = fields[d].view(np.int32)
    groups = [list(range(d + 1))] if layout == "aos" else [[f] for f in range(d + 1)]
    bufs = to_device(n, wl.dtypes, groups, fields)
    sections = P.Sections(wl.sections)
    P.adha_run_section(P.Schema(wl.dtypes), n, P.Layout(groups), bufs, sections.arr[0])
    torch.cuda.synchronize()
    oracle.section(wl.sections[0], wl.dtypes, fields)
    assert_fields_equal(from_device(n, wl.dtypes, groups, bufs), fields, "assign")
