"""adha_run_program with return_to_input under a plan that leaves the input layout and comes back to it: the
result is in the input buffers whatever layout the last section ran in."""
import pytest
import torch

import oracle
import synth
from gpu_util import assert_fields_equal, from_device, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fixed", [[0, 1, 0], [1, 1, 0], [1, 0, 1], [0, 0, 0]])
@pytest.mark.parametrize("n", [4099, 65536])
def test_result_is_in_the_input_buffers(fixed, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    wl = synth.config1(n=n)
    S, aos = P.Schema(wl.dtypes), P.Layout.aos(wl.F)
    cand = P.adha_layout_set_create(wl.F, [aos, P.Layout.soa(wl.F)])
    fields = oracle.initial_fields(wl)
    want = oracle.run_program_fields(wl, [a.copy() for a in fields])
    bufs = to_device(n, wl.dtypes, aos.groups, fields)
    ws = torch.empty(P.adha_program_workspace_bytes(S, n, aos, cand), dtype=torch.uint8, device="cuda")
    plan = P.adha_run_program(S, n, aos, bufs, P.Sections(wl.sections), cand, opts=P.PlanOpts(return_to_input=True),
                              workspace=ws, fixed=fixed)
    torch.cuda.synchronize()
    assert plan.final_ptrs[0] == bufs[0].data_ptr()
    assert_fields_equal(from_device(n, wl.dtypes, aos.groups, bufs), want, "returned program")
