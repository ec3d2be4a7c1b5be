"""GPU parity of sections and fused runs on records near what a 32-record chunk holds: structs that fit twice
only without the room after each staged record, structs that fit once, many small structs that room doubles,
and a forced second chunk buffer; bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_fields_equal, from_device, to_device

pytestmark = pytest.mark.gpu
F32, F64 = synth.workloads.F32, synth.workloads.F64


@pytest.fixture(scope="module")
def P():
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    return P


def _workload(n, dtype, F):
    kind = {F32: "F32_PM1", F64: "F64_PM1"}[dtype]
    everything, some = frozenset(range(F)), frozenset(range(0, F, 3))
    secs = [synth.Section("mix", (), everything, everything), synth.Section("mix", (), everything, some)]
    return synth.Workload("wide", n, [synth.Field("f%d" % k, dtype, kind) for k in range(F)], 13, secs)


@pytest.mark.parametrize("dtype,F,width", [
    (F64, 50, 50), (F64, 52, 52), (F64, 53, 53), (F64, 54, 54), (F64, 56, 56), (F64, 56, 1), (F64, 40, 4), (F64, 64, 64),
    (F32, 64, 8), (F32, 40, 8), (F32, 64, 64),
])
@pytest.mark.parametrize("n", [33, 70001])
@pytest.mark.parametrize("buffers", [0, 2])
def test_wide_records(P, dtype, F, width, n, buffers):
    wl = _workload(n, dtype, F)
    fields = oracle.initial_fields(wl)
    want = oracle.run_program_fields(wl, [a.copy() for a in fields])
    groups = [list(range(f, min(f + width, F))) for f in range(0, F, width)]
    S, lay = P.Schema(wl.dtypes), P.Layout(groups)
    for fused in (False, True):
        bufs = to_device(n, wl.dtypes, groups, fields)
        sections = P.Sections(wl.sections)
        try:
            P.adha_tune_section_buffers(buffers)
            P.adha_tune_fused_buffers(buffers)
            if fused:
                P.adha_run_sections_fused(S, n, lay, bufs, sections)
            else:
                for k in range(2):
                    P.adha_run_section(S, n, lay, bufs, sections.arr[k])
        finally:
            P.adha_tune_section_buffers(0)
            P.adha_tune_fused_buffers(0)
        torch.cuda.synchronize()
        assert_fields_equal(from_device(n, wl.dtypes, groups, bufs), want, "fused" if fused else "sections")
