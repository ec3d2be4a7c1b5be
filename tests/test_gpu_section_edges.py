"""GPU parity of the single-section kernels where their chunking changes: operands that coincide (written
fields read again by a later step), structs of an even number of 16-byte pieces (staged with room after
each record), the K-Means sections at every number of clusters, feature counts around blocks of four, and
record counts around whole chunks, all bit for bit against the oracle (the K-Means sections against numpy,
on features and centroids whose distances are exact)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_fields_equal, from_device, to_device

pytestmark = pytest.mark.gpu
F32, I32 = synth.workloads.F32, synth.workloads.I32


@pytest.fixture(scope="module")
def P():
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    return P


def _workload(n, dtypes, sections):
    kinds = {F32: "F32_PM1", I32: "I32_U20"}
    return synth.Workload("edge", n, [synth.Field("f%d" % k, d, kinds[d]) for k, d in enumerate(dtypes)], 11, sections)


@pytest.mark.parametrize("groups", [[[0, 1, 2, 3, 4, 5, 6, 7]], [[0, 1, 2, 3], [4, 5, 6, 7]], [[k] for k in range(8)]])
@pytest.mark.parametrize("op,args,params", [
    ("drift", (0, 1, 2, 1, 0, 2), (0.5,)), ("drift", (0, 0, 2, 3, 4, 5), (0.5,)), ("drift", (0, 1, 2, 3, 4, 5), (0.5,)),
    ("kick", (0, 1, 0, 2), (0.5, 0.25, -0.125, 1.0)), ("kick", (0, 1, 2, 1), (0.5, 0.25, -0.125, 1.0)),
    ("madd3", (0, 1, 0), ()), ("madd3", (3, 3, 3), ()), ("add", (2, 5, 5), ()),
])
@pytest.mark.parametrize("n", [31, 128, 70001])
def test_operands_that_coincide(P, groups, op, args, params, n):
    write = {"drift": args[:3], "kick": args[:3], "madd3": args[2:], "add": args[2:]}[op]
    sec = synth.Section(op, args, frozenset(args), frozenset(write), params=params)
    wl = _workload(n, [F32] * 8, [sec])
    fields = oracle.initial_fields(wl)
    want = oracle.run_program_fields(wl, [a.copy() for a in fields])
    bufs = to_device(n, wl.dtypes, groups, fields)
    P.adha_run_section(P.Schema(wl.dtypes), n, P.Layout(groups), bufs, P.c_section(sec))
    torch.cuda.synchronize()
    assert_fields_equal(from_device(n, wl.dtypes, groups, bufs), want, op)


@pytest.mark.parametrize("d,K", [(1, 1), (3, 2), (4, 3), (7, 8), (8, 4), (15, 5), (16, 6), (31, 7), (32, 5)])
@pytest.mark.parametrize("layout", ["aos", "soa", "halves"])
@pytest.mark.parametrize("n", [63, 4096 + 65])
def test_kmeans_sections(P, d, K, layout, n):
    rng = np.random.default_rng(d * 10 + K)
    # features and centroids on the 2^-6 grid: every distance is exact, so the memberships are decided
    cent = tuple(float(v) for v in rng.integers(-64, 64, K * d) / 64.0)
    feats = frozenset(range(d))
    secs = [synth.Section("assign", (d, K), feats, frozenset([d]), table=cent),
            synth.Section("reduce", (d, K), feats | frozenset([d]), frozenset())]
    wl = _workload(n, [F32] * d + [I32], secs)
    groups = {"aos": [list(range(d + 1))], "soa": [[f] for f in range(d + 1)],
              "halves": [list(range(d // 2 + 1)), list(range(d // 2 + 1, d + 1))]}[layout]
    fields = [(rng.integers(-64, 64, n) / 64.0).astype(np.float32) for _ in range(d)] + [np.zeros(n, np.int32)]
    S, lay = P.Schema(wl.dtypes), P.Layout(groups)
    member = np.stack([((np.stack(fields[:d], 1) - np.array(cent, np.float32).reshape(K, d)[k]) ** 2).sum(1, dtype=np.float64)
                       for k in range(K)]).argmin(0).astype(np.int32)
    q = np.stack(fields[:d], 1).astype(np.float64) * 2.0 ** 23
    want = np.stack([np.concatenate([[(member == k).sum()], q[member == k].sum(0)]) for k in range(K)]).astype(np.int64)
    for fused in (False, True):
        bufs = to_device(n, wl.dtypes, groups, fields)
        sections = P.Sections(secs)
        if fused:
            P.adha_run_sections_fused(S, n, lay, bufs, sections)
        else:
            for k in range(2):
                P.adha_run_section(S, n, lay, bufs, sections.arr[k])
        torch.cuda.synchronize()
        got = from_device(n, wl.dtypes, groups, bufs)
        assert_fields_equal(got, fields[:d] + [member], "assign")
        assert np.array_equal(sections.outputs[1].cpu().numpy(), want), "reduce, fused %s" % fused
