"""GPU parity of chain runs: a run of axpb / mul / tanh sections and its gradient in one pass each.  The
gradient of the linear loss equals the oracle's chain gradient bit for bit, the forward state its
final state, and the backward hands the state back as it was; at the record counts where chunks of 32,
64 and 128 records end, operands that alias, groups the run does not touch, structs whose size is and
is not a multiple of 16 bytes, and more sections than one run takes."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    return P


def _sections(rng, fields, count):
    """Sections over `fields`; operands drawn with replacement, so x, y and z coincide often."""
    out = []
    for _ in range(count):
        u, (x, y, z) = rng.random(), (int(f) for f in rng.choice(fields, 3))
        if u < 0.4:
            a, b = (float(np.float32(v)) for v in rng.uniform(-1, 1, 2))
            out.append(synth.Section("axpb", (x, z), frozenset([x]), frozenset([z]), params=(a, b)))
        elif u < 0.7:
            out.append(synth.Section("mul", (x, y, z), frozenset([x, y]), frozenset([z])))
        else:
            out.append(synth.Section("tanh", (x, z), frozenset([x]), frozenset([z])))
    return out


LAYOUTS = {"soa": lambda F: [[f] for f in range(F)], "aos": lambda F: [list(range(F))],
           "mixed": lambda F: [[0, 1, 2, 3], [4]] + [[5, 6, 7]] + [[f] for f in range(8, F)]}


@pytest.mark.parametrize("layout", sorted(LAYOUTS))
@pytest.mark.parametrize("F,used,count,n", [
    (3, 3, 1, 1), (9, 9, 7, 31), (12, 6, 40, 32), (24, 24, 64, 127), (24, 10, 64, 128), (10, 10, 129, 129),
    (8, 8, 300, 4099), (64, 64, 128, 4099), (24, 24, 64, (1 << 18) + 33), (12, 5, 16, (1 << 18) - 1),
])
def test_chain_equals_oracle(P, layout, F, used, count, n):
    from paper_1407_4859_gb300.autograd import SegmentFn
    if F < 9 and layout == "mixed":
        pytest.skip("too few fields for this layout")
    rng = np.random.default_rng(F * 1000 + count)
    secs = _sections(rng, np.arange(used), count)
    fields = [np.float32(4.0) * rng.standard_normal(n).astype(np.float32) for _ in range(F)]   # tanh saturates for some
    c = [float(np.float32(v)) for v in rng.uniform(-1, 1, F)]
    st = [a.copy() for a in fields]
    want = oracle.chain_grad(secs, st, c)
    lay = P.Layout(LAYOUTS[layout](F))
    leaves = [torch.from_numpy(np.stack([fields[f] for f in g], axis=1)).cuda().requires_grad_() for g in lay.groups]
    state = [x * 1.0 for x in leaves]   # the segment works in place
    out = SegmentFn.apply((P.Schema([0] * F), n, lay, secs), *state)
    seeds = [torch.tensor([c[f] for f in g], device="cuda").expand(n, len(g)).contiguous() for g in lay.groups]
    for g, t in zip(lay.groups, out):
        for j, f in enumerate(g):
            assert np.array_equal(t.detach()[:, j].cpu().numpy().view(np.uint32), st[f].view(np.uint32)), "state %d" % f
    kept = [s.clone() for s in seeds]
    torch.autograd.backward(out, seeds)
    for g, x, t, s, k in zip(lay.groups, leaves, out, seeds, kept):
        assert torch.equal(s, k)                              # incoming gradients are left alone
        for j, f in enumerate(g):
            assert np.array_equal(x.grad[:, j].cpu().numpy().view(np.uint32), want[f].view(np.uint32)), "grad %d" % f
            assert np.array_equal(t.detach()[:, j].cpu().numpy().view(np.uint32), fields[f].view(np.uint32)), f


def test_tanh_of_every_float(P):
    """The chain run's tanh (packed, with a quotient of its own) equals the section kernel's (one IEEE
    division) for all 2^32 floats, NaN for NaN."""
    n = 1 << 24
    sec = synth.Section("tanh", (0, 1), frozenset([0]), frozenset([1]))
    S, aos, soa = P.Schema([0, 0]), P.Layout.aos(2), P.Layout.soa(2)
    from paper_1407_4859_gb300._lib import adha_section
    secs = (adha_section * 1)(P.c_section(sec))
    saved = torch.empty(n, dtype=torch.float32, device="cuda")
    base = torch.arange(n, dtype=torch.int64, device="cuda")
    for k in range(256):
        x = (base + (k << 24)).to(torch.int32).view(torch.float32)
        both = torch.stack([x, torch.zeros_like(x)], dim=1)
        P.adha_run_section(S, n, aos, [both], secs[0])
        z = torch.zeros_like(x)
        P.adha_chain_forward(S, n, soa, [x, z], secs, saved)
        want, got = both[:, 1].view(torch.int32), z.view(torch.int32)
        same = (want == got) | (torch.isnan(both[:, 1]) & torch.isnan(z))
        assert bool(same.all()), (k, x[~same][:4].tolist(), both[:, 1][~same][:4].tolist(), z[~same][:4].tolist())
