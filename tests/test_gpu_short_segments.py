"""GPU parity of short segments on structs, around where they change between chain runs and single sections:
forward state, gradient and restored state against the oracle, bit for bit; the rule itself on the CPU."""
import numpy as np
import pytest
import torch

import oracle
import synth


def _sections(rng, F, count):
    out = []
    for k in range(count):
        x, y, z = (int(f) for f in rng.choice(F, 3))
        if k % 3 == 0:
            out.append(synth.Section("mul", (x, y, z), frozenset([x, y]), frozenset([z])))
        elif k % 3 == 1:
            out.append(synth.Section("axpb", (x, z), frozenset([x]), frozenset([z]), params=(0.75, -0.5)))
        else:
            out.append(synth.Section("tanh", (x, z), frozenset([x]), frozenset([z])))
    return out


def test_which_segments_run_one_by_one():
    from paper_1407_4859_gb300.api import Layout
    from paper_1407_4859_gb300.autograd import _faster_one_by_one as single
    rng = np.random.default_rng(1)
    for F in (24, 63, 64):
        aos, soa = Layout([list(range(F))]), Layout([[f] for f in range(F)])
        assert single(1 << 22, aos, _sections(rng, F, 1))
        assert not single(1 << 12, aos, _sections(rng, F, 1))      # launches cost more
        assert not single(1 << 22, aos, _sections(rng, F, 8))
        assert not single(1 << 22, soa, _sections(rng, F, 1))      # arrays: a chain run moves what it touches
    assert not single(1 << 22, Layout([[0, 1], [2]]), [])


@pytest.mark.gpu
@pytest.mark.parametrize("F,width,count", [(64, 64, 1), (64, 64, 2), (64, 64, 5), (63, 63, 4), (64, 8, 3), (35, 35, 2), (35, 7, 2)])
@pytest.mark.parametrize("n", [1 << 19, (1 << 20) + 5])
def test_short_segments_equal_oracle(F, width, count, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    from paper_1407_4859_gb300.autograd import SegmentFn
    rng = np.random.default_rng(F + count)
    secs = _sections(rng, F, count)
    lay = P.Layout([list(range(b, min(b + width, F))) for b in range(0, F, width)])
    gen = torch.Generator(device="cuda").manual_seed(3)
    leaves = [torch.randn((n, len(g)), device="cuda", generator=gen).requires_grad_() for g in lay.groups]
    out = SegmentFn.apply((P.Schema([0] * F), n, lay, secs), *[x * 1.0 for x in leaves])
    c = [float(np.float32(v)) for v in rng.uniform(-1, 1, F)]
    seeds = [torch.tensor([c[f] for f in g], device="cuda").expand(n, len(g)).contiguous() for g in lay.groups]
    pick = np.unique(np.concatenate([np.arange(200), n - 1 - np.arange(200), rng.integers(0, n, 2000)]))
    at = torch.from_numpy(pick).cuda()
    fields = [np.ascontiguousarray(np.concatenate([x.detach()[at].cpu().numpy() for x in leaves], axis=1)[:, f]) for f in range(F)]
    state = [a.copy() for a in fields]
    want = oracle.chain_grad(secs, state, c)
    after = torch.cat([t.detach()[at] for t in out], dim=1).cpu().numpy()
    torch.autograd.backward(out, seeds)
    grad = torch.cat([x.grad[at] for x in leaves], dim=1).cpu().numpy()
    for f in range(F):
        assert np.array_equal(after[:, f].copy().view(np.uint32), state[f].view(np.uint32)), "state %d" % f
        assert np.array_equal(grad[:, f].copy().view(np.uint32), want[f].view(np.uint32)), "gradient %d" % f
    for x, t in zip(leaves, out):
        assert torch.equal(t.detach(), x.detach())                # handed back as it was
