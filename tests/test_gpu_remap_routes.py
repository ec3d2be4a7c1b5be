"""GPU parity of the default remap on pairs of layouts around the limits of its rules (the element schedule or by
columns, records per chunk, waves), with as many records as the rules ask for: every byte against the oracle at both
ends and around 2000 places in between, padding included, and back again to the source's bytes."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
SIZE = {"f": 4, "d": 8, "h": 2}
CODE = {"f": 0, "d": 1, "h": 3}


def _groups(F, width):
    return [list(range(k, min(k + width, F))) for k in range(0, F, width)]


@pytest.mark.parametrize("types,width,mb", [
    ("hh", 1, 31), ("hhh", 1, 141), ("hhf", 1, 141), ("fhhfh", 1, 201), ("d" * 40, 1, 81), ("f" * 56, 1, 81), ("f" * 64, 1, 81),
    ("f" * 24, 8, 121), ("f" * 24, 4, 119), ("d" * 24, 8, 121), ("f" * 64, 32, 121), ("fd" * 24, 24, 121), ("d" * 64, 32, 41),
    ("fdh" * 12, 5, 121), ("f" * 8, 4, 61), ("fhf" * 10, 6, 61), ("f" * 24, 6, 601),
])
def test_remap_there_and_back(types, width, mb):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    F = len(types)
    dtypes = [CODE[t] for t in types]
    S, aos, split = P.Schema(dtypes), P.Layout.aos(F), P.Layout(_groups(F, width))
    n = mb * 1000000 // sum(SIZE[t] for t in types) + 5
    (stride,), _ = P.adha_layout_strides(S, aos)
    strides, _ = P.adha_layout_strides(S, split)
    gen = torch.Generator(device="cuda").manual_seed(F)
    parts = [torch.randint(0, 256, (n * s,), dtype=torch.uint8, device="cuda", generator=gen) for s in strides]
    there = torch.full((n * stride,), 0xA5, dtype=torch.uint8, device="cuda")
    P.adha_remap(S, n, split, parts, aos, [there])
    rng = np.random.default_rng(F)
    at = torch.from_numpy(np.unique(np.concatenate([np.arange(300), n - 1 - np.arange(300), rng.integers(0, n, 2000)]))).cuda()

    def records(buf, s):
        return buf.view(n, s)[at].cpu().numpy().reshape(-1)

    some = [records(b, s) for b, s in zip(parts, strides)]
    want = oracle.remap(len(at), dtypes, split.groups, some, aos.groups)
    assert np.array_equal(records(there, stride), want[0])
    back = [torch.full_like(b, 0xA5) for b in parts]
    P.adha_remap(S, n, aos, [there], split, back)
    want = oracle.remap(len(at), dtypes, aos.groups, want, split.groups)
    for b, s, w in zip(back, strides, want):
        assert np.array_equal(records(b, s), w)
    again = torch.full_like(there, 0x5A)
    P.adha_remap(S, n, split, back, aos, [again])
    assert torch.equal(again, there)
