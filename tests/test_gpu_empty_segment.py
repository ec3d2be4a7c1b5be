"""A segment without sections hands the state and its gradients through, in buffers of its own."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4099])
@pytest.mark.parametrize("groups", [[[0, 1, 2]], [[0], [1], [2]]])
def test_segment_without_sections(groups, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    from paper_1407_4859_gb300.autograd import SegmentFn
    leaves = [torch.randn((n, len(g)), device="cuda").requires_grad_() for g in groups]
    out = SegmentFn.apply((P.Schema([0] * 3), n, P.Layout(groups), []), *[x * 2.0 for x in leaves])
    seeds = [torch.randn_like(x) for x in leaves]
    kept = [s.clone() for s in seeds]
    torch.autograd.backward(out, seeds)
    for x, s, k, o in zip(leaves, seeds, kept, out):
        assert torch.equal(o, x * 2.0)
        assert torch.equal(s, k)
        assert torch.equal(x.grad, 2.0 * k)
