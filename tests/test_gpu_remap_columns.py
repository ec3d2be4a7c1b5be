"""GPU parity of the remap by columns, byte for byte against the oracle: each of its forms (structs to
arrays, narrow structs into several structs and back, arrays straight into structs in every batch
remainder, groups carried whole), structs staged with room, records too wide for 128 or 64 of them, dirty
source padding, and record counts around the chunk sizes and where each chunk size begins."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
F32, F64, I32, BF16 = range(4)

PAIRS = {
    "structs_to_arrays": ([F32] * 8 + [F64] * 4 + [I32] * 4, "aos", "soa"),
    "arrays_to_structs": ([F32] * 8 + [F64] * 4 + [I32] * 4, "soa", "aos"),
    "arrays_to_structs_15": ([F32] * 15 + [F64] * 7, "soa", [list(range(9, 22)), list(range(9))]),
    "narrow_structs": ([F32] * 9, "aos", [[0, 1, 2], [3, 4, 5, 7], [6], [8]]),
    "narrow_structs_back": ([F32] * 9, [[0, 1, 2], [3, 4, 5, 7], [6], [8]], "aos"),
    "padding_and_bf16": ([BF16, F64, BF16, F32, BF16, BF16], "aos", [[1, 0], [2], [5, 3], [4]]),
    "padding_back": ([BF16, F64, BF16, F32, BF16, BF16], [[1, 0], [2], [5, 3], [4]], "aos"),
    "room_64": ([F32] * 16, "aos", "soa"),
    "room_32_both": ([F32] * 8, "aos", [[7, 6, 5, 4, 3, 2, 1, 0]]),
    "carried": ([F32] * 6 + [BF16], [[0, 1, 2], [3], [4, 5], [6]], [[4, 5], [2, 1, 0], [3], [6]]),
    "wide": ([F64] * 64, "aos", "soa"),
    "wide_back": ([F64] * 64, "soa", "aos"),
    "two_byte_arrays": ([BF16] * 5 + [F32], "soa", "aos"),
    "one_field": ([BF16], "aos", "soa"),
}


def _groups(x, F):
    return [list(range(F))] if x == "aos" else [[f] for f in range(F)] if x == "soa" else x


@pytest.mark.parametrize("pair", sorted(PAIRS))
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 20011, 50021, 160007, 311301])
def test_bytes_equal_oracle(pair, n):
    from paper_1407_4859_gb300 import build
    build.build()
    import paper_1407_4859_gb300 as P
    dtypes, src, dst = PAIRS[pair]
    if len(dtypes) == 64 and n > 50021:
        n = 50021 + n % 64
    src, dst = _groups(src, len(dtypes)), _groups(dst, len(dtypes))
    S = P.Schema(dtypes)
    rng = np.random.default_rng(n)
    strides, _ = P.adha_layout_strides(S, P.Layout(src))
    host = [rng.integers(0, 256, n * st, dtype=np.uint8) for st in strides]   # padding bytes are dirty too
    want = oracle.remap(n, dtypes, src, host, dst)
    room = [torch.full((w.size + 64,), 0xAB, dtype=torch.uint8, device="cuda") for w in want]
    P.adha_remap(S, n, P.Layout(src), [torch.from_numpy(h).cuda() for h in host], P.Layout(dst), [r[:w.size] for r, w in zip(room, want)])
    torch.cuda.synchronize()
    for g, (r, w) in enumerate(zip(room, want)):
        got = r.cpu().numpy()
        assert np.array_equal(got[:w.size], w), "group %d" % g
        assert (got[w.size:] == 0xAB).all(), "group %d: bytes after its end" % g
