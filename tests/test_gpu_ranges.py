"""Sizes at which the kernels' partitions and variants change: edges of tiles, remainders, the ends of their ranges."""
import numpy as np
import pytest

import locks_synth
import oracle
from common import t2np

pytestmark = pytest.mark.gpu


# Every problem's pages are sliced by its own length: requests of one token, a page less one, and one long request in the
# same row; 4, 16 and 3 heads per KV head; pages of several 16-token tiles that end inside a tile.  The bound is that of
# the attention tests: bf16 P and output.
@pytest.mark.parametrize("lens,Hq,Hkv,B,layout", [([16 * 450 + 3, 1, 33, 16 * 7], 8, 2, 16, "HND"), ([15, 16 * 700], 32, 2, 16, "NHD"),
                                                  ([5000, 16 * 400, 17] * 20, 6, 2, 16, "HND"), ([64 * 130 + 33, 64], 8, 2, 64, "HND"),
                                                  ([32 * 230, 49], 16, 1, 32, "NHD"), ([16 * 385], 4, 1, 16, "HND")])
def test_dense_attention_ragged_rows(lens, Hq, Hkv, B, layout):
    from gpu_util import GpuCase
    gc = GpuCase(locks_synth.Workload("ragged", lens, Hq=Hq, Hkv=Hkv, B=B, budget=16 * B, seed=len(lens) + Hq, layout=layout,
                                      tail_fill=float("nan")))
    out, lse = gc.gpu_attend()
    oout, olse = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm)
    assert np.abs(out - oout).max() <= 2e-2
    assert np.abs(lse - olse).max() <= 1e-3 * max(1.0, np.abs(olse).max() / 10)
    assert gc.status() == 0
