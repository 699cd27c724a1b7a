"""Edges of the kernels chosen by shape: tile remainders, the smallest and largest of a range, empty users, bad ids -
against the fp64 oracle, through the C ABI.  Tolerances as in the parity tests of the same paths."""
import numpy as np
import pytest
import torch

from oracle import lime_oracle as O
from paper_2510_18239_b200 import synth
from tests import lime_helpers as Hh

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _lib():
    from paper_2510_18239_b200 import binding
    return binding


@pytest.mark.parametrize("d,ell", [(32, 8), (32, 64), (64, 16), (128, 32), (256, 32), (256, 64)])
@pytest.mark.parametrize("counts,by_id", [([1], True), ([15, 16, 17], False), ([0, 5, 0, 33, 1, 0], True), ([3] * 70 + [0] * 40 + [400], True)])
def test_score_lists_by_warp(d, ell, counts, by_id):
    """The warp-level scorer: lists around its 16-slot step, many users inside one step, users without candidates, ids
    outside the corpus."""
    Bd = _lib()
    dtype, corpus, B, total = synth.BF16, 500, len(counts), int(sum(counts))
    lime = Bd.Lime(d, max(1, d // 128), ell, 1, dtype=Bd.LIME_BF16, gated_mlp=False)
    off = O.lengths_to_offsets(np.asarray(counts))
    rows = corpus if by_id else total
    LS = synth.normal_storage(5, "ls", (B, ell, d), 1.0, dtype)
    T = synth.normal_storage(5, "t", (rows, d), 1.0, dtype)
    W = synth.to_storage(O.softmax_rows(np.random.default_rng(5).normal(size=(rows, ell))), dtype)
    ids = synth.uniform_ids(5, "ids", total, corpus) if by_id else np.arange(total, dtype=np.int32)
    if by_id:
        ids[total // 2], ids[-1] = -3, corpus
    flag = torch.full((1,), 2 ** 31 - 1, dtype=torch.int32, device="cuda")
    got = Hh.to_f64(lime.score_candidates(Bd.to_device(LS, dtype), Bd.to_device(W, dtype), Bd.to_device(T, dtype),
                                          cand_off=torch.from_numpy(off.astype(np.int32)).cuda(), total_cands=total,
                                          cand_ids=torch.from_numpy(ids).cuda() if by_id else None, dev_flag=flag))
    W64, T64, LS64 = (synth.storage_to_f64(x, dtype) for x in (W, T, LS))
    ok = (ids >= 0) & (ids < rows)
    want = np.zeros(total)
    for b in range(B):
        s = np.arange(off[b], off[b + 1])
        s = s[ok[s]]
        want[s] = O.score_candidates(W64[ids[s]], LS64[b], T64[ids[s]])
    assert np.abs(got - want).max() <= 1e-4 * max(1.0, np.abs(want).max())
    if by_id:
        assert np.all(got[~ok] == 0.0) and int(flag.item()) == total // 2
