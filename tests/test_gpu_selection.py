"""The class-wise top-k at the sizes where its shape changes: one CTA up to 4096 items, a cluster with 4 and with 16
items per thread up to 81920, the larger-problem kernels above; 2048 to 128 buckets per class (G), ties that leave
more than 128 items in one bucket, and budgets of nothing and everything."""

import numpy as np
import pytest
import torch

from oracle import metok_oracle as O
from paper_2506_02850_b200 import binding as B

pytestmark = pytest.mark.gpu

SIZES = [1, 31, 128, 129, 1023, 4095, 4096, 4097, 4100, 32767, 32768, 32769, 81919, 81920, 81921]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("G", [1, 2, 5, 33, 64])
def test_class_topk_at_its_edges(n, G):
    rng = np.random.default_rng(n * 100 + G)
    vis_start, Lt = int(rng.integers(0, 40)), int(rng.integers(1, 40))
    groups = rng.integers(0, G, n).astype(np.int32)
    for kind in ("spread", "ties", "two"):
        s = np.exp(rng.standard_normal(n)).astype(np.float32) / n
        if kind == "ties":
            s = np.round(s * n * 4).astype(np.float32) / 4              # a few dozen distinct values
        elif kind == "two":
            s = (rng.random(n) < 0.5).astype(np.float32)                # two
        pop = np.bincount(groups, minlength=G)
        budgets = [int(rng.integers(0, p + 1)) for p in pop]
        budgets[0] = int(pop[0])                                        # a class that keeps everything
        budgets[-1] = 0 if G > 2 else max(1, int(pop[-1]) // 3)         # and one that keeps nothing
        want = O.weighted_topk(s.astype(np.float64), groups, budgets, vis_start + n + Lt, vis_start)
        got = B.metok_prune_by_scores(torch.from_numpy(s).cuda(), None, vis_start + n + Lt, vis_start,
                                      torch.from_numpy(groups).cuda(), budgets)
        torch.cuda.synchronize()
        m = int(got["S_out"].item())
        assert m == want["S_out"]
        assert np.array_equal(got["keep_idx"][:m].cpu().numpy(), want["keep_idx"]), kind


@pytest.mark.parametrize("T,N,k,lens", [
    (40, 100, 3, [1, 38, 1]),        # one CTA per event, four items per thread
    (50, 161, 40, [11] + [1] * 39),  # more events than fit as clusters: eight items per thread
    (60, 99, 2, [59, 1]),            # a cluster
    (340, 100, 2, [339, 1]),         # a cluster with sixteen items per thread
    (840, 100, 2, [839, 1]),         # beyond it
])
def test_event_topk_at_its_edges(T, N, k, lens):
    rng = np.random.default_rng(T)
    d = 16
    V = rng.standard_normal((T, N, d)).astype(np.float32)
    t = rng.standard_normal(d).astype(np.float32)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    got = B.metok_compress_vision(torch.from_numpy(V).cuda(), torch.from_numpy(offs).cuda(), torch.from_numpy(t).cuda(),
                                  B.vision_params(0.5, 0.01, 0.01))
    torch.cuda.synchronize()
    n_out = int(got["n_out"].item())
    src = got["out_src"][:n_out].cpu().numpy()
    score = got["token_score"].cpu().numpy()
    want = []
    for e in range(k):                                                  # the best of the kernel's own scores, lower index on ties
        lo, hi = int(offs[e]) * N, int(offs[e + 1]) * N
        b = max(1, int(np.ceil(0.01 * (hi - lo) - 1e-9)))
        want += sorted(lo + np.argsort(-score[lo:hi], kind="stable")[:b])
    assert np.array_equal(src, np.asarray(want))
    assign = got["assign"].cpu().numpy()
    assert np.array_equal(assign[src], np.arange(n_out))
    members = got["out_members"][:n_out].cpu().numpy()
    assert np.array_equal(np.bincount(assign, minlength=n_out), members) and int(members.sum()) == T * N
