"""The ray budget's radix select where it can go wrong: path counts around its
steps and beyond its most list tiles, scores that are all equal, special values
and neighbours in their last bits, budgets of nothing, one, all but one and more
than all, and lists out of order or with ids out of range (which are left out).
The reference ranks in numpy: score descending (non-positive scores and NaN as
0), then by place in the list."""
import numpy as np
import pytest

import scenes
import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


def _ref(lst, score, budget):
    lst = lst[lst < score.shape[0]]
    s = score[lst]
    key = np.where(s > 0, s, np.float32(0)).view(np.uint32)
    return np.sort(lst[np.argsort(~key, kind="stable")[:budget]])


def _scores(rng, n):
    special = np.array([np.nan, np.inf, -np.inf, 0.0, -0.0, 1e-45, 1e-38, 3.4e38, 1.0, -1.0], np.float32)
    yield np.full(n, 0.5, np.float32)
    yield special[rng.integers(0, special.size, n)]
    yield (np.float32(1.0).view(np.uint32) + rng.integers(0, 700, n).astype(np.uint32)).view(np.float32)
    yield np.exp(4.0 * rng.standard_normal(n)).astype(np.float32)


@pytest.mark.parametrize("n", [1, 31, 257, 2047, 2049, 6145, 2_200_013])
def test_budget_select_matches_ranking(n):
    import torch
    h = gu.lib_scene(scenes.tiny_box(n_paths=n))
    rng = np.random.default_rng(n)
    out = torch.zeros(n, dtype=torch.int32, device="cuda")
    out_cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    ids = np.arange(n, dtype=np.uint32)
    for k, score in enumerate(_scores(rng, n)):
        lst = ids if k % 2 else np.sort(rng.choice(ids, size=max(1, n // 2), replace=False))
        if k == 3:
            lst = rng.permutation(lst)
            lst[:: 7] = n + 3
        d_list = torch.zeros(n, dtype=torch.int32, device="cuda")
        d_list[: lst.size] = torch.as_tensor(lst.view(np.int32), device="cuda")
        d_cnt = torch.tensor([lst.size], dtype=torch.int32, device="cuda")
        d_score = torch.as_tensor(score, device="cuda")
        for budget in sorted({0, 1, lst.size // 3, lst.size - 1, lst.size, lst.size + 5}):
            pv.pv_budget_list(h, d_list, d_cnt, d_score, budget, out, out_cnt)
            got = out[: int(out_cnt.item())].cpu().numpy().view(np.uint32)
            np.testing.assert_array_equal(got, _ref(lst, score, budget), err_msg=f"scores {k}, budget {budget}")
    assert pv.pv_read_device_status(h) == 0
    pv.pv_destroy_scene(h)
