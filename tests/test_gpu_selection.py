"""The selection kernel of the three-launch step where its ways part: a cut in a bin of exactly and of more than 1024
blocks, scores below the histogram's range, units whose keys just fit and just do not fit into shared memory."""
import pytest
import torch

from paper_2609_26300_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("keys,X", [("spread", 1100), ("spread", 24576), ("spread", 24577), ("alike", 1027), ("alike", 1028),
                                    ("alike", 24577), ("far apart", 4000)])
@pytest.mark.parametrize("K", [4, 200])
def test_selected_ids_are_the_best_of_the_scores(keys, X, K):
    """Exact: the ids against a stable sort of the scores the kernel itself left behind."""
    g = torch.Generator("cuda").manual_seed(X)
    k, v = (torch.randn((X, 1, 16, 128), generator=g, device="cuda") for _ in range(2))
    q = torch.randn((1, 4, 128), generator=g, device="cuda")
    if keys == "alike":
        k.copy_(k[:1].clone().expand_as(k))
    elif keys == "far apart":   # block means far apart, keys of a block close together: e^l stays near e^(mean logit)
        k = 0.1 * k + 30.0 * torch.randn((X, 1, 1, 128), generator=g, device="cuda")
    ckv = binding.CompKV(4, 1, max_batch=1, max_blocks_per_seq=X, num_pages=X, block_size=16, kv_dtype=binding.CKV_F32,
                         sink_blocks=1, recent_blocks=2)   # fp32 pages: always append, scan, select, attention as launches
    table = torch.arange(X, dtype=torch.int32, device="cuda")[None].contiguous()
    lens = torch.tensor([16 * X - 3], dtype=torch.int32, device="cuda")
    ckv.stats_build(k, v, table, lens, 16 * X)
    ids, cnt = ckv.decode(q, k, v, table, lens, 16 * X, 16 * K)[2:4]
    S = ckv.copy_scores(1)[0, 0, :X]
    torch.cuda.synchronize()
    assert ckv.read_status() == 0
    ranked = S[1:X - 2]
    if keys == "alike":
        assert bool((ranked == ranked[0]).all())
    elif keys == "far apart":
        assert int((ranked < 2.0 ** -54).sum()) > 1024
    best = 1 + torch.sort(ranked, descending=True, stable=True).indices[:K - 3]
    want = sorted([0, X - 2, X - 1] + best.tolist())
    assert cnt.tolist() == [[K]] and ids[0, 0, :K].tolist() == want
