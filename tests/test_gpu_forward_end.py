"""The end of the forward scan: every warp counts and writes its share of its
CTA's candidates, in every call.  Scores that rise with the ad keep the
buffers full to the end; the scores are exact, so each call must give the same
ids and scores."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,k", [(12_289, 1), (60_000, 300), (200_000, 1024)])
def test_no_candidate_is_lost_at_the_end(n, k):
    emb = torch.zeros((n, 4), device=DEV)
    emb[:, 1] = torch.arange(n, device=DEV) - n / 2
    h = torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV)
    want = torch.arange(n - 1, n - 1 - k, -1, dtype=torch.int32, device=DEV)
    none = np.zeros(0, np.uint32)
    ix = ebr.build_index(n, 4, none, none, emb)
    q = ebr.Query(h_u=h, k=k, q_w=torch.zeros(4, device=DEV))
    ids = torch.empty((2, 300, k), dtype=torch.int32, device=DEV)
    sc = torch.empty((2, 300, k), device=DEV)
    for i in range(300):
        ebr.score_topk(ix, None, [q], ids[0, i], sc[0, i])
        ebr.scan_topk_noalloc(emb, h, None, None, k, ids[1, i], sc[1, i])
    assert bool((ids == want).all())
    assert bool((sc == emb[:, 1][want.long()]).all())
