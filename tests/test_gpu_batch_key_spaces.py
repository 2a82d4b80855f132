"""Batches over key spaces of millions, where a group's slice of the expanded
weights is longer than 2^31 bytes: every user's top-K against FP64 sums of the
same weights."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import check_topk  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _batch(fields, vocab, B, n_ads=3_000, d=64, k=40):
    """Returns the users served by the batched scan, of B; checks all."""
    n_keys = fields * vocab
    rng = np.random.default_rng(fields + B)
    key = rng.integers(0, vocab, (n_ads, fields)) + vocab * np.arange(fields)
    key[0, -1] = n_keys - 1
    key[:, 0] = rng.integers(0, 5, n_ads)  # an uneven number of ads per key
    short = rng.random(n_ads) < 0.2        # ads with fewer keys: padding
    has = np.ones((n_ads, fields), bool)
    has[short, 1:3] = False
    pa, f = np.nonzero(has)
    pk = key[pa, f].astype(np.uint32)
    pa = pa.astype(np.uint32)
    emb = (rng.standard_normal((n_ads, d)) / 8).astype(np.float32)
    h = (rng.standard_normal((B, d)) / 8).astype(np.float32)
    users = rng.integers(0, 50, (B, 1)).astype(np.uint32)
    ix = ebr.build_index(n_ads, n_keys, pk, pa, emb, dtype="bf16")
    cross = ebr.cross_create([50], [vocab] * fields, [(0, j) for j in range(fields)],
                             (rng.standard_normal(1 << 16) * 0.3).astype(np.float32),
                             hashed=True, hash_bits=16)
    w, row = [], torch.empty((1, n_keys), device=DEV)
    at = torch.from_numpy(pk.astype(np.int64)).to(DEV)
    ud = torch.from_numpy(users.view(np.int32)).to(DEV)
    for b in range(B):
        ebr.expand_query(cross, ud[b:b + 1], row)
        w.append(row[0, at].cpu().numpy().astype(np.float64))
    del row
    hd = torch.from_numpy(h).to(DEV)
    ids = torch.empty((B, k), dtype=torch.int32, device=DEV)
    sc = torch.empty((B, k), device=DEV)
    before = ix.profile_read().batched
    ebr.score_topk(ix, cross, [ebr.Query(h_u=hd[b], k=k, user_vals=ud[b]) for b in range(B)],
                   ids, sc)
    torch.cuda.synchronize()
    ids, sc = ids.cpu().numpy().view(np.uint32), sc.cpu().numpy()
    e64 = emb.astype(np.float64)
    for b in range(B):
        wide, mag = np.zeros(n_ads), np.zeros(n_ads)
        np.add.at(wide, pa, w[b])
        np.add.at(mag, pa, np.abs(w[b]))
        ref = e64 @ h[b].astype(np.float64) + wide
        tol = oracle.tolerance(ref, np.abs(e64) @ np.abs(h[b]).astype(np.float64) + mag, 1e-5)
        check_topk(ids[b], sc[b], ref, tol, k)
    return ix.profile_read().batched - before


@pytest.mark.parametrize("vocab", [932_000, 1_000_000])  # 2.15e9 and 2.3e9 bytes a slice
def test_slices_longer_than_a_2d_memsets_pitch(vocab):
    assert _batch(9, vocab, 70) == 70


@pytest.mark.parametrize("B,batched", [(70, 70), (256, 0)])
def test_the_largest_weights_of_a_batch(B, batched):
    # 17 M keys (no forward table): 128 users' weights are 8.7 GB, 256 users' over the bound
    assert _batch(17, 1_000_000, B) == batched
