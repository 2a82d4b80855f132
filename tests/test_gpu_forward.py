"""The scan over the forward key table, and the block-wise scan that serves the
indexes without one, at the sizes where either can go wrong: every score and
the top-K against FP64 sums of the same terms (the HitMatch equation plus
Eq. 1), with the 1e-5 condition-scale tolerance of the parity tests; and
against Algorithm 2's key-major traversal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import check_scores, check_topk  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _inventory(n_ads, n_keys, most, even, d, seed):
    """Ads with `most` distinct keys each (even) or 0..most of them."""
    rng = np.random.default_rng(seed)
    cnt = np.full(n_ads, most) if even else rng.integers(0, most + 1, n_ads)
    cnt[n_ads // 2] = most
    cnt = np.minimum(cnt, n_keys)
    ad = np.repeat(np.arange(n_ads), cnt)
    start = rng.integers(0, n_keys, n_ads)
    step = np.concatenate([np.arange(c) for c in cnt]) if ad.size else np.zeros(0, np.int64)
    key = (start[ad] + step * max(1, n_keys // (most + 1))) % n_keys
    pairs = np.unique(np.stack([key, ad]), axis=1)
    p = rng.permutation(pairs.shape[1])
    emb = rng.standard_normal((n_ads, d)).astype(np.float32) / np.float32(np.sqrt(d))
    h = rng.standard_normal(d).astype(np.float32)
    w = rng.standard_normal(n_keys).astype(np.float32)
    w[rng.random(n_keys) < 0.1] *= np.float32(1e-6)  # terms of every class
    return pairs[0][p].astype(np.uint32), pairs[1][p].astype(np.uint32), emb, h, w


def _table(ix, emb, dtype):
    if dtype == "f32":
        return emb.astype(np.float64)
    codes, scale = ix.export_emb()
    if dtype == "bf16":
        return (codes.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    vals = np.array([oracle.fp8_e4m3_value(c) for c in range(256)], np.float64)
    return vals[codes] * scale.astype(np.float64)[:, None]


@pytest.mark.parametrize("n_ads,n_keys,most,even,d,dtype", [
    (1, 1, 1, True, 4, "f32"),
    (33, 50, 3, False, 8, "f32"),
    (257, 300, 17, False, 16, "f32"),
    (5_000, 65_535, 16, True, 32, "f32"),      # last key space of 16 bits
    (70_001, 65_536, 16, True, 64, "f32"),     # first of 24 bits; stages of several runs
    (40_000, 200_000, 24, False, 128, "f32"),  # two threads per row
    (9_000, 700, 40, True, 64, "f32"),         # ten quads per run
    (600, 900, 64, True, 64, "f32"),           # the most quads of a window
    (600, 900, 65, True, 64, "f32"),           # one more: no table, the block-wise scan
    (3_000, 400, 300, False, 64, "f32"),       # uneven counts: no table
    (300, 40, 5, False, 8, "bf16"),
    (70_003, 70_000, 33, False, 64, "bf16"),
    (20_001, 480, 32, True, 128, "bf16"),
    (1_000, 80, 9, False, 16, "fp8e4m3"),
    (70_002, 480, 32, True, 64, "fp8e4m3"),
    (20_003, 90_000, 12, False, 128, "fp8e4m3"),
])
def test_every_score_and_top_k(n_ads, n_keys, most, even, d, dtype):
    pk, pa, emb, h, w = _inventory(n_ads, n_keys, most, even, d, seed=n_ads + most)
    ix = ebr.build_index(n_ads, n_keys, pk, pa, emb, dtype=dtype)
    wide = np.zeros(n_ads)
    mag = np.zeros(n_ads)
    np.add.at(wide, pa, w[pk].astype(np.float64))
    np.add.at(mag, pa, np.abs(w[pk]).astype(np.float64))
    out = torch.empty(n_ads, device=DEV)
    q = dict(h_u=_dev(h), q_w=_dev(w))
    table = _table(ix, emb, dtype)
    ref = table @ h.astype(np.float64) + wide
    tol = oracle.tolerance(ref, np.abs(table) @ np.abs(h).astype(np.float64) + mag, 1e-5)
    ebr.score_all(ix, None, ebr.Query(k=1, **q), out)
    check_scores(out.cpu().numpy(), ref, tol, "every score")
    # the key-major traversal of the same query
    km = torch.empty(n_ads, device=DEV)
    ebr.score_all(ix, None, ebr.Query(k=1, flags=ebr.QF_KEY_MAJOR, **q), km)
    check_scores(km.cpu().numpy(), ref, tol, "key-major")
    # top-K (rescored in FP32), with and without a bitmap, K up to past the inventory
    ref = emb.astype(np.float64) @ h.astype(np.float64) + wide
    tol = oracle.tolerance(ref, np.abs(emb).astype(np.float64) @ np.abs(h).astype(np.float64) + mag,
                           1e-5)
    rng = np.random.default_rng(1)
    for k, frac in ((1, None), (min(n_ads, 700), None), (min(2000, n_ads + 5), 0.3)):
        mask = None if frac is None else rng.random(n_ads) < frac
        words = None
        if mask is not None:
            bits = np.zeros((n_ads + 63) // 64 * 64, bool)
            bits[:n_ads] = mask
            words = _dev(np.packbits(bits, bitorder="little").view(np.int64))
        ids = torch.empty(k, dtype=torch.int32, device=DEV)
        sc = torch.empty(k, device=DEV)
        ebr.score_topk(ix, None, [ebr.Query(k=k, filter=words, **q)], ids, sc)
        check_topk(ids.cpu().numpy().view(np.uint32), sc.cpu().numpy(), ref, tol, k, mask)


@pytest.mark.parametrize("dtype", ["bf16", "fp8e4m3"])
def test_user_vectors_of_any_scale(dtype):
    # the three 16-bit pieces of h_u: tiny, huge and widely spread entries
    n_ads, d = 3_000, 64
    pk, pa, emb, h, w = _inventory(n_ads, 60, 4, True, d, seed=3)
    ix = ebr.build_index(n_ads, 60, pk, pa, emb, dtype=dtype)
    table = _table(ix, emb, dtype)
    w[:] = 0
    out = torch.empty(n_ads, device=DEV)
    for scale in (1e-20, 1.0, 1e20):
        hs = (h * scale * 10.0 ** np.linspace(-6, 0, d)).astype(np.float32)
        ebr.score_all(ix, None, ebr.Query(h_u=_dev(hs), k=1, q_w=_dev(w)), out)
        ref = table @ hs.astype(np.float64)
        tol = 1e-5 * (np.abs(table) @ np.abs(hs).astype(np.float64))
        check_scores(out.cpu().numpy(), ref, tol, "scale %g" % scale)
    ebr.score_all(ix, None, ebr.Query(h_u=_dev(np.zeros(d, np.float32)), k=1, q_w=_dev(w)), out)
    assert not out.cpu().numpy().any()
