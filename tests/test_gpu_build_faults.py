"""Failures inside the index build, made to happen by ebr_debug_build_index: an
error comes back, the context stays usable and the next build is right."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu


def _pairs(n_ads, n_keys, nnz, seed=0):
    rng = np.random.default_rng(seed)
    return (rng.integers(0, n_keys, nnz).astype(np.uint32),
            rng.integers(0, n_ads, nnz).astype(np.uint32))


@pytest.mark.parametrize("fault", [ebr.FAULT_SORT_PAIRS, ebr.FAULT_SORT_KEYS,
                                   ebr.FAULT_SORT_BLOCKS, 7])
@pytest.mark.parametrize("n_ads,n_keys,nnz", [(3_000, 5_000, 30_000), (70_000, 70_000, 400_000)])
def test_a_sort_that_gives_up_is_an_error(fault, n_ads, n_keys, nnz):
    pk, pa = _pairs(n_ads, n_keys, nnz)
    emb = np.zeros((n_ads, 4), np.float32)
    with pytest.raises(ebr.EbrError) as e:
        ebr.build_index(n_ads, n_keys, pk, pa, emb, debug_faults=fault)
    assert e.value.code == ebr.EBR_ETIMEDOUT
    torch.cuda.synchronize()
    ix = ebr.build_index(n_ads, n_keys, pk, pa, emb)
    ref = oracle.build_index(n_keys, n_ads, pk, pa)
    for g in range(9):
        for got, want in zip(ix.export(g), (ref["keys"][g], ref["header"][g], ref["values"][g])):
            np.testing.assert_array_equal(got, want, err_msg="g=%d" % g)


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8e4m3"])
def test_without_memory_for_the_forward_table_the_index_is_built_without(dtype):
    n_ads, n_keys, d, k = 20_001, 300, 64, 50
    pk, pa = _pairs(n_ads, n_keys, 10 * n_ads)
    rng = np.random.default_rng(1)
    emb = rng.standard_normal((n_ads, d)).astype(np.float32)
    h = rng.standard_normal(d).astype(np.float32)
    w = rng.standard_normal(n_keys).astype(np.float32)
    dev = torch.device("cuda:0")
    q = ebr.Query(h_u=torch.from_numpy(h).to(dev), k=k, q_w=torch.from_numpy(w).to(dev))
    pairs = np.unique(np.stack([pk, pa]), axis=1)
    wide = np.zeros(n_ads)
    np.add.at(wide, pairs[1], w[pairs[0]].astype(np.float64))
    ref = emb.astype(np.float64) @ h + wide
    for faults in (0, ebr.FAULT_FORWARD_MEM):
        ix = ebr.build_index(n_ads, n_keys, pk, pa, emb, dtype=dtype, debug_faults=faults)
        ids = torch.empty(k, dtype=torch.int32, device=dev)
        sc = torch.empty(k, device=dev)
        ebr.score_topk(ix, None, [q], ids, sc)
        got = ids.cpu().numpy()
        assert np.unique(got).size == k
        # 1e-5 of the products' sizes is far below the gap that a lost ad would leave
        np.testing.assert_allclose(sc.cpu().numpy(), np.sort(ref)[::-1][:k], atol=1e-3)
        np.testing.assert_allclose(sc.cpu().numpy(), ref[got], atol=1e-3)
