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
