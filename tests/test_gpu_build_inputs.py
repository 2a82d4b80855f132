"""Where the posting arrays of an index build may lie: host or device memory, on
any byte."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off_key,off_ad", [(0, 0), (1, 0), (0, 2), (3, 1)])
def test_postings_on_any_byte_of_device_memory(off_key, off_ad):
    n_ads, n_keys, nnz = 700, 50, 5_000
    rng = np.random.default_rng(1)
    pk = rng.integers(0, n_keys, nnz).astype(np.uint32)
    pa = rng.integers(0, n_ads, nnz).astype(np.uint32)

    def put(a, off):
        buf = torch.zeros(4 * nnz + 8, dtype=torch.uint8, device="cuda:0")
        buf[off:off + 4 * nnz] = torch.from_numpy(a.view(np.uint8)).to(buf.device)
        return buf

    bk, ba = put(pk, off_key), put(pa, off_ad)
    emb = np.zeros((n_ads, 4), np.float32)
    torch.cuda.synchronize()
    d = ebr.IndexDesc(n_ads, n_keys, nnz, bk.data_ptr() + off_key, ba.data_ptr() + off_ad, 4,
                      ebr.F32, emb.ctypes.data, 0, 0, None)
    h = ctypes.c_void_p()
    assert ebr.ebr_build_index(ctypes.byref(d), ctypes.byref(h)) == ebr.EBR_OK
    ix = ebr.Index(h)
    ref = oracle.build_index(n_keys, n_ads, pk, pa)
    for g in range(9):
        for got, want in zip(ix.export(g), (ref["keys"][g], ref["header"][g], ref["values"][g])):
            np.testing.assert_array_equal(got, want, err_msg="g=%d" % g)
