"""The inner products of quantised tables in the forward scan (tensor pipe) are
no further from FP64 than the FP32 multiply-adds of the block-wise scan."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("decades", [0, 5])  # of the user vector, first element to last
@pytest.mark.parametrize("dtype,d", [("bf16", 8), ("bf16", 16), ("bf16", 32), ("bf16", 64),
                                     ("bf16", 128), ("fp8e4m3", 16), ("fp8e4m3", 32),
                                     ("fp8e4m3", 64), ("fp8e4m3", 128)])
def test_error_is_no_larger_than_that_of_fp32_multiply_adds(dtype, d, decades):
    n = 100_000
    rng = np.random.default_rng(d)
    emb = (rng.standard_normal((n, d)) / np.sqrt(d)).astype(np.float32)
    pk = rng.integers(0, 300, 4 * n).astype(np.uint32)
    pa = np.repeat(np.arange(n), 4).astype(np.uint32)
    rms = []
    for faults in (0, ebr.FAULT_FORWARD_MEM):
        ix = ebr.build_index(n, 300, pk, pa, emb, dtype=dtype, debug_faults=faults)
        codes, scale = ix.export_emb()
        if dtype == "bf16":
            table = (codes.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
        else:
            table = oracle.fp8_e4m3_value(np.arange(256))[codes] * scale[:, None].astype(np.float64)
        table = torch.from_numpy(table).to(DEV)
        sq = 0.0
        for seed in range(6):
            h = np.random.default_rng(seed).standard_normal(d) * np.logspace(0, -decades, d)
            h = torch.from_numpy(h.astype(np.float32)).to(DEV)
            out = torch.empty(n, device=DEV)
            ebr.score_all(ix, None, ebr.Query(h_u=h, q_w=torch.zeros(300, device=DEV), k=1), out)
            mag = table.abs() @ h.double().abs()
            sq += float((((out.double() - table @ h.double()) / mag) ** 2).mean())
        rms.append(np.sqrt(sq / 6))
    assert rms[0] <= rms[1], rms
