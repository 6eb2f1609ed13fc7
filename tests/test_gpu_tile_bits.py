"""A plan's values keep their bits (GPU): NaNs of every kind in dense tiles and in the residual, the
pattern of all ones and the one beside it among them, in windows that hold all of A and in selections."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2606_22482_gb300 as ns  # noqa: E402
from nsutil import compare_plan, oracle_tune, to_dev, tune_from  # noqa: E402

DEV = torch.device("cuda", 0)
BITS = np.array([0xFFFFFFFF, 0xFFFFFFFE, 0xFFFFFFFD, 0x7FFFFFFF, 0x7FC00000, 0x7F800001, 0xFF800000, 0x80000000, 0,
                 1, 0x3F800000], np.uint32)


@pytest.mark.parametrize("form", [dict(), dict(tau_col=1), dict(tau_row=3), dict(reorder=2), dict(col_order=1)])
@pytest.mark.parametrize("TM,TK", [(16, 16), (64, 32)])
@pytest.mark.parametrize("K", [32, 264])
def test_values_keep_their_bits(form, TM, TK, K):
    if TM * K > 16384:
        pytest.skip("dense tiles need TM * K <= 16384")
    rng = np.random.default_rng(TM + K)
    m = 500
    rows = np.repeat(np.arange(m), rng.integers(0, 10, m))
    cols = np.clip(rows // 16 * 16 + rng.integers(0, 24, rows.size), 0, m - 1)
    key = np.unique(rows * m + cols)
    A = synth.csr_from_coo(m, m, key // m, (key % m).astype(np.int32), rng.choice(BITS, key.size).view(np.float32))
    tune = tune_from(ns, tau_tile=TM + 4, TM=TM, TK=TK, **form)
    with ns.spmm_plan(to_dev(A, DEV), K, ns.NS_F32, tune) as p:
        assert p.stats()["n_dtiles"] > 0
        compare_plan(p, oracle.plan(A, K, **oracle_tune(tune)), A, tune)
