"""The planner's dense-tile passes at the edges of their forms (GPU): window counts around one turn and
the limit of the single-block scans, plans with and without expanded tiles, windows that hold all of A
in CSR order and windows that hold a selection, more tiles in a window than shared memory ranks, and
values whose bits are those of the mark for an absent one.  Every plan is the oracle's bit for bit."""
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


def check(A, K, dtype, **kw):
    tune = tune_from(ns, **kw)
    with ns.spmm_plan(to_dev(A, DEV), K, dtype, tune) as p:
        assert p.stats()["n_dtiles"] > 0
        compare_plan(p, oracle.plan(A, K, b_bf16=dtype == ns.NS_BF16, **oracle_tune(tune)), A, tune)


def banded(m, seed):
    """Rows of 0 to 9 nonzeros near the diagonal, every third window of 16 rows left sparse."""
    rng = np.random.default_rng(seed)
    n = rng.integers(0, 10, m)
    n[(np.arange(m) // 16) % 3 == 1] //= 8
    rows = np.repeat(np.arange(m), n)
    cols = np.clip(rows // 16 * 16 + rng.integers(0, 24, rows.size), 0, m - 1)
    key = np.unique(rows * m + cols)
    return synth.csr_from_coo(m, m, key // m, (key % m).astype(np.int32),
                              rng.standard_normal(key.size).astype(np.float32))


@pytest.mark.parametrize("windows", [1, 1023, 1024, 1025, 8192, 8193])
@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_window_counts(windows, dtype):
    check(banded(16 * windows - 3, windows), 32, dtype, tau_tile=40, TM=16, TK=16, reorder=0)


@pytest.mark.parametrize("form", [dict(), dict(tau_col=1), dict(tau_row=3), dict(reorder=2), dict(absorb_cap=0)])
@pytest.mark.parametrize("TM,TK", [(16, 16), (32, 16), (64, 32)])
@pytest.mark.parametrize("K,dtype", [(40, ns.NS_F32), (264, ns.NS_F32), (40, ns.NS_BF16), (264, ns.NS_BF16)])
def test_forms(form, TM, TK, K, dtype):
    if TM * K > 16384:
        pytest.skip("dense tiles need TM * K <= 16384")
    check(banded(1500, TM + TK), K, dtype, tau_tile=TM + 4, TM=TM, TK=TK, **form)


@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_more_tiles_than_shared_ranks(dtype):
    rng = np.random.default_rng(5)
    n = 700_000
    cols = [np.sort(rng.choice(n, 30_000, replace=False)) for _ in range(20)]
    rows = np.repeat(np.arange(20), 30_000)
    A = synth.csr_from_coo(20, n, rows, np.concatenate(cols).astype(np.int32),
                           rng.standard_normal(rows.size).astype(np.float32))
    check(A, 32, dtype, tau_tile=17, TM=16, TK=16, reorder=0)


@pytest.mark.parametrize("K,dtype", [(32, ns.NS_F32), (264, ns.NS_F32), (32, ns.NS_BF16)])
def test_values_like_the_mark(K, dtype):
    A = banded(200, 9)
    at = np.nonzero(np.diff(A["rowptr"]) > 0)[0]
    row = int(at[at % 48 < 16][5])
    bits = A["vals"].view(np.uint32)
    bits[A["rowptr"][row]:A["rowptr"][row + 1]] = 0xFFFFFFFF
    B = torch.ones(200, K, device=DEV, dtype=torch.bfloat16 if dtype == ns.NS_BF16 else torch.float32)
    C = torch.zeros(200, K, device=DEV)
    with ns.spmm_plan(to_dev(A, DEV), K, dtype, tune_from(ns, tau_tile=20, TM=16, TK=16)) as p:
        assert p.stats()["n_dtiles"] > 0
        p.execute(B, C)
    nan = torch.isnan(C).cpu().numpy()
    assert nan[row].all()
    assert not np.delete(nan, row, axis=0).any()
