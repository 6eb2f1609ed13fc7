"""Rows of B (and C) 4 GB and more apart (GPU): every item that gathers B keeps the distance in 64 bits."""
import numpy as np
import pytest

import synth
from parity import check_result

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2606_22482_gb300 as ns  # noqa: E402
from nsutil import to_dev, tune_from  # noqa: E402

DEV = torch.device("cuda", 0)
FAR = (1 << 32) + 32  # bytes between rows: 32 where only 32 bits are kept


def matrix(m, n):
    """Rows with every column in the first windows of 16, with one in the later ones."""
    rng = np.random.default_rng(1)
    row, col = np.nonzero(np.ones((m, n), bool))
    keep = (row < m // 2) | (col == row % n)
    row, col = row[keep], col[keep]
    return synth.csr_from_coo(m, n, row, col.astype(np.int32), rng.uniform(-1, 1, row.size).astype(np.float32))


@pytest.mark.parametrize("K,dtype,kw", [
    (40, ns.NS_F32, dict()), (40, ns.NS_BF16, dict()), (128, ns.NS_BF16, dict(l2_hints=2)),
    (512, ns.NS_F32, dict()), (512, ns.NS_BF16, dict(chunk_nnz=2)),
    (40, ns.NS_F32, dict(tau_tile=20)), (40, ns.NS_BF16, dict(tau_tile=20)),           # dense windows and chunks
    (200, ns.NS_F32, dict(tau_tile=20, absorb_cap=0)), (200, ns.NS_BF16, dict(tau_tile=20, absorb_cap=0)),
    (264, ns.NS_F32, dict(tau_tile=20)), (264, ns.NS_BF16, dict(tau_tile=20))])
def test_far_rows_of_b(K, dtype, kw):
    A = matrix(96, 3)
    bf16 = dtype == ns.NS_BF16
    B = synth.dense_b(3, K, seed=2)
    h = synth.bf16_bits(B) if bf16 else B
    flat = torch.empty(2 * FAR + 4 * K, dtype=torch.uint8, device=DEV).view(torch.bfloat16 if bf16 else torch.float32)
    Bd = flat.as_strided((3, K), (FAR // (2 if bf16 else 4), 1))
    Bd.copy_(torch.from_numpy(h.view(np.int16)).to(DEV).view(torch.bfloat16) if bf16 else torch.from_numpy(h).to(DEV))
    C = torch.full((96, K), float("nan"), device=DEV)
    with ns.spmm_plan(to_dev(A, DEV), K, dtype, tune_from(ns, **kw)) as p:
        assert (p.stats()["n_dtiles"] > 0) == ("tau_tile" in kw)
        p.execute(Bd, C)
        torch.cuda.synchronize()
    tiles = bf16 and "tau_tile" in kw
    check_result(C.cpu().numpy(), A, h, b_bf16=bf16, bf16_tiles=tiles, tol=2e-2 if tiles else 1e-5)


@pytest.mark.parametrize("kw", [dict(), dict(tau_tile=20)])
def test_far_rows_of_c(kw):
    A = synth.csr_from_coo(3, 96, *(lambda M: (M["colidx"], np.repeat(np.arange(96), np.diff(M["rowptr"])).astype(np.int32),
                                              M["vals"]))(matrix(96, 3)))
    B = synth.dense_b(96, 40, seed=3)
    C = torch.empty(2 * FAR + 160, dtype=torch.uint8, device=DEV).view(torch.float32).as_strided((3, 40), (FAR // 4, 1))
    C.fill_(float("nan"))
    with ns.spmm_plan(to_dev(A, DEV), 40, ns.NS_F32, tune_from(ns, **kw)) as p:
        p.execute(torch.from_numpy(B).to(DEV), C)
        torch.cuda.synchronize()
    check_result(C.cpu().numpy(), A, B)
