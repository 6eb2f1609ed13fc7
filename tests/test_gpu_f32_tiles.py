"""FP32 dense tiles on the 5th-generation tensor cores at the edges of their forms (GPU): every tile
shape, one and two feature blocks, ragged widths and windows, column slices, residual chunks beside
the windows, and rows of B that no column names."""
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
# products of three-piece operands keep six of nine terms: what is left out is below 2^-22 of |a||b|,
# and each piece's products are summed as FP32 within a tile of 32 columns
TOL = 1e-6


def product(A, B, **tune):
    K = B.shape[1]
    C = torch.full((A["m"], K), float("nan"), device=DEV)
    with ns.spmm_plan(to_dev(A, DEV), K, ns.NS_F32, tune_from(ns, **tune)) as p:
        p.execute(torch.from_numpy(B).to(DEV), C)
        torch.cuda.synchronize()
        st = p.stats()
    assert st["n_dtiles"] > 0
    return C.cpu().numpy(), st


@pytest.mark.parametrize("TM,TK", [(16, 16), (16, 32), (32, 16), (32, 32), (64, 16), (64, 32)])
@pytest.mark.parametrize("K", [8, 40, 128, 136, 256])
def test_shapes_and_widths(TM, TK, K):
    A = synth.block_sparse_csr(700 // 64 * 64 + 64, seed=TM + TK, band=2, p_random=0.05)
    A = synth.csr_from_coo(701, A["n"], *_rows(A, 701))      # a last window that is not full
    B = synth.dense_b(A["n"], K, seed=K)
    c, _ = product(A, B, tau_tile=TM * TK // 4, TM=TM, TK=TK)
    check_result(c, A, B, tol=TOL)


def _rows(A, m):
    keep = A["rowptr"][m]
    rows = np.repeat(np.arange(m), np.diff(A["rowptr"][:m + 1]))
    return rows, A["colidx"][:keep], A["vals"][:keep]


@pytest.mark.parametrize("kw", [dict(TN=64), dict(TN=72), dict(absorb_cap=0, chunk_nnz=16), dict(tau_row=3),
                                dict(chunk_nnz=1024, absorb_cap=0)])
def test_slices_and_residual_chunks(kw):
    A = synth.rmat_csr(11, 60000, seed=3)
    B = synth.dense_b(A["n"], 136, seed=4)
    c, st = product(A, B, tau_tile=24, **kw)
    assert "absorb_cap" not in kw or st["n_chunks"] > 0
    check_result(c, A, B, tol=TOL)


def test_wide_slices_of_a_wide_plan():
    # K = 512 in slices of 304: the last slice, 208 columns wide, runs on the planes
    A = synth.block_sparse_csr(512, seed=1, band=2)
    B = synth.dense_b(512, 512, seed=2)
    c, _ = product(A, B, tau_tile=64, TM=16, TK=32, TN=304)
    check_result(c, A, B, tol=TOL)


def test_padding_reads_no_row_of_b():
    # the columns that pad a window's last tile multiply nothing: a NaN in a row of B that A does not
    # use (row 0 among them) stays out of every result
    A = synth.block_sparse_csr(320, seed=7, band=1, p_random=0.0)
    rows = np.repeat(np.arange(320), np.diff(A["rowptr"]))
    used = A["colidx"] >= 64
    A = synth.csr_from_coo(320, 320, rows[used], A["colidx"][used], A["vals"][used])
    B = synth.dense_b(320, 64, seed=8)
    B[:64] = np.nan
    c, _ = product(A, B, tau_tile=8, TM=16, TK=32)
    assert np.isfinite(c).all()
    check_result(c, A, np.nan_to_num(B), tol=TOL)
