"""The contiguous-stream kernel at the edges of its forms (GPU): lane groups of every width, column
slices above K = 256, chunks shared by a CTA and by a warp, 16-byte aligned B, and rows that
straddle shares of a chunk or chunks, each element within the forward error bound of a dot product."""
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


def rows_csr(lens, n, seed):
    """Rows of the given lengths, distinct uniform columns."""
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lens]
    rows = np.repeat(np.arange(len(lens)), lens)
    vals = rng.uniform(-1, 1, size=len(rows)).astype(np.float32)
    return synth.csr_from_coo(len(lens), n, rows, np.concatenate(cols) if len(rows) else rows, vals)


# empty rows at both ends and in runs, rows of one, rows as long as a share and a chunk, one hub
LENS = [0, 0, 3, 0, 1, 1, 40, 0, 0, 0, 0, 700, 2, 0, 64, 64, 5, 0, 129, 1, 0, 33] * 4 + [0] * 70 + [17, 0, 0]


def product(A, B, dtype, W, offset=0):
    K = B.shape[1]
    h = synth.bf16_bits(B) if dtype == ns.NS_BF16 else B
    flat = torch.zeros(h.size + offset, dtype=torch.bfloat16 if dtype == ns.NS_BF16 else torch.float32, device=DEV)
    flat[offset:] = torch.from_numpy(h.view(np.int16).reshape(-1)).to(DEV).view(torch.bfloat16) \
        if dtype == ns.NS_BF16 else torch.from_numpy(h.reshape(-1)).to(DEV)
    Bt = flat[offset:].view(A["n"], K)
    C = torch.full((A["m"], K), float("nan"), device=DEV)
    with ns.spmm_plan(to_dev(A, DEV), K, dtype, tune_from(ns, chunk_nnz=W, absorb_cap=W)) as p:
        p.execute(Bt, C)
        torch.cuda.synchronize()
        n_chunks = p.stats()["n_chunks"]
    return C.cpu().numpy(), h, n_chunks


@pytest.mark.parametrize("K", [8, 32, 40, 64, 72, 128, 136, 256, 264, 512, 1024])
@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_widths_and_shares(K, dtype):
    A = rows_csr(LENS, 800, seed=K)
    B = synth.dense_b(800, K, seed=K + 1)
    for W in (3, 16, 256, 1024):  # W = 3 gives more chunks than the cooperative form takes
        c, h, nc = product(A, B, dtype, W)
        assert (nc > 8 * 152) == (W == 3)
        check_result(c, A, h, b_bf16=dtype == ns.NS_BF16, tol=1e-6)


@pytest.mark.parametrize("K", [32, 64, 128, 192])
def test_b_on_a_16_byte_boundary(K):
    A = rows_csr(LENS, 800, seed=K)
    B = synth.dense_b(800, K, seed=K + 1)
    aligned, _, _ = product(A, B, ns.NS_F32, 64)
    shifted, _, _ = product(A, B, ns.NS_F32, 64, offset=4)
    assert np.array_equal(aligned, shifted)      # the same sums in the same order


@pytest.mark.parametrize("W", [3, 64])
def test_nonfinite_rows_stay_their_own(W):
    # columns 0 and 1 of A hold an infinity and a NaN in B: exactly the rows with them are not finite
    A = rows_csr([5, 9, 0, 1, 30, 4, 0, 77, 2] * 20, 90, seed=5)
    B = synth.dense_b(90, 64, seed=6)
    B[0], B[1] = np.inf, np.nan
    c, _, _ = product(A, B, ns.NS_F32, W)
    hit = np.array([np.any(A["colidx"][a:b] < 2) for a, b in zip(A["rowptr"][:-1], A["rowptr"][1:])])
    assert np.array_equal(~np.isfinite(c).all(axis=1), hit) and hit.any() and not hit.all()
