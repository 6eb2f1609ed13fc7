"""The contiguous-stream kernel where its forms meet (GPU): rows of many pieces summed by all lane groups,
16-byte aligned B at ragged widths, wide rows with more and fewer chunks than a CTA shares, wide rows in
short chunks, and B past L2."""
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
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lens]
    rows = np.repeat(np.arange(len(lens)), lens)
    return synth.csr_from_coo(len(lens), n, rows, np.concatenate(cols).astype(np.int32),
                              rng.uniform(-1, 1, size=rows.size).astype(np.float32))


def on_device(h, dtype, off=0):
    """`h` on the device, `off` elements past a 32-byte boundary."""
    td = torch.bfloat16 if dtype == ns.NS_BF16 else torch.float32
    flat = torch.zeros(h.size + off, dtype=td, device=DEV)
    flat[off:] = torch.from_numpy(h.view(np.int16 if dtype == ns.NS_BF16 else np.float32).reshape(-1)).to(DEV).view(td)
    return flat[off:].view(h.shape)


def products(A, h, dtype, W, offs=(0,)):
    out = []
    with ns.spmm_plan(to_dev(A, DEV), h.shape[1], dtype, tune_from(ns, chunk_nnz=W)) as p:
        for off in offs:
            C = torch.full((A["m"], h.shape[1]), float("nan"), device=DEV)
            p.execute(on_device(h, dtype, off), C)
            torch.cuda.synchronize()
            out.append(C.cpu().numpy())
        st = p.stats()
    assert all(np.array_equal(out[0], c) for c in out[1:])
    check_result(out[0], A, h, b_bf16=dtype == ns.NS_BF16, tol=1e-6)
    return st


# pieces of a row: 2, 3, around 4 and 8 times the lane groups, hundreds
PIECES = [1, 40, 70, 150, 260, 270, 530, 1100, 0, 2100, 9000, 5, 16, 33]


@pytest.mark.parametrize("K", [8, 24, 40, 64, 72, 104, 128, 136, 200, 256, 264, 520])
@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_rows_of_many_pieces(K, dtype):
    h = synth.dense_b(10_000, K, seed=K)
    h = synth.bf16_bits(h) if dtype == ns.NS_BF16 else h
    A = rows_csr(PIECES * 2, 10_000, seed=K)
    st = products(A, h, dtype, 32, offs=(0, 4, 0) if dtype == ns.NS_F32 else (0, 8))
    assert st["n_split"] > 0 and st["n_slots"] > 700


@pytest.mark.parametrize("K", [136, 192, 256])
@pytest.mark.parametrize("copies", [5, 16])  # a CTA a chunk up to 8 chunks an SM, a warp past it
def test_wide_rows_a_warp_or_a_cta_a_chunk(K, copies):
    A = rows_csr(([0, 0, 3, 0, 1, 40, 0, 300, 2, 64, 5, 0, 33] * copies), 800, seed=K)
    h = synth.dense_b(800, K, seed=1)
    st = products(A, h, ns.NS_F32, 2, offs=(0, 4))
    assert (st["n_chunks"] > 8 * 152) == (copies == 16)


@pytest.mark.parametrize("W", [4, 32, 33])  # short chunks at several slices a row are not cut into slices
@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_wide_rows_in_short_chunks(W, dtype):
    A = rows_csr([0, 0, 3, 0, 1, 40, 0, 300, 2, 64, 5, 0, 33] * 6, 800, seed=W)
    h = synth.dense_b(800, 520, seed=1)
    products(A, synth.bf16_bits(h) if dtype == ns.NS_BF16 else h, dtype, W)


@pytest.mark.parametrize("K", [72, 128])
def test_b_past_l2(K):
    n = (300 << 20) // (4 * K)
    A = rows_csr([0, 7, 300, 1, 0, 2500, 19] * 300, n, seed=K)
    products(A, synth.dense_b(n, K, seed=2), ns.NS_F32, 256, offs=(0, 4))
