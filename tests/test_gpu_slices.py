"""Launches of more than 256 columns run as column slices (GPU): served, with an arrival counter per split
row and slice, and with the hot-row map, in the form whose warps share chunks and in the one-warp form."""
import time

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


def hubs(m, seed):
    """A power-law graph with a few rows that many chunks share."""
    rng = np.random.default_rng(seed)
    A = synth.rmat_csr(int(np.log2(m)), 6 * m, seed=seed)
    rows = np.repeat(np.arange(m), np.diff(A["rowptr"]))
    hub = np.repeat([3, m // 2, m - 1], m // 2)
    cols = np.concatenate([rng.permutation(m)[:m // 2] for _ in range(3)])
    key = np.unique(np.concatenate([rows * m + A["colidx"], hub * m + cols]))
    return synth.csr_from_coo(m, m, key // m, (key % m).astype(np.int32), rng.uniform(-1, 1, key.size).astype(np.float32))


@pytest.mark.parametrize("m", [512, 65536])  # chunks shared by a CTA, and by a warp
def test_served_slices(m):
    A = hubs(m, seed=1)
    sv = ns.Server(max_inflight=6)
    gid = sv.register(A)
    work = []
    for i, K in enumerate([264, 512, 64, 264, 512, 1024, 264]):
        B = synth.dense_b(m, K, seed=K)
        bf16 = i % 2 == 1
        h = synth.bf16_bits(B) if bf16 else B
        C = np.full((m, K), np.nan, np.float32)
        work.append((sv.submit(gid, h, C, ns.NS_BF16 if bf16 else ns.NS_F32), h, bf16, C))
    t0 = time.time()
    for t, h, bf16, C in work:
        while not sv.poll(t)[0]:
            assert time.time() - t0 < 60
            time.sleep(0.001)
        check_result(C, A, h, b_bf16=bf16, tol=1e-6)
    assert np.array_equal(work[0][3], work[6][3])  # the same request twice
    sv.close()


@pytest.mark.parametrize("K", [32, 264, 512])
@pytest.mark.parametrize("m,W", [(512, 16), (65536, 128)])
@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_hot_row_map(K, m, W, dtype):
    A = hubs(m, seed=2)
    h = synth.dense_b(m, K, seed=3)
    if dtype == ns.NS_BF16:
        h = synth.bf16_bits(h)
        Bd = torch.from_numpy(h.view(np.int16)).to(DEV).view(torch.bfloat16)
    else:
        Bd = torch.from_numpy(h).to(DEV)
    out = []
    for hints in (1, 2):
        C = torch.full((m, K), float("nan"), device=DEV)
        with ns.spmm_plan(to_dev(A, DEV), K, dtype, tune_from(ns, chunk_nnz=W, l2_hints=hints)) as p:
            for _ in range(2):
                p.execute(Bd, C)
            torch.cuda.synchronize()
            assert (p.stats()["n_chunks"] > 8 * 152) == (m > 512) and p.stats()["n_split"] > 0
        out.append(C.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    check_result(out[1], A, h, b_bf16=dtype == ns.NS_BF16, tol=1e-6)
