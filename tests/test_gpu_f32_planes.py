"""FP32 plans whose dense tiles' planes do not fit (GPU): past their bound on memory, when their
allocation fails, or in a launch with such a plan, the product runs from the packed tiles; the plan is
the oracle's either way."""
import time

import numpy as np
import pytest

import oracle
import synth
from parity import check_result

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2606_22482_gb300 as ns  # noqa: E402
from nsutil import compare_plan, oracle_tune, to_dev, tune_from  # noqa: E402

DEV = torch.device("cuda", 0)


def plane_bytes(st):
    return 6 * st["TM"] * st["TK"] * st["n_dtiles"]


def scattered(m, per_row, n, seed):
    """Rows of a few distinct uniform columns: tiles with one nonzero a column."""
    rng = np.random.default_rng(seed)
    key = np.unique(np.repeat(np.arange(m), per_row) * n + rng.integers(0, n, m * per_row))
    return synth.csr_from_coo(m, n, key // n, (key % n).astype(np.int32), rng.uniform(-1, 1, key.size).astype(np.float32))


def execute(p, A, B):
    C = torch.full((A["m"], B.shape[1]), float("nan"), device=DEV)
    p.execute(torch.from_numpy(B).to(DEV), C)
    torch.cuda.synchronize()
    return C.cpu().numpy()


@pytest.fixture(autouse=True)
def _injection_off():
    yield
    ns.inject_alloc_failure(-1)


def survives(A, K, tune):
    """The plan made with its planes' allocation failing (the first failure that planning survives),
    and which allocation that is."""
    At = to_dev(A, DEV)
    for after in range(16):
        ns.inject_alloc_failure(after)
        try:
            return ns.spmm_plan(At, K, ns.NS_F32, tune), after
        except ns.NsError as e:
            assert e.code == 3
        finally:
            ns.inject_alloc_failure(-1)


def test_planes_past_their_bound():
    A = scattered(48_000, 64, 60_000, seed=1)  # 1.1 GB of planes, 47 times the CSR
    K = 8
    B = synth.dense_b(A["n"], K, seed=1)
    tune = tune_from(ns, tau_tile=1, TM=64, TK=32)
    with ns.spmm_plan(to_dev(A, DEV), K, ns.NS_F32, tune) as p:
        st = p.stats()
        assert plane_bytes(st) > 1 << 30 and st["device_bytes"] < plane_bytes(st)
        compare_plan(p, oracle.plan(A, K, **oracle_tune(tune)), A, tune)
        check_result(execute(p, A, B), A, B)


@pytest.mark.parametrize("TM,TK", [(16, 16), (64, 32)])
@pytest.mark.parametrize("K", [8, 40, 128, 256])
def test_failed_allocation_of_planes(TM, TK, K):
    A = synth.block_sparse_csr(512, seed=2, block=16, band=2, p_random=0.05)
    B = synth.dense_b(A["n"], K, seed=3)
    tune = tune_from(ns, tau_tile=40, TM=TM, TK=TK)
    with ns.spmm_plan(to_dev(A, DEV), K, ns.NS_F32, tune) as p:
        full = p.stats()
    with survives(A, K, tune)[0] as p:
        assert full["device_bytes"] - p.stats()["device_bytes"] >= plane_bytes(full) > 0
        compare_plan(p, oracle.plan(A, K, **oracle_tune(tune)), A, tune)
        check_result(execute(p, A, B), A, B)


def test_batch_of_both_kinds():
    graphs = [synth.block_sparse_csr(640, seed=1, band=2), scattered(2000, 2, 30_000, seed=2),
              synth.uniform_csr(300, 300, 5, seed=3)]
    K = 40
    Bs = [synth.dense_b(g["n"], K, seed=i) for i, g in enumerate(graphs)]
    tune = tune_from(ns, tau_tile=1, TM=64, TK=32)
    for failing in (False, True):
        if failing:  # the first plan without planes, the others with theirs
            p, after = survives(graphs[0], K, tune)
            p.close()
            ns.inject_alloc_failure(after)
        Cd = [torch.full((g["m"], K), float("nan"), device=DEV) for g in graphs]
        bt = ns.Batch([to_dev(g, DEV) for g in graphs], [K] * 3, ns.NS_F32, tune)
        bt.execute([torch.from_numpy(b).to(DEV) for b in Bs], Cd)
        torch.cuda.synchronize()
        for g, b, c in zip(graphs, Bs, Cd):
            check_result(c.cpu().numpy(), g, b)
        bt.close()


@pytest.mark.parametrize("budget", [4 << 20, 1 << 30])  # planes past an eighth of it, and within
def test_served_hybrid(budget):
    graphs = [synth.block_sparse_csr(1024, seed=1, band=2), scattered(2000, 2, 3000, seed=2)]
    sv = ns.Server(hbm_budget_bytes=budget, max_inflight=8, tune=tune_from(ns, tau_tile=64, TM=64, TK=32))
    gids = [sv.register(g) for g in graphs]
    work = []
    for i in range(6):
        g = graphs[i % 2]
        B = synth.dense_b(g["n"], 64, seed=i)
        C = np.full((g["m"], 64), np.nan, np.float32)
        work.append((sv.submit(gids[i % 2], B, C), g, B, C))
    t0 = time.time()
    for t, g, B, C in work:
        while not sv.poll(t)[0]:
            assert time.time() - t0 < 30
            time.sleep(0.001)
        check_result(C, g, B)
    sv.close()
