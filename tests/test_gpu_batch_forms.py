"""A batch whose B move between 32- and 16-byte boundaries (GPU): the launches take the form that the
operands allow, in one captured graph, and the results keep their bits."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2606_22482_gb300 as ns  # noqa: E402
from nsutil import to_dev  # noqa: E402

DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("dtype", [ns.NS_F32, ns.NS_BF16])
def test_operands_change_alignment(dtype):
    td, per16 = (torch.bfloat16, 8) if dtype == ns.NS_BF16 else (torch.float32, 4)
    graphs = synth.batch_graphs(8, seed=3, n_lo=200, n_hi=6000) + [synth.csr_from_coo(5, 5, np.zeros(0), np.zeros(0))]
    Ks = [8, 24, 64, 24, 8, 264, 64, 264, 40]
    Bs = [torch.randn(g["n"], k, device=DEV).to(td) for g, k in zip(graphs, Ks)]

    def at(B, off):  # a copy of B, `off` 16-byte units past a 32-byte boundary
        flat = torch.empty(B.numel() + per16 * off, dtype=td, device=DEV)
        assert flat.data_ptr() % 32 == 0
        flat[per16 * off:] = B.reshape(-1)
        return flat[per16 * off:].view(B.shape)

    bt = ns.Batch([to_dev(g, DEV) for g in graphs], Ks, dtype)
    first = None
    for offs in ([0] * 9, [1] * 9, [0] * 9, [1, 0, 0, 0, 0, 0, 0, 0, 0], [0, 1, 0, 1, 0, 1, 0, 0, 1], [0] * 9, [1] * 9):
        Cs = [torch.full((g["m"], k), float("nan"), device=DEV) for g, k in zip(graphs, Ks)]
        bt.execute([at(B, o) for B, o in zip(Bs, offs)], Cs)
        torch.cuda.synchronize()
        Cs = [c.cpu().numpy() for c in Cs]
        if first is None:
            first = Cs
            for g, B, c in zip(graphs, Bs, Cs):
                assert oracle.rel_frobenius(c, oracle.spmm(g, B.float().cpu().numpy())) <= 1e-5
        assert all(np.array_equal(a, b) for a, b in zip(first, Cs))
    bt.close()


def test_plan_operand_changes_alignment():
    A = synth.uniform_csr(900, 700, 9, seed=1)
    B = torch.randn(700, 48, device=DEV)
    flat = torch.empty(B.numel() + 4, device=DEV)
    flat[4:] = B.reshape(-1)
    t = ns.tune_default()
    t.TN = 32  # slices of 32 and 16 columns
    for tune in (None, t):
        with ns.spmm_plan(to_dev(A, DEV), 48, ns.NS_F32, tune) as p:
            Cs = [torch.full((900, 48), float("nan"), device=DEV) for _ in range(4)]
            for C, b in zip(Cs, (B, flat[4:].view(700, 48), B, flat[4:].view(700, 48))):
                p.execute(b, C)
            torch.cuda.synchronize()
        assert all(torch.equal(Cs[0], C) for C in Cs[1:])
        assert oracle.rel_frobenius(Cs[0].cpu().numpy(), oracle.spmm(A, B.cpu().numpy())) <= 1e-5
