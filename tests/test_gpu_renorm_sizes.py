"""GPU: enlargement and renormalization of the block operators at the edges of their size classes
(enlarged sectors around 16, 32 and 128 states, several columns of 32, blocks of more than 2048
elements), through the product at the first position after dmrg_build_blocks: every right-block
operator of the chain has gone through them.  Against the oracle's product on identical inputs,
1e-12 of the norm (the bar of the product tests)."""
import numpy as np
import pytest

from gen import make_problem, initial_mps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Np,Nn,M0", [(2, 2, 6), (3, 3, 70), (3, 2, 260), (4, 4, 420), (3, 3, 1500)])
def test_build_blocks_sizes(Np, Nn, M0):
    from paper_1507_00161_gb300.build import build
    build()
    import paper_1507_00161_gb300 as P
    from oracle.dmrg import OracleDMRG
    prob = make_problem("sd", Np, Nn, (Np + Nn) % 2, seed=51)
    init = initial_mps(prob, M0, 52)
    sb = OracleDMRG(prob, init).superblock(1)
    d = P.DMRG(prob)
    d.build_blocks(init)
    x = np.random.default_rng(3).standard_normal(d.psi_layout(1)["size"])
    y = torch.empty(x.size, dtype=torch.float64, device="cuda")
    d.heff_apply(1, torch.tensor(x, device="cuda"), y)
    ref = sb.apply(x)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    d.close()
