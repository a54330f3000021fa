"""GPU: the FP64 tile kernel of the product (every block wider than 16, heff_big_edge = 0) at the
edges of its tiles, chunks, groups of terms and slots.

* First position: against the oracle's product on identical inputs, right sectors of 17 to
  ~100 states, left blocks of one or two; 1e-12 of the norm, the bar of the product tests.
* Further in (complete left blocks, so the basis is the inputs'): blocks wide on both sides,
  both associations, fewer terms than slots up to several groups; against the grouped GEMM
  passes (heff_big_edge = 1) on the same superblock, whose sums run in another order: 1e-12."""
import numpy as np
import pytest

from gen import make_problem, initial_mps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1507_00161_gb300.build import build
    build()
    import paper_1507_00161_gb300 as P
    return P


def _product(d, p, x, edge):
    d.set_tuning(heff_big_edge=edge)
    y = torch.full_like(x, float("nan"))
    d.heff_apply(p, x, y)
    z = torch.full_like(x, float("nan"))
    d.heff_apply(p, x, z)          # replayed from the graph
    assert torch.equal(y, z)
    return y.cpu().numpy()


@pytest.mark.parametrize("Np,Nn,M0", [(2, 2, 300), (3, 2, 520), (4, 4, 900)])
def test_first_position(P, Np, Nn, M0):
    from oracle.dmrg import OracleDMRG
    prob = make_problem("sd", Np, Nn, (Np + Nn) % 2, seed=41)
    init = initial_mps(prob, M0, 42)
    sb = OracleDMRG(prob, init).superblock(1)
    d = P.DMRG(prob)
    d.build_blocks(init)
    lay = d.psi_layout(1)
    assert max(lay["dr"]) > 16
    x = np.random.default_rng(1).standard_normal(lay["size"])
    ref = sb.apply(x)
    y = _product(d, 1, torch.tensor(x, device="cuda"), 0)
    assert np.linalg.norm(y - ref) <= 1e-12 * np.linalg.norm(ref)
    d.close()


@pytest.mark.parametrize("space,Np,Nn,M0,p", [("sd", 4, 4, 400, 5), ("sd", 5, 4, 256, 11),
                                              ("pf", 4, 4, 1100, 4), ("pf", 4, 5, 900, 10)])
def test_inner_positions(P, space, Np, Nn, M0, p):
    prob = make_problem(space, Np, Nn, (Np + Nn) % 2, seed=43)
    d = P.DMRG(prob, dav_max_iter=1)
    d.build_blocks(initial_mps(prob, M0, 44))
    for q in range(1, p):
        d.step(q, 0, 4096)
    lay = d.psi_layout(p)
    assert max(max(lay["dl"]), max(lay["dr"])) > 16   # (wider than the small-block kernel)
    x = torch.tensor(np.random.default_rng(2).standard_normal(lay["size"]), device="cuda")
    ref = _product(d, p, x, 1)
    y = _product(d, p, x, 0)
    assert np.linalg.norm(y - ref) <= 1e-12 * np.linalg.norm(ref)
    d.close()
