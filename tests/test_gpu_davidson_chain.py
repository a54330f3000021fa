"""GPU: the fused chain of a Davidson iteration (dots, Ritz problem, residual, correction,
orthogonalisation) through dmrg_davidson, at subspace sizes around its edges (restart at 4
vectors, an odd size whose Jacobi rounds have a bye, the largest one) and vector lengths below
and above the 264 chunks of its sums.  Against numpy's lowest eigenpair of the oracle's dense
H_eff: both stop at |H x - theta x| <= 1e-8, so theta is within 1e-8 of the eigenvalue, and the
returned vector is normalised and has that residual (1e-12 |H| allowed for rounding)."""
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


@pytest.mark.parametrize("space,Np,Nn,M0,p", [("p", 2, 2, 5, 1), ("p", 1, 2, 6, 2),
                                              ("sd", 3, 2, 96, 1), ("sd", 2, 2, 400, 1)])
@pytest.mark.parametrize("sub", [4, 5, 9, 64])
def test_davidson_chain(P, space, Np, Nn, M0, p, sub):
    from oracle.dmrg import OracleDMRG
    prob = make_problem(space, Np, Nn, (Np + Nn) % 2, seed=31)
    init = initial_mps(prob, M0, 32)
    o = OracleDMRG(prob, init)
    d = P.DMRG(prob, dav_max_sub=sub, dav_max_iter=600)
    d.build_blocks(init)
    for q in range(1, p):
        d.step(q, 0, 64)
    n = d.psi_layout(p)["size"]
    if p == 1:
        sb = o.superblock(1)
        H = np.stack([sb.apply(e) for e in np.eye(n)], axis=1)
    else:   # the library's own matrix (its products are pinned elsewhere)
        H = np.zeros((n, n))
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        for i in range(n):
            e = torch.zeros(n, dtype=torch.float64, device="cuda")
            e[i] = 1.0
            d.heff_apply(p, e, y)
            H[:, i] = y.cpu().numpy()
    w = np.linalg.eigvalsh((H + H.T) / 2)
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    energy, st = d.davidson(p, guess=torch.ones(n, dtype=torch.float64, device="cuda"), out=out)
    x = out.cpu().numpy()
    assert st["converged"] == 1
    assert abs(np.linalg.norm(x) - 1.0) <= 1e-12
    assert np.linalg.norm(H @ x - energy * x) <= 1e-8 + 1e-12 * np.abs(w).max()
    assert abs(energy - w[0]) <= 1e-8
    d.close()
