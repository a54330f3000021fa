"""GPU: the subspace size of Davidson changed between runs of one context, on the same superblock:
the largest, smaller ones (the workspace of the larger one stays), and in between.  Every run stops
at |H x - theta x| <= 1e-8 against the oracle's dense H_eff, so theta is within 1e-8 of the
eigenvalue and the returned vector has that residual (1e-12 |H| allowed for rounding)."""
import numpy as np
import pytest

from gen import make_problem, initial_mps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_subspace_size_changes():
    from paper_1507_00161_gb300.build import build
    build()
    import paper_1507_00161_gb300 as P
    from oracle.dmrg import OracleDMRG
    prob = make_problem("sd", 3, 2, 1, seed=31)
    init = initial_mps(prob, 96, 32)
    sb = OracleDMRG(prob, init).superblock(1)
    d = P.DMRG(prob)
    d.build_blocks(init)
    n = d.psi_layout(1)["size"]
    H = np.stack([sb.apply(e) for e in np.eye(n)], axis=1)
    w = np.linalg.eigvalsh((H + H.T) / 2)
    guess = torch.ones(n, dtype=torch.float64, device="cuda")
    out = torch.empty_like(guess)
    for sub in (64, 5, 24, 4, 9):
        d.set_options(dav_max_sub=sub, dav_max_iter=600)
        energy, st = d.davidson(1, guess=guess, out=out)
        x = out.cpu().numpy()
        assert st["converged"] == 1, sub
        assert np.linalg.norm(H @ x - energy * x) <= 1e-8 + 1e-12 * np.abs(w).max(), sub
        assert abs(energy - w[0]) <= 1e-8, sub
    d.close()
