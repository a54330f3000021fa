"""GPU: the mixed tile kernel of the product (split-TF32 MMAs, heff_big_edge = 0) element by element
against the oracle's FP64 product, at the edges of its tiles, pieces and copies: tiles of up to 16 and of
more columns, inner dimensions that are odd, multiples of 8, and beyond 32 with rows that do and do not
start on 16 bytes.  Left blocks are complete, so the basis is the inputs'.

Tolerance of an element, relative to S = sum of |L| |psi| |R| over its products: the operands are
FP32 and the a_lo b_lo terms are left out (together below 4 x 2^-21), and every MMA step of 8 inner
elements rounds the running sum, at worst by 2^-21 of its absolute sum (9 addends cut at the largest
one's 24 bits).  A sum runs through 3 ceil(dR / 8) steps of psi R^T, 3 ceil(dL / 8) steps per term for
the at most 16 terms of a slot and group, and at most 6 additions of slots and groups."""
import numpy as np
import pytest

from gen import make_problem, initial_mps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # space, Np, Nn, M0, p, and what its blocks must contain
    ("sd", 4, 4, 400, 5, {"narrow", "wide", "odd"}),
    ("sd", 4, 4, 1200, 4, {"narrow", "wide", "odd", "of 8", "rows of 4", "other rows"}),
    ("sd", 4, 4, 1200, 10, {"narrow", "wide", "odd", "of 8", "tall"}),
    ("sd", 5, 4, 256, 11, {"narrow", "odd", "of 8", "rows of 4", "other rows", "tall"}),
]


@pytest.mark.parametrize("space,Np,Nn,M0,p,contains", CASES)
def test_elements(space, Np, Nn, M0, p, contains):
    from paper_1507_00161_gb300.build import build
    build()
    import paper_1507_00161_gb300 as P
    from oracle.dmrg import Block, OracleDMRG, SuperBlock, enlarge_left
    prob = make_problem(space, Np, Nn, (Np + Nn) % 2, seed=41)
    init = initial_mps(prob, M0, 42)
    o = OracleDMRG(prob, init)
    for q in range(1, p):
        o.left[q] = enlarge_left(o.left[q - 1], q, o.mpo, o.ch)
    sb = o.superblock(p)
    dl = np.array([b[2] for b in sb.layout.blocks])
    dr = np.array([b[3] for b in sb.layout.blocks])
    inner = np.concatenate([dl, dr])
    has = {"narrow": np.any((dr <= 16) & (dl > 16)) or np.any(dr % 32 > 0) and np.any(dr[dr > 16] % 32 <= 16),
           "wide": np.any(dr > 16), "tall": np.any(dl > 16), "odd": np.any(inner % 2 == 1),
           "of 8": np.any(inner[inner > 7] % 8 == 0),
           "rows of 4": np.any((inner > 32) & (inner % 4 == 0)),
           "other rows": np.any((inner > 32) & (inner % 4 != 0))}
    assert all(has[c] for c in contains), has
    d = P.DMRG(prob, dav_max_iter=1)
    d.build_blocks(init)
    for q in range(1, p):
        d.step(q, 0, 4096)
    d.set_options(precision=P.MIXED_FP32)
    d.set_tuning(heff_big_edge=0)
    assert d.psi_layout(p)["size"] == sb.layout.size
    x = np.random.default_rng(5).standard_normal(sb.layout.size)
    xd = torch.tensor(x, device="cuda")
    y, z = (torch.full_like(xd, float("nan")) for _ in range(2))
    d.heff_apply(p, xd, y)
    d.heff_apply(p, xd, z)          # replayed from the graph
    assert torch.equal(y, z)
    ref = sb.apply(x)

    def sizes(b):
        return Block(b.sectors, b.dims, [{k: np.abs(v) for k, v in op.items()} for op in b.ops], b.pieces)

    S = SuperBlock(sizes(sb.L), sizes(sb.R), [0] * len(sb.parity), sb.qT).apply(np.abs(x))
    steps = 3 * -(-dr.max() // 8) + 16 * 3 * -(-dl.max() // 8) + 6
    err = np.abs(y.cpu().numpy() - ref)
    worst = np.max(err / np.maximum(S, 1e-300))
    print(f"\n[mixed tiles] {space} {Np}p+{Nn}n M0={M0} p={p}: worst {worst:.2e} of S, bar {(steps + 4) * 2.0 ** -21:.2e}")
    assert np.all(err <= (steps + 4) * 2.0 ** -21 * S)
    d.close()
