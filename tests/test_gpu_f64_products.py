"""FP64 products (gemm_f64.cu) at the edges of their tiles.  Sigma of a
four-orbital chain whose bonds carry chosen dimensions runs every form of FP64
task through both kernels (batches folded into rows and into columns, swapped
operands, K runs, K splits, several scaling blocks); the block-sparse oracle
gives the reference."""
import numpy as np
import pytest

import synth
from oracle import blocksparse as bs

pytestmark = pytest.mark.gpu

# Both sides round each of three nested products (fused operators, phase 1,
# phase 2): the library to 2^-53 per product, the oracle's FP64 chains to about
# sqrt(K) 2^-53 each with K <= 1e4 terms, together below 4e-14 in the 2-norm.
RTOL = 1e-13


def _wide_mps(dl, dr, seed):
    """Four orbitals, four electrons; one sector of bonds 1 and 3 has dimension
    dl and dr, the others a few."""
    rng = np.random.default_rng(seed)
    masks = synth.site_masks(4)
    bonds = synth.bond_sectors(masks, 4, 0, 10 ** 6)
    bonds[1] = [(n, z, dl if (n, z) == (1, 1) else 1 + i) for i, (n, z, _) in enumerate(bonds[1])]
    bonds[2] = [(n, z, 2 + i % 3) for i, (n, z, _) in enumerate(bonds[2])]
    bonds[3] = [(n, z, dr if (n, z) == (3, -1) else 3 - i % 2) for i, (n, z, _) in enumerate(bonds[3])]
    sites = []
    for p in range(4):
        at = {q[:2]: j for j, q in enumerate(bonds[p + 1])}
        blocks = {}
        for ia, (n, z, da) in enumerate(bonds[p]):
            for s in range(4):
                q = (n + synth.LOCAL_N[s], z + synth.LOCAL_2SZ[s])
                if q in at:
                    db = bonds[p + 1][at[q]][2]
                    blocks[(ia, s, at[q])] = rng.standard_normal((da, db)) / np.sqrt(da + db)
        sites.append(blocks)
    return dict(bonds=bonds, sites=sites, masks=masks)


def _case(mpslcc, dl, dr):
    h, V = synth.ab_initio(4, 12, seed=5)
    m = _wide_mps(dl, dr, 1000 * dl + dr)
    mpo = bs.Mpo(h, V, "H", 0, 4)
    L = bs.update_left(mpo, bs.boundary_left(mpo), m, m, 0)
    R = bs.update_right(mpo, bs.boundary_right(mpo), m, m, 3)
    ctx = mpslcc.Context(device=0)
    ctx.build_mpo(h, V, 4, 0)
    ctx.load_mps(1, m)
    return ctx, lambda psi: bs.sigma(mpo, m, m, 1, psi, L, R)


@pytest.mark.parametrize("dl,dr", [(1, 1), (5, 300), (31, 33), (32, 64), (65, 63), (127, 129), (128, 128), (300, 7)])
def test_f64_products_match_the_oracle_at_tile_edges(mpslcc, dl, dr):
    ctx, oracle = _case(mpslcc, dl, dr)
    with ctx:
        n, _ = ctx.local_dim(1, mpslcc.OP_H_11)
        psi = synth.random_vector(n, dl + dr)
        s = ctx.apply_heff(1, mpslcc.OP_H_11, psi)
    r = oracle(psi)
    assert np.linalg.norm(s - r) <= RTOL * np.linalg.norm(r)


@pytest.mark.parametrize("scale", [1e-280, 1e280])
def test_f64_products_keep_their_accuracy_at_the_ends_of_the_range(mpslcc, scale):
    """Rows are scaled by powers of two of their own, so an input of extreme
    magnitude gives the scaled result to the same accuracy."""
    ctx, oracle = _case(mpslcc, 65, 63)
    with ctx:
        n, _ = ctx.local_dim(1, mpslcc.OP_H_11)
        psi = synth.random_vector(n, 3)
        s = ctx.apply_heff(1, mpslcc.OP_H_11, psi * scale)
    r = oracle(psi)
    assert np.linalg.norm(s / scale - r) <= RTOL * np.linalg.norm(r)


def test_f64_products_with_a_non_finite_row(mpslcc):
    """A row that holds an infinity goes through plain multiply-adds: what does
    not touch it is unchanged, what does is not finite."""
    torch = pytest.importorskip("torch")
    ctx, oracle = _case(mpslcc, 65, 63)
    with ctx:
        n, _ = ctx.local_dim(1, mpslcc.OP_H_11)
        psi = synth.random_vector(n, 9)
        ref = ctx.apply_heff(1, mpslcc.OP_H_11, psi)
        x = torch.from_numpy(psi).cuda()
        x[n // 2] = float("inf")
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.apply_heff_device(1, mpslcc.OP_H_11, x.data_ptr(), y.data_ptr(), n, n)
        torch.cuda.synchronize()
        s = y.cpu().numpy()
    ok = np.isfinite(s)
    assert not ok.all()
    assert ok.any() and np.linalg.norm(s[ok] - ref[ok]) <= RTOL * np.linalg.norm(ref)
