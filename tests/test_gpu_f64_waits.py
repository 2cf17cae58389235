"""The waits of the tensor-core FP64 products run out on valid work: the bound is
the caller's, the call reports E_TIMEOUT, the kernel leaves the GPU usable and
small products, which wait for nothing, still run."""
import numpy as np
import pytest

import synth

from oracle import blocksparse as bs
from test_gpu_f64_products import RTOL, _wide_mps

pytestmark = pytest.mark.gpu


def _case(mpslcc, dl, dr, **opts):
    h, V = synth.ab_initio(4, 12, seed=5)
    m = _wide_mps(dl, dr, 1000 * dl + dr)
    mpo = bs.Mpo(h, V, "H", 0, 4)
    L = bs.update_left(mpo, bs.boundary_left(mpo), m, m, 0)
    R = bs.update_right(mpo, bs.boundary_right(mpo), m, m, 3)
    ctx = mpslcc.Context(device=0, **opts)
    ctx.build_mpo(h, V, 4, 0)
    ctx.load_mps(1, m)
    return ctx, lambda psi: bs.sigma(mpo, m, m, 1, psi, L, R)


def test_an_expired_wait_of_an_fp64_product_returns_timeout(mpslcc):
    ctx, _ = _case(mpslcc, 300, 200, wait_timeout_s=1e-9)
    with ctx:
        n, _ = ctx.local_dim(1, mpslcc.OP_H_11)
        psi = synth.random_vector(n, 1)
        for _ in range(2):
            with pytest.raises(mpslcc.MpsLccError) as e:
                ctx.apply_heff(1, mpslcc.OP_H_11, psi)
            assert e.value.status == 6, str(e.value)
    small, oracle_small = _case(mpslcc, 5, 6, wait_timeout_s=1e-9)
    with small:
        m, _ = small.local_dim(1, mpslcc.OP_H_11)
        phi = synth.random_vector(m, 2)
        s = small.apply_heff(1, mpslcc.OP_H_11, phi)
    assert np.linalg.norm(s - oracle_small(phi)) <= RTOL * np.linalg.norm(s)
    ctx, oracle = _case(mpslcc, 300, 200)
    with ctx:
        s = ctx.apply_heff(1, mpslcc.OP_H_11, psi)
    r = oracle(psi)
    assert np.linalg.norm(s - r) <= RTOL * np.linalg.norm(r)
