"""The allocation-free GEMM at the edges of its tiles: it picks its N tile by
the number of tiles and writes FP64 rows itself, and must equal the FP32 result
of the allocating entry point bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name", ["BF16", "TF32", "BF16X3"])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 31, 9), (129, 17, 64), (128, 64, 65), (257, 300, 33), (2500, 20, 16),
                                   (640, 1000, 40), (2049, 1409, 24)])
def test_noalloc_gemm_equals_the_fp32_product_at_tile_edges(mpslcc, prec_name, m, n, k):
    torch = pytest.importorskip("torch")
    prec = getattr(mpslcc, prec_name)
    rng = np.random.default_rng(m + 7 * n + k)
    A = rng.standard_normal((m, k))
    B = rng.standard_normal((n, k))
    with mpslcc.Context(device=0) as ctx:
        ref = ctx.debug_tc_gemm(A, B, prec=prec, mode=2)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    dC = torch.full((m * n + 2,), float("nan"), dtype=torch.float64, device="cuda")
    mpslcc.tc_gemm_noalloc(0, torch.cuda.current_stream().cuda_stream, prec, m, n, k, dA.data_ptr(), dB.data_ptr(),
                           dC[1:].data_ptr())
    out = dC.cpu().numpy()
    assert np.isnan(out[0]) and np.isnan(out[-1])   # nothing beside C is written
    assert np.array_equal(out[1:-1].reshape(m, n), ref)
