"""The products' accounting (tlr_gemm_stats) counts the work that ran."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_2108_11932_gb300 as T
    T.build()
    return T


@pytest.mark.parametrize("n,bs,nops", [(96, 8, 5), (64, 12, 3)])
def test_a_converged_slot_counts_no_second_pass(T, n, bs, nops):
    """Zero operands converge in their first round: a sample of 2 n^2 bs and a Gram matrix of 2 n bs^2 each, and nothing
    of the second orthogonalization (block widths without the fused kernel)."""
    import torch
    ctx = T.Context(0)
    ctx.gemm_stats(True)
    _, _, r = ctx.ara_dense(torch.zeros((nops, n, n), dtype=torch.float64, device="cuda:0"), bs, 1e-6, 1)
    st = ctx.gemm_stats(False)
    assert int(r.max()) == 0
    assert st["fp64_NN"]["flops"] == 2 * n * n * bs * nops
    assert st["fp64_TN"]["flops"] == 2 * n * bs * bs * nops
    ctx.close()
