"""FP64 orthonormalisation of more rows than the digit sums are proven for (2^27)
runs on the FP64 kernels, which nothing smaller reaches.  Their sums run over
the rows of a chunk (of 2 per SM) in order, so rows per chunk times eps bounds
the error of the Gram matrix, and with it of Q."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,split", [((1 << 27) + 1, False), (1 << 20, True)])
def test_route_and_result(n, split):
    import paper_2511_06600_gb300 as hef
    K = 2
    V = torch.randn(n, K, dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(1)) + 0.5
    A = V - V.mean(0)
    torch.cuda.synchronize()
    hef.trace_read()
    hef.trace_kernels("k_")
    try:
        Q, R, rank = hef.orthonormalize(V, K, want_R=True)
        torch.cuda.synchronize()
    finally:
        hef.trace_kernels(None)
    names = set(hef.trace_read())
    assert ("k_gram_split" in names, "k_apply_split" in names) == (split, split)
    assert ("k_gram" in names, "k_apply" in names) == (not split, not split)
    assert int(rank) == K
    tol = 2 * 2.2e-16 * (n / (2 * torch.cuda.get_device_properties(0).multi_processor_count) + 100)
    assert float((Q.T @ Q - torch.eye(K, device="cuda", dtype=Q.dtype)).abs().max()) <= tol
    assert float((A - Q @ R).abs().max()) <= tol * float(A.abs().max())
    assert float(R[1, 0]) == 0 and float(R.diagonal().min()) > 0
