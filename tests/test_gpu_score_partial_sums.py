"""Q_H of the FP32 form: how many hyperedges an FP32 partial sum of the staged pass
may cover before FP64 takes over.  Every window of 64 pins holds 32 two-pin
hyperedges of spread 1; one hyperedge in 32 windows weighs 2^26, where FP32 steps
by 8, the others 1.  The others that share the heavy one's partial sum are lost;
all later sums are FP64 and exact.  Eight windows of 32 hyperedges over 15
warps, in quads, are at most 5 quads: 19 others."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 100])
def test_partial_sums_cover_few_hyperedges(K):
    import paper_2511_06600_gb300 as hef
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks, per = sms, 32 * 32  # one heavy hyperedge per CTA's 32 windows
    m = blocks * per
    pins = torch.arange(2 * m, dtype=torch.int32, device="cuda")
    eptr = torch.arange(0, 2 * m + 1, 2, dtype=torch.int64, device="cuda")
    w = torch.ones(m, dtype=torch.float64, device="cuda")
    w[::per] = 2.0 ** 26
    inc = hef.build_incidence(2 * m, eptr, pins, w)
    inc.check()
    Q = torch.zeros(2 * m, hef.padded_ld(K, torch.float32), device="cuda")
    Q[1::2, :K] = 1.0
    QH = hef.edge_resistance(inc, Q, K)["QH"].cpu()
    inc.check()
    lost = blocks * 2.0 ** 26 + (m - blocks) - QH
    assert (lost.abs() <= 19 * blocks).all(), (lost / blocks).tolist()
