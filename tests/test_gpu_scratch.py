"""Device memory that read-outs take beside their result: the partial sums of
a marginal are at most 2^18 doubles (2 MiB), whatever its size."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


@pytest.mark.parametrize("m", [3, 8, 12, 17])
def test_marginal_scratch(sv, m):
    import torch

    n = 23
    masks = ((1 << m) - 1, ((1 << m) - 1) << (n - m))  # with and without physical bit 0
    out = torch.empty(1 << m, dtype=torch.float64, device="cuda")
    with sv.State(n, sv.SV_C64) as s:  # the kernels' code is loaded on their first use
        for mask in masks:
            sv.sv_probabilities_device(s.h, mask, out.data_ptr())
        torch.cuda.synchronize()
    with sv.State(n, sv.SV_C64) as s:
        sv.sv_info(s.h)
        torch.cuda.synchronize()
        for mask in masks:
            free = torch.cuda.mem_get_info()[0]
            sv.sv_probabilities_device(s.h, mask, out.data_ptr())
            torch.cuda.synchronize()
            # 2 MiB of sums, in 2 MiB pages
            assert free - torch.cuda.mem_get_info()[0] <= 4 << 20
        assert abs(float(out.sum()) - 1.0) < 1e-12
