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


def test_slot_values_one_pass_at_a_time(sv, orc):
    """Without room for the slot values of all passes the call computes them
    pass by pass: one refused allocation is survived, and the amplitudes are
    those of an undisturbed call."""
    import numpy as np

    from paper_2605_15098_gb300 import circuits as C

    n = 19
    g = C.random_circuit(n, 8, 4)
    cfg = sv.make_config(sv.SV_MODE_PARTITIONED)
    with sv.State(n, sv.SV_C64) as s:
        s.apply(g, cfg)
        want = s.amplitudes()
    survived = 0
    for after in range(5):  # three allocations of the apply, two of a new handle
        with sv.State(n, sv.SV_C64) as s:
            sv.sv_fault_inject(sv.SV_FAULT_ALLOC, after)
            try:
                s.apply(g, cfg)
                sv.sv_destroy(sv.sv_create(3, sv.SV_C64))  # refused if the fault is still to come
            except sv.SvError as e:
                assert e.code == sv.SV_ERR_OOM
                continue
            finally:
                sv.sv_fault_inject(sv.SV_FAULT_ALLOC, -1)
            survived += 1
            assert np.array_equal(s.amplitudes(), want)
    assert survived == 1


@pytest.mark.parametrize("dt,n,m", [("c64", 20, 15), ("c64", 24, 15), ("c64", 24, 16), ("c128", 21, 16)])
def test_many_outcomes_without_scratch(sv, orc, dt, n, m):
    """A marginal of 2^15 outcomes or more without physical bit 0 needs no device
    memory but its result: it survives a refused allocation, and it can be
    captured into a graph on a handle that has not run one before."""
    import numpy as np
    import torch

    rng = np.random.default_rng(n + m)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dt == "c64" else np.complex128)
    mask = ((1 << m) - 1) << (n - m)
    ref = orc.marginal(n, psi.astype(np.complex128), mask)
    code = sv.SV_C64 if dt == "c64" else sv.SV_C128
    out = torch.empty(1 << m, dtype=torch.float64, device="cuda")

    def check():
        torch.cuda.synchronize()
        assert np.max(np.abs(out.cpu().numpy() - ref)) <= 2e-13 * np.max(ref)  # as tests/test_gpu_readout.py
        out.zero_()
        torch.cuda.synchronize()

    with sv.State(n, code) as s:
        sv.sv_copy_in(s.h, psi)
        sv.sv_fault_inject(sv.SV_FAULT_ALLOC, 0)
        try:
            sv.sv_probabilities_device(s.h, mask, out.data_ptr())
        finally:
            sv.sv_fault_inject(sv.SV_FAULT_ALLOC, -1)
        check()

    amps = torch.from_numpy(psi).cuda()
    stream = torch.cuda.Stream()
    with sv.State(n, code, tensor=amps, stream=stream) as s:
        sv.sv_info(s.h)
        torch.cuda.synchronize()
        amps.copy_(torch.from_numpy(psi))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            sv.sv_probabilities_device(s.h, mask, out.data_ptr())
        g.replay()
        check()
