"""Amplitude retrieval at N = 2048: one CTA per row (schedule 16) against a cluster
of one mask per CTA (schedule 1).  The line search evaluates the row's fields at
about ten points an iteration, from registers; where they overflow, the layout
loses what it is there for."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402


def test_one_cta_per_row_stays_ahead():
    N, M, J = 2048, 1216, 4
    g = torch.Generator("cuda").manual_seed(0)
    T, E = (torch.view_as_complex(torch.randn(M, N, 2, generator=g, device="cuda")) / math.sqrt(2 * N) for _ in range(2))
    d = torch.polar(torch.ones(J, N, device="cuda"), 2 * math.pi * torch.rand(J, N, generator=g, device="cuda"))
    Y = torch.fft.fft(d * T[:, None]).abs().square().contiguous()
    T0, To, ms = T + 0.2 * E, torch.empty_like(T), {}
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for G in (1, 16):
        with tmr.tmr_create(N, M, J, d, None, dict(cost="amplitude", schedule=G)) as h:
            ms[G] = 1e9
            for _ in range(5):
                a.record()
                tmr.tmr_retrieve_from(h, T0, Y, None, 10, To)
                b.record()
                torch.cuda.synchronize()
                ms[G] = min(ms[G], a.elapsed_time(b))
    # measured 0.81; 1.06 with the square roots of the intensities taken anew at every point
    assert ms[16] <= 0.93 * ms[1], ms
