"""GPU: requests that follow others on one server (stream sets and memory blocks taken over from retired
engines) give bitwise the results of the first wave."""
import numpy as np
import pytest

from paper_2106_03872_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_second_wave_same_results():
    from paper_2106_03872_gb300 import ks
    specs = [(12.0, 32, 20, 0, 3), (15.0, 48, 12, 1, 3), (12.0, 32, 9, 1, 4), (12.0, 32, 17, 1, 4), (10.0, 24, 5, 0, 2)]
    srv = ks.Server(budget_bytes=6 << 30, workers=4)
    waves = []
    for _ in range(3):
        tickets = []
        for k, (L, N, n, kind, count) in enumerate(specs):
            cell = inputs.small_cell(L, N, 3, n, 40 + k, depth=-3.0)
            c0 = np.linalg.qr(inputs.random_coeffs(40 + k, n, ks.count_gvectors(L, N, 20.0)).T)[0].T
            tickets.append(srv.submit(cell, kind, count, c0=c0, nstates=n))
        out = []
        for t in tickets:
            st, res, states, _ = srv.poll(t, timeout_ms=60000, want_states=True)
            assert st == ks.KS_OK
            out.append((res, states))
        waves.append(out)
    srv.close()
    for w in waves[1:]:
        for (r0, s0), (r1, s1) in zip(waves[0], w):
            assert np.array_equal(r0, r1) and np.array_equal(s0, s1)
