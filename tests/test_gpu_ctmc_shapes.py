"""Exponential-service model: every number of replications per warp (1 to 32) and class counts up to eight against the oracle:
counters and end state exact, time integrals within 1e-9.  Requests that meet an empty buffer and a free slot are placed in
the event that ends their prefill, so both backlogged and empty buffers are among the cases."""
import numpy as np
import pytest

from qsim_inputs import presets
from qsim_inputs.spec import GATE_OCCUPANCY, GATE_PRIORITY, ROUTER_SLI, ROUTER_SOLO_FIRST

pytestmark = pytest.mark.gpu

RECORD = 3816      # bytes of a replication's record in the workspace


def instance(I, R, router, gate, n=12, M=None):
    rng = np.random.default_rng(100 * I + R % 97)
    inp = presets.ctmc_instance(n=n, R=R, router=router, gate=gate, P=tuple(rng.integers(200, 3000, I)), D=tuple(rng.integers(50, 600, I)),
                                lam=tuple(np.full(I, 1.5 / I)), theta=tuple(np.full(I, 0.3)))
    return inp if M is None else inp.with_(M=M)


@pytest.mark.parametrize("I,R,router,gate,M", [
    (1, 1, ROUTER_SOLO_FIRST, GATE_OCCUPANCY, None),
    (2, 887, ROUTER_SLI, GATE_OCCUPANCY, None),              # one replication per warp
    (2, 1777, ROUTER_SLI, GATE_PRIORITY, None),              # two
    (3, 3553, ROUTER_SOLO_FIRST, GATE_OCCUPANCY, 4),         # four
    (5, 7105, ROUTER_SLI, GATE_OCCUPANCY, 6),                # eight
    (2, 14209, ROUTER_SOLO_FIRST, GATE_PRIORITY, 11),        # sixteen; one solo GPU: the buffers fill
    (2, 28449, ROUTER_SLI, GATE_OCCUPANCY, 12),              # thirty-two; no solo GPU: the solo pool only drains by abandonment
    (8, 70, ROUTER_SLI, GATE_OCCUPANCY, 6),
])
def test_replications_per_warp_and_class_counts(I, R, router, gate, M):
    from oracle import run_ctmc_oracle
    from paper_2602_02987_b200 import QSimCTMC
    inp = instance(I, R, router, gate, M=M)
    sim = QSimCTMC(inp)
    sim.run_until(7.0)
    sim.run_until(19.0)
    got = sim.stats()
    sim.close()
    for r in sorted({0, 1, R // 3, R // 2, R - 2, R - 1} & set(range(R))):
        ref = run_ctmc_oracle(inp.with_(R=1, rep_offset=inp.rep_offset + r), 19.0)
        for k, v in ref.items():
            if v.dtype.kind in "ui":
                assert np.array_equal(got[k][r], v[0]), (r, k)
            else:
                assert np.allclose(got[k][r], v[0], rtol=1e-9, atol=1e-300), (r, k)


@pytest.mark.parametrize("router", [ROUTER_SOLO_FIRST, ROUTER_SLI])
def test_a_state_whose_clocks_of_intensity_zero_stood_still(router):
    # A workspace saved by an earlier build without patience: the abandonment clocks were never brought up to date there, while the
    # time integrals were.  The record: 40 bytes of scalars, then clocks [7][8] of (acc, lvl, t_last, t_fire, m), 8 bytes each.
    import torch
    from paper_2602_02987_b200 import QSimCTMC
    inp = instance(2, 5, router, GATE_OCCUPANCY).with_(theta=np.zeros(2))
    got = []
    for old in (False, True):
        sim = QSimCTMC(inp)
        sim.run_until(7.0)
        if old:
            first = sim.ptr - sim.ws.data_ptr()
            rec = sim.ws[first:first + inp.R * RECORD].view(inp.R, RECORD)
            for k in (1, 2, 3):
                for i in range(2):
                    at = 40 + (k * 8 + i) * 40 + 16
                    rec[:, at:at + 8] = 0
            torch.cuda.synchronize()
        sim.run_until(19.0)
        got.append(sim.stats())
        sim.close()
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k]), k


@pytest.mark.parametrize("I", [1, 2, 8])
def test_statistics_formed_on_the_host_and_on_the_device(I):
    # 767 replications are read out on the host and 768 on the device; a replication does not depend on how many there are
    from paper_2602_02987_b200 import QSimCTMC
    got = []
    for R in (767, 768):
        sim = QSimCTMC(instance(I, 5, ROUTER_SLI, GATE_OCCUPANCY).with_(R=R))
        sim.run_until(11.0)
        got.append(sim.stats())
        sim.close()
    assert (got[0]["events"] > 0).all()
    for k in got[0]:
        assert got[0][k].shape[0] == 767 and got[1][k].shape[0] == 768
        assert np.array_equal(got[0][k], got[1][k][:767]), k
