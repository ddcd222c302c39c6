"""Fleets' forward dynamics with three lanes per request (FP32 plans, double-float
updates): units of ten sorted positions with chains of different lengths, with and
without double-float bias sweeps in one unit, partial units, against the FP64 oracle
(bar 1e-3, as test_fleet_gpu.py) and bit for bit across schedules and block shapes.
"""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[1], [3, 2, 1], list(range(1, 24)), [65, 64] * 10 + [7] * 25,
                                     [128, 100, 66, 65, 64, 63, 33, 2, 1, 1, 1]])
@pytest.mark.parametrize("ids", [0, 5])
def test_units_of_uneven_chains(cuda_lib, lengths, ids):
    import torch

    rd = cuda_lib
    kinds = [rd.RD_REQ_FD] * len(lengths) + [rd.RD_REQ_ID] * ids
    lengths = lengths + [9] * ids
    chains = [chaingen.make_chain(n, seed=50 + k) for k, n in enumerate(lengths)]
    plan = rd.Plan(rd.Fleet(chains), np.arange(len(chains)), kinds)
    rng = np.random.default_rng(3)
    host = [rng.standard_normal(plan.total_joints).astype(np.float32) for _ in range(3)]
    dev = [torch.from_numpy(h).cuda() for h in host]
    base = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                     2.0, -1.0, 0.5, 0.3, 0.2, -0.6])
    status = torch.full((plan.R,), 7, dtype=torch.int32, device="cuda")
    out = rd.fleet_batch(plan, *dev, base=base, status=status)
    for r, (ch, kind) in enumerate(zip(chains, kinds)):
        at = slice(plan.offsets[r], plan.offsets[r] + ch.n)
        x = [h[at].astype(np.float64)[None] for h in host]
        ref = (oracle.fd_aba if kind == rd.RD_REQ_FD else oracle.rnea)(ch, *x, base=base)
        err = oracle.rel_err(out[at].cpu().double().numpy()[None], ref)
        assert err <= (1e-3 if kind == rd.RD_REQ_FD else 1e-4), (r, ch.n, kind, err)
    assert not status[:len(lengths) - ids].any()
    for kw in ({"schedule": rd.RD_SCHED_PER_GROUP}, {"tune": rd.RD_FLEET_TUNE(5, 1)},
               {"tune": rd.RD_FLEET_TUNE(6, 1)}, {"tune": rd.RD_FLEET_TUNE(7, 2)},
               {"tune": rd.RD_FLEET_TUNE(9, 1)}):
        assert torch.equal(out, rd.fleet_batch(plan, *dev, base=base, **kw)), kw
