"""Plans whose forward dynamics stays at one thread per request (many chains of like
length) and plans without forward dynamics (the last, of many short rows, runs the
three-lane kernel): against the FP64 oracle (bars of test_fleet_gpu.py) and bit for bit
across schedules and block shapes, 512-thread blocks included."""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,count,fd", [([7], 15000, 15000), ([3, 5], 30000, 30000),
                                              ([6, 9, 12], 30000, 24000), ([32], 3000, 0), ([2, 30], 700, 0),
                                              ([3, 5], 45000, 0)])
def test_one_thread_plans(cuda_lib, lengths, count, fd):
    import torch

    rd = cuda_lib
    chains = [chaingen.make_chain(n, seed=70 + n) for n in lengths]
    robot = np.arange(count) % len(chains)
    kinds = np.where(np.arange(count) < fd, rd.RD_REQ_FD, rd.RD_REQ_ID)
    plan = rd.Plan(rd.Fleet(chains), robot, kinds)
    rng = np.random.default_rng(9)
    host = [rng.standard_normal(plan.total_joints).astype(np.float32) for _ in range(3)]
    dev = [torch.from_numpy(h).cuda() for h in host]
    status = torch.full((count,), 7, dtype=torch.int32, device="cuda")
    out = rd.fleet_batch(plan, *dev, status=status)
    for r in np.r_[0:20, count // 2:count // 2 + 20, count - 20:count]:
        at = slice(plan.offsets[r], plan.offsets[r] + plan.lengths[r])
        x = [h[at].astype(np.float64)[None] for h in host]
        f, bar = (oracle.fd_aba, 1e-3) if kinds[r] == rd.RD_REQ_FD else (oracle.rnea, 1e-4)
        assert oracle.rel_err(out[at].cpu().double().numpy()[None], f(chains[robot[r]], *x)) <= bar, r
    assert not status[:fd].any()
    for kw in ({"schedule": rd.RD_SCHED_PER_GROUP}, {"tune": rd.RD_FLEET_TUNE(5, 1)},
               {"tune": rd.RD_FLEET_TUNE(7, 1)}, {"tune": rd.RD_FLEET_TUNE(8, 2)}, {"tune": rd.RD_FLEET_TUNE(9, 1)}):
        assert torch.equal(out, rd.fleet_batch(plan, *dev, **kw)), kw
