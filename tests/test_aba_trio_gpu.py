"""GPU parity of forward dynamics with three lanes per instance
(RD_ABA_THREE_LANES: Eq. (abi) and the solves of Eq. recursive-fd by axis). Against
the FP64 oracle's fd_aba (bar 1e-3, as in test_aba_gpu.py) and the one-thread
kernel. The bias sweeps of the two are the same FP32 operations up to 64 links, so
they differ by the double-float updates alone, of which FP32 output shows an ulp
or two of the largest value (2e-6, the bar of test_three_warps_agree_with_two).
"""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


def run(rd, n, B, flags, base=None, status=None):
    import torch

    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + 9 * n)
    st = chaingen.make_states(B, n, seed=73, kinds=("q", "qd", "tau"))
    host = [st[k].astype(np.float32) for k in ("q", "qd", "tau")]
    qdd = rd.aba(rd.Model(ch), *(torch.from_numpy(v).cuda() for v in host), base=base,
                 status=status, flags=flags)
    return qdd.cpu().double().numpy(), ch, [v.astype(np.float64) for v in host]


# block edges: 30 instances with FP32 bias sweeps, 20 with double-float ones, warps of 10
@pytest.mark.parametrize("B", [1, 9, 20, 30, 31, 77])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 64, 65, 128])
def test_trio_matches_oracle_and_one_thread(cuda_lib, n, B):
    import torch

    rd = cuda_lib
    status = torch.full((B,), 7, dtype=torch.int32, device="cuda")
    qdd, ch, h = run(rd, n, B, rd.RD_ABA_THREE_LANES, base=BASE, status=status)
    assert oracle.rel_err(qdd, oracle.fd_aba(ch, *h, base=BASE)) <= 1e-3
    assert not status.cpu().numpy().any()
    one, _, _ = run(rd, n, B, rd.RD_ABA_THREAD_PER_INSTANCE, base=BASE)
    assert np.max(np.abs(qdd - one)) <= 2e-6 * max(np.max(np.abs(one)), 1.0)


@pytest.mark.parametrize("n", [5, 20])
def test_trio_double_float_bias_short_chains(cuda_lib, n):
    rd = cuda_lib
    ext = rd.RD_ABA_EXTENDED_BIAS
    qdd, ch, h = run(rd, n, 41, rd.RD_ABA_THREE_LANES | ext)
    one, _, _ = run(rd, n, 41, rd.RD_ABA_THREAD_PER_INSTANCE | ext)
    assert oracle.rel_err(qdd, oracle.fd_aba(ch, *h)) <= 1e-3
    assert np.max(np.abs(qdd - one)) <= 2e-6 * max(np.max(np.abs(one)), 1.0)


@pytest.mark.parametrize("n,B", [(64, 18240), (64, 18241), (100, 24320), (3, 16384)])
def test_trio_is_chosen_up_to_its_range(cuda_lib, n, B):
    """Without a mapping flag the library takes it while the batch is resident at
    once (B <= 120 per SM, 160 with double-float bias sweeps; 152 SMs)."""
    import torch

    rd = cuda_lib
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    st = chaingen.make_states(64, n, seed=5, kinds=("q", "qd", "tau"))
    x = [torch.from_numpy(st[k].astype(np.float32)).cuda().repeat(-(-B // 64), 1)[:B].contiguous()
         for k in ("q", "qd", "tau")]
    model = rd.Model(chaingen.make_chain(n))
    auto = rd.aba(model, *x)
    trio = rd.aba(model, *x, flags=rd.RD_ABA_THREE_LANES)
    if B <= (160 if n > 64 else 120) * sms:
        assert torch.equal(auto, trio)
    assert torch.equal(trio[:64], trio[64:128])  # the same states, in other lanes and blocks


def test_trio_flags_a_singular_joint(cuda_lib):
    """A point mass on the last joint's axis: Omega = 0 there."""
    import torch

    rd = cuda_lib
    ch = chaingen.make_chain(4)
    ch.inertia[3] = 0.0
    ch.inertia[3, 0] = 1.0  # at the origin of frame 3
    ch.S[3, :3] = 0.0       # the axis through the origin
    status = torch.zeros(33, dtype=torch.int32, device="cuda")
    x = [torch.zeros(33, 4, device="cuda") for _ in range(3)]
    rd.aba(rd.Model(ch), *x, status=status, flags=rd.RD_ABA_THREE_LANES)
    assert np.all(status.cpu().numpy() == rd.RD_WARN_SINGULAR)


def test_trio_rejects_what_it_does_not_take(cuda_lib):
    import torch

    rd = cuda_lib
    model = rd.Model(chaingen.make_chain(4))
    x = torch.zeros(3, 4, device="cuda")
    for other in (rd.RD_ABA_TWO_WARPS, rd.RD_ABA_THREAD_PER_INSTANCE, rd.RD_ABA_FP64_UPDATE,
                  rd.RD_ABA_JOINT_FRAMES, rd.RD_ABA_SCANS_IN_DTYPE):
        with pytest.raises(rd.RdError):
            rd.aba(model, x, x, x, flags=rd.RD_ABA_THREE_LANES | other)
    assert rd.aba(model, x[:0], x[:0], x[:0], flags=rd.RD_ABA_THREE_LANES).numel() == 0


@pytest.mark.parametrize("B", [1, 29, 31])
@pytest.mark.parametrize("n", [1, 3, 7, 64, 128])
def test_trio_fp64_matches_oracle(cuda_lib, n, B):
    """FP64 data: the bars of test_aba_gpu.py (1e-8) with a moving base."""
    import torch

    rd = cuda_lib
    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + 9 * n)
    st = chaingen.make_states(B, n, seed=73, kinds=("q", "qd", "tau"))
    x = [torch.from_numpy(st[k]).cuda() for k in ("q", "qd", "tau")]
    ref = oracle.fd_aba(ch, *(st[k] for k in ("q", "qd", "tau")), base=BASE)
    trio = rd.aba(rd.Model(ch), *x, base=BASE, flags=rd.RD_ABA_THREE_LANES)
    one = rd.aba(rd.Model(ch), *x, base=BASE, flags=rd.RD_ABA_THREAD_PER_INSTANCE)
    assert oracle.rel_err(trio.cpu().numpy(), ref) <= 1e-8
    assert oracle.rel_err(one.cpu().numpy(), ref) <= 1e-8
