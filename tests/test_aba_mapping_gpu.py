"""Forward dynamics by two and by three warps per 32 instances with double-float updates
at the sizes where the library's choice is three lanes per instance
(RD_ABA_EXACT_MAPPING). Against the FP64 oracle at the bar of test_aba_gpu.py (1e-3), the two
against each other at the bar of test_three_warps_agree_with_two (2e-6 of the largest
value), and not bit for bit equal to three lanes: their sums are formed in another
order, which some of 65536 outputs or more show in their last bit.
"""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


def inputs(n, B, seed=73):
    import torch

    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + 9 * n)
    st = chaingen.make_states(B, n, seed=seed, kinds=("q", "qd", "tau"))
    host = [st[k].astype(np.float32) for k in ("q", "qd", "tau")]
    return ch, [h.astype(np.float64) for h in host], [torch.from_numpy(h).cuda() for h in host]


@pytest.mark.parametrize("bias", [0, 0x8])  # FP32, double-float bias sweeps (longer chains: always)
@pytest.mark.parametrize("n", [1, 3, 7, 33, 64, 65, 100, 128])
def test_both_mappings_match_oracle_and_each_other(cuda_lib, n, bias):
    rd = cuda_lib
    ch, h, x = inputs(n, 70)
    ref = oracle.fd_aba(ch, *h, base=BASE)
    model = rd.Model(ch)
    got = [rd.aba(model, *x, base=BASE, flags=bias | f | rd.RD_ABA_EXACT_MAPPING).cpu().double().numpy()
           for f in (rd.RD_ABA_TWO_WARPS, rd.RD_ABA_THREE_WARPS)]
    for g in got:
        assert oracle.rel_err(g, ref) <= 1e-3
    assert np.max(np.abs(got[0] - got[1])) <= 2e-6 * max(np.max(np.abs(got[0])), 1.0)


@pytest.mark.parametrize("n,B,replaced", [(64, 1024, "three"), (64, 8192, "two"), (80, 1536, "two")])
def test_the_named_kernel_runs(cuda_lib, n, B, replaced):
    """With the flag the named kernel; without it three lanes where they replaced that
    mapping as the library's choice, and else the named kernel too."""
    import torch

    rd = cuda_lib
    ch, _, x = inputs(n, B, seed=23)
    model = rd.Model(ch)
    lanes = rd.aba(model, *x, flags=rd.RD_ABA_THREE_LANES)
    assert torch.equal(rd.aba(model, *x), lanes)
    for name, f in (("two", rd.RD_ABA_TWO_WARPS), ("three", rd.RD_ABA_THREE_WARPS)):
        plain = rd.aba(model, *x, flags=f)
        assert torch.equal(plain, lanes) == (name == replaced)
        exact = rd.aba(model, *x, flags=f | rd.RD_ABA_EXACT_MAPPING)
        assert not torch.equal(exact, lanes)
        assert name == replaced or torch.equal(plain, exact)
        assert float((exact - lanes).abs().max()) <= 2e-6 * max(float(lanes.abs().max()), 1.0)


def test_workload_batch_sampled(cuda_lib):
    """n = 64 and 100, B = 16384: every 64th instance against the oracle."""
    rd = cuda_lib
    for n in (64, 100):
        ch, h, x = inputs(n, 16384, seed=1609)
        idx = np.arange(0, 16384, 64)
        ref = oracle.fd_aba(ch, *(v[idx] for v in h))
        for f in (rd.RD_ABA_TWO_WARPS, rd.RD_ABA_THREE_WARPS):
            g = rd.aba(rd.Model(ch), *x, flags=f | rd.RD_ABA_EXACT_MAPPING).cpu().double().numpy()
            assert oracle.rel_err(g[idx], ref) <= 1e-3


def test_exact_is_for_a_named_mapping(cuda_lib):
    import torch

    rd = cuda_lib
    ch, _, x = inputs(6, 40)
    model = rd.Model(ch)
    with pytest.raises(rd.RdError):
        rd.aba(model, *x, flags=rd.RD_ABA_EXACT_MAPPING)
    for f in (rd.RD_ABA_THREAD_PER_INSTANCE, rd.RD_ABA_WARP_PER_INSTANCE, rd.RD_ABA_THREE_LANES):
        assert torch.equal(rd.aba(model, *x, flags=f), rd.aba(model, *x, flags=f | rd.RD_ABA_EXACT_MAPPING))
