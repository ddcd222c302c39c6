"""Which mapping forward dynamics takes without a flag, on both sides of each of its lines
(rd_aba_last_mapping), batches by the device's SM count; every row equals the row with
the same state in another lane or block, and the first rows the FP64 oracle's (bars of
test_aba_gpu.py)."""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
TOL = {"float32": 1e-3, "float64": 1e-8}


def sms():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


def route(rd, n, B, dtype="float32", flags=0, bar=TOL):
    """bar None: FP32 bias sweeps on a long chain, which do not reach the bar (and serve
    comparisons): only finite."""
    import torch

    few = min(B, 48)
    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + 9 * n)
    host = [v.astype(dtype) for v in chaingen.make_states(few, n, seed=5, kinds=("q", "qd", "tau")).values()]
    x = [torch.from_numpy(h).cuda().repeat(-(-B // few), 1)[:B].contiguous() for h in host]
    qdd = rd.aba(rd.Model(ch), *x, flags=flags)
    took = rd.aba_last_mapping()
    if bar:
        ref = oracle.fd_aba(ch, *(h.astype(np.float64) for h in host))
        assert oracle.rel_err(qdd[:few].cpu().numpy().astype(np.float64), ref) <= bar[dtype]
    else:
        assert torch.isfinite(qdd).all()
    whole = qdd[: B // few * few].view(-1, few, n)
    assert torch.equal(whole, whole[:1].expand_as(whole))
    return took


@pytest.mark.parametrize("n,per_sm", [(3, 120), (7, 120), (64, 120), (65, 160), (128, 160)])
def test_fp32_three_lanes_end(cuda_lib, n, per_sm):
    B = per_sm * sms()
    assert route(cuda_lib, n, B) == cuda_lib.RD_ABA_THREE_LANES
    assert route(cuda_lib, n, B + 1) == cuda_lib.RD_ABA_THREAD_PER_INSTANCE


@pytest.mark.parametrize("n", [3, 7, 49, 128])
def test_fp64_three_lanes_end(cuda_lib, n):
    B = 60 * sms()
    assert route(cuda_lib, n, B, "float64") == cuda_lib.RD_ABA_THREE_LANES
    assert route(cuda_lib, n, B + 1, "float64") == cuda_lib.RD_ABA_THREAD_PER_INSTANCE


def test_double_float_bias_of_short_chains(cuda_lib):
    """Beyond one wave two warps lead up to five links, and the line ends sooner."""
    rd = cuda_lib
    ext, wave = rd.RD_ABA_EXTENDED_BIAS, 80 * sms()
    for n, last in ((3, 136), (4, 160), (5, 150), (11, 150), (12, 160)):
        assert route(rd, n, wave, flags=ext) == rd.RD_ABA_THREE_LANES
        assert route(rd, n, wave + 1, flags=ext) == (rd.RD_ABA_TWO_WARPS if n <= 5 else rd.RD_ABA_THREE_LANES)
        assert route(rd, n, last * sms(), flags=ext) == rd.RD_ABA_THREE_LANES
        assert route(rd, n, last * sms() + 1, flags=ext) == rd.RD_ABA_THREAD_PER_INSTANCE


def test_fp32_bias_of_long_chains(cuda_lib):
    """Three blocks per SM from 90 links on: two warps lead in between up to 99."""
    rd = cuda_lib
    bias, resident = rd.RD_ABA_FP32_BIAS, 90 * sms()
    for n, between in ((89, rd.RD_ABA_THREE_LANES), (90, rd.RD_ABA_TWO_WARPS), (99, rd.RD_ABA_TWO_WARPS),
                       (100, rd.RD_ABA_THREE_LANES)):
        took = [route(rd, n, B, flags=bias, bar=None) for B in (resident, resident + 1, 120 * sms())]
        assert took == [rd.RD_ABA_THREE_LANES, between, rd.RD_ABA_THREE_LANES], n


def test_fp64_one_warp_leads_for_long_chains_in_small_batches(cuda_lib):
    rd = cuda_lib
    assert route(rd, 48, 512, "float64") == rd.RD_ABA_WARP_PER_INSTANCE
    assert route(rd, 48, 513, "float64") == rd.RD_ABA_THREE_LANES
    assert route(rd, 47, 512, "float64") == rd.RD_ABA_THREE_LANES
    assert route(rd, 2, 512, "float64") == rd.RD_ABA_THREAD_PER_INSTANCE


def test_short_chains_and_other_precisions(cuda_lib):
    rd = cuda_lib
    assert route(rd, 2, 2048) == rd.RD_ABA_THREE_WARPS
    assert route(rd, 2, 2049) == rd.RD_ABA_TWO_WARPS
    assert route(rd, 2, 16385) == rd.RD_ABA_THREAD_PER_INSTANCE
    assert route(rd, 64, 512, flags=rd.RD_ABA_FP64_UPDATE) == rd.RD_ABA_WARP_PER_INSTANCE
    assert route(rd, 64, 4096, flags=rd.RD_ABA_FP64_UPDATE) == rd.RD_ABA_THREE_WARPS
    assert route(rd, 64, 4097, flags=rd.RD_ABA_FP64_UPDATE) == rd.RD_ABA_TWO_WARPS
    assert route(rd, 16, 512, flags=rd.RD_ABA_JOINT_FRAMES) == rd.RD_ABA_JOINT_FRAMES


@pytest.mark.parametrize("mapping", ["lanes", "thread"])
@pytest.mark.parametrize("n", [1, 3, 7, 16, 33, 64, 128])
def test_fp64_solves_the_equations_of_motion(cuda_lib, n, mapping):
    """ID(q, qd, qdd) gives tau back to within 2^10 n units of rounding of the largest
    torque in play (tau and the bias torques): n links, each a sum of some tens of
    products, and up to a few digits that the rank-one updates of the inertia cancel.
    The qdd bar of 1e-8 would let six more digits go."""
    import torch

    rd = cuda_lib
    B = 200
    base = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1, 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])
    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + 9 * n)
    st = chaingen.make_states(B, n, seed=8, kinds=("q", "qd", "tau"))
    x = [torch.from_numpy(v).cuda() for v in st.values()]
    flag = rd.RD_ABA_THREE_LANES if mapping == "lanes" else rd.RD_ABA_THREAD_PER_INSTANCE
    qdd = rd.aba(rd.Model(ch), *x, base=base, flags=flag).cpu().numpy()
    tau = oracle.rnea(ch, st["q"], st["qd"], qdd, base=base)
    bias = oracle.rnea(ch, st["q"], st["qd"], np.zeros_like(qdd), base=base)
    scale = np.max(np.abs(bias), 1) + np.max(np.abs(st["tau"]), 1)
    assert np.max(np.max(np.abs(tau - st["tau"]), 1) / scale) <= 2.0 ** 10 * n * 2.0 ** -53
