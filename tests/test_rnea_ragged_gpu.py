"""Inverse dynamics on rows that fill no whole 16-byte chunks (n % 4 != 0, or arrays off
a 16-byte boundary): the common-normal kernel with warp-wide staging, AUTO past the
lane-parallel kernel's batches. Lengths on both sides of its layouts (no, four and
eight register links; every link stored up to 32; re-derived beyond; 108 for FP64),
batches that leave lanes of the last block idle, against the FP64 oracle at the usual
bars (FP32 1e-4, FP64 1e-10).
"""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
TOL = {"float32": 1e-4, "float64": 1e-10}
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


def run(rd, n, B, dtype, offset=0, variant=0):
    """tau on arrays that start `offset` elements into their allocation."""
    import torch

    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + n)
    npdt = np.dtype(dtype)
    host = [v.astype(npdt) for v in chaingen.make_states(B, n, seed=7).values()]

    def place(a):
        flat = torch.full((B * n + offset + 8,), float("nan"), dtype=getattr(torch, dtype), device="cuda")
        view = flat[offset:offset + B * n].view(B, n)
        if a is not None:
            view.copy_(torch.from_numpy(a))
        return flat, view

    x = [place(a)[1] for a in host]
    flat, out = place(None)
    rd.rnea(rd.Model(ch), *x, out=out, base=BASE, variant=variant)
    tau = out.cpu().numpy().astype(np.float64)
    rest = torch.cat([flat[:offset], flat[offset + B * n:]])
    assert torch.isnan(rest).all()  # nothing written outside the rows
    idx = np.r_[0:min(B, 64), max(0, B - 40):B]
    ref = oracle.rnea(ch, *(h[idx].astype(np.float64) for h in host), base=BASE)
    return oracle.rel_err(tau[idx], ref)


@pytest.mark.parametrize("dtype,B", [("float32", 2049), ("float32", 40000), ("float64", 8161)])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 6, 7, 9, 11, 30, 31, 33, 63, 65, 107, 109, 127])
def test_ragged_lengths(cuda_lib, n, dtype, B):
    if B == 40000 and n > 33:
        B = 2080
    assert run(cuda_lib, n, B, dtype) <= TOL[dtype]


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n,offset", [(4, 1), (8, 3), (32, 1), (36, 2), (7, 1), (29, 3)])
def test_unaligned_rows(cuda_lib, n, offset, dtype):
    assert run(cuda_lib, n, 8161, dtype, offset=offset) <= TOL[dtype]
    assert cuda_lib.rnea_last_config()[0] == cuda_lib.RD_RNEA_KERNEL_DH_PARAM


def test_ragged_fast_trig(cuda_lib):
    # the special-function sines are within 4e-7, three times the polynomial's error
    assert run(cuda_lib, 13, 5001, "float32", variant=cuda_lib.RD_FLAG_FAST_TRIG) <= 3e-4
