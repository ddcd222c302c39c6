"""The adjoint on rows that fill no whole 16-byte chunks or start off a 16-byte boundary:
the common-normal kernel with streamed pieces, re-deriving its state and with it in the
workspace, FP32 and FP64, against the oracle's complex-step gradient at the bars of
test_vjp_gpu.py (1e-3 and 1e-9 per gradient)."""
import numpy as np
import pytest

import chaingen
import oracle
from gradcheck import grad_err

pytestmark = pytest.mark.gpu
TOL = {"float32": 1e-3, "float64": 1e-9}
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


def check(rd, n, B, dtype, mode, offset=0):
    import torch

    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + n)
    host = [v.astype(dtype) for v in chaingen.make_states(B, n, seed=9, kinds=("q", "qd", "qdd", "w")).values()]

    def place(a=None):
        flat = torch.full((B * n + offset + 8,), float("nan"), dtype=getattr(torch, dtype), device="cuda")
        view = flat[offset:offset + B * n].view(B, n)
        if a is not None:
            view.copy_(torch.from_numpy(a))
        return flat, view

    out = [place() for _ in range(3)]
    g = rd.rnea_vjp(rd.Model(ch), *(place(a)[1] for a in host), base=BASE, mode=mode,
                    out=[v for _, v in out])
    for flat, _ in out:  # nothing written outside the rows
        assert torch.isnan(flat[:offset]).all() and torch.isnan(flat[offset + B * n:]).all()
    idx = np.r_[0:min(B, 20), max(0, B - 20):B]
    ref = oracle.rnea_grad(ch, *(a[idx].astype(np.float64) for a in host), base=BASE)
    assert grad_err([a.cpu().numpy()[idx] for a in g], ref) <= TOL[dtype], (n, B, dtype, mode)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 6, 7, 31, 33, 66, 127])
def test_ragged_lengths(cuda_lib, n, dtype):
    for B in (1, 33, 70):
        check(cuda_lib, n, B, dtype, cuda_lib.RD_VJP_RECOMPUTE)
        check(cuda_lib, n, B, dtype, cuda_lib.RD_VJP_STORE)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n,offset", [(4, 1), (32, 3), (7, 1), (29, 2)])
def test_unaligned_rows(cuda_lib, n, offset, dtype):
    check(cuda_lib, n, 50, dtype, cuda_lib.RD_VJP_RECOMPUTE, offset=offset)
