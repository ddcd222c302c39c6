"""FP64 inverse dynamics on the common-normal kernel with eight links' state in
registers (AUTO for whole 16-byte chunks): every length at which its layout changes
(no register links below 8, 32 and 128 constants, stored and re-derived links, the
joint-frame kernels beyond 108) against the FP64 oracle at the FP64 bar, 1e-10, and
with the recursion by origin accelerations a moving base.
"""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


@pytest.mark.parametrize("base", [None, BASE])
@pytest.mark.parametrize("n", [4, 8, 12, 32, 36, 64, 100, 108, 112, 128])
def test_auto_fp64_matches_oracle(cuda_lib, n, base):
    import torch

    B = 8161  # above the batches of sixteen lanes per instance, a ragged last block
    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + n)
    st = chaingen.make_states(B, n, seed=11)
    x = [torch.from_numpy(st[k]).cuda() for k in ("q", "qd", "qdd")]
    tau = cuda_lib.rnea(cuda_lib.Model(ch), *x, base=base).cpu().numpy()
    here = cuda_lib.rnea_last_config()[0]
    assert (here == cuda_lib.RD_RNEA_KERNEL_DH_PARAM) == (n <= 108)
    idx = np.r_[0:64, B - 64:B]
    ref = oracle.rnea(ch, *(st[k][idx] for k in ("q", "qd", "qdd")), base=base)
    assert oracle.rel_err(tau[idx], ref) <= 1e-10
