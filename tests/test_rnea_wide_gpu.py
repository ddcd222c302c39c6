"""FP64 inverse dynamics with sixteen lanes per instance (AUTO for small batches): lengths
around its sixteen links a pass and the shortest, batches that leave half a warp idle,
a moving base, rows off a 16-byte boundary, against the FP64 oracle (bar 1e-10)."""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


@pytest.mark.parametrize("B", [1, 2, 33, 1000])
@pytest.mark.parametrize("n", [1, 2, 7, 15, 16, 17, 32, 33, 100, 108])
def test_wide_matches_oracle(cuda_lib, n, B):
    import torch

    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + n)
    st = chaingen.make_states(B, n, seed=3)
    dev = []
    for v in st.values():  # one element off the allocation's start
        flat = torch.empty(B * n + 1, dtype=torch.float64, device="cuda")
        flat[1:].copy_(torch.from_numpy(v.reshape(-1)))
        dev.append(flat[1:].view(B, n))
    for base in (None, BASE):
        tau = cuda_lib.rnea(cuda_lib.Model(ch), *dev, base=base).cpu().numpy()
        assert cuda_lib.rnea_last_config()[0] == cuda_lib.RD_RNEA_KERNEL_WIDE
        assert oracle.rel_err(tau, oracle.rnea(ch, *st.values(), base=base)) <= 1e-10


def test_wide_beyond_the_common_normal_kernel(cuda_lib):
    """n = 128 between the lane scans' batches and 44 per SM."""
    import torch

    B, n = 5000, 128
    ch = chaingen.make_chain(n)
    st = chaingen.make_states(B, n, seed=3)
    tau = cuda_lib.rnea(cuda_lib.Model(ch), *(torch.from_numpy(v).cuda() for v in st.values()))
    assert cuda_lib.rnea_last_config()[0] == cuda_lib.RD_RNEA_KERNEL_WIDE
    ref = oracle.rnea(ch, *(v[-50:] for v in st.values()))
    assert oracle.rel_err(tau[-50:].cpu().numpy(), ref) <= 1e-10
