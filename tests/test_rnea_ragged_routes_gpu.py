"""FP32 inverse dynamics on rows that fill no whole 16-byte chunks: which kernel and state
layout AUTO takes on both sides of each of its lines, and the layouts of large batches
(eight register links; few or no links stored beyond 32, so that most chunks are
re-derived), against the FP64 oracle at the usual bar (1e-4)."""
import numpy as np
import pytest

import chaingen
import oracle

pytestmark = pytest.mark.gpu
BASE = np.array([0.2, -0.1, 0.3, 0.5, -0.4, 0.25, 0.3, 1.1, 9.81, -0.2, 0.4, 0.1,
                 2.0, -1.0, 0.5, 0.3, 0.2, -0.6])


def run(rd, n, B, offset=0):
    """Relative error of the first and last instances, NaN guards checked; the route taken."""
    import torch

    ch = chaingen.make_chain(n, seed=chaingen.BASE_SEED + n)
    few = chaingen.make_states(80, n, seed=7)
    host = [few[k].astype(np.float32) for k in ("q", "qd", "qdd")]

    def place(a=None):
        flat = torch.full((B * n + offset + 8,), float("nan"), device="cuda")
        view = flat[offset:offset + B * n].view(B, n)
        if a is not None:  # the 80 states in turn
            t = torch.from_numpy(a).cuda()
            view.copy_(t.repeat(-(-B // 80), 1)[:B])
        return flat, view

    x = [place(a)[1] for a in host]
    flat, out = place()
    rd.rnea(rd.Model(ch), *x, out=out, base=BASE)
    route = rd.rnea_last_config(), rd.rnea_last_state_layout()
    assert torch.isnan(flat[:offset]).all() and torch.isnan(flat[offset + B * n:]).all()
    ref = oracle.rnea(ch, *(h.astype(np.float64) for h in host), base=BASE)
    idx = np.r_[0:min(B, 80), max(0, B - 80):B]
    err = oracle.rel_err(out.cpu().numpy().astype(np.float64)[idx], ref[idx % 80])
    # every row equals the row with the same state in the first eighty
    full = out[: B // 80 * 80].view(-1, 80, n)
    assert torch.equal(full, full[:1].expand_as(full))
    return err, route


@pytest.mark.parametrize("n,most", [(3, 2048), (9, 2048), (13, 16), (15, 24), (17, 16), (31, 24), (33, 2048), (45, 2048),
                                    (63, 16), (65, 2048), (66, 16), (127, 16)])
def test_scans_up_to_their_last_batch(cuda_lib, n, most):
    """most: the batch, or (16, 24) instances per SM."""
    import torch

    if most < 100:
        most *= torch.cuda.get_device_properties(0).multi_processor_count
    err, ((kernel, _, _), _) = run(cuda_lib, n, most)
    assert err <= 1e-4 and kernel & 0xf00 == 0x100, kernel
    err, ((kernel, _, _), _) = run(cuda_lib, n, most + 1)
    assert err <= 1e-4 and kernel == cuda_lib.RD_RNEA_KERNEL_DH_PARAM


@pytest.mark.parametrize("n", [1, 2])
@pytest.mark.parametrize("B", [5000, 70001])
def test_one_and_two_links_stay_in_joint_frames(cuda_lib, n, B):
    err, ((kernel, _, _), _) = run(cuda_lib, n, B)
    assert err <= 1e-4 and kernel == cuda_lib.RD_VARIANT_SERIAL


@pytest.mark.parametrize("n,B,offset,stored,registers", [
    (31, 8200, 0, 31, 4), (28, 100003, 1, 28, 8), (30, 100003, 0, 30, 8), (31, 100003, 0, 31, 8),
    (32, 100003, 3, 32, 8), (63, 65537, 0, 12, 0), (64, 65537, 1, 12, 0), (99, 65537, 0, 0, 0),
    (127, 65537, 0, 0, 0), (128, 40001, 2, 0, 0)])
def test_layouts_of_large_batches(cuda_lib, n, B, offset, stored, registers):
    err, ((kernel, block, got), (reg, _)) = run(cuda_lib, n, B, offset)
    assert err <= 1e-4
    assert (kernel, block, got, reg) == (cuda_lib.RD_RNEA_KERNEL_DH_PARAM, 32, stored, registers)
