"""Device memory that lb_msd_trajectory needs: 16 doubles per record and body
(centres 3, quaternions 4, work 9) beside the results."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_sixteen_doubles_per_record_are_enough():
    """16 million records (2.05 GB) with 2.8 GB of device memory left."""
    import torch
    from paper_1604_01829_gb300 import lb
    nb, nrec = 64, 250000
    rng = np.random.default_rng(1)
    X = np.cumsum(rng.standard_normal((nb, nrec, 3)), axis=1)
    q = np.zeros((nb, nrec, 4))
    q[..., 0] = 1.0
    few = lb.lb_msd_trajectory(X[:2, :100], q[:2, :100], 3)      # modules loaded, context warm
    assert few.shape[1] == 3
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - 2800 * 2 ** 20, dtype=torch.uint8, device="cuda")
    try:
        msd = lb.lb_msd_trajectory(X, q, 2)
    finally:
        del held
        torch.cuda.empty_cache()
    ref = np.stack([np.ascontiguousarray(((X[:, l:] - X[:, :-l]) ** 2).transpose(0, 2, 1)).mean(axis=2) for l in (1, 2)], axis=1)
    # the reference's pairwise sums (over the last axis) of 250,000 terms: 2^-52 log2(250000)
    assert np.abs(msd[:, :, :3] - ref).max() <= 18 * 2.0 ** -52 * ref.max()
